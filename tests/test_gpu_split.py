"""Calls of 3 to 16 tokens: K split over the CTAs of a cluster.  One quantisation group and many, numbers of groups that no
cluster divides, an odd number (scales that are read 2 bytes at a time), rows past the last whole tile, grids so small that the
tiles of a cluster go through in several passes, x and scales at the least alignment that is accepted, and the wait for t."""
import pytest

import oracle
from gpu_utils import DeviceLinear, REL_F_TOL, check_parity, compare, torch_to_f64
from workloads import make_linear

pytestmark = pytest.mark.gpu

FBQ_ERR_TIMEOUT = -5


@pytest.fixture(scope="module")
def fbq():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    import paper_2501_16385_b200 as lib
    yield lib
    for name in ("gemv_ctas", "test_skip_t_arrive", "t_poll_limit"):
        lib.set_option(name, 0)


@pytest.mark.parametrize("bits,dtype,M,N,K,rank", [
    (4, "f16", 3, 8, 128, 16), (3, "bf16", 16, 24, 128, 0), (4, "bf16", 9, 40, 3 * 128, 112), (3, "f16", 8, 72, 5 * 128, 128),
    (4, "f16", 16, 1000, 7 * 128, 64), (3, "f16", 9, 2056, 11 * 128, 48), (4, "bf16", 7, 520, 17 * 128, 32), (3, "bf16", 16, 136, 43 * 128, 96),
    (4, "f16", 16, 264, 86 * 128, 128), (4, "bf16", 11, 2312, 40 * 128, 16), (3, "f16", 13, 48, 108 * 128, 64), (4, "f16", 5, 4104, 32 * 128, 0),
    (4, "f16", 4, 40, 560 * 128, 64), (3, "bf16", 8, 24, 577 * 128, 0)])        # the last two: clusters of sixteen
def test_shapes(fbq, bits, dtype, M, N, K, rank):
    inp = make_linear(M, N, K, bits, rank, dtype=dtype, seed=7000 + M + N + K, outlier_frac=0.01)
    before = fbq.launch_count()
    check_parity(inp, fbq, threads=16, floor=2e-5)
    assert fbq.launch_count() - before == 2                   # one of them packs the codes


@pytest.mark.parametrize("bits,dtype,M,N,K,rank,ctas", [(4, "f16", 16, 1096, 1024, 64, 2), (3, "bf16", 8, 1608, 9 * 128, 128, 1), (4, "bf16", 12, 3000, 2048, 32, 4)])
def test_few_ctas_and_several_passes(fbq, bits, dtype, M, N, K, rank, ctas):
    import torch
    inp = make_linear(M, N, K, bits, rank, dtype=dtype, seed=7300 + M)
    dev = DeviceLinear(inp, fbq)
    want = oracle.linear_inputs(inp, threads=16)
    fbq.set_option("gemv_ctas", ctas)
    try:
        ys = [dev.run(fbq) for _ in range(3)]
        torch.cuda.synchronize()
    finally:
        fbq.set_option("gemv_ctas", 0)
    assert fbq.poll_status() == 0
    assert all(torch.equal(ys[0], y) for y in ys)
    rel, mx, lim = compare(torch_to_f64(ys[0], dtype), want, inp.x_f64(), K)
    lim += 2.0 ** -8 * float(abs(want).max()) if dtype == "bf16" else 0.0      # half an ulp of the largest output
    assert rel <= REL_F_TOL and mx <= lim


@pytest.mark.parametrize("bits,M", [(4, 4), (3, 12)])
def test_least_alignment(fbq, bits, M):
    # x 16 and not 32 bytes aligned, scales and zero points 2 and not 4: the same bits as from aligned buffers
    import torch
    inp = make_linear(M, 328, 6 * 128, bits, 32, seed=7400 + M)
    dev = DeviceLinear(inp, fbq)
    want = dev.run(fbq)

    def shifted(t, elements):
        room = torch.zeros(t.numel() + 64, dtype=t.dtype, device="cuda")
        first = (32 - room.data_ptr() % 32) % 32 // t.element_size() + elements
        out = room[first: first + t.numel()].view(t.shape)
        out.copy_(t)
        return out

    x = shifted(dev.x, 8)
    assert x.data_ptr() % 32 == 16
    assert torch.equal(dev.run(fbq, x=x), want)
    dev.scales, dev.zeros = shifted(dev.scales, 1), shifted(dev.zeros, 1)
    assert torch.equal(dev.run(fbq), want)
    torch.cuda.synchronize()
    assert fbq.poll_status() == 0


def test_wait_for_t_runs_out(fbq):
    import torch
    inp = make_linear(8, 512, 1024, 4, 32, seed=7500)
    dev = DeviceLinear(inp, fbq)
    want = dev.run(fbq)
    torch.cuda.synchronize()
    fbq.set_option("test_skip_t_arrive", 1)
    fbq.set_option("t_poll_limit", 2000)
    try:
        dev.run(fbq)
        torch.cuda.synchronize()                              # the kernel returned
        assert fbq.poll_status() == FBQ_ERR_TIMEOUT           # ... and said why
    finally:
        fbq.set_option("test_skip_t_arrive", 0)
        fbq.set_option("t_poll_limit", 0)
    assert fbq.poll_status() == 0
    for _ in range(3):
        assert torch.equal(dev.run(fbq), want)                # t of an earlier launch is never taken for this one's
    check_parity(inp, fbq)


def test_huge_and_non_finite_t(fbq):
    # t beyond the fp16 range enters the up-projection as it is; an infinite one makes infinite outputs, and no NaN
    import torch
    M, N, K, r = 4, 64, 256, 16
    inp = make_linear(M, N, K, 4, r, seed=7600)
    dev = DeviceLinear(inp, fbq)
    dev.x = torch.full((M, K), 100.0, dtype=torch.float16, device="cuda")
    dev.A = torch.full((r, K), 50.0, dtype=torch.float16, device="cuda")
    dev.B = torch.full((N, r), 2.0 ** -14, dtype=torch.float16, device="cuda")
    dev.scales = torch.zeros_like(dev.scales)
    y = dev.run(fbq)
    assert torch.all(y == 1250.0)                             # 16 ranks x 1 280 000 x 2^-14
    z = torch.zeros((M, K), dtype=torch.float16, device="cuda")
    z[1, 7] = float("inf")
    y = dev.run(fbq, x=z)
    torch.cuda.synchronize()
    assert torch.all(y[0] == 0) and torch.all(y[2:] == 0) and not torch.any(torch.isfinite(y[1]))
    assert fbq.poll_status() == 0


@pytest.mark.parametrize("M,K,rank", [(3, 100480, 16), (8, 100480, 64), (5, 131200, 0)])
def test_just_past_the_deepest_layer(fbq, M, K, rank):
    check_parity(make_linear(M, 40, K, 4, rank, seed=7700 + M), fbq, threads=16, floor=2e-5)
