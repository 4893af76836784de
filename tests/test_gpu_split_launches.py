"""The split kernel's count of launches, whose numbers the words of t carry: grids of more than 65536 CTAs, and
counts at which a number of 32 bits, or of 31, comes round; calls whose grid is bounded to less than holds their rows."""
import pytest

from gpu_utils import DeviceLinear, REL_F_TOL, check_parity
from workloads import make_linear

pytestmark = pytest.mark.gpu


def _codes(words, rows, K):
    """INT4 codes of some rows, [rows][K]."""
    import torch
    w = words.view(-1, K // 8)[rows]
    return (w[:, :, None] >> torch.arange(0, 32, 4, device="cuda", dtype=torch.int32)).bitwise_and(15).reshape(len(rows), K)


def test_more_than_65536_ctas():
    import torch
    import paper_2501_16385_b200 as fbq
    M, N, K, r = 16, 15_000_000, 128, 128
    ctas, _ = fbq.split_plan(M, N, K, 128, 4, r)
    assert ctas > 65536
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    words = torch.randint(-2**31, 2**31, (fbq.packed_words(N, K, 4),), dtype=torch.int32, device="cuda", generator=g)
    scales = (torch.rand((N, 1), device="cuda", generator=g) * 0.015 + 0.005).half()
    zeros = torch.randint(6, 10, (N, 1), device="cuda", generator=g).half()
    x = torch.randn((M, K), device="cuda", generator=g).half()
    A = (torch.randn((r, K), device="cuda", generator=g) * 0.2).half()
    B = torch.randn((N, r), dtype=torch.float16, device="cuda", generator=g) * 0.1
    small = slice(0, 4096)
    for _ in range(2):                                        # the second launch has the number after the first one's
        y = fbq.linear(x, words, scales, zeros, A, B, N, 128, 4)
        torch.cuda.synchronize()
        assert fbq.poll_status() == 0
        y_small = fbq.linear(x, words[: 4096 * K // 8], scales[small], zeros[small], A, B[small], 4096, 128, 4)
        rows = torch.cat([torch.arange(0, N, N // 20000, device="cuda"), torch.arange(N - 200, N, device="cuda")])
        w = scales[rows].double() * (_codes(words, rows, K).double() - zeros[rows].double())
        want = x.double() @ w.T + (x.double() @ A.double().T) @ B[rows].double().T
        got = y[:, rows].double()
        assert float((got - want).norm() / want.norm()) <= REL_F_TOL
        # row by row: most of an output comes from t, which a row without it would show
        assert float(((got - want).norm(dim=0) / want.norm(dim=0)).max()) < 0.02
        assert torch.equal(y_small, y[:, small])              # (one tile's sums do not depend on the grid: one K slice)
    assert fbq.poll_status() == 0


@pytest.mark.parametrize("launches", [-2, -1, 2**31 - 2, 2**31 - 1, -2**31])
@pytest.mark.parametrize("M,N,K,rank,ctas", [(16, 200, 1024, 64, 0), (8, 40, 512, 128, 0), (16, 1096, 1024, 64, 2)])
def test_number_comes_round(launches, M, N, K, rank, ctas):
    # fewer tiles than warps, so that some warps multiply no tile and have not looked at t when they take it in, and (the last
    # one) tiles in several passes, where none has: each launch around the turn waits for its own t
    import torch
    import paper_2501_16385_b200 as fbq
    inp = make_linear(M, N, K, 4, rank, seed=7700 + M + N, ab_std=0.141)
    dev = DeviceLinear(inp, fbq)
    assert fbq.split_plan(M, N, K, 128, 4, rank) is not None
    fbq.set_option("gemv_ctas", ctas)
    try:
        check_parity(inp, fbq, threads=16)
        want = dev.run(fbq)
        other = -dev.x                                        # in between: another t in the same words
        negative = dev.run(fbq, x=other)
        torch.cuda.synchronize()
        fbq.set_option("test_split_launches", launches)
        for _ in range(4):
            assert torch.equal(dev.run(fbq), want)
            assert torch.equal(dev.run(fbq, x=other), negative)
        torch.cuda.synchronize()
    finally:
        fbq.set_option("gemv_ctas", 0)
    assert fbq.get_option("test_split_launches") == 0 and fbq.poll_status() == 0


@pytest.mark.parametrize("bits,dtype,M,N,K,rank,ctas", [(4, "bf16", 8, 11008, 512, 128, 3), (3, "f16", 16, 4104, 1024, 64, 5), (4, "f16", 5, 90008, 128, 0, 1),
                                                       (3, "bf16", 12, 2056, 5120, 32, 8)])
def test_rows_in_several_launches(bits, dtype, M, N, K, rank, ctas):
    import torch
    import paper_2501_16385_b200 as fbq
    inp = make_linear(M, N, K, bits, rank, dtype=dtype, seed=7900 + M + N)
    assert fbq.split_plan(M, N, K, 128, bits, rank, dtype == "bf16", ctas)[0] <= ctas
    dev = DeviceLinear(inp, fbq)
    whole = dev.run(fbq)
    fbq.set_option("gemv_ctas", ctas)
    try:
        before = fbq.launch_count()
        ys = [dev.run(fbq) for _ in range(2)]
        assert fbq.launch_count() - before > 2
        torch.cuda.synchronize()
    finally:
        fbq.set_option("gemv_ctas", 0)
    assert fbq.poll_status() == 0 and torch.equal(*ys)
    # fp32 sums in another order, one rounding each
    d = (ys[0].double() - whole.double()).norm(dim=0) / whole.double().norm(dim=0)
    assert float(d.max()) < (2.0 ** -7 if dtype == "bf16" else 2.0 ** -10)
