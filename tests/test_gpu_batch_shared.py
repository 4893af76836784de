"""Batches whose problems share x: one launch of the streaming kernel over all of them.  Row counts from one tile to many,
ragged ones, every form of the kernel; the same through host buffers, pinned and pageable."""
import numpy as np
import pytest

import oracle
from gpu_utils import DeviceLinear, REL_F_TOL, compare, torch_to_f64
from workloads import make_linear

pytestmark = pytest.mark.gpu


def _shared(M, bits, rank, dtype, K, rows):
    inps = [make_linear(M, N, K, bits, rank, dtype=dtype, seed=8000 + N) for N in rows]
    for i in inps[1:]:
        i.x = inps[0].x
    return inps


def _check(inps, ys, dtype):
    for inp, y in zip(inps, ys):
        want = oracle.linear_inputs(inp, threads=8)
        rel, mx, lim = compare(torch_to_f64(y, dtype), want, inp.x_f64(), inp.K)
        lim += 2.0 ** -8 * float(np.max(np.abs(want))) if dtype == "bf16" else 0.0
        assert rel <= REL_F_TOL and mx <= lim


@pytest.mark.parametrize("M,bits,rank,dtype,K,rows", [(1, 3, 64, "f16", 1024, (8, 1000, 4096)), (1, 4, 0, "bf16", 2048, (16, 24)),
                                                      (2, 4, 128, "f16", 640, (512, 512, 512)), (4, 4, 64, "bf16", 1024, (40, 2048, 8)),
                                                      (3, 3, 0, "f16", 256, (16, 32)), (12, 4, 16, "f16", 512, (1376, 1376)),
                                                      (2, 3, 32, "bf16", 384, (64,) * 8)])
def test_shared_x_is_one_launch(M, bits, rank, dtype, K, rows):
    import torch
    import paper_2501_16385_b200 as fbq
    inps = _shared(M, bits, rank, dtype, K, rows)
    devs = [DeviceLinear(i, fbq) for i in inps]
    ys = [torch.full((M, i.N), float("nan"), dtype=devs[0].x.dtype, device="cuda") for i in inps]
    probs = [(devs[0].x, d.qweight, d.scales, d.zeros, d.A if rank else None, d.B if rank else None, y) for d, y in zip(devs, ys)]
    fits = all(i.N > 16 for i in inps) or M <= 2          # the 16-bit form pairs its CTAs: a single tile goes alone
    for _ in range(3):                                   # scratch and counters are back at zero each time
        before = fbq.launch_count()
        fbq.linear_batch(probs, 128, bits)
        torch.cuda.synchronize()
        assert fbq.launch_count() - before == (1 if fits else len(rows))
        assert fbq.poll_status() == 0
    _check(inps, ys, dtype)
    # the same from and to host memory, pinned (shared and not) and pageable
    hx = devs[0].x.cpu().pin_memory()
    for pin_x, pin_y in ((True, True), (False, True), (True, False)):
        x = hx if pin_x else devs[0].x.cpu()
        hy = [torch.zeros((M, i.N), dtype=x.dtype) for i in inps]
        hy = [y.pin_memory() for y in hy] if pin_y else hy
        fbq.linear_batch([(x, *p[1:6], y) for p, y in zip(probs, hy)], 128, bits, host_io=True)
        torch.cuda.synchronize()
        assert fbq.poll_status() == 0
        for d, h in zip(ys, hy):
            assert torch.allclose(d.cpu().float(), h.float(), rtol=2e-2, atol=2e-3)


@pytest.mark.parametrize("M,bits,rank,dtype,K,rows", [(1, 4, 128, "f16", 4096, (4096, 1000, 40)), (2, 3, 112, "bf16", 1024, (2056, 2056)),
                                                      (1, 3, 128, "f16", 13824, (640, 640)), (2, 4, 64, "f16", 13824, (640, 520)),
                                                      (1, 4, 128, "f16", 4096, (4096,) * 4 + (11008,) * 2)])
def test_shared_x_with_ctas_that_fill_an_sm(M, bits, rank, dtype, K, rows):
    # t CTAs of rank 112 and 128, or x of a long K, take more than half of an SM's shared memory: one CTA per SM; in the last
    # case the t CTAs of six problems would leave too few SMs, and some main CTAs start when they are through
    test_shared_x_is_one_launch(M, bits, rank, dtype, K, rows)
