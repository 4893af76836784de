"""Calls whose large scratch cannot be allocated are still served: prompts by the prefill kernel that needs none, the Gram matrix
and the reconstruction step with smaller slabs, the step at last in the unused half of the caller's workspace.  The device's
memory is taken by one large tensor for the length of a call, after the kernels have been loaded."""
import contextlib

import numpy as np
import pytest

from gpu_utils import DeviceLinear
from workloads import make_linear

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def free_megabytes(fbq, n):
    import torch
    torch.cuda.synchronize()
    fbq.release_workspaces()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (n << 20), dtype=torch.uint8, device="cuda")
    try:
        yield
        torch.cuda.synchronize()
        assert fbq.poll_status() == 0
    finally:
        del hog
        torch.cuda.empty_cache()
        fbq.release_workspaces()


def test_long_prompt_without_memory_for_16_bit_weights():
    import torch
    import paper_2501_16385_b200 as fbq
    dev = DeviceLinear(make_linear(1100, 13064, 2560, 4, 64, seed=9100), fbq)       # 67 MB in 16 bits
    want = dev.run(fbq)
    i = dev.inp
    ys = [torch.full_like(want, float("nan")) for _ in range(2)]
    DeviceLinear(make_linear(1100, 512, 2560, 4, 64, seed=9101), fbq).run(fbq)       # loads the kernel of few tiles
    with free_megabytes(fbq, 40):
        for y in ys:
            fbq.linear(dev.x, dev.qweight, dev.scales, dev.zeros, dev.A, dev.B, i.N, 128, 4, y=y)
    assert torch.equal(*ys)
    y = ys[0]
    # the same rounded weights and t, sums in another order: one rounding to fp16 apart
    assert float((y.float() - want.float()).norm() / want.float().norm()) < 2 ** -10
    assert torch.equal(dev.run(fbq), want)                                           # with memory again, the kernel of before


@pytest.mark.parametrize("left", [100, 10])            # 201 MB wanted, 128 with the lowered bound, 17 at least
def test_step_without_memory_for_its_scratch(left):
    import torch
    import paper_2501_16385_b200 as fbq
    N, K, rank = 2048, 4096, 16
    g = torch.Generator(device="cuda")
    g.manual_seed(left)
    X = torch.randn((512, K), device="cuda", generator=g)
    W = torch.randn((N, K), device="cuda", generator=g) * 0.05
    A = torch.randn((rank, K), device="cuda", generator=g) * 0.05
    B = torch.randn((N, rank), device="cuda", generator=g) * 0.05
    H = fbq.gram(X)
    a, b = A.clone(), B.clone()
    loss, ws = fbq.reconstruct_step(W, H, a, b, 1e-7, 128, 4)
    want = [float(loss.item()), a, b]
    a2, b2, loss2 = A.clone(), B.clone(), torch.zeros(1, device="cuda")
    with free_megabytes(fbq, left):
        fbq.reconstruct_step(W, H, a2, b2, 1e-7, 128, 4, workspace=ws, loss=loss2)
    # fp32 sums in another order (tests/test_gpu_products.py has the bounds of either against float64)
    assert np.isclose(float(loss2.item()), want[0], rtol=4e-6)
    assert float((a2 - want[1]).norm() / want[1].norm()) < 2e-6 and float((b2 - want[2]).norm() / want[2].norm()) < 2e-6


def test_gram_without_memory_for_its_scratch():
    import torch
    import paper_2501_16385_b200 as fbq
    X = torch.randn((20000, 1024), device="cuda")                                    # 123 MB of split operands
    want = X.double().T @ X.double()
    fbq.gram(X[:512].contiguous())
    H = torch.empty((1024, 1024), device="cuda")
    with free_megabytes(fbq, 40):
        assert fbq.lib().fbq_gram(X.data_ptr(), H.data_ptr(), 20000, 1024, torch.cuda.current_stream().cuda_stream) == 0
    assert float((H.double() - want).norm() / want.norm()) < 3e-7
