"""The grid bound of one stream's linears: it changes that stream alone, outlives the scratch buffers, and is taken back by 0."""
import pytest

from gpu_utils import DeviceLinear, check_parity
from workloads import make_linear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,bits,rank", [(1, 3, 64), (2, 4, 0), (4, 4, 32)])
def test_stream_option_bounds_the_grid_of_one_stream(M, bits, rank):
    import torch
    import paper_2501_16385_b200 as fbq
    inp = make_linear(M, 4096, 1024, bits, rank, seed=9000 + M)
    check_parity(inp, fbq, expect_kernel=fbq.KERNEL_DECODE)
    dev = DeviceLinear(inp, fbq)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]

    def run(s):
        with torch.cuda.stream(s):
            y = dev.run(fbq)
        s.synchronize()
        assert fbq.poll_status(s) == 0
        return y

    default = [run(s) for s in streams]
    assert torch.equal(*default)
    try:
        fbq.set_option("gemv_ctas", 24)
        bounded = run(streams[0])                    # what a grid of 24 CTAs gives, bit for bit
    finally:
        fbq.set_option("gemv_ctas", 0)
    fbq.set_stream_option("gemv_ctas", 24, streams[0])
    assert torch.equal(run(streams[0]), bounded) and torch.equal(run(streams[1]), default[1])
    fbq.release_workspaces()
    assert torch.equal(run(streams[0]), bounded)
    fbq.set_stream_option("gemv_ctas", 0, streams[0])
    assert torch.equal(run(streams[0]), default[0])
    assert float((bounded.float() - default[0].float()).norm() / default[0].float().norm()) < 2 ** -10


def test_stream_option_rejects_what_it_does_not_know():
    import paper_2501_16385_b200 as fbq
    for name, value in (("batch_ctas", 1), ("gemv_ctas", -1)):
        with pytest.raises(fbq.FbqError) as err:
            fbq.set_stream_option(name, value)
        assert err.value.code == -1
