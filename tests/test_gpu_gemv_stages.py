"""3 to 8 tokens of few, ragged output features: K in slices over one, two and eight CTAs of a cluster that are not of one length,
warps with stages of one and of two quantisation groups, with a group more than others, and with none."""
import pytest

from gpu_utils import check_parity
from workloads import make_linear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,dtype,M,N,K,rank", [
    (4, "f16", 3, 40, 17 * 128, 0), (3, "bf16", 8, 24, 9 * 128, 16), (4, "bf16", 4, 8, 128, 64),       # 17 and 9 groups over two CTAs, one group
    (4, "f16", 7, 72, 86 * 128, 64), (3, "f16", 8, 40, 86 * 128, 0),                                    # eight CTAs of 10 and 11 groups,
    (4, "bf16", 8, 56, 86 * 128, 128), (3, "f16", 6, 24, 129 * 128, 32), (4, "f16", 3, 40, 193 * 128, 128)])   # ... 16 and 17, 24 and 25
def test_stage_sizes_and_slices(bits, dtype, M, N, K, rank):
    import paper_2501_16385_b200 as fbq
    inp = make_linear(M, N, K, bits, rank, dtype=dtype, seed=4000 + M + K, outlier_frac=0.01)
    check_parity(inp, fbq, expect_kernel=fbq.KERNEL_DECODE, threads=16, floor=2e-5)
