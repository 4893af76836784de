"""Streaming decode of 3 to 8 tokens: stages of sixteen or of eight quantisation groups, whole K or K slices, with K just
past a stage and just past a warp's share of it, and few, ragged output features."""
import pytest

from gpu_utils import check_parity
from workloads import make_linear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,dtype,M,N,K,rank", [
    (4, "f16", 3, 40, 17 * 128, 0), (3, "bf16", 8, 24, 9 * 128, 16), (4, "bf16", 4, 8, 128, 64),       # whole K, sixteen
    (4, "f16", 7, 72, 86 * 128, 64), (3, "f16", 8, 40, 86 * 128, 0),                                    # whole K, eight
    (4, "bf16", 8, 56, 86 * 128, 128), (3, "f16", 6, 24, 129 * 128, 32), (4, "f16", 3, 40, 193 * 128, 128)])   # slices
def test_stage_sizes_and_slices(bits, dtype, M, N, K, rank):
    import paper_2501_16385_b200 as fbq
    inp = make_linear(M, N, K, bits, rank, dtype=dtype, seed=4000 + M + K, outlier_frac=0.01)
    check_parity(inp, fbq, expect_kernel=fbq.KERNEL_DECODE, threads=16, floor=2e-5)
