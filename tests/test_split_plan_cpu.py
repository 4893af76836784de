"""Plans of calls of 3 to 16 tokens (host logic): their grids under a bound on the CTAs, and where there is none."""
import pytest

import paper_2501_16385_b200 as fbq


@pytest.mark.parametrize("M,N,K,rank", [(8, 4096, 4096, 64), (8, 1608, 1152, 128), (8, 11008, 4096, 128), (4, 11008, 4096, 64), (16, 4096, 13824, 64),
                                        (16, 5120, 13824, 128), (3, 8, 128, 16), (16, 32000, 8192, 0), (5, 4096, 28672, 32)])
def test_grid_stays_within_the_bound(M, N, K, rank):
    least = None                                              # CTAs without which there is no plan
    for bound in list(range(1, 65)) + [74, 148, 296, 1000]:
        ctas, cluster = fbq.split_plan(M, N, K, 128, 4, rank, max_ctas=bound)
        least = ctas if least is None else least
        assert ctas <= max(bound, least)
        assert ctas % cluster == 0
    # one cluster for t (two hold the largest), one for the rows, of as many CTAs as hold x of all tokens
    assert least <= (3 if rank else 1) * max(1, 2 ** (((M + 7) // 8 * K // 128 + 63) // 64 - 1).bit_length())


@pytest.mark.parametrize("rank", [0, 16, 64, 128])
@pytest.mark.parametrize("M", [3, 4, 5, 8])
def test_deep_layers_without_a_plan(M, rank):
    for N in (8, 1024, 100000):
        assert fbq.split_plan(M, N, 65536, 128, 4, rank) is not None
    deepest = 131072 if rank == 0 else 100352
    assert fbq.split_plan(M, 1024, deepest, 128, 4, rank) is not None
    assert fbq.select_kernel(M, 1024, deepest, 128, 4, rank) == fbq.KERNEL_DECODE
    assert fbq.split_plan(M, 1024, deepest + 128, 128, 4, rank) is None
    # there the other decode kernel only where it is ahead of the tensor cores
    assert fbq.select_kernel(M, 1024, deepest + 128, 128, 4, rank) == (fbq.KERNEL_DECODE if M == 3 and rank <= 16 else fbq.KERNEL_PREFILL)
