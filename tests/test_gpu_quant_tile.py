"""The quantiser's kernel for groups of 128 where its tiles end: rows beside a multiple of 128, ranks beside the 32 indices
it stages at a time, rows of B that are not 16-byte aligned, weights that sit on rounding boundaries."""
import numpy as np
import pytest

import oracle
from test_gpu_quantizer import _dev16, _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("want_wf", [False, True])
@pytest.mark.parametrize("N,K,rank,dtype", [(1, 128, 1, "f16"), (127, 256, 31, "f16"), (129, 128, 32, "bf16"), (130, 384, 33, "f16"),
                                           (256, 128, 72, "bf16"), (128, 256, 0, "f16")])
def test_tile_edges_bit_for_bit(N, K, rank, dtype, want_wf):
    import torch
    import paper_2501_16385_b200 as fbq
    bits = 3 + N % 2
    W, A, B = _inputs(N, K, rank, dtype, seed=7000 + N)
    # a row of exact ties: range 15/4 (7/4), scale 1/4, values on multiples of 1/8
    W[-1] = np.random.default_rng(N).integers(0, 8 * ((1 << bits) - 1) // 4 + 1, K) / 8.0
    W[-1, ::128], W[-1, 1::128] = 0.0, ((1 << bits) - 1) / 4.0
    if rank:
        B[-1] = 0
    Wd = torch.from_numpy(W).cuda()
    codes, s, z, wf = fbq.quantize_feedback(Wd, None if A is None else _dev16(A, dtype), None if B is None else _dev16(B, dtype), 128, bits,
                                            want_wf=want_wf)
    c_or, s_or, z_or, _, wf_or = oracle.quantize_feedback(W, A, B, 128, bits, dtype=dtype)
    assert np.array_equal(s.view(torch.int16).cpu().numpy().view(np.uint16), s_or)
    assert np.array_equal(z.view(torch.int16).cpu().numpy().view(np.uint16), z_or)
    assert np.array_equal(codes.cpu().numpy(), c_or)
    if want_wf:
        assert np.array_equal(wf.cpu().numpy().view(np.uint32), wf_or.view(np.uint32))
    q = fbq.pack(codes, bits)
    assert np.array_equal(q.cpu().numpy().view(np.uint32), oracle.pack(c_or, bits))
