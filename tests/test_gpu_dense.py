"""The prefill kernel that dequantises the weights once per call (many tiles): ragged tokens and features, K that is not
a multiple of its dequantisation units, every sub-branch width of its blocks, both activation types; call after call."""
import numpy as np
import pytest

import oracle
from gpu_utils import DeviceLinear, check_parity, torch_to_f64
from workloads import make_exact_class, make_linear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,dtype,M,N,K,rank", [(4, "bf16", 2090, 7432, 384, 64), (3, "f16", 3001, 5128, 256, 200),
                                                   (4, "f16", 2500, 6920, 128, 0), (3, "bf16", 700, 22024, 640, 8)])
def test_dense_prefill_edges(bits, dtype, M, N, K, rank):
    import paper_2501_16385_b200 as fbq
    inp = make_linear(M, N, K, bits, rank, dtype=dtype, seed=3000 + M, outlier_frac=0.01)
    rows = np.unique(np.concatenate([np.arange(9), np.arange(N - 9, N), np.random.default_rng(M).choice(N, 20)]))
    check_parity(inp, fbq, expect_kernel=fbq.KERNEL_PREFILL, n_list=rows, threads=16, floor=2e-5)


def test_dense_prefill_exact_class_is_bitwise_and_repeats():
    import paper_2501_16385_b200 as fbq
    inp = make_exact_class(1100, 13064, 512, 4, 64, seed=3100, x_nnz=32, x_max=2)
    dev = DeviceLinear(inp, fbq)
    rows = np.arange(5, inp.N, 97)
    want = oracle.linear_inputs(inp, n_list=rows, threads=16)
    for _ in range(3):
        y = torch_to_f64(dev.run(fbq), "f16")
        assert fbq.poll_status() == 0
        assert np.array_equal(y[:, rows], want)


def test_dense_prefill_on_streams_that_share_the_sms():
    # 6000 tokens are 47 t tiles: more than half of the pairs, so launches that share the SMs cannot each have a pair per
    # t tile.  The waits of a launch must not depend on that: every call returns without a time-out and with the same bits
    # as alone (sums of a tile are made by one pair in a fixed order, whichever pair that is).
    import torch
    import paper_2501_16385_b200 as fbq
    devs = [DeviceLinear(make_linear(6000, 5128 + 256 * i, 384, 4, 64, dtype="bf16", seed=3200 + i), fbq) for i in range(3)]
    alone = [d.run(fbq) for d in devs]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in devs]
    for s in streams:
        s.wait_stream(torch.cuda.current_stream())
    for _ in range(10):
        got = []
        for s, d in zip(streams, devs):
            with torch.cuda.stream(s):
                got.append([d.run(fbq) for _ in range(3)])
        torch.cuda.synchronize()
        for s in streams:
            assert fbq.poll_status(s) == 0
        for ys, want in zip(got, alone):
            assert all(torch.equal(y, want) for y in ys)


def test_dense_prefill_of_a_matrix_wider_than_the_scratch():
    # 62000 x 4352 weights are 540 MB in 16 bits: two launches of 31232 and 30768 rows
    import torch
    import paper_2501_16385_b200 as fbq
    M, N, K = 1000, 62000, 4352
    inp = make_linear(M, N, K, 3, 16, dtype="f16", seed=3300)
    rows = np.unique(np.concatenate([[0, 1, 32767, 32768, N - 1], np.arange(31224, 31240), np.random.default_rng(1).choice(N, 12)]))
    fbq.release_workspaces()
    before = fbq.launch_count()
    check_parity(inp, fbq, expect_kernel=fbq.KERNEL_PREFILL, n_list=rows, threads=16, floor=2e-5)
    assert fbq.launch_count() - before == 3                  # one of them packs the codes
    dev = DeviceLinear(inp, fbq)
    dev.run(fbq)
    torch.cuda.synchronize()
    y = dev.run(fbq)
    assert torch.equal(y, dev.run(fbq))


def test_dense_prefill_without_its_scratch_runs_the_other_kernel():
    # In a capture on a stream that has no room for the 16-bit weights the call is still served.  Counters and t are warmed up
    # by calls that never use that scratch: 222 tiles of 256 features (three waves) and a call of few features.
    import torch
    import paper_2501_16385_b200 as fbq
    inp = make_linear(1030, 11520, 256, 4, 16, dtype="f16", seed=3400)
    dev = DeviceLinear(inp, fbq)
    want = dev.run(fbq)                                      # with the scratch, on the current stream
    warm = [DeviceLinear(make_linear(129, 56832, 128, 4, 0, seed=3401), fbq), DeviceLinear(make_linear(1030, 512, 128, 4, 16, seed=3402), fbq)]
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    y = torch.full((1030, 11520), float("nan"), dtype=torch.float16, device="cuda")
    with torch.cuda.stream(stream):
        for d in warm:
            d.run(fbq)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            fbq.linear(dev.x, dev.qweight, dev.scales, dev.zeros, dev.A, dev.B, 11520, 128, 4, y=y)
        for _ in range(2):
            y.fill_(float("nan"))
            graph.replay()
            stream.synchronize()
            assert fbq.poll_status(stream) == 0
            # the same products of the same rounded weights and t, sums in another order: one rounding to fp16 apart
            assert float((y.float() - want.float()).norm() / want.float().norm()) < 2 ** -10


def test_pair_option_holds_for_many_tiles():
    # the option's kernel dequantises in place: the call takes none of the 16-bit weights' scratch (67 MB here)
    import torch
    import paper_2501_16385_b200 as fbq
    inp = make_linear(1100, 13064, 2560, 4, 64, seed=3500)
    rows = np.arange(3, inp.N, 501)
    dev = DeviceLinear(inp, fbq)
    taken = []
    for pair in (0, 1):
        fbq.set_option("prefill_pair", pair)
        try:
            dev.run(fbq)                                     # the output's memory is with torch, the kernel is loaded
            torch.cuda.synchronize()
            fbq.release_workspaces()
            before = torch.cuda.mem_get_info()[0]
            dev.run(fbq)
            torch.cuda.synchronize()
            taken.append(before - torch.cuda.mem_get_info()[0])
            check_parity(inp, fbq, expect_kernel=fbq.KERNEL_PREFILL, n_list=rows, threads=16, floor=2e-5)
        finally:
            fbq.set_option("prefill_pair", 0)
    assert taken[0] >= inp.N * inp.K * 2 > taken[1]


@pytest.mark.parametrize("K,rank", [(128, 0), (128, 64), (256, 8)])
def test_dense_prefill_of_many_short_tiles(K, rank):
    # 55 x 32 tiles, some twenty per pair, each of one to three stages: the ring of claimed tiles wraps around while the copies
    # run as many tiles ahead of the epilogue as they can
    import torch
    import paper_2501_16385_b200 as fbq
    M, N = 8000, 14008
    inp = make_linear(M, N, K, 4, rank, dtype="f16", seed=3600 + K + rank)
    rows = np.unique(np.concatenate([np.arange(4), np.arange(N - 4, N), np.random.default_rng(K).choice(N, 24)]))
    check_parity(inp, fbq, expect_kernel=fbq.KERNEL_PREFILL, n_list=rows, threads=16, floor=2e-5)
    dev = DeviceLinear(inp, fbq)
    want = dev.run(fbq)
    for _ in range(20):
        assert torch.equal(dev.run(fbq), want)
    assert fbq.poll_status() == 0
