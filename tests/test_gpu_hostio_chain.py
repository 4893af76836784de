"""Host-buffer calls queued one behind the other on one stream, without a synchronisation between them, where each call's
x_host is the y_host of the call before: every call has to see what the one before it wrote (calls on one stream run in
order).  The buffers start as NaN, so a value read too early shows in every output that depends on it."""
import pytest

pytestmark = pytest.mark.gpu


def _weights(fbq, K, N, bits, rank, g):
    import torch
    words = torch.randint(-2**31, 2**31, (fbq.packed_words(N, K, bits),), dtype=torch.int32, device="cuda", generator=g)
    scales = torch.full((N, K // 128), 0.005, device="cuda").half()
    zeros = torch.full((N, K // 128), 8.0 if bits == 4 else 4.0, device="cuda").half()
    A = (torch.randn((rank, K), device="cuda", generator=g) * 0.02).half() if rank else None
    B = (torch.randn((N, rank), device="cuda", generator=g) * 0.02).half() if rank else None
    return words, scales, zeros, A, B


@pytest.mark.parametrize("M,bits,rank", [(1, 3, 64), (1, 4, 0), (2, 4, 32), (8, 4, 64)])
@pytest.mark.parametrize("batch", [False, True])
def test_chained_host_calls_run_in_order(M, bits, rank, batch):
    import torch
    import paper_2501_16385_b200 as fbq
    g = torch.Generator(device="cuda")
    g.manual_seed(M * 10 + bits)
    widths = (1024, 8192, 1024, 4096, 512)              # a long kernel ahead of a short one and the reverse
    chain = [_weights(fbq, K, N, bits, rank, g) for K, N in zip(widths, widths[1:])]
    other = _weights(fbq, widths[0], 256, bits, rank, g)          # second member of each batch: reads the chain's first x
    x0 = torch.randn((M, widths[0]), device="cuda", generator=g).half()
    want, x = [], x0
    for w, N in zip(chain, widths[1:]):
        x = fbq.linear(x, *w, N, 128, bits)
        want.append(x.float().cpu())
    first = x0.cpu().pin_memory()
    for _ in range(25):
        ys = [torch.full((M, N), float("nan")).half().pin_memory() for N in widths[1:]]
        aside = torch.zeros((M, 256)).half().pin_memory()
        torch.cuda.synchronize()
        src = first
        for w, y in zip(chain, ys):
            if batch:
                fbq.linear_batch([(src, *w, y), (first, *other, aside)], 128, bits, host_io=True)
            else:
                fbq.linear_hostio(src, *w, y, y.shape[1], 128, bits)
            src = y
        torch.cuda.synchronize()
        assert fbq.poll_status() == 0
        for y, ref in zip(ys, want):
            # the same kernels on the same inputs, up to the order of the sub-branch's partial sums (another share of the
            # grid): fp16 rounding of each step, amplified by at most the four steps of the chain
            assert torch.isfinite(y).all()
            assert float((y.float() - ref).norm() / ref.norm()) < 4 * 2 ** -10


@pytest.mark.parametrize("M,pin", [(13, True), (13, False), (40, True), (300, True)])
def test_host_batches_of_mixed_kernels_and_shared_x(M, pin):
    # a batch whose problems run one after the other (some of them the tensor-core kernel's): x of all of them is staged at the
    # start of the call where it is small, per problem where it is large (300 tokens here), shared x once
    import torch
    import paper_2501_16385_b200 as fbq
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    shapes = [(1024, 512), (1024, 768), (13824, 256), (1024, 264)]
    weights = [_weights(fbq, K, N, 4, 16, g) for K, N in shapes]
    assert len({fbq.select_kernel(13, N, K, 128, 4, 16) for K, N in shapes}) == 2
    a, b, c = (torch.randn((M, K), device="cuda", generator=g).half() for K in (1024, 13824, 1024))
    xs = [a, a, b, c]
    want = [fbq.linear(x, *w, N, 128, 4) for x, w, (K, N) in zip(xs, weights, shapes)]
    host = {id(x): (x.cpu().pin_memory() if pin else x.cpu()) for x in xs}
    for _ in range(5):
        ys = [torch.full((M, N), float("nan")).half() for K, N in shapes]
        ys = [y.pin_memory() if pin else y for y in ys]
        fbq.linear_batch([(host[id(x)], *w, y) for x, w, y in zip(xs, weights, ys)], 128, 4, host_io=True)
        torch.cuda.synchronize()
        assert fbq.poll_status() == 0
        assert all(torch.equal(y, ref.cpu()) for y, ref in zip(ys, want))
