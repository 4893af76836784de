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
