"""Calls of 3 to 16 tokens on inputs at the ends of the formats: x so small that its quotients by the field weights of the codes
are subnormal in fp16, in all of a token, in some of its groups, beside larger ones, and in some tokens only; x so large that it
cannot be scaled up against that; columns of x that are large in every group, and x of one sign; infinities and NaN."""
import pytest

pytestmark = pytest.mark.gpu


def _problem(fbq, M, N, K, bits, rank, dtype, seed):
    """Weights as the library takes them, and dequantised in 64 bits."""
    import torch
    act = torch.float16 if dtype == "f16" else torch.bfloat16
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    codes = torch.randint(0, 2 ** bits, (N, K), device="cuda", generator=g).to(torch.uint8)
    scales = (torch.rand((N, K // 128), device="cuda", generator=g) * 0.4 + 0.2).half()
    zeros = torch.randint(2 ** bits // 2 - 2, 2 ** bits // 2 + 2, (N, K // 128), device="cuda", generator=g).half()
    A = (torch.randn((rank, K), device="cuda", generator=g) * 0.2).to(act) if rank else None
    B = (torch.randn((N, rank), device="cuda", generator=g) * 0.2).to(act) if rank else None
    w = (codes.double().view(N, -1, 128) - zeros.double()[:, :, None]) * scales.double()[:, :, None]

    def run(x):
        return fbq.linear(x, fbq.pack(codes, bits), scales, zeros, A, B, N, 128, bits)

    return run, w.view(N, K), A, B, g


@pytest.mark.parametrize("rank", [0, 32])
@pytest.mark.parametrize("M,K", [(3, 1152), (8, 1152), (9, 2048), (16, 5120)])
@pytest.mark.parametrize("bits", [3, 4])
def test_small_x(bits, M, K, rank):
    import torch
    import paper_2501_16385_b200 as fbq
    N = 264
    run, w, A, B, g = _problem(fbq, M, N, K, bits, rank, "f16", 100 * bits + M)
    n = torch.randn((M, K), device="cuda", generator=g)
    cases = [n * s for s in (1.0, 1e-2, 1e-3, 3e-4, 1e-4, 3e-5, 1e-5)]
    cases.append(n * 10.0 ** -(torch.arange(M, device="cuda") % 6)[:, None])                        # every token its own size
    cases.append(n * 10.0 ** -(torch.arange(K, device="cuda") // 128 % 6)[None])                   # every group
    cases.append(n * 1e-4 * (torch.arange(K, device="cuda") >= K - 128)[None])                     # all zero but a group's
    cases.append(n * (torch.arange(M, device="cuda") % 3)[:, None] * 1e-4)                         # zero tokens among others
    line = 1024.0 if bits == 3 else 4096.0                    # from here on x times the largest field weight is not finite
    for large in (line - 1, line, 5000.0):
        x = n * 1e-4
        x[1:, 200] = large                                    # in one group of all tokens but one,
        cases.append(x)
        x = n * 0.03
        x[M // 2, ::1200] = -large                            # in several of one token
        cases.append(x)
    for x in cases:
        x = x.half()
        want = x.double() @ w.T
        if rank:
            want = want + (x.double() @ A.double().T) @ B.double().T
        y = run(x)
        some = want.norm(dim=1) > 0
        assert torch.all(y[~some] == 0)
        err = ((y.double() - want).norm(dim=1) / want.norm(dim=1))[some]
        # the roundings of y (below 2^-14 to multiples of 2^-24) and of x, the latter below 1e-4
        rms = want[some].square().mean(dim=1).sqrt()
        assert torch.all(err <= 2.0 ** -11 + 2.0 ** -25 / rms + 1e-4)
    torch.cuda.synchronize()
    assert fbq.poll_status() == 0


@pytest.mark.parametrize("M,K", [(8, 4096), (16, 13824)])
@pytest.mark.parametrize("bits", [3, 4])
def test_large_columns(bits, M, K):
    # what a token's sums lose where one column of every group is far larger than the rest, or all x have one sign: about the
    # rounding of y (2.1e-4) and no more once again, 4e-4 in all; the prefill kernel, which rounds the weights, has 2.9e-4
    import torch
    import paper_2501_16385_b200 as fbq
    run, w, _, _, g = _problem(fbq, M, 1024, K, bits, 0, "f16", 300 * bits + M)
    n = torch.randn((M, K), device="cuda", generator=g)
    cases = [n.abs(), n + 2]
    for column in (0, 77, 127):
        x = n * 0.02
        x.view(M, -1, 128)[:, :, column] = 20.0
        cases.append(x)
    for x in cases:
        x = x.half()
        want = x.double() @ w.T
        assert float(((run(x).double() - want).norm(dim=1) / want.norm(dim=1)).max()) <= 4e-4
    assert fbq.poll_status() == 0


@pytest.mark.parametrize("bits,dtype,M,K,rank", [(3, "f16", 16, 5120, 0), (4, "bf16", 16, 5120, 0), (4, "f16", 12, 5120, 32), (3, "bf16", 9, 13824, 0),
                                                 (3, "f16", 4, 1152, 32), (4, "bf16", 8, 128, 0)])
def test_infinite_and_huge_x(bits, dtype, M, K, rank):
    # infinities of the sign of x times the weight, NaN where such meet or the weight is 0, in the tokens that hold them and no others
    import torch
    import paper_2501_16385_b200 as fbq
    run, w, A, B, g = _problem(fbq, M, 72, K, bits, rank, dtype, 500 * bits + M)
    act = torch.float16 if dtype == "f16" else torch.bfloat16
    x = torch.randn((M, K), device="cuda", generator=g).to(act)
    clean = run(x)
    inf = float("inf")
    x[0, 3], x[0, K - 1] = inf, inf
    x[1, 77] = -inf
    x[2, 5], x[2, K - 1 - 127] = inf, -inf
    if M > 3:
        x[M - 1, K // 2] = float("nan")
    if M > 8 and dtype == "bf16":
        x[8] = 2e35 * torch.rand((K,), device="cuda", generator=g).to(act)     # 128 times their sum is beyond fp32, y is not
    want = (x.double()[:, None, :] * w[None]).sum(-1)
    if rank:
        t = (x.double()[:, None, :] * A.double()[None]).sum(-1)
        want = want + (t[:, None, :] * B.double()[None]).sum(-1)
    y = run(x)
    assert torch.equal(y.isnan(), want.isnan()) and torch.equal(y.isinf(), want.isinf())
    assert torch.equal(y[y.isinf()].sign().double(), want[want.isinf()].sign())
    assert y[:2].isinf().any() or rank
    same = [m for m in range(3, M - 1) if m != 8]
    assert torch.equal(y[same], clean[same])
    if M > 8 and dtype == "bf16":
        assert float((y[8].double() - want[8]).norm() / want[8].norm()) < 2.0 ** -8
    torch.cuda.synchronize()
    assert fbq.poll_status() == 0
