"""The tensor-core products behind fbq_gram and fbq_reconstruct_step where their tiles end, and how close to float64 they come."""
import numpy as np
import pytest

from oracle import reconstruct as rec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,K", [(1, 5), (65, 257), (300, 512), (129, 255), (1000, 770)])
def test_gram_tile_edges(T, K):
    import torch
    import paper_2501_16385_b200 as fbq
    rng = np.random.default_rng(T)
    X = (rng.standard_normal((T, K)) * (1.0 + 4.0 * (rng.random(K) < 0.05))).astype(np.float32)
    H = fbq.gram(torch.from_numpy(X).cuda()).cpu().numpy()
    assert fbq.poll_status() == 0
    want = X.astype(np.float64).T @ X.astype(np.float64)
    assert np.linalg.norm(H - want) <= 3e-7 * np.linalg.norm(want)
    assert np.abs(H - want).max() <= 1e-6 * np.abs(want).max()
    assert np.array_equal(H, H.T)


@pytest.mark.parametrize("N,K,rank", [(1, 128, 1), (257, 384, 33), (130, 640, 260)])
def test_step_tile_edges(N, K, rank):
    import torch
    import paper_2501_16385_b200 as fbq
    rng = np.random.default_rng(N)
    W = (rng.standard_normal((N, K)) * 0.05).astype(np.float32)
    X = rng.standard_normal((200, K)).astype(np.float32)
    A = (rng.standard_normal((rank, K)) * 0.05).astype(np.float32)
    B = (rng.standard_normal((N, rank)) * 0.05).astype(np.float32)
    H = rec.gram(X)
    lr = 0.05 / (np.linalg.eigvalsh(H)[-1] * max(np.linalg.norm(A, 2), np.linalg.norm(B, 2)) ** 2)
    Ad, Bd = torch.from_numpy(A.copy()).cuda(), torch.from_numpy(B.copy()).cuda()
    loss, _ = fbq.reconstruct_step(torch.from_numpy(W).cuda(), torch.from_numpy(H.astype(np.float32)).cuda(), Ad, Bd, lr, 128, 4)
    assert fbq.poll_status() == 0
    loss_o, A_o, B_o = rec.step(W, H, A, B, lr, 128, 4)
    assert np.isclose(float(loss.item()), loss_o, rtol=2e-6)
    assert np.linalg.norm(Ad.cpu().numpy() - A_o) <= 1e-6 * np.linalg.norm(A_o)
    assert np.linalg.norm(Bd.cpu().numpy() - B_o) <= 1e-6 * np.linalg.norm(B_o)


def test_gram_captured_before_the_stream_has_scratch():
    import torch
    import paper_2501_16385_b200 as fbq
    X = torch.randn((96, 320), device="cuda")
    fbq.gram(X[:, :64].contiguous())                   # the kernels are loaded
    H = torch.zeros((320, 320), device="cuda")
    stream = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        with torch.cuda.graph(g, stream=stream):
            H.copy_(fbq.gram(X))
    g.replay()
    torch.cuda.synchronize()
    want = X.double().T @ X.double()
    assert float((H.double() - want).norm() / want.norm()) < 3e-7


@pytest.mark.parametrize("N,K,rank", [(70, 384, 16), (300, 640, 40)])
def test_step_takes_any_h(N, K, rank):
    # H with an antisymmetric part as large as the symmetric one: G = -2 Delta_F H and tr(Delta_F H Delta_F^T) as they stand
    import torch
    import paper_2501_16385_b200 as fbq
    rng = np.random.default_rng(N + 1)
    W = (rng.standard_normal((N, K)) * 0.05).astype(np.float32)
    A = (rng.standard_normal((rank, K)) * 0.05).astype(np.float32)
    B = (rng.standard_normal((N, rank)) * 0.05).astype(np.float32)
    H = (rng.standard_normal((K, K)) + 8.0 * np.eye(K)).astype(np.float32)
    lr = 0.05 / (np.linalg.norm(H.astype(np.float64), 2) * max(np.linalg.norm(A, 2), np.linalg.norm(B, 2)) ** 2)
    Ad, Bd = torch.from_numpy(A.copy()).cuda(), torch.from_numpy(B.copy()).cuda()
    loss, _ = fbq.reconstruct_step(torch.from_numpy(W).cuda(), torch.from_numpy(H).cuda(), Ad, Bd, lr, 128, 4)
    assert fbq.poll_status() == 0
    loss_o, A_o, B_o = rec.step(W, H, A, B, lr, 128, 4)
    # the loss is a sum of K^2 terms of both signs, of which the diagonal's 8 |Delta|^2 remains: an error of 2^-24 of their
    # root sum of squares, sqrt(K) / 8 of the loss, is far inside this
    assert np.isclose(float(loss.item()), loss_o, rtol=1e-5)
    for got, want, old in ((Ad, A_o, A), (Bd, B_o, B)):
        assert np.linalg.norm(got.cpu().numpy() - want) <= 1e-6 * np.linalg.norm(want)
        # the step by itself: its error is that of the products plus one fp32 rounding of the updated matrix
        step = want - old.astype(np.float64)
        err = np.linalg.norm((got.cpu().numpy().astype(np.float64) - old) - step)
        assert err <= 1e-5 * np.linalg.norm(step) + 2.0 ** -24 * np.linalg.norm(want)


@pytest.fixture
def one_megabyte():
    import paper_2501_16385_b200 as fbq
    fbq.set_option("scratch_mb", 1)
    yield
    fbq.set_option("scratch_mb", 0)


@pytest.mark.parametrize("T,K", [(1000, 770), (257, 1000), (700, 64)])
def test_gram_in_slabs(one_megabyte, T, K):
    test_gram_tile_edges(T, K)


@pytest.mark.parametrize("N,K,rank", [(700, 1152, 33), (100, 1152, 8), (3000, 128, 16), (257, 640, 260)])
def test_step_in_slabs(one_megabyte, N, K, rank):
    # several slabs of both matrices (ragged last ones), of H alone, of Delta alone; more rank than a tile
    import paper_2501_16385_b200 as fbq
    fbq.release_workspaces()
    test_step_tile_edges(N, K, rank)
    test_step_takes_any_h(N, K, rank)


def test_scratch_of_a_large_step_is_bounded():
    # Delta, its transpose and H of 3072 x 12288 split as a whole are 1.36 GB; the default bound is 1 GB beyond what the rank needs.
    # Reference in float64 from the library's own Delta, which the tests of the quantiser pin.
    import torch
    import paper_2501_16385_b200 as fbq
    N, K, rank = 3072, 12288, 16
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    W = torch.randn((N, K), device="cuda", generator=g) * 0.05
    A = (torch.randn((rank, K), device="cuda", generator=g) * 0.05).half().float()
    B = (torch.randn((N, rank), device="cuda", generator=g) * 0.05).half().float()
    H = torch.randn((K, K), device="cuda", generator=g) + 50.0 * torch.eye(K, device="cuda")
    WF = fbq.quantize_feedback(W, A.half(), B.half(), 128, 4, want_wf=True)[3]
    D = W.double() - WF.double()
    lr = 1e-5
    DH = D @ H.double()
    want_a, want_b, want_loss = A.double() + 2 * lr * (B.double().T @ DH), B.double() + 2 * lr * (DH @ A.double().T), float((DH * D).sum())
    ws = torch.empty(int(fbq.lib().fbq_reconstruct_workspace_floats(N, K, rank)), device="cuda")
    fbq.release_workspaces()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    loss, _ = fbq.reconstruct_step(W, H, A, B, lr, 128, 4, workspace=ws)
    assert fbq.poll_status() == 0
    assert free - torch.cuda.mem_get_info()[0] < 1100 << 20
    # W_F and Delta are rounded to fp32 differently (W_F has 2^-24 of |W|, about 2^-20 of |Delta|)
    assert abs(float(loss.item()) - want_loss) <= 1e-5 * want_loss
    assert float((A.double() - want_a).norm() / want_a.norm()) < 1e-6
    assert float((B.double() - want_b).norm() / want_b.norm()) < 1e-6


def test_products_without_dependent_launch_are_the_same():
    import torch
    import paper_2501_16385_b200 as fbq
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    X, W = torch.randn((500, 512), device="cuda", generator=g), torch.randn((300, 512), device="cuda", generator=g) * 0.05
    A, B = torch.randn((24, 512), device="cuda", generator=g) * 0.05, torch.randn((300, 24), device="cuda", generator=g) * 0.05
    got = []
    for pdl in (1, 0):
        fbq.set_option("pdl", pdl)
        try:
            a, b, H = A.clone(), B.clone(), fbq.gram(X)
            loss, _ = fbq.reconstruct_step(W, H, a, b, 1e-6, 128, 4)
            got.append((H, a, b, loss))
        finally:
            fbq.set_option("pdl", 1)
    assert fbq.poll_status() == 0
    assert all(torch.equal(u, v) for u, v in zip(*got))
