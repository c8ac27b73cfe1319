"""The FP32 products' form for few output tiles (K cut over a cluster of
blocks), the Grams and sums that a launch's last block finishes, and the HALS
normalisation in one launch, at the sizes where they can go wrong: one row or
column past a tile, K one past a slab, a split or the fit into shared memory,
rows that are not 16-byte aligned, every column width.

Tolerance as in test_gpu_parity.py: a K-term FP32 dot product is within
K u (|A| |B|) of the exact one (u = 2^-24); the tests allow 2 K u."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ax():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf.Handle()


def rnd(g, *shape):
    return torch.rand(shape, generator=g, device="cuda") - 0.25


def check(got, A, B, K):
    ref = A.double() @ B.double()
    tol = 2 * K * U32 * (A.double().abs() @ B.double().abs()) + 1e-30
    assert bool(((got.double() - ref).abs() <= tol).all())


# (m, n, k): A H^T has m rows and contracts n, W^T A the other way round
SHAPES = [(127, 128, 16), (128, 129, 17), (129, 1024, 32), (1, 4, 1), (257, 1025, 33), (300, 4096, 64),
          (260, 4100, 64), (64, 8192, 32), (130, 8196, 20), (90, 17408, 10), (131, 17412, 16),
          (1000, 903, 65), (2000, 1500, 10), (4864, 260, 50), (4865, 260, 64), (9729, 132, 12)]


@pytest.mark.parametrize("m,n,k", SHAPES)
def test_products(ax, m, n, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + 7 * n + k)
    A, H, W = rnd(g, m, n), rnd(g, k, n), rnd(g, m, k)
    check(ax.aht(A, H), A, H.T, n)
    check(ax.wta(A, W), W.T, A, m)
    # the transposed sides, whose long axis is the other operand's
    At = A.T.contiguous()
    check(ax.wta(At, H.T.contiguous()), H, A.T, n)
    check(ax.aht(At, W.T.contiguous()), At, W, m)


@pytest.mark.parametrize("rows", [1, 63, 64, 65, 128, 129, 4097, 9729, 38912, 38913])
@pytest.mark.parametrize("k", [1, 10, 17, 50])
def test_gram(ax, rows, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(rows + k)
    X = rnd(g, rows, k)
    for _ in range(2):  # twice: the last block's counter is back at its start
        G = ax.gram_w(X)
        check(G, X.T, X, rows)
        assert torch.equal(G, G.T)


@pytest.mark.parametrize("m,n,k", [(33, 20, 3), (500, 333, 8), (1201, 804, 50), (700, 900, 130)])
def test_residual_loss_and_hals_normalisation(ax, m, n, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    A = torch.rand((m, n), generator=g, device="cuda") + 1.0
    W, H = (torch.rand(s, generator=g, device="cuda") * 0.1 for s in ((m, k), (k, n)))
    W[:, 0] = 0.0  # a zero column stays as it is
    D = (A.double() - W.double() @ H.double()).norm()
    # far from a fit nothing cancels: u-sized terms, plus the sums' own
    for _ in range(2):
        assert ax.relres(A, W, H) == pytest.approx(float(D / A.double().norm()), rel=1e-6)
        loss, _ = ax.loss_fwd(A, W, H)
        assert float(loss) == pytest.approx(0.5 * float(D) ** 2, rel=2e-6)
    GH = (H.double() @ H.double().T).float()
    P = (A.double() @ H.double().T).float()
    P[:, 0] = -1.0
    W2, H2 = W.clone(), H.clone()
    ax.update_w("hals", W2, P, GH, H2)
    s = W2.double().norm(dim=0)
    live = s > 0
    # unit columns: k u for the Gram's entry and the product, well inside 1e-5
    assert bool(((s[live] - 1).abs() <= 1e-5).all()) and not bool(live[0])
    W3 = W.clone()
    ax.update_w("hals", W3, P, GH)
    assert torch.equal(W3, W2)
    scale = (H2.double() / H.double())
    row = scale.mean(dim=1, keepdim=True)
    assert bool(((scale - row).abs() <= 4 * U32 * row.abs()).all())
    assert torch.equal(H2[0], H[0])
