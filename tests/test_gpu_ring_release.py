"""The rings of the kernels that read TMA-copied tiles with ordinary loads
(FP32 products and wide Grams, direct tensor-core products): a stage that is
given back too early is overwritten under the loads.  A fits in L2, so the next
copy lands soon; the entries are small whole numbers, so every sum is exact in
FP32 and any misplaced tile shows, in every one of the repeated calls."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ax():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf.Handle()


def ints(g, *shape):
    return torch.randint(-3, 4, shape, generator=g, device="cuda").float()


# equal runs of slabs (64, 56, 48 columns), one block per tile in a cluster,
# unaligned rows (register-staged; clusters filled by 4-byte copies)
@pytest.mark.parametrize("m,n,k", [(40000, 400, 64), (40000, 404, 50), (30000, 512, 48), (2000, 1500, 10),
                                   (600, 9000, 64), (40000, 403, 50), (2000, 1501, 20)])
@pytest.mark.parametrize("prec", ["fp32", "tf32", "bf16"])
def test_single_products(ax, m, n, k, prec):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n + k)
    A, H, W = ints(g, m, n), ints(g, k, n), ints(g, m, k)
    P, Q = (A.double() @ H.double().T).float(), (W.double().T @ A.double()).float()
    for _ in range(10):
        assert torch.equal(ax.aht(A, H, prec), P) and torch.equal(ax.wta(A, W, prec), Q)


@pytest.mark.parametrize("rows,k", [(60000, 256), (40000, 96), (2048, 512)])
def test_wide_gram(ax, rows, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(rows)
    X = ints(g, rows, k)
    G = (X.double().T @ X.double()).float()
    for _ in range(10):
        assert torch.equal(ax.gram_w(X), G)


# whole tiles; slabs kept and folded
@pytest.mark.parametrize("m,n,k", [(40000, 400, 64), (15000, 1200, 20)])
def test_factorisation(ax, m, n, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    A, W0, H0 = (torch.rand(s, generator=g, device="cuda") for s in ((m, n), (m, k), (k, n)))
    W, H, rel, _ = ax.run(A, k, "mu", 3, W0, H0, prec="fp32")
    for _ in range(5):
        W1, H1, rel1, _ = ax.run(A, k, "mu", 3, W0, H0, prec="fp32")
        assert torch.equal(W, W1) and torch.equal(H, H1) and (rel == rel1).all()
