"""FP32 products whose tiles are cut into equal runs of K slabs, one per SM: one
tile over many SMs, a tile or two per SM with a remainder, exactly one tile per
SM, fewer K steps than a slab, a last slab and a last step that are not full,
several column tiles.

Tolerance: a K-term FP32 dot product is within K u (|A| |B|) of the exact one
(u = 2^-24); the tests allow 2 K u."""
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


def check(got, A, B, K):
    ref = A.double() @ B.double()
    tol = 2 * K * U32 * (A.double().abs() @ B.double().abs()) + 1e-30
    assert bool(((got.double() - ref).abs() <= tol).all())


# (rows of the product, K, columns)
@pytest.mark.parametrize("M,K,k", [(40, 60004, 64), (257, 200000, 20), (512, 131072, 100), (12000, 1000, 64),
                                   (32000, 300, 50), (38912, 128, 33), (38913, 144, 40), (20000, 1028, 100),
                                   (9988, 20, 10), (60000, 68, 130), (77824, 260, 16), (39168, 2052, 7)])
def test_products(ax, M, K, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K + k)
    A, H = (torch.rand(s, generator=g, device="cuda") - 0.25 for s in ((M, K), (k, K)))
    for _ in range(2):
        check(ax.aht(A, H), A, H.T, K)
    if M % 4 == 0:
        check(ax.wta(A.T.contiguous(), H.T.contiguous()), H, A.T, K)


@pytest.mark.parametrize("m,n,k", [(15000, 1200, 20), (516, 40000, 32), (7000, 7000, 16), (9728, 9732, 10),
                                   (39000, 300, 7)])
def test_factorisation_sums_keep_their_order(ax, m, n, k):
    """The products of a factorisation split K in one way, whether the slabs' sums
    are folded where they are formed (rows that are not 16-byte aligned) or kept
    in memory and folded by a second launch: the same bits."""
    from paper_1609_09154_gb300.aunmf import Matrix

    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    A, W0, H0 = (torch.rand(s, generator=g, device="cuda") for s in ((m, n), (m, k), (k, n)))
    wide = torch.zeros((m, n + 1), device="cuda")  # stays alive: V holds its address
    wide[:, :n].copy_(A)
    V = Matrix(m, n, wide.data_ptr(), n + 1, None, None, None, 0)
    W, H, _, _ = ax.run(A, k, "mu", 2, W0, H0, prec="fp32")
    W1, H1, _, _ = ax.run(V, k, "mu", 2, W0, H0, prec="fp32")
    assert torch.equal(W, W1) and torch.equal(H, H1)
