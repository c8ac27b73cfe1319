"""The FP32 products' column tiles of 48, 56 and 64 columns, at the ranks where
the choice between them changes and one column to either side, with a last row
tile and a last K step that are not full.

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


# enough rows that the output tiles are not few
@pytest.mark.parametrize("m,n", [(9988, 260), (19716, 1028)])
@pytest.mark.parametrize("k", [33, 47, 48, 49, 50, 55, 56, 57, 64, 65, 96, 97, 100, 112, 113, 128, 150])
def test_products(ax, m, n, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + k)
    A, H = (torch.rand(s, generator=g, device="cuda") - 0.25 for s in ((m, n), (k, n)))
    check(ax.aht(A, H), A, H.T, n)
    At = A.T.contiguous()
    check(ax.wta(At, H.T.contiguous()), H, A.T, n)
