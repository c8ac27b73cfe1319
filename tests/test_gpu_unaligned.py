"""FP32 products of matrices whose rows are not 16-byte aligned, at the edges of
the 128-row tile, of the four-element loads and of the 16-K step, every column
width, enough rows that the output tiles are not few.

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


@pytest.mark.parametrize("M,K,k", [(9985, 1003, 64), (9987, 1009, 50), (20001, 17, 33), (20002, 15, 16),
                                   (12289, 1027, 10), (38913, 259, 32), (10001, 1, 5), (39001, 129, 130)])
def test_products(ax, M, K, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K + k)
    A, H = (torch.rand(s, generator=g, device="cuda") - 0.25 for s in ((M, K), (k, K)))
    check(ax.aht(A, H), A, H.T, K)  # rows of K floats
    At = A.T.clone(memory_format=torch.contiguous_format)  # K = 1: a view of A keeps its stride of 1
    check(ax.wta(At, H.T.contiguous()), H, A.T, K)  # rows of M floats
