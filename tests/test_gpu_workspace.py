"""Device memory that a handle keeps: no form's workspace is taken by a call that
does not run that form."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def aunmf():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf


def growth(aunmf, call):
    """Bytes that a new handle's call takes (kernels loaded by a first handle)."""
    for _ in range(2):
        h = aunmf.Handle()
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        call(h)
        torch.cuda.synchronize()
        used = before - torch.cuda.mem_get_info()[0]
        h.close()
    return used


# 38 row tiles of W^T A in 107 slabs: kept slab sums would be 266 MB.  Rows that
# are not 16-byte aligned; whole splits that fill the SMs
@pytest.mark.parametrize("n", [9701, 9728])
def test_fp32_products_without_kept_slabs(aunmf, n):
    m, k = 13600, 33
    A, W, H = (torch.rand(s, device="cuda") for s in ((m, n), (m, k), (k, n)))
    # factors and products 3 n k, Gram partials 304 k^2, split partials 4 m k, the
    # factor's copy m (k + 3): 4 bytes each, and some 2 MB pages
    need = 4 * (3 * n * k + 304 * k * k + 4 * m * k + m * (k + 3))
    assert growth(aunmf, lambda h: h.relres(A, W, H)) <= need + (40 << 20)

@pytest.mark.parametrize("k", [50, 512])
def test_sparse_products(aunmf, k):
    """The CSC (8 bytes a nonzero) and its sort (24) are all that grows with the
    nonzeros, besides the list of long rows (at worst 72 / 512 + 28 / 512): the
    long rows' partial sums, at worst 12 k / 512 bytes, share the sort's memory."""
    m, n, per = 1 << 19, 3000, 32
    nnz = m * per
    ptr = torch.arange(0, nnz + 1, per, device="cuda", dtype=torch.int64)
    idx = (torch.arange(m, device="cuda")[:, None] * 7 + torch.arange(per, device="cuda") * 93) % n
    idx = idx.sort(1).values.int().reshape(-1).contiguous()
    val = torch.rand(nnz, device="cuda")
    S = aunmf.csr_matrix(ptr, idx, val, (m, n))
    W = torch.rand((m, k), device="cuda")
    torch.empty((k, n), device="cuda")  # (wta's output then comes from torch's cache)
    used = growth(aunmf, lambda h: h.wta(S, W))
    assert used <= 32.2 * nnz + 4 * 2 * n * k + (24 << 20)
