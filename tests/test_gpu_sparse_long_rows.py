"""Sparse products whose rows (of the CSR, or of the CSC: columns of A) lie at
the edges of the chunked form: 512 nonzeros is the longest row a warp walks,
chunks hold 256 (512 above 32,768 nonzeros), a row's chunks are added by eight
warps.  Against a 64-bit product; FP32 sums of d terms are within d u (|S| |X|)
of it, the test allows 2 d u (u = 2^-24, d the longest row)."""
import pytest

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24
torch = pytest.importorskip("torch")

N = 70001
LENGTHS = [0, 1, 255, 256, 511, 512, 513, 768, 769, 1024, 2047, 2048, 2049, 4097, 32768, 32769, 33280, 70001, 0, 513]


@pytest.fixture(scope="module")
def ax():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf


@pytest.mark.parametrize("k", [1, 31, 33, 64, 100, 300])
def test_row_lengths(ax, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(k)
    m = len(LENGTHS)
    cols, ptr = [], [0]
    for d in LENGTHS:
        cols.append(torch.randperm(N, generator=g, device="cuda")[:d].sort().values)
        ptr.append(ptr[-1] + d)
    idx = torch.cat(cols).int().contiguous()
    val = torch.rand(ptr[-1], generator=g, device="cuda") - 0.25
    ptr = torch.tensor(ptr, device="cuda", dtype=torch.int64)
    D = torch.zeros((m, N), device="cuda", dtype=torch.float64)
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), ptr[1:] - ptr[:-1])
    D[rows, idx.long()] = val.double()
    h = ax.Handle()
    tol = 2 * max(LENGTHS) * U32

    def check(got, ref, mag):
        assert bool(((got.double() - ref).abs() <= tol * mag + 1e-30).all())

    H = torch.rand((k, N), generator=g, device="cuda") - 0.25
    W = torch.rand((m, k), generator=g, device="cuda") - 0.25
    S = ax.csr_matrix(ptr, idx, val, (m, N))
    P = h.aht(S, H)
    check(P, D @ H.double().T, D.abs() @ H.double().T.abs())
    check(h.wta(S, W), W.double().T @ D, W.double().T.abs() @ D.abs())
    assert torch.equal(P, h.aht(S, H))
    # the same matrix transposed: the long rows are the CSC's
    order = torch.argsort(idx.long() * m + rows)
    tptr = torch.zeros(N + 1, device="cuda", dtype=torch.int64)
    tptr[1:] = torch.cumsum(torch.bincount(idx.long(), minlength=N), 0)
    tidx, tval, Ht = rows[order].int().contiguous(), val[order].contiguous(), H.T.contiguous()
    T = ax.csr_matrix(tptr, tidx, tval, (N, m))  # (holds pointers: the tensors stay alive here)
    Q = h.wta(T, Ht)
    check(Q.T, D @ H.double().T, D.abs() @ H.double().T.abs())
    torch.cuda.synchronize()
    assert torch.equal(Q, h.wta(T, Ht))
    # the CSR's and the CSC's sums are the same sums in the same order
    assert torch.equal(Q.T, P)
    h.close()
