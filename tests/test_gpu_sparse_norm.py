"""||A||^2 of a CSR matrix over the whole range of its entries: squares that FP32
cannot hold, sums of many equal entries, an infinite or NaN entry.

Tolerance of the scaled cases: the residual of a factor pair far from a fit is 1
to the products' FP32 rounding, the norm itself is an FP64 sum of exact squares
(nnz 2^-53)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ax():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf


def csr(ax, vals, m=300, n=200, per=7):
    """m rows of `per` nonzeros, values cycled from vals; the tensors stay alive
    with the returned tuple."""
    ptr = torch.arange(0, m * per + 1, per, device="cuda", dtype=torch.int64)
    idx = ((torch.arange(m, device="cuda")[:, None] * 3 + torch.arange(per, device="cuda") * 11) % n).sort(1).values
    idx = idx.int().reshape(-1).contiguous()
    v = torch.tensor(vals, device="cuda", dtype=torch.float32).repeat(m * per // len(vals) + 1)[:m * per].contiguous()
    return ax.csr_matrix(ptr, idx, v, (m, n)), v, (ptr, idx)


@pytest.mark.parametrize("val", [1e20, 3e19, 1.0, 1e-19, 1e-20, 1e-22, 1e-23, 1e-30])
def test_loss_of_zero_factors_is_the_norm(ax, val):
    S, v, keep = csr(ax, [val, 0.5 * val, 0.3 * val])
    h = ax.Handle()
    Z, Y = torch.zeros((300, 3), device="cuda"), torch.zeros((3, 200), device="cuda")
    loss, _ = h.loss_fwd(S, Z, Y)
    ref = 0.5 * float((v.double() ** 2).sum())
    assert float(loss) == pytest.approx(ref, rel=2100 * 2.0 ** -52, abs=0)
    assert h.relres(S, Z, Y) == pytest.approx(1.0, rel=1e-12)
    h.close()


def test_many_equal_entries(ax):
    """4.9e6 entries of one value: no rounding of one sign accumulates."""
    S, v, keep = csr(ax, [0.1], m=700000, n=5000)
    h = ax.Handle()
    Z, Y = torch.zeros((700000, 2), device="cuda"), torch.zeros((2, 5000), device="cuda")
    loss, _ = h.loss_fwd(S, Z, Y)
    assert float(loss) == pytest.approx(0.5 * float((v.double() ** 2).sum()), rel=1e-12)
    h.close()


@pytest.mark.parametrize("algo", ["mu", "hals"])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_nonfinite_entry_is_an_error(ax, algo, bad):
    S, v, keep = csr(ax, [1.0])
    v[777] = bad
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    W0, H0 = (torch.rand(s, generator=g, device="cuda") for s in ((300, 5), (5, 200)))
    h = ax.Handle()
    with pytest.raises(ax.AunmfError) as e:
        h.run(S, 5, algo, 2, W0, H0, prec="fp32")
    assert e.value.code == ax.E_NUMERIC
    assert not np.isfinite(h.relres(S, W0, H0))
    h.close()


def test_nonfinite_dense_entry_is_an_error(ax):
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    A, W0, H0 = (torch.rand(s, generator=g, device="cuda") for s in ((300, 200), (300, 5), (5, 200)))
    h = ax.Handle()
    for bad in (np.inf, np.nan):
        B = A.clone()
        B[17, 9] = bad
        with pytest.raises(ax.AunmfError) as e:
            h.run(B, 5, "mu", 2, W0, H0, prec="fp32")
        assert e.value.code == ax.E_NUMERIC
    h.close()
