"""Block principal pivoting at the ranks where a lane's part changes: one or two
entries a lane (k = 32, 33), a full last lane, factorisations of up to k / 2
rows (k = 1 .. 3, 63, 64).

Checked by the optimality conditions of each solution x >= 0 with y = G x - r:
x is rounded to FP32 on output (2^-24 of each entry), so y is off by at most 2^-23
|G| x of its true value, which is 0 where x > 0 and >= 0 elsewhere."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ax():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf.Handle()


@pytest.mark.parametrize("k", [1, 2, 3, 16, 31, 32, 33, 48, 63, 64])
def test_optimality(ax, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(k)
    C = torch.rand((8 * k + 8, k), generator=g, device="cuda").double()
    G = (C.T @ C).float()
    G = torch.maximum(G, G.T)
    X = torch.randn((700, k), generator=g, device="cuda").clamp_(min=0)
    E = torch.randn((700, k), generator=g, device="cuda")
    R = (X.double() @ G.double() + 2.0 * E.double()).float()
    Z, _, unsolved = ax.nls_bpp(G, R)
    assert unsolved == 0
    x, Gd, r = Z.double(), G.double(), R.double()
    y = x @ Gd - r
    tol = 2.0 ** -23 * (x.abs() @ Gd.abs() + r.abs())
    assert bool((Z >= 0).all())
    assert bool((y >= -tol).all())
    assert bool((y.abs()[Z > 0] <= tol[Z > 0]).all())
