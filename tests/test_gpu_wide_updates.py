"""The updates and gradient rows of ranks above 64 on blocked products: row
counts at the tile edges (64, 128, 256 rows), ranks at the ends of a block of
16 coordinates and of a 128-entry chain step, ranks and rows that are not whole
16-byte groups (HALS then takes the warp-per-row form).

Against 64-bit references.  MU and gradient rows: one k-term FP32 sum (k u of
its terms' magnitudes, 2 k u allowed) and a few roundings.  HALS: the bar of the
parity tests, (1e-4 of the entry + 1e-5 of the largest) x k / 64."""
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


def problem(rows, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(rows * 1000 + k)
    X = torch.rand((rows, k), generator=g, device="cuda")
    F = torch.rand((3 * k, k), generator=g, device="cuda")
    G = (F.double().T @ F.double()).float()
    G = torch.maximum(G, G.T)
    Y = torch.rand((rows, k), generator=g, device="cuda")
    P = (Y.double() @ G.double()).float()
    return X, P, G


CASES = [(1, 65), (63, 66), (64, 80), (65, 96), (127, 100), (129, 108), (255, 109), (257, 112), (64, 128),
         (200, 129), (130, 132), (90, 144), (300, 255), (70, 256), (65, 260), (128, 384), (66, 388), (129, 512),
         (12000, 112), (20000, 68)]


@pytest.mark.parametrize("rows,k", CASES)
def test_updates(ax, rows, k):
    X, P, G = problem(rows, k)
    Xd, Pd, Gd = X.double(), P.double(), G.double()
    W = X.clone()
    ax.update_w("mu", W, P, G)
    ref = Xd * Pd / (Xd @ Gd + 1e-16)
    assert bool(((W.double() - ref).abs() <= (2 * k + 8) * U32 * ref + 1e-30).all())
    W = X.clone()
    W[:, 3] = 0.0
    Z = W.double()
    G0, G0d = G.clone(), Gd.clone()
    G0[5, 5] = G0d[5, 5] = 0.0  # a coordinate without a diagonal stays as it is
    # (update_w normalises the columns afterwards: the H side does not)
    H = W.T.contiguous()
    ax.update_h("hals", H, P.T.contiguous(), G0)
    for i in range(k):
        if float(G0d[i, i]) > 0:
            Z[:, i] = (Z[:, i] + (Pd[:, i] - Z @ G0d[:, i]) / G0d[i, i]).clamp(min=0)
    tol = max(1.0, k / 64.0) * (1e-4 * Z.abs() + 1e-5 * Z.abs().max())
    assert bool(((H.T.double() - Z).abs() <= tol).all())
    assert torch.equal(H[5], W[:, 5])


@pytest.mark.parametrize("m,n,k", [(65, 130, 66), (300, 257, 100), (129, 90, 260), (200, 140, 512)])
def test_gradient_rows(ax, m, n, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(k)
    A, W, H = (torch.rand(s, generator=g, device="cuda") for s in ((m, n), (m, k), (k, n)))
    dW, dH = ax.loss_bwd(A, W, H)
    Ad, Wd, Hd = A.double(), W.double(), H.double()
    GH, GW = Hd @ Hd.T, Wd.T @ Wd
    # the Gram (n or m terms), its product (k terms) and the product with A
    tw = (2 * (n + k) + 8) * U32 * (Wd @ GH + Ad @ Hd.T)
    th = (2 * (m + k) + 8) * U32 * (GW @ Hd + Wd.T @ Ad)
    assert bool(((dW.double() - (Wd @ GH - Ad @ Hd.T)).abs() <= tw).all())
    assert bool(((dH.double() - (GW @ Hd - Wd.T @ Ad)).abs() <= th).all())
