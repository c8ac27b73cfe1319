"""||A||^2 inside the TF32 / BF16 loss (k <= 64, where the W^T A product sums it on
the way): entries of one value, whose FP32 rounding does not average out, and
entries past the range of FP32 squares.

With zero factors the loss is half of ||A||^2 + 2 <round(A) - A, A>.  Tolerance: a
chain of 16 FP32 FMAs of one value errs by a factor that is worked out here, in
64 bits (the products are exact there); the chains' own sums and the rounding term
add 16 u 2^-8 = 4e-9 at most (u = 2^-24, |round(A) - A| <= 2^-9 |A|)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ax():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf.Handle()


def loss_of(ax, A, prec):
    m, n = A.shape
    loss, _ = ax.loss_fwd(A, torch.zeros((m, 5), device="cuda"), torch.zeros((5, n), device="cuda"), prec)
    return float(loss)


def chain(c, terms):
    """Relative error of `terms` FMAs s = fl(s + c c)."""
    s, sq = np.float32(0), np.float64(c) * np.float64(c)
    for _ in range(terms):
        s = np.float32(np.float64(s) + sq)
    return abs(float(s) / (terms * sq) - 1)


def constants():
    """Values whose chain of 64 errs at least three times as much as that of 16."""
    rng = np.random.default_rng(3)
    cs = [np.float32(c) for c in rng.uniform(0.1, 2.0, 400)]
    cs = [c for c in cs if chain(c, 64) > 3 * chain(c, 16) + 1e-7]
    return sorted(cs, key=lambda c: -chain(c, 64))[:4]


@pytest.mark.parametrize("prec", ["tf32", "bf16"])
@pytest.mark.parametrize("m,n", [(4096, 1000), (4096, 1001), (1920, 259)])
def test_entries_of_one_value(ax, prec, m, n):
    cs = constants()
    assert len(cs) == 4
    for c in cs:
        A = torch.full((m, n), float(c), device="cuda")
        if prec == "bf16":
            r = float(A[0, 0].bfloat16())
        else:
            b = A[0, 0].view(torch.int32)
            r = float(((b + 0x1000) & ~0x1FFF).view(torch.float32))
        c = float(c)
        ref = 0.5 * m * n * (c * c + 2 * c * (r - c))
        assert abs(loss_of(ax, A, prec) - ref) <= (chain(c, 16) + 4e-9) * 0.5 * m * n * c * c


@pytest.mark.parametrize("prec", ["tf32", "bf16"])
@pytest.mark.parametrize("n", [500, 501])
def test_entries_past_the_range_of_their_squares(ax, prec, n):
    A = torch.rand((700, n), device="cuda")
    A[333, 77] = 2e19
    assert loss_of(ax, A, prec) == np.inf
    # squares that FP32 holds, their sum it does not
    A[:] = 2e18
    ref = 0.5 * A.numel() * 4e36
    assert loss_of(ax, A, prec) == pytest.approx(ref, rel=1e-2)  # (the rounding term: 2^-8)
    A[333, 77] = np.nan
    assert np.isnan(loss_of(ax, A, prec))
