"""The tensor-core products that read the FP32 A themselves (k <= 64): ragged
tiles, contractions that end inside an operand stage or a raw tile, every MMA
width class, rows that are not 16-byte aligned, K splits.

The reference rounds A as the kernel does (TF32 to nearest, ties away; BF16 to
nearest even) and multiplies in 64 bits, so what is left is the FP32 summation
(2 K u of |A| |F|, u = 2^-24) and the factor's two-term split, which carries it
to 2^-22 (TF32) or 2^-16 (BF16): a wrongly rounded A (2^-12, 2^-9) shows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24
SPLIT = {"tf32": 2.0 ** -22, "bf16": 2.0 ** -16}
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ax():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf.Handle()


def rounded(A, prec):
    if prec == "bf16":
        return A.bfloat16().double()
    b = A.view(torch.int32)
    return ((b + 0x1000) & ~0x1FFF).view(torch.float32).double()


def check(got, A, B, Ar, K, prec):
    ref, mag = Ar @ B.double(), A.double().abs() @ B.double().abs()
    tol = (2 * K * U32 + SPLIT[prec]) * mag + 1e-30
    assert bool(((got.double() - ref).abs() <= tol).all())


SHAPES = [(1, 1, 1), (255, 31, 8), (256, 32, 9), (257, 33, 48), (300, 63, 56), (513, 64, 57),
          (130, 65, 64), (700, 96, 10), (1200, 1000, 50), (39000, 260, 20), (260, 39001, 33),
          (5000, 4999, 64)]


@pytest.mark.parametrize("prec", ["tf32", "bf16"])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_products(ax, m, n, k, prec):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n + k)
    r = lambda *s: torch.rand(s, generator=g, device="cuda") - 0.25  # noqa: E731
    A, H, W = r(m, n), r(k, n), r(m, k)
    Ar = rounded(A, prec)
    check(ax.aht(A, H, prec), A, H.T, Ar, n, prec)
    check(ax.wta(A, W, prec).T, A.T, W, Ar.T, m, prec)
    At = A.T.contiguous()
    check(ax.aht(At, W.T.contiguous(), prec), At, W, Ar.T, m, prec)
    check(ax.wta(At, H.T.contiguous(), prec).T, A, H.T, Ar, n, prec)


@pytest.mark.parametrize("n", [1600, 1601])
def test_repeated_products_are_equal(ax, n):
    """Many units per CTA, tiles that hit L2: the ring slots are refilled while
    the warps are far apart, and every call gives the same bits."""
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    A = torch.rand((40000, n), generator=g, device="cuda")
    H, W = torch.rand((50, n), generator=g, device="cuda"), torch.rand((40000, 50), generator=g, device="cuda")
    for prec in ("tf32", "bf16"):
        P, Q = ax.aht(A, H, prec), ax.wta(A, W, prec)
        check(P, A, H.T, rounded(A, prec), n, prec)
        for _ in range(10):
            assert torch.equal(P, ax.aht(A, H, prec)) and torch.equal(Q, ax.wta(A, W, prec))


def test_unaligned_base(ax):
    """A starts 4 bytes past a 16-byte boundary, rows of 16-byte multiples."""
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    m, n, k = 515, 260, 24
    A = torch.rand(m * n + 1, generator=g, device="cuda")[1:].view(m, n)
    H, W = torch.rand((k, n), generator=g, device="cuda"), torch.rand((m, k), generator=g, device="cuda")
    for prec in ("tf32", "bf16"):
        Ar = rounded(A.clone(), prec)
        check(ax.aht(A, H, prec), A, H.T, Ar, n, prec)
        check(ax.wta(A, W, prec).T, A.T, W, Ar.T, m, prec)


@pytest.mark.parametrize("m,n,k,last", [(700, 512, 20, 12), (611, 503, 64, 3)])
def test_run_equals_the_form_with_copies(ax, m, n, k, last):
    """A run of up to 12 TF32 iterations (3 when A's rows are not 16-byte aligned)
    reads A directly, a longer one keeps rounded copies: the same factors and
    residuals to the bit."""
    from paper_1609_09154_gb300 import synth

    A, _, _ = synth.dense_lowrank_torch(m, n, k, 3, "cuda")
    W0, H0 = synth.init_factors_torch(m, n, k, 3, "cuda")
    W, H, rel, _ = ax.run(A, k, "hals", last, W0, H0, prec="tf32")
    W1, H1, rel1, _ = ax.run(A, k, "hals", last + 1, W0, H0, prec="tf32")
    np.testing.assert_array_equal(rel, rel1[:last])
    W2, H2, rel2, _ = ax.run(A, k, "hals", 1, W, H, prec="tf32")
    assert torch.equal(W2, W1) and torch.equal(H2, H1) and rel2[0] == rel1[last]
    # BF16: one iteration reads A directly, more keep copies
    _, _, r1, _ = ax.run(A, k, "mu", 1, W0, H0, prec="bf16")
    _, _, r2, _ = ax.run(A, k, "mu", 2, W0, H0, prec="bf16")
    assert r1[0] == r2[0]
