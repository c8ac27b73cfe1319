"""Products whose every sum is exact in FP32, at contractions so long that a rounding
bound (which grows with them) would hide a lost or repeated slab, operand stage or
chunk: whole numbers, compared bit for bit.  And rounding of A to TF32 and BF16:
entries in [1, 2) that rounding to nearest and dropping bits take apart, ties among
them, whose rounded sums are exact (multiples of 2^-10 or 2^-7 below 2^13)."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ax():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf.Handle()


def rnd(g, lo, hi, *shape):
    return torch.randint(lo, hi, shape, generator=g, device="cuda").float()


# (rows, contraction, columns): one tile over many SMs, a last slab and a last step
# that are not full, several column tiles, one K past a stage; rows of other alignments
@pytest.mark.parametrize("M,K,k", [(40, 60004, 64), (257, 200000, 20), (512, 131072, 100), (38913, 144, 40),
                                   (20000, 1028, 100), (90, 17408, 10), (131, 17409, 16), (260, 39001, 33),
                                   (5000, 4999, 64), (1, 300001, 3)])
def test_long_contractions(ax, M, K, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K + k)
    A, H = rnd(g, -4, 5, M, K), rnd(g, -4, 5, k, K)
    P = (A.double() @ H.double().T).float()
    At, Ht = A.T.contiguous(), H.T.contiguous()
    for prec in ("fp32", "tf32", "bf16"):
        assert torch.equal(ax.aht(A, H, prec), P)
        assert torch.equal(ax.wta(At, Ht, prec), P.T)


@pytest.mark.parametrize("prec,bits", [("tf32", 10), ("bf16", 7)])
@pytest.mark.parametrize("m,n,k", [(700, 4999, 50), (4999, 300, 64), (513, 2048, 7), (300, 1000, 90)])
def test_a_is_rounded_to_nearest(ax, prec, bits, m, n, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n)
    # 1 + j / 2^(bits + 3): below, at and above the middle between two neighbours
    A = 1.0 + rnd(g, 0, 2 ** (bits + 3), m, n) / 2.0 ** (bits + 3)
    if prec == "bf16":
        Ar = A.bfloat16().float()
    else:
        Ar = ((A.view(torch.int32) + 0x1000) & ~0x1FFF).view(torch.float32)
    assert not torch.equal(A, Ar)
    H, W = rnd(g, -1, 2, k, n), rnd(g, -1, 2, m, k)
    assert torch.equal(ax.aht(A, H, prec), (Ar.double() @ H.double().T).float())
    assert torch.equal(ax.wta(A, W, prec), (W.double().T @ Ar.double()).float())
