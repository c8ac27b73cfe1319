"""Right-hand sides that reach the exchange cap on an ill-conditioned Gram: they go
on in FP64 from the set they had reached, alone and in a batch, with warm and with
cold starts; a cap below 10 k ends them.

The problems are uniform low-rank ones at full rank of the fit, whose Gram matrices
reach cond 1e9 in the second iteration; rows of each were seen to reach the cap
(as many as below, in TF32), which ones depends on the sums' last bits.  A row's
solution is unique, so single and batched runs agree to the bar of
test_gpu_batched.py (1e-5 of the relative residual)."""
import pytest

from paper_1609_09154_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
PROBLEMS = [(588, 3909, 64, 960778), (2858, 3131, 48, 661596), (2717, 4099, 64, 564196), (2129, 5120, 32, 180537)]


@pytest.fixture(scope="module")
def ax():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf.Handle()


def problem(m, n, k, seed):
    A, _, _ = synth.dense_lowrank_torch(m, n, k, seed=seed, device="cuda")
    _, H0 = synth.init_factors_torch(m, n, k, seed=seed, device="cuda")
    return A, H0


@pytest.mark.parametrize("cold", [False, True])
def test_batched_and_single_agree(ax, cold):
    ps = [problem(*p) for p in PROBLEMS]
    ks = [p[2] for p in PROBLEMS]
    # (an unconverged right-hand side would raise)
    _, _, rel, info = ax.run_batched([A for A, _ in ps], ks, 4, [H0 for _, H0 in ps], bpp_cold_start=cold)
    assert info["bpp_nonconverged"] == 0 and info["bpp_numeric"] == 0
    for i, (A, H0) in enumerate(ps):
        Z = torch.zeros((A.shape[0], ks[i]), device="cuda")
        _, _, r, one = ax.run(A, ks[i], "abpp", 4, Z, H0, prec="tf32", bpp_cold_start=cold)
        assert one["bpp_nonconverged"] == 0
        assert abs(r[-1] - rel[i, -1]) <= 1e-5 * r[-1]


@pytest.mark.parametrize("cold", [False, True])
def test_cap_and_count(ax, cold):
    """With the cap one below 10 k the rows end at it; at 10 k they go on, and
    the exchanges of both solvers are counted."""
    m, n, k, seed = 2522, 5235, 32, 5577
    A, H0 = problem(m, n, k, seed)
    Z = torch.zeros((m, k), device="cuda")
    kw = dict(prec="tf32", bpp_cold_start=cold)
    _, _, _, low = ax.run(A, k, "abpp", 2, Z, H0, bpp_max_pivots=10 * k - 1, allow_noconverge=True, **kw)
    _, _, _, full = ax.run(A, k, "abpp", 2, Z, H0, **kw)
    assert low["bpp_nonconverged"] > 0 and full["bpp_nonconverged"] == 0
    assert full["bpp_pivots"] > low["bpp_pivots"] and full["bpp_redone"] > low["bpp_redone"]
