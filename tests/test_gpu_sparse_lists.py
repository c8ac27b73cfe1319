"""The list of a sparse matrix's long rows (more than 512 nonzeros), in segments of
the rows, and the product that works it off beside the short ones: hundreds of long
rows in many segments, rows of one segment only, none at all.

Values are small whole numbers, so every sum is exact in FP32: a chunk that is
lost, added twice or out of place shows.  A matrix without long rows costs no
launch more than one too small to have any."""
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


def matrix(ax, lens, n, seed):
    """CSR with row lengths `lens` (each row's columns equally spaced from a random
    start), its parts and its dense product in 64 bits."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    lens = torch.as_tensor(lens, device="cuda", dtype=torch.int64)
    m = lens.numel()
    ptr = torch.zeros(m + 1, device="cuda", dtype=torch.int64)
    ptr[1:] = torch.cumsum(lens, 0)
    row = torch.repeat_interleave(torch.arange(m, device="cuda"), lens)
    pos = torch.arange(int(ptr[-1]), device="cuda") - ptr[row]
    step = n // lens.clamp(min=1)
    start = torch.randint(0, n, (m,), generator=g, device="cuda") % step.clamp(min=1)
    idx = start[row] + pos * step[row]
    val = torch.randint(-3, 4, idx.shape, generator=g, device="cuda").float()
    order = torch.argsort(idx * m + row)
    tptr = torch.zeros(n + 1, device="cuda", dtype=torch.int64)
    tptr[1:] = torch.cumsum(torch.bincount(idx, minlength=n), 0)
    tidx, tval = row[order].int().contiguous(), val[order].contiguous()
    T = ax.csr_matrix(tptr, tidx, tval, (n, m))
    D = torch.sparse_coo_tensor(torch.stack([row, idx]), val.double(), (m, n)).coalesce()
    idx32 = idx.int().contiguous()
    S = ax.csr_matrix(ptr, idx32, val, (m, n))
    return S, T, D, (ptr, val, idx32, tptr, tidx, tval)


def ints(shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(-3, 4, shape, generator=g, device="cuda").float()


def lengths(kind):
    rng = np.random.default_rng(5)
    if kind == "many":  # 300,000 rows: 256 segments of 1172 rows
        lens = rng.integers(0, 20, 300000)
        at = rng.choice(300000, 700, replace=False)
        lens[at] = rng.choice([512, 513, 600, 768, 769, 1025, 5000, 33000, 40000], 700)
        lens[[0, 1171, 1172, 299999]] = [513, 514, 515, 2000]
    elif kind == "one segment":
        lens = rng.integers(0, 5, 140000)
        lens[70000:70400] = 700
    elif kind == "all long":
        lens = np.full(900, 1030)
    else:
        lens = np.full(5000, 9)
    return lens


@pytest.mark.parametrize("k", [10, 50, 130])
@pytest.mark.parametrize("kind", ["many", "one segment", "all long", "none"])
def test_products_are_exact(ax, kind, k):
    n = 60000
    lens = lengths(kind)
    S, T, D, keep = matrix(ax, lens, n, 1)
    m = len(lens)
    H, W = ints((k, n), 2), ints((m, k), 3)
    P = (D @ H.double().T).float()
    Q = (D.t() @ W.double()).float().T.contiguous()
    h = ax.Handle()
    Ht, Wt = H.T.contiguous(), W.T.contiguous()
    for _ in range(3):
        assert torch.equal(h.aht(S, H), P) and torch.equal(h.wta(S, W), Q)
        # the transpose: the long rows are the other form's
        assert torch.equal(h.wta(T, Ht), P.T) and torch.equal(h.aht(T, Wt), Q.T)
    torch.cuda.synchronize()
    h.close()


def test_repeated_iterations_reuse_the_list(ax):
    """A run's products use one list over and over (eager and as a graph)."""
    lens = lengths("one segment")
    S, T, D, keep = matrix(ax, lens, 3000, 4)
    keep[1].abs_()
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    W0 = torch.rand((len(lens), 8), generator=g, device="cuda")
    H0 = torch.rand((8, 3000), generator=g, device="cuda")
    h = ax.Handle()
    W, H, rel, _ = h.run(S, 8, "mu", 6, W0, H0)
    W1, H1, rel1, _ = h.run(S, 8, "mu", 6, W0, H0, use_graph=False)
    assert torch.equal(W, W1) and torch.equal(H, H1) and (rel == rel1).all()
    a, b = W0, H0
    for _ in range(6):
        a, b, _, _ = h.run(S, 8, "mu", 1, a, b)
    assert torch.equal(W, a) and torch.equal(H, b)
    h.close()


def test_no_launch_for_long_rows_that_do_not_exist(ax):
    h = ax.Handle()

    def per_iteration(m):
        S, T, D, keep = matrix(ax, np.full(m, 5), 400, 7)
        W0, H0 = ints((m, 4), 8).abs() + 1, ints((4, 400), 9).abs() + 1
        n = [h.run(S, 4, "mu", it, W0, H0, use_graph=False)[3]["launches"] for it in (1, 3)]
        torch.cuda.synchronize()
        return (n[1] - n[0]) / 2

    assert per_iteration(600) == per_iteration(100)
    h.close()
