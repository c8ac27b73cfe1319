"""Performance cases: the calls a program makes into this library, over the sizes it makes them at.

Each case goes through the Python binding (`aunmf.Handle`, `autograd.nmf_loss`) with device tensors, as a user's
program does.  The families (`kind`) are

  steps    one iteration of a custom driver, written with the step calls, and its residual
  run      a whole dense factorisation (`Handle.run`)
  product  one product with A (`Handle.aht`, `Handle.wta`)
  loss     the differentiable objective, forward and backward
  sparse   a whole factorisation of a CSR matrix
  spmm     both products with a CSR matrix that has power-law hubs
  nls      nonnegative least squares for many right-hand sides (`Handle.nls_bpp`)
  batched  many uneven problems at once (`Handle.run_batched`)

Inputs are the synthetic recipes of `synth` (planted low rank plus noise, uniform or power-law sparse).  A program
holds one handle and gives it one input after another; so do these cases.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_1609_09154_gb300 import aunmf, autograd, synth

DEV = "cuda"
F64 = torch.float64
_handles = []


def _handle():
    """The program's one handle, on torch's current stream."""
    if not _handles:
        _handles.append(aunmf.Handle())
    return _handles[0]


def listed():
    return [
        # The smallest work: a user's own loop over the step calls on the 2,000 x 1,500 validation size.
        {"name": "steps_2000x1500_k10_hals", "kind": "steps", "m": 2000, "n": 1500, "k": 10, "algo": "hals"},
        # A whole small factorisation with the paper's flagship update.
        {"name": "run_2000x1500_k10_abpp", "kind": "run", "m": 2000, "n": 1500, "k": 10, "algo": "abpp",
         "prec": "fp32", "iters": 10},
        # The same size with multiplicative updates: what most callers of an NMF routine run first.
        {"name": "run_2000x1500_k10_mu", "kind": "run", "m": 2000, "n": 1500, "k": 10, "algo": "mu",
         "prec": "fp32", "iters": 30},
        # A quarter of the benchmark's sides at its rank, tensor-core products.
        {"name": "run_24000x16000_k50_hals_tf32", "kind": "run", "m": 24000, "n": 16000, "k": 50, "algo": "hals",
         "prec": "tf32", "iters": 10},
        # A wide rank of the k sweep (topic models): wide products, Grams and sweeps, ragged sides.
        {"name": "run_12001x7999_k256_hals_bf16", "kind": "run", "m": 12001, "n": 7999, "k": 256, "algo": "hals",
         "prec": "bf16", "iters": 4},
        # One product at the benchmark's full size: a driver that brings its own updates.
        {"name": "aht_96000x64000_k50_tf32", "kind": "product", "op": "aht", "m": 96000, "n": 64000, "k": 50,
         "prec": "tf32"},
        # The other product in reference precision.
        {"name": "wta_32000x24000_k50_fp32", "kind": "product", "op": "wta", "m": 32000, "n": 24000, "k": 50,
         "prec": "fp32"},
        # Gradient-based training of the factors: the loss workload, and a ragged one in mixed precision.
        {"name": "loss_20000x10000_k100_fp32", "kind": "loss", "m": 20000, "n": 10000, "k": 100, "prec": "fp32"},
        {"name": "loss_9999x12001_k32_tf32", "kind": "loss", "m": 9999, "n": 12001, "k": 32, "prec": "tf32"},
        # The sparse workload: 5e7 nonzeros at uniform positions.
        {"name": "sparse_1000000x500000_k50_mu", "kind": "sparse", "m": 1000000, "n": 500000, "k": 50,
         "nnz": 50000000, "algo": "mu", "iters": 5},
        # A driver's two products with a web-graph-like matrix (hub rows and columns).
        {"name": "spmm_300001x200003_k32", "kind": "spmm", "m": 300001, "n": 200003, "k": 32, "nnz": 20000000},
        # The local solver on its own: one factor's rows against a fixed Gram matrix.
        {"name": "nls_64000_k50", "kind": "nls", "rows": 64000, "k": 50},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["steps", "run", "run", "product", "product", "loss", "sparse", "spmm", "nls", "batched"])
    c = {"kind": kind}
    if kind == "steps":
        c.update(m=_log(rng, 300, 8000), n=_log(rng, 300, 8000), k=rng.randint(4, 64), algo=rng.choice(["mu", "hals"]))
    elif kind == "run":
        algo = rng.choice(["mu", "hals", "abpp"])
        if algo == "abpp":
            c.update(m=_log(rng, 500, 8000), n=_log(rng, 500, 8000), k=rng.randint(4, 16), prec="fp32")
        else:
            c.update(m=_log(rng, 500, 24000), n=_log(rng, 500, 16000), k=_log(rng, 4, 300),
                     prec=rng.choice(["fp32", "tf32", "bf16"]))
        c.update(algo=algo, iters=rng.randint(3, 8))
    elif kind == "product":
        c.update(op=rng.choice(["aht", "wta"]), m=_log(rng, 1000, 64000), n=_log(rng, 1000, 32000),
                 k=_log(rng, 4, 512), prec=rng.choice(["fp32", "tf32", "bf16"]))
    elif kind == "loss":
        c.update(m=_log(rng, 1000, 20000), n=_log(rng, 1000, 16000), k=_log(rng, 4, 200),
                 prec=rng.choice(["fp32", "tf32", "bf16"]))
    elif kind == "sparse":
        # (HALS on structureless sparse input subtracts nearly equal sums: two FP32 runs of it are not comparable)
        c.update(m=_log(rng, 20000, 1000000), n=_log(rng, 20000, 500000), k=rng.randint(8, 64),
                 nnz=_log(rng, 500000, 40000000), algo="mu", iters=rng.randint(2, 5))
    elif kind == "spmm":
        c.update(m=_log(rng, 20000, 600000), n=_log(rng, 20000, 400000), k=_log(rng, 8, 128),
                 nnz=_log(rng, 500000, 20000000))
    elif kind == "nls":
        c.update(rows=_log(rng, 1000, 96000), k=rng.randint(6, 64))
    else:
        # many uneven problems, ABPP with tensor-core products
        c.update(count=rng.randint(8, 24), lo=500, hi=_log(rng, 1000, 4000), kmax=rng.choice([16, 32, 64]),
                 prec=rng.choice(["tf32", "bf16"]), iters=2)
    return c


# ---------------------------------------------------------------- inputs
def _dense(c, seed):
    A, _, _ = synth.dense_lowrank_torch(c["m"], c["n"], c["k"], seed, DEV)
    W, H = synth.init_factors_torch(c["m"], c["n"], c["k"], seed, DEV)
    return A, W, H


def _batch_dims(c):
    """The problems' sizes: part of the case, the same for every seed."""
    g = np.random.default_rng(c["count"] * 100003 + c["hi"])
    ks = [k for k in (8, 16, 32, 64) if k <= c["kmax"]]
    return [(int(g.integers(c["lo"], c["hi"] + 1)), int(g.integers(c["lo"], c["hi"] + 1)), int(g.choice(ks)))
            for _ in range(c["count"])]


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c, "h": _handle()}
    if kind in ("steps", "run"):
        s["A"], s["W"], s["H"] = _dense(c, seed)
    elif kind == "product":
        s["A"], W, H = _dense(c, seed)
        s["F"] = H if c["op"] == "aht" else W
    elif kind == "loss":
        s["A"], W, H = _dense(c, seed)
        # a small start, as gradient descent takes
        s["W"] = (0.1 * W).requires_grad_(True)
        s["H"] = (0.1 * H).requires_grad_(True)
    elif kind in ("sparse", "spmm"):
        if kind == "sparse":
            s["csr"] = synth.sparse_uniform_torch(c["m"], c["n"], c["nnz"] / (c["m"] * c["n"]), seed, DEV)
        else:
            s["csr"] = synth.sparse_powerlaw_torch(c["m"], c["n"], c["nnz"], seed, DEV)
        s["A"] = aunmf.csr_matrix(*s["csr"], (c["m"], c["n"]))
        s["W"], s["H"] = synth.init_factors_torch(c["m"], c["n"], c["k"], seed, DEV)
    elif kind == "nls":
        # the middle of an ABPP run: a factor's Gram matrix, and right-hand sides whose solutions have about half
        # of their entries at zero
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed))
        C = torch.rand((4096, c["k"]), generator=g, device=DEV)
        G = (C.to(F64).T @ C.to(F64)).to(torch.float32).contiguous()
        X = torch.randn((c["rows"], c["k"]), generator=g, device=DEV).clamp_(min=0)
        E = torch.randn((c["rows"], c["k"]), generator=g, device=DEV)
        s["G"] = G
        s["R"] = (X.to(F64) @ G.to(F64) + 20.0 * E.to(F64)).to(torch.float32).contiguous()
    else:
        s["As"], s["H0"], s["ks"] = [], [], []
        for i, (m, n, k) in enumerate(_batch_dims(c)):
            A, _, _ = synth.dense_lowrank_torch(m, n, k, seed + 31 * i, DEV)
            s["As"].append(A)
            s["H0"].append(synth.init_factors_torch(m, n, k, seed + 31 * i, DEV)[1])
            s["ks"].append(k)
    return s


# ---------------------------------------------------------------- one pass
def _curve(rel):
    """The residual curve in the digits it carries: the library forms it from FP32 products."""
    return rel.astype(np.float32)


def run(state):
    s, c = state, state["case"]
    h, kind = s["h"], c["kind"]
    if kind == "steps":
        A, W, H = s["A"], s["W"], s["H"]
        GH = h.gram_h(H)
        PW = h.aht(A, H)
        h.update_w(c["algo"], W, PW, GH, H)
        GW = h.gram_w(W)
        PH = h.wta(A, W)
        h.update_h(c["algo"], H, PH, GW)
        return {"GH": GH, "PW": PW, "GW": GW, "PH": PH, "W": W, "H": H, "relres": h.relres(A, W, H)}
    if kind in ("run", "sparse"):
        W, H, rel, _ = h.run(s["A"], c["k"], c["algo"], c["iters"], s["W"], s["H"], prec=c.get("prec", "fp32"),
                             allow_noconverge=c["algo"] == "abpp")
        return {"W": W, "H": H, "relres": _curve(rel)}
    if kind == "product":
        return h.aht(s["A"], s["F"], c["prec"]) if c["op"] == "aht" else h.wta(s["A"], s["F"], c["prec"])
    if kind == "loss":
        s["W"].grad = s["H"].grad = None
        loss = autograd.nmf_loss(s["A"], s["W"], s["H"], c["prec"])
        loss.backward()
        return {"loss": loss.detach(), "dW": s["W"].grad, "dH": s["H"].grad}
    if kind == "spmm":
        return {"PW": h.aht(s["A"], s["H"]), "PH": h.wta(s["A"], s["W"])}
    if kind == "nls":
        X, _, unsolved = h.nls_bpp(s["G"], s["R"])
        return {"X": X, "unsolved": unsolved}
    Ws, Hs, rel, _ = h.run_batched(s["As"], s["ks"], c["iters"], s["H0"], prec=c["prec"], allow_noconverge=True)
    return {"W": Ws, "H": Hs, "relres": _curve(rel)}


# ---------------------------------------------------------------- floors
def work(case):
    """Bytes: inputs once and outputs once for each pass of A that the method cannot do without (every product of an
    iteration needs the result of the one before).  Flops: the products, the Gram matrices and the k x k part of the
    updates; block principal pivoting's solves depend on the data and count as one such part."""
    c, kind = case, case["kind"]
    if kind == "batched":
        b = f = 0.0
        for m, n, k in _batch_dims(c):
            b += c["iters"] * 2 * 4.0 * m * n + 4.0 * k * (m + 2 * n)
            f += c["iters"] * (4.0 * m * n * k + 3.0 * (m + n) * k * k)
        return {"bytes": b, "flops": f}
    k = c["k"]
    if kind == "nls":
        return {"bytes": 8.0 * c["rows"] * k + 4.0 * k * k, "flops": 2.0 * c["rows"] * k * k}
    m, n = c["m"], c["n"]
    factors = 4.0 * k * (m + n)
    part = 3.0 * (m + n) * k * k  # Grams (half of k x k each) and updates
    if kind == "steps":
        return {"bytes": 2 * 4.0 * m * n + 4 * factors, "flops": 6.0 * m * n * k + part}
    if kind == "run":
        it = c["iters"]
        ea = 2.0 if c["prec"] == "bf16" else 4.0  # a program's A is FP32; a kept BF16 copy is the least each pass reads
        return {"bytes": max(4.0 * m * n, it * 2 * ea * m * n) + 2 * factors, "flops": it * (4.0 * m * n * k + part)}
    if kind == "product":
        return {"bytes": 4.0 * m * n + factors, "flops": 2.0 * m * n * k}
    if kind == "loss":
        return {"bytes": 2 * 4.0 * m * n + 2 * factors, "flops": 4.0 * m * n * k + 3.0 * (m + n) * k * k}
    nnz = c["nnz"]
    if kind == "spmm":
        return {"bytes": 2 * 8.0 * nnz + 16.0 * m + 2 * factors, "flops": 4.0 * nnz * k}
    it = c["iters"]
    return {"bytes": it * (2 * 8.0 * nnz + 8.0 * (m + n) + 2 * factors), "flops": it * (4.0 * nnz * k + part)}


# ---------------------------------------------------------------- 64-bit values
class _Mat:
    """A in 64 bits, dense (row block by row block) or sparse, for exact()."""

    def __init__(self, s):
        c = s["case"]
        self.shape = (c["m"], c["n"])
        if "csr" in s:
            ptr, idx, val = s["csr"]
            self.val = val.to(F64)
            self.S = torch.sparse_csr_tensor(ptr, idx.to(torch.int64), self.val, self.shape)
            rows = torch.repeat_interleave(torch.arange(c["m"], device=DEV), ptr[1:] - ptr[:-1])
            self.St = torch.sparse_coo_tensor(torch.stack([idx.to(torch.int64), rows]), self.val,
                                              (c["n"], c["m"])).coalesce().to_sparse_csr()
            self.n2 = float((self.val ** 2).sum())
        else:
            self.A, self.S = s["A"], None
            self.n2 = sum(float((b.to(F64) ** 2).sum()) for _, b in self.blocks())

    def blocks(self):
        step = max(1, 100_000_000 // self.shape[1])
        for r in range(0, self.shape[0], step):
            yield slice(r, r + step), self.A[r:r + step]

    def times(self, Ht):
        """A Ht (m x k)"""
        if self.S is not None:
            return self.S @ Ht
        return torch.cat([b.to(F64) @ Ht for _, b in self.blocks()])

    def t_times(self, W):
        """A^T W (n x k)"""
        if self.S is not None:
            return self.St @ W
        out = torch.zeros((self.shape[1], W.shape[1]), dtype=F64, device=DEV)
        for r, b in self.blocks():
            out += b.to(F64).T @ W[r]
        return out


def _nls(G, R):
    """argmin_{x >= 0} of each row of R by block principal pivoting, all rows at once, in 64 bits."""
    rows, k = R.shape
    out = torch.empty_like(R)
    eye = torch.eye(k, dtype=F64, device=DEV)
    for r0 in range(0, rows, 16384):
        r = R[r0:r0 + 16384]
        pas = torch.linalg.solve(G, r.T).T > 0
        alpha = torch.full((len(r),), 3, device=DEV)
        beta = torch.full((len(r),), k + 1, device=DEV)
        for _ in range(10 * k):
            f = pas.to(F64)
            M = G * f[:, :, None] * f[:, None, :] + eye * (1 - f)[:, None, :]
            x = torch.linalg.solve(M, (r * f)[:, :, None])[:, :, 0] * f
            y = (x @ G - r) * (1 - f)
            tol = 1e-11 * (r.abs() + x.abs() @ G.abs())
            bad = (pas & (x < 0)) | (~pas & (y < -tol))
            nv = bad.sum(1)
            if not bool(nv.any()):
                break
            less = nv < beta
            whole = less | (alpha >= 1)
            alpha = torch.where(less, torch.full_like(alpha, 3), alpha - 1)
            beta = torch.where(less, nv, beta)
            last = bad & (torch.cumsum(bad.flip(1), 1).flip(1) == 1)
            pas = pas ^ torch.where(whole[:, None], bad, last)
        out[r0:r0 + 16384] = x.clamp(min=0)
    return out


def _update(algo, X, P, G):
    """X <- the local update of its rows; in place for HALS."""
    if algo == "mu":
        return X * P / (X @ G + 1e-16)
    if algo == "abpp":
        return _nls(G, P)
    for i in range(X.shape[1]):
        if float(G[i, i]) > 0:
            X[:, i] = (X[:, i] + (P[:, i] - X @ G[:, i]) / G[i, i]).clamp(min=0)
    return X


def _iterate(A, W, Ht, algo):
    GH = Ht.T @ Ht
    PW = A.times(Ht)
    W = _update(algo, W, PW, GH)
    GW = W.T @ W
    if algo == "hals":
        n = torch.sqrt(torch.diagonal(GW))
        n = torch.where(n > 0, n, torch.ones_like(n))
        W, Ht, GW = W / n, Ht * n, GW / n / n[:, None]
    PHt = A.t_times(W)
    Ht = _update(algo, Ht.clone(), PHt, GW)
    r2 = A.n2 - 2 * float((PHt * Ht).sum()) + float((GW * (Ht.T @ Ht)).sum())
    return W, Ht, GH, PW, GW, PHt, (max(0.0, r2) / A.n2) ** 0.5


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "batched":
        # tensor-core operand rounding (2^-12, 2^-9) times the condition of the factors' Grams: the factors of two
        # precisions differ although both fit A alike
        return None
    s = prepare(case, seed)
    if kind == "nls":
        return {"X": _nls(s["G"].to(F64), s["R"].to(F64)), "unsolved": None}
    A = _Mat(s)
    if kind == "product":
        F = s["F"].to(F64)
        return A.times(F.T.contiguous()) if c["op"] == "aht" else A.t_times(F).T.contiguous()
    W, Ht = s["W"].detach().to(F64), s["H"].detach().to(F64).T.contiguous()
    if kind == "spmm":
        return {"PW": A.times(Ht), "PH": A.t_times(W).T.contiguous()}
    if kind == "loss":
        PW, PHt, GH, GW = A.times(Ht), A.t_times(W), Ht.T @ Ht, W.T @ W
        loss = 0.5 * (A.n2 - 2 * (PHt * Ht).sum() + (GW * GH).sum())
        return {"loss": loss, "dW": W @ GH - PW, "dH": (Ht @ GW - PHt).T.contiguous()}
    if kind == "steps":
        W, Ht, GH, PW, GW, PHt, rel = _iterate(A, W, Ht, c["algo"])
        return {"GH": GH, "PW": PW, "GW": GW, "PH": PHt.T.contiguous(), "W": W, "H": Ht.T.contiguous(),
                "relres": rel}
    rel = []
    for _ in range(c["iters"]):
        W, Ht, _, _, _, _, r = _iterate(A, W, Ht, c["algo"])
        rel.append(r)
    return {"W": W, "H": Ht.T.contiguous(), "relres": np.array(rel)}
