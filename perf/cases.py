"""The work that a program of this library has it do, as measurable cases.

A case names a sparsity pattern (kind and size), what is asked of it (op) and
the number m of matrices of a Hessian-type call:

  op           one pass                                            stands for
  factor       refactor(X), log det, gradient                      a line search: f and its gradient at a new X
  hessian      H(Y_i), i < m, on a factor that is kept             conjugate gradients, many directions at one X
  inv_hessian  H^{-1}(T_i), i < m, on a factor that is kept        preconditioned solves at one X
  newton       refactor(X), log det, gradient, H^{-1}(T_i), i < m  one Newton (predictor-corrector) iteration
  complete     completion of S, f*(S) and the values of X-hat      dual iterate: dual value and dual gradient
  schur        A_i . H(A_j) of m sparse A_i                        coefficients of an interior-point iteration
  step         refactor, log det, gradient, H, H^{-1}, completion  a primal-dual iteration, every operation once

Values follow the benchmark's recipe: X with off-diagonals uniform[-1, 1] on
the filled pattern and diagonal = row abs-sum + 1, Y and T uniform[-1, 1],
S = P(G G^T + c I) with G Gaussian, A_i with eight nonzeros.  Analysis
options are the defaults with the ordering of each kind.  Buffers of inputs
and outputs are kept over the passes, as an iterating program keeps them.
"""
import math

import numpy as np
import torch

import workloads as W
from paper_1203_2742_gb300 import binding as B


def listed():
    return [
        # the smallest program: one band of 200 columns, where latency and launches are everything
        {"name": "band200 step", "kind": "band", "n": 200, "w": 8, "op": "step", "m": 1},
        # a band of ordinary size and width, several directions at once
        {"name": "band3000 hessian", "kind": "band", "n": 3000, "w": 24, "op": "hessian", "m": 8},
        # a long, wide band: one elimination chain of 12000 columns
        {"name": "band12000 newton", "kind": "band", "n": 12000, "w": 61, "op": "newton", "m": 2},
        # block arrow: thousands of identical leaves under one small root
        {"name": "arrow5000 step", "kind": "arrow", "n": 5000, "w": 32, "op": "step", "m": 4},
        # a small grid with sparse constraint matrices, odd sides
        {"name": "grid63x41 schur", "kind": "grid2d", "nx": 63, "ny": 41, "op": "schur", "m": 12},
        # the benchmark's grid: many directions in one batched call, both ways
        {"name": "grid150 hessian", "kind": "grid2d", "nx": 150, "ny": 150, "op": "hessian", "m": 64},
        {"name": "grid150 inv_hessian", "kind": "grid2d", "nx": 150, "ny": 150, "op": "inv_hessian", "m": 64},
        # a 3D grid, ragged sides: middle-sized and large dense fronts
        {"name": "grid17x20x13 newton", "kind": "grid3d", "nx": 17, "ny": 20, "nz": 13, "op": "newton", "m": 2},
        # the benchmark's random pattern: value and gradient, many directions, the dual side
        {"name": "er5000 factor", "kind": "er", "n": 5000, "op": "factor", "m": 1},
        {"name": "er5000 hessian", "kind": "er", "n": 5000, "op": "hessian", "m": 8},
        {"name": "er5000 complete", "kind": "er", "n": 5000, "op": "complete", "m": 1},
        # independent uneven problems in one object
        {"name": "batch24 hessian", "kind": "batch", "count": 24, "nmin": 300, "nmax": 5000, "op": "hessian", "m": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["band", "arrow", "grid2d", "grid3d", "er", "batch"])
    op = rng.choice(["factor", "hessian", "inv_hessian", "newton", "complete", "schur", "step"])
    many = op in ("hessian", "inv_hessian", "schur")
    m = _log(rng, 1, 16) if many else 1 if op in ("factor", "complete") else rng.choice([1, 1, 2, 3])
    if kind == "band":
        c = {"n": _log(rng, 200, 12000 if not many else 6000), "w": rng.randint(4, 62)}
        if op == "step":
            c["n"] = min(c["n"], 5000)
    elif kind == "arrow":
        c = {"n": _log(rng, 300, 10000), "w": rng.randint(8, 48)}
    elif kind == "grid2d":
        c = {"nx": _log(rng, 12, 150), "ny": _log(rng, 12, 150)}
    elif kind == "grid3d":
        c = {"nx": rng.randint(6, 18), "ny": rng.randint(6, 18), "nz": rng.randint(6, 18)}
        m = min(m, 6)
    elif kind == "er":
        c = {"n": _log(rng, 400, 4500)}
        m = min(m, 8)
    else:
        c = {"count": rng.randint(4, 24), "nmin": 300, "nmax": _log(rng, 1000, 4000)}
        m = min(m, 4)
    return {"kind": kind, **c, "op": op, "m": m}


# ---------------------------------------------------------------------------
# patterns and values
# ---------------------------------------------------------------------------

def _symbolic(case):
    k = case["kind"]
    if k == "band":
        return B.Symbolic(*W.band(case["n"], case["w"]))
    if k == "arrow":
        return B.Symbolic(*W.arrow(case["n"], case["w"]))
    if k == "grid2d":
        d = (case["nx"], case["ny"])
        return B.Symbolic(*W.grid2d(*d), **W.nd_options(d))
    if k == "grid3d":
        d = (case["nx"], case["ny"], case["nz"])
        return B.Symbolic(*W.grid3d(*d), **W.nd_options(d))
    if k == "er":  # five neighbours a vertex: density 0.1 % at n = 5000
        pat = W.erdos_renyi(case["n"], 5.0 / case["n"], np.random.default_rng(1))
        return B.Symbolic(*pat, ordering="mindeg", relax=16)
    rng = np.random.default_rng(case["count"])
    pats, ords = [], []
    for i in range(case["count"]):
        n = int(round(np.exp(rng.uniform(np.log(case["nmin"]), np.log(case["nmax"])))))
        if i % 3 == 0:
            pats.append(W.band(n, int(rng.integers(4, 63))))
            ords.append("natural")
        elif i % 3 == 1:
            pats.append(W.arrow(n, 32))
            ords.append("natural")
        else:
            d = W.grid_dims("grid", n)
            pats.append(W.grid2d(*d))
            ords.append(W.nd_options(d))
    return B.SymbolicBatch(pats, orderings=ords)


def _cols(sym):
    return np.repeat(np.arange(sym.n), np.diff(np.asarray(sym.colptr, np.int64)))


def _values(case, seed, sym):
    """x, y (m x nnz) and s on the GPU, from the seed alone."""
    op, m = case["op"], case["m"]
    r, c = np.asarray(sym.rowind, np.int64), _cols(sym)
    rng = np.random.default_rng(seed)
    v = {}
    if op != "complete":
        x = rng.uniform(-1.0, 1.0, sym.nnz)
        off = r != c
        x[~off] = 0.0
        ab = np.abs(x)
        x[~off] = np.bincount(r, ab, sym.n) + np.bincount(c, ab, sym.n) + 1.0
        v["x"] = torch.from_numpy(x).cuda()
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if op == "schur":
        y = np.zeros((m, sym.nnz))
        for i in range(m):
            y[i, rng.choice(sym.nnz, 8, replace=False)] = rng.uniform(-1.0, 1.0, 8)
        v["y"] = torch.from_numpy(y).cuda()
    elif op in ("hessian", "inv_hessian", "newton", "step"):
        v["y"] = torch.rand((m, sym.nnz), generator=gen, device="cuda", dtype=torch.float64) * 2 - 1
    if op in ("complete", "step"):
        g = torch.randn((sym.n, 20), generator=gen, device="cuda", dtype=torch.float64)
        rt, ct = torch.from_numpy(r).cuda(), torch.from_numpy(c).cuda()
        s = torch.cat([(g[rt[i:i + 500000]] * g[ct[i:i + 500000]]).sum(1) for i in range(0, sym.nnz, 500000)])
        v["s"] = s + 0.5 * (rt == ct)
    return v


def prepare(case, seed):
    sym = _symbolic(case)
    st = {"op": case["op"], "m": case["m"], "sym": sym, **_values(case, seed, sym)}
    if "x" in st:
        st["fac"] = sym.factor(st["x"])
        st["g"] = st["fac"].gradient()
    if "s" in st:
        st["comp"], _ = sym.complete(st["s"])
        st["xhat"] = torch.empty_like(st["s"])
    if "y" in st:
        st["t"] = torch.empty_like(st["y"])
        st["u"] = torch.empty_like(st["y"])
        st["h"] = torch.empty((case["m"], case["m"]), dtype=torch.float64, device="cuda")
    if case["op"] == "inv_hessian":  # the factor's blocks for H^{-1} are there before the first of many calls
        st["fac"].inv_hessian(st["y"], out=st["t"])
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    op, f = st["op"], st.get("fac")
    if op == "hessian":
        return {"t": f.hessian(st["y"], out=st["t"])}
    if op == "inv_hessian":
        return {"t": f.inv_hessian(st["y"], out=st["t"])}
    if op == "schur":
        h, t = f.schur(st["y"], t=st["t"], h=st["h"])
        return {"h": h, "t": t}
    out = {}
    if op in ("factor", "newton", "step"):
        f.refactor(st["x"])
        out["logdet"] = f.logdet()
        out["g"] = f.gradient(out=st["g"])
    if op == "step":
        out["t"] = f.hessian(st["y"], out=st["t"])
    if op in ("newton", "step"):
        out["u"] = f.inv_hessian(st["y"], out=st["u"])
    if op in ("complete", "step"):
        out["fstar"] = st["comp"].recomplete(st["s"])
        out["xhat"] = st["comp"].product(out=st["xhat"])
    return out


def work(case):
    """Values read and written once (8 bytes each), and the flops of the
    supernodal algorithms on the unsplit partition."""
    op, m = case["op"], case["m"]
    sym = _symbolic(case)
    f, nnz = sym.flops(), sym.nnz
    # in, out, flops: the factor's own blocks are read once where a call starts from them
    parts = {"factor": (1, 1, f["factor"] + f["gradient"]),
             "hessian": (2 + m, m, m * f["hessian"]),
             "inv_hessian": (2 + m, m, m * f["inv_hessian"]),
             "schur": (2 + m, m, m * f["hessian"] + 2.0 * m * m * nnz),
             "newton": (1 + m, 1 + m, f["factor"] + f["gradient"] + m * f["inv_hessian"]),
             "complete": (1, 1, f["completion"]),
             "step": (2 + m, 2 + 2 * m, f["factor"] + f["gradient"] + m * (f["hessian"] + f["inv_hessian"]) +
                      f["completion"])}
    i, o, fl = parts[op]
    return {"bytes": 8.0 * nnz * (i + o), "flops": float(fl)}


# ---------------------------------------------------------------------------
# the same in 64 bits, by dense matrices and the clique sums of a chordal pattern
# ---------------------------------------------------------------------------

class _Dense:
    """One instance: columns [a, b), values [z0, z1) of the analysed pattern."""

    def __init__(self, sym, a, b, z0, z1):
        self.n, self.z0, self.z1 = b - a, z0, z1
        self.cp = np.asarray(sym.colptr, np.int64)[a:b + 1] - z0
        self.ri = np.asarray(sym.rowind, np.int64)[z0:z1] - a
        self.r = torch.from_numpy(self.ri).cuda()
        self.c = torch.from_numpy(np.repeat(np.arange(self.n), np.diff(self.cp))).cuda()

    def full(self, v):
        d = torch.zeros((self.n, self.n), dtype=torch.float64, device="cuda")
        d[self.r, self.c] = v
        d[self.c, self.r] = v
        return d

    def project(self, d):
        return d[self.r, self.c]

    def cliques(self):
        """(sign, J) of the clique sum: + every column's clique, - its
        separator, without the pairs that cancel, grouped by size."""
        cnt = np.diff(self.cp)
        groups = {}
        for j in range(self.n):
            J = self.ri[self.cp[j]:self.cp[j + 1]]
            # the separator of column j - 1 is this very clique: both drop out
            if not (j > 0 and cnt[j - 1] == cnt[j] + 1 and self.ri[self.cp[j - 1] + 1] == j):
                groups.setdefault((1.0, len(J)), []).append(J)
            last = j + 1 == self.n or not (cnt[j] == cnt[j + 1] + 1 and len(J) > 1 and J[1] == j + 1)
            if last and len(J) > 1:
                groups.setdefault((-1.0, len(J) - 1), []).append(J[1:])
        for (sign, k), js in groups.items():
            step = max(1, 20_000_000 // (k * k))
            for i in range(0, len(js), step):
                yield sign, torch.from_numpy(np.stack(js[i:i + step])).cuda()

    def clique_sum(self, s, ts):
        """Values on V of sum +-S_JJ^-1 T_JJ S_JJ^-1 for every T of ts, of
        sum +-S_JJ^-1, and sum -+log det S_JJ."""
        S = self.full(s)
        outs = [torch.zeros_like(S) for _ in ts]
        xhat = torch.zeros_like(S)
        Ts = [self.full(t) for t in ts]
        ld = 0.0
        for sign, J in self.cliques():
            i, j = J[:, :, None].expand(-1, -1, J.shape[1]), J[:, None, :].expand(-1, J.shape[1], -1)
            L = torch.linalg.cholesky(S[i, j])
            inv = torch.cholesky_inverse(L)
            ld -= sign * 2.0 * float(torch.log(torch.diagonal(L, dim1=1, dim2=2)).sum())
            xhat.index_put_((i, j), sign * inv, accumulate=True)
            for o, T in zip(outs, Ts):
                o.index_put_((i, j), sign * (inv @ T[i, j] @ inv), accumulate=True)
        return [self.project(o) for o in outs], self.project(xhat), ld


def exact(case, seed):
    op, m = case["op"], case["m"]
    sym = _symbolic(case)
    v = _values(case, seed, sym)
    if isinstance(sym, B.SymbolicBatch):
        parts = [_Dense(sym, int(sym.n_off[i]), int(sym.n_off[i + 1]), int(sym.nnz_off[i]), int(sym.nnz_off[i + 1]))
                 for i in range(sym.count)]
    else:
        parts = [_Dense(sym, 0, sym.n, 0, sym.nnz)]
    # about 20 seconds of dense 64-bit arithmetic at 1 TFLOP/s
    cost = sum(float(p.n) ** 3 * (1 + (4 * m if op in ("hessian", "schur", "step") else 0)) for p in parts)
    room = max(8.0 * p.n * p.n * (2 * m + 4) for p in parts)
    if cost > 1.2e13 or room > 1e11:
        return None
    out = {"logdet": 0.0, "fstar": 0.0}
    keep = {k: [] for k in ("g", "t", "u", "xhat")}
    for p in parts:
        seg = lambda w: w[..., p.z0:p.z1]
        if op != "complete":
            L = torch.linalg.cholesky(p.full(seg(v["x"])))
            out["logdet"] += 2.0 * float(torch.log(torch.diagonal(L)).sum())
            Z = torch.cholesky_inverse(L)
            del L
            S = p.project(Z)
            keep["g"].append(-S)
            if op in ("hessian", "schur", "step"):
                keep["t"].append(torch.stack([p.project(Z @ p.full(seg(v["y"])[i]) @ Z) for i in range(m)]))
            del Z
            if op in ("inv_hessian", "newton", "step"):
                u, _, _ = p.clique_sum(S, [seg(v["y"])[i] for i in range(m)])
                keep["u"].append(torch.stack(u))
        if op in ("complete", "step"):
            _, xh, ld = p.clique_sum(seg(v["s"]), [])
            keep["xhat"].append(xh)
            out["fstar"] += ld - p.n
    cat = {k: torch.cat(w, dim=-1) for k, w in keep.items() if w}
    if op == "hessian":
        return {"t": cat["t"]}
    if op == "inv_hessian":
        return {"t": cat["u"]}
    if op == "schur":
        wt = torch.full((sym.nnz,), 2.0, dtype=torch.float64, device="cuda")
        wt[torch.from_numpy(np.asarray(sym.colptr, np.int64)[:-1].copy()).cuda()] = 1.0
        return {"h": (v["y"] * wt) @ cat["t"].T, "t": cat["t"]}
    names = {"factor": ("logdet", "g"), "newton": ("logdet", "g", "u"), "complete": ("fstar", "xhat"),
             "step": ("logdet", "g", "t", "u", "fstar", "xhat")}[op]
    return {k: out[k] if k in out else cat[k] for k in names}
