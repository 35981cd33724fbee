"""Many short chain runs in one object beside one long enough to be cut into
segments: more of them than a grid dimension of a launch holds, every value
against dense references (the long band alone on the CPU oracle); and the time
of a call stays near that of the two kinds on their own."""
import numpy as np
import pytest

import workloads as W
from oracle import dense as OD
from test_gpu_grouped_fronts import _dev, _host

pytestmark = pytest.mark.gpu
COUNT, SIZE = 65540, 12  # 65540 tridiagonal patterns: a run of ten columns each


def _pattern(long, count):
    """One block-diagonal pattern: the long band first, then the tridiagonal ones."""
    n1, cp1, ri1 = long
    cs = np.concatenate([np.repeat([2], SIZE - 1), [1]])
    rs = np.concatenate([np.column_stack([np.arange(SIZE - 1), np.arange(1, SIZE)]).ravel(), [SIZE - 1]])
    off = n1 + SIZE * np.arange(count)
    cp = np.concatenate([[0], np.cumsum(np.concatenate([np.diff(cp1), np.tile(cs, count)]))])
    ri = np.concatenate([ri1, (rs[None, :] + off[:, None]).ravel()]).astype(np.int32)
    return (n1 + count * SIZE, cp, ri), rs, np.repeat(np.arange(SIZE), cs)


def test_more_runs_than_a_grid_dimension():
    from paper_1203_2742_gb300 import binding as B
    n1, cp1, ri1 = W.band(1300, 24)
    (N, cp, ri), rs, cols = _pattern((n1, cp1, ri1), COUNT)
    nz1, nz = len(ri1), len(rs)
    sym = B.Symbolic(N, cp, ri)
    assert np.array_equal(sym.colptr, cp) and np.array_equal(sym.rowind, ri)
    assert sym.schedule()["lvl_counts"][0][0] > 65535
    rng = np.random.default_rng(3)
    x = W.diag_dominant(N, cp, ri, rng)
    y = W.uniform_sym(N, cp, ri, rng, count=1)[0]
    f = sym.factor(_dev(x))
    g = _host(f.gradient())
    td = f.hessian(_dev(y[None]))
    t = _host(td)[0]
    assert OD.rel_err(N, cp, ri, _host(f.inv_hessian(td))[0], y) < 1e-9
    assert OD.rel_err(N, cp, ri, _host(f.product()), x) < 1e-12
    assert f.status() == 0
    err = lambda p, q: OD.rel_err(n1, cp1, ri1, p[:nz1], q)
    assert err(g, OD.gradient(n1, cp1, ri1, x[:nz1])) < 1e-10
    assert err(t, OD.hessian(n1, cp1, ri1, x[:nz1], [y[:nz1]])[0]) < 1e-10

    def full(v):
        d = np.zeros((COUNT, SIZE, SIZE))
        d[:, rs, cols] = v[nz1:].reshape(COUNT, nz)
        d[:, cols, rs] = d[:, rs, cols]
        return d

    z = np.linalg.inv(full(x))
    h = z @ full(y) @ z
    assert np.abs(g[nz1:].reshape(COUNT, nz) + z[:, rs, cols]).max() < 1e-12 * np.abs(z).max()
    assert np.abs(t[nz1:].reshape(COUNT, nz) - h[:, rs, cols]).max() < 1e-12 * np.abs(h).max()


def test_short_runs_beside_a_long_one_cost_no_more():
    """Kernels over all columns of all runs: time by columns, not by runs times the
    longest run (a factor of ten and more here)."""
    import torch
    from paper_1203_2742_gb300 import binding as B

    def times(pattern):
        sym = B.Symbolic(*pattern)
        rng = np.random.default_rng(4)
        x = _dev(W.diag_dominant(sym.n, sym.colptr, sym.rowind, rng))
        y = _dev(W.uniform_sym(sym.n, sym.colptr, sym.rowind, rng, count=2))
        f = sym.factor(x)
        g, t, u = f.gradient(), f.hessian(y), None
        u = f.inv_hessian(t)
        p = f.product()
        out = []
        for call in (lambda: f.refactor(x), lambda: f.gradient(out=g), lambda: f.hessian(y, out=t),
                     lambda: f.inv_hessian(t, out=u), lambda: f.product(out=p)):
            best = 1e30
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                call()
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
            out.append(best)
        return out

    long = W.band(1300, 24)
    short = _pattern((0, np.zeros(1, np.int64), np.zeros(0, np.int32)), 30000)[0]
    both = times(_pattern(long, 30000)[0])
    for t, a, b in zip(both, times(long), times(short)):
        assert t < 3.0 * (a + b), (both, a, b)
