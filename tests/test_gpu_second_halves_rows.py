"""Repeated calls on dense fronts whose second halves run on side streams: the
first, the captured and the replayed calls, then one right-hand side at a time,
outputs overwritten in between, give every row of the outputs again."""
import numpy as np
import pytest

import workloads as W
from oracle import dense as OD
from test_gpu_dense_second_halves import OPTS
from test_gpu_grouped_fronts import _cliques, _dev, _host

pytestmark = pytest.mark.gpu
M = 5


@pytest.mark.parametrize("kids", [1, 2, 3])
def test_every_row_again(kids):
    from paper_1203_2742_gb300 import binding as B
    sym = B.Symbolic(*_cliques(70, 60, kids), **OPTS)
    n, cp, ri = sym.n, sym.colptr, sym.rowind
    rng = np.random.default_rng(20 + kids)
    xh = W.diag_dominant(n, cp, ri, rng)
    yh = W.uniform_sym(n, cp, ri, rng, count=M)
    x, y = _dev(xh), _dev(yh)
    f = sym.factor(x)
    g, t = f.gradient(), f.hessian(y)
    b, w = f.inv_hessian(t), f.hessian_factor(y)
    want = OD.hessian(n, cp, ri, xh, list(yh))
    adj = _host(f.hessian_factor_adj(w))
    first_w = _host(w).copy()
    grad = OD.gradient(n, cp, ri, xh)
    for limit in (0, 0, 0, 1):
        if limit:
            f.set_workspace_limit(limit)
        for v in (g, t, b, w):
            v.fill_(float("nan"))
        f.refactor(x)
        f.gradient(out=g)
        f.hessian(y, out=t)
        f.inv_hessian(t, out=b)
        f.hessian_factor(y, out=w)
        assert f.status() == 0
        for v in (g, t, b, w):
            assert np.isfinite(_host(v)).all()
        assert OD.rel_err(n, cp, ri, _host(g), grad) < 1e-10
        for i in range(M):
            assert OD.rel_err(n, cp, ri, _host(t)[i], want[i]) < 1e-10
            assert OD.rel_err(n, cp, ri, _host(b)[i], yh[i]) < 1e-9
            assert OD.rel_err(n, cp, ri, adj[i], want[i]) < 1e-10
            assert OD.rel_err(n, cp, ri, _host(w)[i], first_w[i]) < 1e-12
