"""Dense fronts whose second halves (what no other front waits for) run on side
streams of their own: levels of one and two fronts, the most that are queued
there, and of more, which keep both halves together; pieces of split supernodes
form chains, so several second halves are pending at once."""
import numpy as np
import pytest

import workloads as W
from oracle import dense as OD
from test_gpu_grouped_fronts import _check, _cliques, _dev, _host

pytestmark = pytest.mark.gpu
OPTS = {"big_rows": 48, "big_cols": 48, "split_cols": 24}


@pytest.mark.parametrize("kids", [1, 2, 3, 5])
@pytest.mark.parametrize("tc", [0, -1])
def test_operations(kids, tc):
    _check(_cliques(70, 60, kids), seed=kids, tc_products=tc, **OPTS)


@pytest.mark.parametrize("kids", [2, 3])
def test_repeated_calls(kids):
    """The same calls again (the second captures the sequence, the third
    replays it), outputs overwritten in between; then limited scratch."""
    import torch
    from paper_1203_2742_gb300 import binding as B
    sym = B.Symbolic(*_cliques(70, 60, kids), **OPTS)
    N, cp, ri = sym.n, sym.colptr, sym.rowind
    rng = np.random.default_rng(7 + kids)
    x = _dev(W.diag_dominant(N, cp, ri, rng))
    y = _dev(W.uniform_sym(N, cp, ri, rng, count=5))
    f = sym.factor(x)
    g, t, b = f.gradient(), f.hessian(y), None
    b = f.inv_hessian(t)
    first = [_host(v).copy() for v in (g, t, b)]
    assert OD.rel_err(N, cp, ri, first[0], OD.gradient(N, cp, ri, _host(x))) < 1e-10
    assert max(OD.rel_err(N, cp, ri, p, q) for p, q in zip(first[2], _host(y))) < 1e-9
    for limit in (0, 0, 1):
        if limit:
            f.set_workspace_limit(limit)  # one right-hand side at a time
        for v in (g, t, b):
            v.fill_(float("nan"))
        torch.cuda.synchronize()
        f.refactor(x)
        f.gradient(out=g)
        f.hessian(y, out=t)
        f.inv_hessian(t, out=b)
        for v, w in zip((g, t, b), first):
            assert OD.rel_err(N, cp, ri, np.atleast_2d(_host(v))[0], np.atleast_2d(w)[0]) < 1e-12
