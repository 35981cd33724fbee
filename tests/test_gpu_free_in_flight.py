"""A factor object may be freed while its last call is still running, on the default
stream and on others: the free waits for the call, whose outputs are complete."""
import numpy as np
import pytest

import workloads as W
from oracle import dense as OD
from test_gpu_grouped_fronts import _cliques, _dev, _host

pytestmark = pytest.mark.gpu

PATTERNS = {
    "band": lambda: W.band(900, 8),
    "grouped": lambda: _cliques(40, 100, 3),
    "dense": lambda: W.band(500, 499),
}


@pytest.mark.parametrize("name", list(PATTERNS))
@pytest.mark.parametrize("own_stream", [False, True])
def test_free_in_flight(name, own_stream):
    import torch
    from paper_1203_2742_gb300 import binding as B
    pattern = PATTERNS[name]()
    sym = B.Symbolic(*pattern)  # values are in the analysed order
    n, cp, ri = sym.n, sym.colptr, sym.rowind
    rng = np.random.default_rng(n)
    xh = W.diag_dominant(n, cp, ri, rng)
    yh = W.uniform_sym(n, cp, ri, rng, count=8)
    x, y = _dev(xh), _dev(yh)
    torch.cuda.synchronize()
    st = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
    outs = []
    with torch.cuda.stream(st):
        for i in range(4):
            sym = B.Symbolic(*pattern)
            f = sym.factor(x)
            g, t = f.gradient(), f.hessian(y)
            outs.append((g, t, f.inv_hessian(t)))
            if i % 2:
                f.free()
            del f, sym
    torch.cuda.synchronize()
    grad, want = OD.gradient(n, cp, ri, xh), OD.hessian(n, cp, ri, xh, [yh[7]])[0]
    for g, t, u in outs:
        assert OD.rel_err(n, cp, ri, _host(g), grad) < 1e-10
        assert OD.rel_err(n, cp, ri, _host(t)[7], want) < 1e-10
        assert OD.rel_err(n, cp, ri, _host(u)[7], yh[7]) < 1e-9
