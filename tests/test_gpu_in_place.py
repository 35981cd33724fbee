"""Inverse Hessian with the output in the place of the input: the same values
as into an array of its own, in every tier (chain runs, whose columns are all in
work at once and read each other's input, warp tier, grouped and dense fronts,
leaf groups), directly, captured and replayed."""
import numpy as np
import pytest

import workloads as W
from test_gpu_grouped_fronts import _cliques, _dev

pytestmark = pytest.mark.gpu

CASES = {
    "chain8": (lambda: W.band(400, 8), {}),
    "chain40": (lambda: W.band(3000, 40), {}),
    "chain64": (lambda: W.band(1200, 64), {}),
    "no_chain": (lambda: W.band(400, 8), {"chain_runs": False}),
    "grid": (lambda: W.grid2d(24, 31), W.nd_options((24, 31))),
    "leaf_group": (lambda: W.arrow(600, 20), {}),
    "grouped": (lambda: _cliques(33, 65, 3), {}),
    "dense": (lambda: _cliques(70, 60, 2), {"big_rows": 48, "big_cols": 48, "split_cols": 24}),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("m", [1, 3])
def test_inverse_hessian_in_place(name, m):
    import torch
    from paper_1203_2742_gb300 import binding as B
    make, opts = CASES[name]
    sym = B.Symbolic(*make(), **opts)
    rng = np.random.default_rng(m)
    f = sym.factor(_dev(W.diag_dominant(sym.n, sym.colptr, sym.rowind, rng)))
    t = f.hessian(_dev(W.uniform_sym(sym.n, sym.colptr, sym.rowind, rng, count=m)))
    want = f.inv_hessian(t)
    buf = torch.empty_like(t)
    for _ in range(3):
        buf.copy_(t)
        assert f.inv_hessian(buf, out=buf) is buf
        assert torch.equal(buf, want)  # the same operations on the same numbers
    assert f.status() == 0
