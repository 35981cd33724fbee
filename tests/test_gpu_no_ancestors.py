"""Independent dense matrices in one object: fronts of the grouped tier without
ancestors have no row products, and calls on them launch none."""
import numpy as np
import pytest

import workloads as W
from oracle import dense as OD
from test_gpu_grouped_fronts import _dev, _host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,count", [(9, 40), (16, 40), (17, 40), (30, 300), (33, 20), (64, 7)])
def test_dense_blocks(n, count):
    from paper_1203_2742_gb300 import binding as B
    sym = B.SymbolicBatch([W.band(n, n - 1)] * count)
    N, cp, ri = sym.n, sym.colptr, sym.rowind
    rng = np.random.default_rng(n)
    x = W.diag_dominant(N, cp, ri, rng)
    ys = W.uniform_sym(N, cp, ri, rng, count=3)
    f = sym.factor(_dev(x))
    f.gradient()
    y, t = _dev(ys), None
    l0 = B.chd_kernel_launches()
    t = f.hessian(y)
    l1 = B.chd_kernel_launches()
    u = f.inv_hessian(t)
    l2 = B.chd_kernel_launches()
    # Hessian: counters, (assembly,) update blocks, M_NN, top-down; inverse: gather, K_NN, update blocks
    assert l1 - l0 <= (4 if n <= 16 else 5) and l2 - l1 <= 3
    w = f.hessian_factor(y)
    ta = _host(f.hessian_factor_adj(w))
    nz = n * (n + 1) // 2
    c0, r0 = cp[:n + 1], ri[:nz]
    for b in (0, count - 1):
        p = slice(b * nz, (b + 1) * nz)
        want = OD.hessian(n, c0, r0, x[p], [v[p] for v in ys])
        for i in range(3):
            assert OD.rel_err(n, c0, r0, _host(t)[i][p], want[i]) < 1e-10
            assert OD.rel_err(n, c0, r0, ta[i][p], want[i]) < 1e-10
    for i in range(3):
        assert OD.rel_err(N, cp, ri, _host(u)[i], ys[i]) < 1e-9
