"""Completions with many CTA-tier fronts of more than 64 columns: they end in one
CTA each and all at once, a few of them by launch sequences, so the number of
launches does not grow with the number of fronts.  P(X-hat^{-1}) = S by the
gradient, f* against log det of a factor of X-hat."""
import numpy as np
import pytest

import workloads as W
from oracle import dense as OD
from test_gpu_grouped_fronts import _cliques, _dev, _host

pytestmark = pytest.mark.gpu

BATCHES = {
    "roots66": (lambda: [W.band(66, 65)] * 40, 30),       # without ancestors
    "roots150": (lambda: [W.band(150, 149)] * 7, 30),
    "one150": (lambda: [W.band(150, 149)], 60),           # a launch sequence
    "one_of_each": (lambda: [W.band(150, 149)] + [W.band(66, 65)] * 20 + [W.band(40, 39)] * 3, 60),
    "ancestors": (lambda: [_cliques(70, 60, 3)] * 6, 30),  # grouped panels, then one CTA each
    "long_ancestors": (lambda: [_cliques(97, 130, 2)] * 4, 50),
    "with_dense": (lambda: [W.band(400, 399)] + [W.band(90, 89)] * 60, 150),
}


@pytest.mark.parametrize("name", list(BATCHES))
def test_wide_fronts(name):
    from paper_1203_2742_gb300 import binding as B
    make, most = BATCHES[name]
    sym = B.SymbolicBatch(make())
    n, cp, ri = sym.n, sym.colptr, sym.rowind
    rng = np.random.default_rng(n)
    s = W.projected_gram(n, cp, ri, rng.standard_normal((n, 12)), 0.7)
    l0 = B.chd_kernel_launches()
    fx, fstar = sym.complete(_dev(s))
    assert B.chd_kernel_launches() - l0 <= most
    x = fx.product()
    for _ in range(3):  # again, captured, replayed
        fx.recomplete(_dev(s), want_fstar=False)
        assert fx.status() == 0
        assert OD.rel_err(n, cp, ri, -_host(fx.gradient()), s) < 1e-9
    want = sym.factor(x).logdet() - n
    assert abs(fstar - want) <= 1e-9 * max(1.0, abs(want))
    ys = W.uniform_sym(n, cp, ri, rng, count=1)
    back = _host(fx.inv_hessian(fx.hessian(_dev(ys))))[0]
    assert OD.rel_err(n, cp, ri, back, ys[0]) < 1e-7
    bad = s.copy()
    bad[cp[-2]] = -1.0  # the last instance's last pivot
    fx.recomplete(_dev(bad), want_fstar=False)
    assert fx.status() == 3
