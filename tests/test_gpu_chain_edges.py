"""The chain tier at the edges of its register layouts (window sizes where the
number of threads or of slots per thread changes, the shortest run, the widest
window) against the same pattern without chain runs, and leaf groups long
enough for their products to be split, against the oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import dense as OD

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _host(t):
    import torch
    torch.cuda.synchronize()
    return t.cpu().numpy()


def _all(sym, x, ys, y2):
    f = sym.factor(_dev(x))
    l, d = f.export()
    out = {"l": _host(l), "d": _host(d), "logdet": f.logdet(), "g": _host(f.gradient()), "xp": _host(f.product()),
           "t": _host(f.hessian(_dev(ys))), "u": _host(f.inv_hessian(_dev(ys))), "w": _host(f.hessian_factor(_dev(ys))),
           "w2": _host(f.hessian_factor(_dev(y2), sparse=True)), "ta": _host(f.hessian_factor_adj(_dev(ys)))}
    assert f.status() == 0
    return out


@pytest.mark.parametrize("a,extra", [(1, 9), (2, 9), (3, 40), (7, 9), (8, 30), (9, 23), (10, 23), (15, 9), (16, 41),
                                     (17, 30), (31, 50), (32, 50), (33, 9), (48, 70), (63, 40), (64, 9), (64, 90)])
def test_chain_window_sizes(a, extra):
    from paper_1203_2742_gb300 import binding as B
    pattern = W.band(a + extra, a)  # a run of extra - 1 columns under a dense front
    rng = np.random.default_rng(a)
    on, off = B.Symbolic(*pattern, chain_runs=True), B.Symbolic(*pattern, chain_runs=False)
    n, cp, ri = on.n, on.colptr, on.rowind
    x = W.diag_dominant(n, cp, ri, rng)
    ys = W.uniform_sym(n, cp, ri, rng, count=2)
    y2 = np.zeros_like(ys)
    for i in range(2):  # the first nonzero inside the run: a pruned prefix
        y2[i, rng.integers(len(ri) // 2, len(ri), size=2)] = 1.0 + i
    r_on, r_off = _all(on, x, ys, y2), _all(off, x, ys, y2)
    err = lambda p, q: OD.rel_err(n, cp, ri, p, q)
    assert err(r_on["l"], r_off["l"]) < 1e-12 and np.allclose(r_on["d"], r_off["d"], rtol=1e-12)
    assert abs(r_on["logdet"] - r_off["logdet"]) <= 1e-12 * max(1.0, abs(r_off["logdet"]))
    assert err(r_on["g"], r_off["g"]) < 1e-12 and err(r_on["xp"], x) < 1e-12
    for k in ("t", "u", "w", "w2", "ta"):
        for i in range(2):
            assert err(r_on[k][i], r_off[k][i]) < 1e-11, k


@pytest.mark.parametrize("bands", [[(5000, 1)], [(2500, 8)], [(1300, 24)], [(701, 61)], [(900, 64)],
                                   [(1500, 30), (200, 5), (620, 47), (1400, 12)]])
def test_chain_segments(bands):
    """Runs long enough to be cut into segments (alone, and of several lengths
    in one object): the gradient and both Hessian passes against the same
    patterns without chain runs, on a factor and on a completion (whose
    segments' matrices do not come from a gradient)."""
    from paper_1203_2742_gb300 import binding as B
    pats = [W.band(n, w) for n, w in bands]
    make = (lambda **o: B.Symbolic(*pats[0], **o)) if len(pats) == 1 else (lambda **o: B.SymbolicBatch(pats, **o))
    rng = np.random.default_rng(len(pats) + bands[0][0])
    on, off = make(chain_runs=True), make(chain_runs=False)
    n, cp, ri = on.n, on.colptr, on.rowind
    x = W.diag_dominant(n, cp, ri, rng)
    ys = W.uniform_sym(n, cp, ri, rng, count=2)
    s = W.projected_gram(n, cp, ri, rng.standard_normal((n, 6)), 1.0)
    err = lambda p, q: OD.rel_err(n, cp, ri, p, q)
    res = []
    for sym in (on, off):
        f = sym.factor(_dev(x))
        fx, _ = sym.complete(_dev(s))
        res.append((_host(f.gradient()), _host(f.hessian(_dev(ys))), _host(f.inv_hessian(f.hessian(_dev(ys)))),
                    _host(fx.hessian(_dev(ys))), _host(fx.gradient())))
        assert f.status() == 0 and fx.status() == 0
    assert err(res[0][0], res[1][0]) < 1e-12
    assert err(-res[0][4], s) < 1e-10
    for i in range(2):
        assert err(res[0][1][i], res[1][1][i]) < 1e-12
        assert err(res[0][2][i], ys[i]) < 1e-9
        assert err(res[0][3][i], res[1][3][i]) < 1e-9


@pytest.mark.parametrize("col", [0, 1, 2, 17])
def test_chain_not_pd(col):
    """A non-positive pivot inside a run is reported with its column."""
    from paper_1203_2742_gb300 import binding as B
    sym = B.Symbolic(*W.band(60, 12))
    x = W.diag_dominant(sym.n, sym.colptr, sym.rowind, np.random.default_rng(3))
    x[sym.colptr[col]] = -1.0
    f = sym.factor(_dev(x))
    rc, _, c = f.error_detail()
    assert rc == 2 and c == col


@pytest.mark.parametrize("n,w", [(300, 20), (700, 33)])
def test_long_leaf_group(n, w):
    """One leaf group of n - w members: its products are long enough to split."""
    from paper_1203_2742_gb300 import binding as B
    sym = B.Symbolic(*W.arrow(n, w))
    rng = np.random.default_rng(n)
    nn, cp, ri = sym.n, sym.colptr, sym.rowind
    x = W.diag_dominant(nn, cp, ri, rng)
    ys = W.uniform_sym(nn, cp, ri, rng, count=3)
    s0 = B.chd_split_k_launches()
    f = sym.factor(_dev(x))
    err = lambda p, q: OD.rel_err(nn, cp, ri, p, q)
    assert abs(f.logdet() - OD.logdet(nn, cp, ri, x)) <= 1e-10 * abs(OD.logdet(nn, cp, ri, x))
    assert err(_host(f.gradient()), OD.gradient(nn, cp, ri, x)) < 1e-10
    t = f.hessian(_dev(ys))
    want = OD.hessian(nn, cp, ri, x, list(ys))
    back = _host(f.inv_hessian(t))
    for i in range(3):
        assert err(_host(t)[i], want[i]) < 1e-10
        assert err(back[i], ys[i]) < 1e-9  # H^{-1}(H(Y)) = Y
    assert err(_host(f.product()), x) < 1e-12
    assert B.chd_split_k_launches() > s0
