"""The grouped tier (fronts between the warp tier and the large dense fronts)
at the edges of its blocks: columns around the thin, one-panel and widest
fronts, ancestor counts around multiples of the row blocks and of the panels of
the grouped inverse, several children with overlapping ancestor sets -- every
operation against the dense oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import dense as OD

pytestmark = pytest.mark.gpu
TOL = 1e-10


def _dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _host(t):
    import torch
    torch.cuda.synchronize()
    return t.cpu().numpy()


def _cliques(n, a, kids=2, extra=5):
    """`kids` leaf cliques of n columns, each with a rows of a common clique of
    a + extra vertices (every second kid skips the first rows), and a tail of
    one more vertex under the last rows of the common clique."""
    p = a + extra
    N = kids * n + p
    rows, cols = [], []
    for k in range(kids):
        own = np.arange(k * n, (k + 1) * n)
        anc = kids * n + (np.arange(a) if k % 2 == 0 else np.arange(p - a, p))
        J = np.concatenate([own, anc])
        r, c = np.meshgrid(J, own, indexing="ij")
        rows.append(r.ravel()); cols.append(c.ravel())
    common = np.arange(kids * n, N)
    r, c = np.meshgrid(common, common, indexing="ij")
    rows.append(r.ravel()); cols.append(c.ravel())
    r, c = np.concatenate(rows), np.concatenate(cols)
    keep = r >= c
    return W.lower_csc_from_pairs(N, r[keep], c[keep])


SIZES = [(1, 40), (1, 65), (9, 7), (9, 8), (8, 33), (15, 16), (16, 31), (17, 32), (31, 33), (32, 64), (33, 65), (40, 96),
         (64, 15), (65, 97), (100, 70), (128, 20), (129, 20), (159, 3)]


@pytest.mark.parametrize("n,a", SIZES)
@pytest.mark.parametrize("kids", [1, 3])
def test_grouped_front_sizes(n, a, kids):
    _check(_cliques(n, a, kids), seed=1000 * n + a)


@pytest.mark.parametrize("n,a,opts", [(10, 330, {}), (3, 513, {}), (16, 320, {"tc_products": -1}),
                                      (12, 40, {"big_rows": 48, "big_cols": 48}),
                                      (40, 70, {"big_rows": 4096, "big_cols": 4096, "split_cols": -1}),
                                      (256, 9, {"big_rows": 4096, "big_cols": 4096, "split_cols": -1}),
                                      (257, 40, {"big_rows": 4096, "big_cols": 4096, "split_cols": -1})])
def test_grouped_dense_thin_fronts(n, a, opts):
    """Thin fronts of the dense tier, and CTA-tier fronts of any size."""
    _check(_cliques(n, a, 2), seed=a, **opts)


def _check(pattern, seed, **opts):
    from paper_1203_2742_gb300 import binding as B
    sym = B.Symbolic(*pattern, **opts)
    N, cp, ri = sym.n, sym.colptr, sym.rowind
    rng = np.random.default_rng(seed)
    x = W.diag_dominant(N, cp, ri, rng)
    ys = W.uniform_sym(N, cp, ri, rng, count=3)
    y2 = np.zeros_like(ys)
    for i in range(3):
        y2[i, rng.choice(len(ri), 2, replace=False)] = 1.0
    err = lambda p, q: OD.rel_err(N, cp, ri, p, q)
    f = sym.factor(_dev(x))
    assert abs(f.logdet() - OD.logdet(N, cp, ri, x)) <= TOL * max(1.0, abs(OD.logdet(N, cp, ri, x)))
    assert err(_host(f.product()), x) < 1e-12  # L D L^T
    assert err(_host(f.gradient()), OD.gradient(N, cp, ri, x)) < TOL
    t = f.hessian(_dev(ys))
    want = OD.hessian(N, cp, ri, x, list(ys))
    back = _host(f.inv_hessian(t))
    w, ws = _host(f.hessian_factor(_dev(y2))), _host(f.hessian_factor(_dev(y2), sparse=True))
    ta = _host(f.hessian_factor_adj(f.hessian_factor(_dev(ys))))
    for i in range(3):
        assert err(_host(t)[i], want[i]) < TOL
        assert err(back[i], ys[i]) < 1e-9  # H^{-1}(H(Y)) = Y
        assert err(ws[i], w[i]) < 1e-12
        assert err(ta[i], want[i]) < TOL  # R^adj(R(Y)) = H(Y)
    assert f.status() == 0
    # completion: P(X-hat^{-1}) = S, f* and the factor's other blocks
    s = W.projected_gram(N, cp, ri, rng.standard_normal((N, 12)), 0.7)
    fx, fstar = sym.complete(_dev(s))
    xh = _host(fx.product())
    assert err(-OD.gradient(N, cp, ri, xh), s) < 1e-9 and err(-_host(fx.gradient()), s) < 1e-9
    assert abs(fstar - (OD.logdet(N, cp, ri, xh) - N)) <= 1e-9 * max(1.0, abs(fstar))
    back = _host(fx.inv_hessian(fx.hessian(_dev(ys[:1]))))[0]
    assert err(back, ys[0]) < 1e-7
    bad = s.copy()
    bad[cp[-2]] = -1.0  # the last pivot of the root: in every V_k, or in the root's P
    fx.recomplete(_dev(bad), want_fstar=False)
    assert fx.status() == 3
    # a failing pivot in the last column of the first supernode
    bad = x.copy()
    col = int(sym.supernodes()[0][1]) - 1
    bad[cp[col]] = -1.0
    f.refactor(_dev(bad))
    rc, _, c = f.error_detail()
    assert rc == 2 and c == col
