"""Completion of dense fronts of one to four columns whose ancestor set is so
long that the back substitution of one launch no longer holds the rows in
shared memory: the longest sets it takes, the next longer ones and the ones
around 40 KiB of rows.  Reference: P(X-hat^{-1}) = S on a dense matrix."""
import numpy as np
import pytest

import workloads as W
from test_gpu_grouped_fronts import _cliques, _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,a", [(4, 1263), (4, 1264), (4, 1279), (4, 1280), (3, 1684), (3, 1685), (3, 1706), (2, 2527),
                                 (2, 2528), (2, 2560), (1, 5056)])
def test_long_ancestor_sets(n, a):
    import torch
    from paper_1203_2742_gb300 import binding as B
    sym = B.Symbolic(*_cliques(n, a, 1))
    sp, _, rp, _ = sym.supernodes()
    assert (sp[1] - sp[0], rp[1] - rp[0]) == (n, n + a)
    N, cp, ri = sym.n, sym.colptr, sym.rowind
    rng = np.random.default_rng(a)
    s = _dev(W.projected_gram(N, cp, ri, rng.standard_normal((N, 12)), 0.7))
    fx, fstar = sym.complete(s)
    assert fx.status() == 0
    r = torch.as_tensor(np.asarray(ri, np.int64), device="cuda")
    c = torch.as_tensor(np.repeat(np.arange(N), np.diff(cp)), device="cuda")
    X = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    x = fx.product()
    X[r, c] = x
    X[c, r] = x
    L = torch.linalg.cholesky(X)
    want = 2.0 * float(torch.log(torch.diagonal(L)).sum()) - N
    assert abs(fstar - want) <= 1e-9 * max(1.0, abs(want))
    # the cliques of S have condition up to (N + 12) / 0.7 = 7300, two solves: 10 eps cond = 2e-11
    got = torch.cholesky_inverse(L)[r, c]
    assert float((got - s).norm() / s.norm()) < 1e-9
