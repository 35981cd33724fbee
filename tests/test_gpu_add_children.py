"""Fronts of more than 64 children in the grouped tier: their blocks are added two at
a time without barriers, in every pass, thin and wide fronts, with and without
ancestors, pruned arguments included; and one with 64, which takes them one by one."""
import numpy as np
import pytest

import workloads as W
from test_gpu_grouped_fronts import _check, _cliques

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,a,kids,extra", [(3, 20, 200, 0), (3, 12, 64, 0), (3, 12, 65, 0), (5, 40, 130, 5), (2, 61, 97, 3)])
def test_root(n, a, kids, extra):
    _check(_cliques(n, a, kids, extra), seed=kids)


@pytest.mark.parametrize("n,own,top,kids", [(3, 10, 40, 100), (2, 24, 70, 90), (3, 45, 33, 70)])
def test_front_with_ancestors(n, own, top, kids):
    """`kids` leaves under a front of `own` columns, which has `top` ancestors."""
    rng = np.random.default_rng(own)
    first = kids * n
    N = first + own + top
    rows, cols = [], []
    for k in range(kids):
        mine = np.arange(k * n, (k + 1) * n)
        J = np.concatenate([mine, [first], np.sort(rng.choice(np.arange(first + 1, N), (own + top) // 2, replace=False))])
        r, c = np.meshgrid(J, mine, indexing="ij")
        rows.append(r.ravel()); cols.append(c.ravel())
    rest = np.arange(first, N)
    r, c = np.meshgrid(rest, rest, indexing="ij")
    r, c = r.ravel(), c.ravel()
    keep = ~((c < first + own) & (r == N - 1))  # the last vertex belongs to the ancestors only
    rows.append(r[keep]); cols.append(c[keep])
    r, c = np.concatenate(rows), np.concatenate(cols)
    keep = (r >= c) & ~((r == N - 1) & (c < first + own))
    _check(W.lower_csc_from_pairs(N, r[keep], c[keep]), seed=kids)
