"""Grouped fronts whose last tile has up to 16 rows or more: quarters of the update
tiles that hold nothing are left out, in the thin and in the wide form."""
import pytest

from test_gpu_grouped_fronts import _check, _cliques

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,a", [(5, 16), (5, 17), (12, 48), (12, 49), (16, 32), (20, 16), (20, 17), (20, 48), (20, 49),
                                 (40, 80), (40, 81)])
def test_ragged_tiles(n, a):
    _check(_cliques(n, a, 2), seed=100 * n + a)
