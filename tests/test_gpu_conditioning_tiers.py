"""Condition number 1e6 where the arithmetic depends on the length of a run or on
the width of a front: runs cut into segments (their windows are composed through
the segments' transfer matrices), grouped fronts of several panels, and thin fronts
with long ancestor sets.  Inputs, references and bounds are those of
test_gpu_conditioning; the oracle's own error on these patterns, against the inverse
of the planted factor, is 4e-11 (inverse) and 2e-10 (inverse Hessian) at most."""
import pytest

import test_gpu_conditioning as C
import workloads as W
from test_gpu_grouped_fronts import _cliques
from tests.helpers import lib

pytestmark = pytest.mark.gpu

SEGMENTS = {"band8": (900, 8), "band24": (700, 24), "band61": (500, 61)}
GROUPED = {"panels3": (70, 60, 3), "panels2": (40, 100, 2), "thin_long": (12, 330, 2)}


@pytest.mark.parametrize("name", list(SEGMENTS))
def test_segmented_runs(name, monkeypatch):
    B = lib()
    monkeypatch.setitem(C.CASES, name, (lambda: W.band(*SEGMENTS[name]), {}))
    C.test_condition_1e6_all_operations(name)
    # the runs are long enough for segments: two launches per inner segment
    sym = B.Symbolic(*W.band(*SEGMENTS[name]))
    import numpy as np
    f = sym.factor(C.dev(W.diag_dominant(sym.n, sym.colptr, sym.rowind, np.random.default_rng(0))))
    l0 = B.chd_kernel_launches()
    f.gradient()
    assert B.chd_kernel_launches() - l0 >= 12


@pytest.mark.parametrize("name", list(GROUPED))
def test_grouped_fronts(name, monkeypatch):
    monkeypatch.setitem(C.CASES, name, (lambda: _cliques(*GROUPED[name]), {}))
    C.test_condition_1e6_all_operations(name)
