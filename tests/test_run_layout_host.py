"""Chain runs on the host: the kernels address the columns of a run from the record
of any one of them, by constant steps through the values and the per-front
regions, and keep two a x a matrices of a segment in its first two fronts."""
import numpy as np
import pytest

import workloads as W
from tests.helpers import lib

CASES = {
    "band1": lambda B: B.Symbolic(*W.band(60, 1)),
    "band8": lambda B: B.Symbolic(*W.band(200, 8)),
    "band64": lambda B: B.Symbolic(*W.band(700, 64)),
    "uneven": lambda B: B.SymbolicBatch([W.band(1300, 24), W.band(40, 5), W.grid2d(14, 14), W.band(90, 33), W.band(30, 24)]),
}


@pytest.mark.parametrize("name", list(CASES))
def test_constant_steps(name):
    sym = CASES[name](lib())
    sp, par, rp, rows = [np.asarray(v) for v in sym.supernodes()]
    f_off, d_off, v_off = [np.asarray(v) for v in sym.offsets()]
    s = sym.schedule()
    cp = np.asarray(sym.colptr)
    runs = int(s["lvl_counts"][0][0] + s["lvl_counts"][0][1])
    assert runs > 0
    for t in range(runs):
        ks = np.asarray(s["task_fronts"])[s["task_ptr"][t]:s["task_ptr"][t + 1]]
        J = int(rp[ks[0] + 1] - rp[ks[0]])
        a = J - 1
        up4 = lambda v: (v + 3) // 4 * 4
        step = np.arange(len(ks))
        assert np.array_equal(ks, ks[0] + step) and np.all(sp[ks + 1] - sp[ks] == 1)
        assert np.array_equal(sp[ks], sp[ks[0]] + step)
        assert np.array_equal(cp[sp[ks]], cp[sp[ks[0]]] + J * step)
        assert np.array_equal(f_off[ks], f_off[ks[0]] + up4(J * J + 2 * J) * step)
        assert np.array_equal(v_off[ks], v_off[ks[0]] + up4(a * a) * step)
        assert np.array_equal(d_off[ks], d_off[ks[0]] + 4 * step)
        for i, k in enumerate(ks):
            assert np.array_equal(rows[rp[k]:rp[k + 1]], sp[k] + np.arange(J)) or i + a >= len(ks)
        assert par[ks[-1]] > ks[-1]  # a run hands over to a parent
        assert a * a <= f_off[ks[0] + 1] - f_off[ks[0]]  # a window fits a front's region
