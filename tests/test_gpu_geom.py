"""Classification and body intercepts with the triangle prefilter and the
single-precision bounds of the intercept search: the oracle's bits on meshes of
several batches, with ragged grids, far from the origin and at small scale."""
import numpy as np
import pytest

from oracle import geom
from paper_2505_17287_gb300 import ibm, synth

pytestmark = pytest.mark.gpu


def _cases():
    out = {}
    # 20,480 triangles, more than one run of 128 columns, an odd remainder
    v, e = synth.icosphere(5, 0.31, (0.013, -0.021, 0.017))
    out["sphere_fine"] = (3, np.linspace(-1, 1, 142), np.linspace(-0.9, 0.9, 30), np.linspace(-0.8, 0.8, 28), v, e)
    # few triangles (a batch is not full); the largest distance bounds
    v, e = synth.box((-0.31, -0.27, -0.22), (0.29, 0.33, 0.24))
    out["box"] = (3, np.linspace(-1, 1, 24), np.linspace(-1, 1, 27), np.linspace(-1, 1, 22), v, e)
    w = synth.wing_case(72, 56, 40, n_chord=60, n_span=20)
    out["wing"] = (3, w.xf, w.yf, w.zf, w.verts, w.elems)
    # coordinates far larger than the distances: the bounds' rounding margin
    s = np.array([1000.0, -2500.0, 400.0])
    out["wing_far"] = (3, w.xf + s[0], w.yf + s[1], w.zf + s[2], w.verts + s, w.elems)
    out["wing_small"] = (3, w.xf * 1e-6, w.yf * 1e-6, w.zf * 1e-6, w.verts * 1e-6, w.elems)
    v, e = synth.ellipse_polyline(0.7, 0.2, 0.5, 700)
    out["ellipse"] = (2, np.linspace(-4, 6, 131), np.linspace(-3, 3, 77), np.array([0.0, 1.0]), v, e)
    out["ellipse_far"] = (2, np.linspace(-4, 6, 131) + 5e4, np.linspace(-3, 3, 77), np.array([0.0, 1.0]),
                          v + np.array([5e4, 0, 0]), e)
    return out


CASES = _cases()


@pytest.mark.parametrize("name", list(CASES))
def test_tables_equal_the_oracle(name):
    nd, xf, yf, zf, v, e = CASES[name]
    case = synth.Case(name, nd, xf, yf, zf, v, e, 100.0, 1e-3, 1)
    s = ibm.Solver(case)
    s.set_body(v, e)
    s.classify()
    got, ref = s.tables(), geom.body_tables(nd, xf, yf, zf, v, e)
    s.close()
    assert np.array_equal(got["type"], ref["type"]) and np.array_equal(got["gidx"], ref["gidx"])
    assert got["gidx"].size > 0
    for k in ("bi", "nrm", "ip", "dist", "kind", "sidx", "wv", "wp"):
        assert np.array_equal(got[k], ref[k]), k
