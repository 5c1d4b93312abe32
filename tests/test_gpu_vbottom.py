"""The V-cycle's coarse levels in one shared-memory launch (k_vbottom) and the
coarsest level's solution operator: the same bits as the persistent tail,
whose passes go through global memory, over ragged extents, one block to
sixteen, both precisions and the smoother variants; grids that are their own
coarsest level; a sweep count changed between steps."""
import numpy as np
import pytest
import torch

from oracle import flow, geom
from paper_2505_17287_gb300 import ibm, synth

pytestmark = pytest.mark.gpu

ALL = 1 << 30   # every level below the finest in the tail


def _case(nx, ny, nz):
    if nz == 1:
        v, e = synth.ellipse_polyline(0.7, 0.5, 0.4, 128)
        return synth.Case("c", 2, synth.uniform_faces(-4.0, 6.0, nx), synth.stretched_faces(-4.0, 4.0, ny, -1, 1, 1.01),
                          np.array([0.0, 1.0]), v, e, 100.0, 0.01, 2)
    v, e = synth.icosphere(2, 0.5, (0.03, 0.02, 0.01))
    return synth.Case("c", 3, synth.uniform_faces(-2.0, 3.0, nx), synth.uniform_faces(-2.0, 2.0, ny),
                      synth.uniform_faces(-2.0, 2.0, nz), v, e, 100.0, 0.01, 2)


def _run(case, precision, steps=2, stream=None, **opts):
    s = ibm.Solver(case, precision=precision, stream=stream)
    s.set_opts(precision=precision, **opts)
    s.set_body(case.verts, case.elems)
    s.classify()
    r = s.step(steps)
    assert r["status"] == ibm.IBM_OK, r
    out = {k: s.get(k) for k in (("u", "v", "w", "p") if case.ndim == 3 else ("u", "v", "p"))}
    s.close()
    return out


# one block (its largest level and one cell more), several blocks with a
# shorter last one, odd rows, and levels too large for the cluster above them
@pytest.mark.parametrize("precision", [ibm.IBM_FP64, ibm.IBM_MIXED])
@pytest.mark.parametrize("shape,opts", [((128, 128, 1), {}), ((130, 127, 1), {"smooth_omega": 1.1}), ((257, 203, 1), {}),
                                        ((601, 301, 1), {"nu_coarse": 1}), ((40, 37, 1), {}), ((33, 29, 31), {}),
                                        ((65, 57, 71), {"smooth_omega": 1.1}), ((96, 80, 99), {"nu_coarse": 2})])
def test_bottom_equals_tail(precision, shape, opts):
    case = _case(*shape)
    a = _run(case, precision, **opts)
    b = _run(case, precision, tail_cells=ALL, **opts)
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("precision", [ibm.IBM_FP64, ibm.IBM_MIXED])
@pytest.mark.parametrize("n", [7, 8, 9, 13, 20])
def test_tiny_grids_match_oracle(precision, n):
    """At most 64 cells: the grid is its own coarsest level; then two levels."""
    v, e = synth.circle_polyline(64, 0.4, 0.013, 0.007)
    f = synth.uniform_faces(-1.0, 1.0, n)
    case = synth.Case("tiny", 2, f, f.copy(), np.array([0.0, 1.0]), v, e, 50.0, 0.02, 2)
    T = geom.body_tables(2, case.xf, case.yf, case.zf, case.verts, case.elems)
    g = flow.Grid(2, case.xf, case.yf, case.zf)
    ost = flow.run(g, T["type"], T, 2, case.Re, case.dt)
    got = _run(case, precision, rtol=1e-13, helm_rtol=1e-14)
    p_ref = flow.normalise(g, T["type"], ost.p)
    for k, ref in (("u", ost.u[0]), ("v", ost.u[1]), ("p", p_ref)):
        assert np.linalg.norm(got[k] - ref) <= 1e-8 * np.linalg.norm(ref), k


@pytest.mark.parametrize("graph", [1, 2])
def test_changed_sweep_count_takes_effect(graph):
    """coarse_sweeps changed and changed back between steps (captured step
    graphs are reused): the bits of a run without the detour."""
    case = _case(96, 64, 1)
    outs = []
    for detour in (False, True):
        s = ibm.Solver(case, precision=ibm.IBM_MIXED, stream=torch.cuda.Stream())
        s.set_opts(precision=ibm.IBM_MIXED, graph=graph)
        s.set_body(case.verts, case.elems)
        s.classify()
        s.step(2)
        st = s.get_state()
        if detour:
            s.set_opts(coarse_sweeps=1)
            s.step(2)
            s.set_opts(coarse_sweeps=32)
            s.set_state(st)
        s.step(2)
        outs.append(s.get("p"))
        s.close()
    assert np.array_equal(outs[0], outs[1])
