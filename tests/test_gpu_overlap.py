"""Overlapped launches (programmatic dependent launch on a stream of one's
own): the bits of plain launches (the legacy default stream), on grids whose
kernels are all overlapped, some and few, and the same bits in every run of
the captured step."""
import numpy as np
import pytest
import torch

from paper_2505_17287_gb300 import ibm, synth

pytestmark = pytest.mark.gpu


def _case(name):
    if name == "small2d":
        return synth.cylinder_case(96, 50, 128, dt=0.01)
    if name == "large2d":
        return synth.cylinder_case(760, 384, 256, dt=0.005)
    return synth.sphere_case(n=76, radius=0.3)


def _run(case, precision, stream, graph, steps=3):
    s = ibm.Solver(case, precision=precision, stream=stream)
    s.set_opts(precision=precision, graph=graph)
    s.set_body(case.verts, case.elems)
    s.classify()
    r = s.step(steps)
    assert r["status"] == ibm.IBM_OK, r
    out = {k: s.get(k) for k in (("u", "v", "w", "p") if case.ndim == 3 else ("u", "v", "p"))}
    s.close()
    return out


@pytest.mark.parametrize("precision", [ibm.IBM_FP64, ibm.IBM_MIXED])
@pytest.mark.parametrize("name", ["small2d", "large2d", "sphere"])
def test_overlapped_launches_give_the_bits_of_plain_ones(name, precision):
    case = _case(name)
    a = _run(case, precision, None, 1)
    for graph in (0, 1):
        b = _run(case, precision, torch.cuda.Stream(), graph)
        for k in a:
            assert np.array_equal(a[k], b[k]), (graph, k)


@pytest.mark.parametrize("precision", [ibm.IBM_FP64, ibm.IBM_MIXED])
def test_captured_steps_repeat_bit_for_bit(precision):
    case = _case("small2d")
    ref = _run(case, precision, torch.cuda.Stream(), 2)
    for _ in range(4):
        b = _run(case, precision, torch.cuda.Stream(), 2)
        assert all(np.array_equal(ref[k], b[k]) for k in ref)


@pytest.mark.parametrize("precision", [ibm.IBM_FP64, ibm.IBM_MIXED])
def test_graphs_kept_over_classifications_and_options(precision):
    """V-cycle graphs captured for one body position and option set, used
    again after a move, a new classification and a changed relaxation factor:
    the bits of a context that launches every kernel."""
    case = synth.wing_case(112, 96, 98, n_chord=30, n_span=10)   # above 2^20 cells: a graph per Krylov vector
    verts = np.array(case.verts)
    verts[:, 1] += 0.03
    outs = []
    for graph in (0, 1):
        s = ibm.Solver(case, precision=precision, stream=torch.cuda.Stream())
        s.set_opts(precision=precision, graph=graph)
        s.set_body(case.verts, case.elems)
        s.classify()
        s.step(1)
        s.move_body(verts, U=(0.0, 0.1, 0.0))
        s.step(1)
        s.set_opts(smooth_omega=1.1)
        s.step(1)
        u = s.get("u")
        s.classify()
        s.step(1)
        outs.append((u, s.get("p")))
        s.close()
    assert all(np.array_equal(a, b) for a, b in zip(*outs))
