"""Device memory of a served case: what it reports to hold, what the budget is
charged, the same result where its block of memory is too small, and the
footprint estimate against the bytes that a case allocates."""
import dataclasses

import numpy as np
import pytest

from paper_2505_17287_gb300 import ibm, synth

pytestmark = pytest.mark.gpu


def _case(extra):
    """A small cylinder whose mesh has `extra` vertices that no segment uses
    (24 bytes each on the device and 16 more during the classification; the
    footprint estimate does not know them)."""
    c = synth.cylinder_case(96, 48, 128, nsteps=3)
    v = np.asarray(c.verts)
    return dataclasses.replace(c, verts=np.vstack([v, np.zeros((extra, v.shape[1]))]))


def _serve(case):
    srv = ibm.Server(max_slots=1)
    r = srv.wait(srv.submit(case, outputs=True))
    st = srv.stats()
    srv.close()
    assert r["status"] == ibm.IBM_OK, r["error"]
    return r, st


# none; the block nearly filled by the vertices, the rest beside it; the
# vertices alone larger than the block
@pytest.mark.parametrize("extra", [0, 2_400_000, 6_000_000])
def test_held_bytes_and_results_past_the_estimate(extra):
    ref, _ = _serve(_case(0))
    r, st = _serve(_case(extra))
    # (vertices at the origin, inside the body's box: the same geometry)
    for n in ref["outputs"]:
        assert np.array_equal(ref["outputs"][n], r["outputs"][n]), n
    est = r["bytes_estimate"]
    if extra == 0:
        # the case holds its whole estimate, and no more
        assert r["bytes_peak"] == est and st["peak_admitted_bytes"] == est
    else:
        # the excess beside the block is reported and charged
        assert r["bytes_peak"] >= est + 16 * extra
        assert st["peak_admitted_bytes"] >= r["bytes_peak"]
    assert st["admitted_bytes"] == 0


def _spheres8(n):
    """Eight spheres that fill the box: more ghost cells than any one body."""
    at = [(0.4, (x, y, z)) for x in (-0.5, 0.5) for y in (-0.5, 0.5) for z in (-0.5, 0.5)]
    c = synth.sphere_case(n=n)
    vs, ts, base = [], [], 0
    for r, o in at:
        v, t = synth.icosphere(3, r)
        vs.append(v + np.array(o))
        ts.append(t + base)
        base += len(v)
    return dataclasses.replace(c, verts=np.vstack(vs), elems=np.vstack(ts).astype(np.int32))


# small grids (what does not scale with the cells), a large single body, many
@pytest.mark.parametrize("precision", [ibm.IBM_FP64, ibm.IBM_MIXED])
@pytest.mark.parametrize("case", [synth.cylinder_case(96, 48, 128), synth.cylinder_case(512, 256, 512),
                                  synth.sphere_case(n=32, radius=0.8), synth.sphere_case(n=64, radius=0.85, level=4),
                                  _spheres8(64)],
                         ids=["cyl96", "cyl512", "sphere32", "sphere64", "spheres64"])
def test_estimate_counts_what_a_case_allocates(case, precision, monkeypatch):
    """The counted terms alone cover the allocations: the estimate's quarter
    and its 56 MiB on top stay margin."""
    import torch
    alloc, delete = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete
    live, top = {}, [0, 0]

    def count(nbytes, dev, stream):
        p = alloc(nbytes, dev, stream)
        live[p] = nbytes
        top[0] += nbytes
        top[1] = max(top)
        return p

    def uncount(p):
        top[0] -= live.pop(p)
        delete(p)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", count)
    monkeypatch.setattr(torch.cuda, "caching_allocator_delete", uncount)
    s = ibm.Solver(case, precision=precision, stream=torch.cuda.Stream())
    s.set_opts(precision=precision)
    s.set_body(case.verts, case.elems)
    s.classify()
    r = s.step(2)
    s.close()
    assert r["status"] == ibm.IBM_OK and top[0] == 0, (r, top)
    nx, ny = len(case.xf) - 1, len(case.yf) - 1
    nz = len(case.zf) - 1 if case.ndim == 3 else 1
    est = ibm.ibm_case_bytes(case.ndim, nx, ny, nz, precision, len(case.elems))
    assert est >= 1.25 * top[1] + (56 << 20), (est, top[1])
