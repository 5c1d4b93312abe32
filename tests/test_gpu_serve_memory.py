"""Device memory of a served case: what it reports to hold, what the budget is
charged, and the same result where its block of memory is too small."""
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
