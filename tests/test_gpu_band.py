"""The near-body band sweeps in their three forms (one block, a cluster, one
launch per sweep), which the band's size chooses: the pressure is the one that
the solver finds without them, in fewer iterations."""
import numpy as np
import pytest
import torch

from paper_2505_17287_gb300 import ibm, synth

pytestmark = pytest.mark.gpu


def _solve(case, precision, rhs, **opts):
    s = ibm.Solver(case, precision=precision, stream=torch.cuda.Stream())
    s.set_opts(precision=precision, max_outer=1000, **opts)
    s.set_body(case.verts, case.elems)
    s.classify()
    phi = torch.zeros_like(rhs)
    torch.cuda.synchronize()
    r = s.poisson_solve(rhs, phi, rtol=1e-12)
    assert r["status"] == ibm.IBM_OK and r["rel_residual"] <= 1e-12, r
    s.close()
    return phi.cpu().numpy(), r["outer_iters"]


# cells of the band, from about 60 to 60,000: one block with one, two and four
# rows a thread; clusters of two to sixteen blocks; too large for a cluster
@pytest.mark.parametrize("precision", [ibm.IBM_FP64, ibm.IBM_MIXED])
@pytest.mark.parametrize("n,radius", [(0, 0.0), (20, 0.17), (25, 0.25), (31, 0.35), (40, 0.4), (50, 0.5), (64, 0.6), (97, 0.62)])
def test_band_sweeps_keep_the_solution(precision, n, radius):
    case = synth.cylinder_case(192, 96, 128) if n == 0 else synth.sphere_case(n=n, radius=radius, level=3)
    rng = np.random.default_rng(n)
    rhs = torch.from_numpy(rng.uniform(-1, 1, case.ncells)).cuda()
    a, ia = _solve(case, precision, rhs)
    b, ib = _solve(case, precision, rhs, band_sweeps=0)
    assert np.linalg.norm(a - b) <= 1e-8 * np.linalg.norm(b)
    assert ia < ib
    # the same bits again, and one sweep is a band too
    c, ic = _solve(case, precision, rhs)
    assert np.array_equal(a, c) and ic == ia
    d, _ = _solve(case, precision, rhs, band_sweeps=1)
    assert np.linalg.norm(d - b) <= 1e-8 * np.linalg.norm(b)
