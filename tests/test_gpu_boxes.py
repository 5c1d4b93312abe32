"""Passes over boxes of quads and warps with shared edges on rows that do not
fill them: the colour-split finest level against the cell-ordered kernels bit
for bit, the FP32 operator product through the mixed solve, and the solution
update on a vector aligned to its type only."""
import numpy as np
import pytest
import torch

from paper_2505_17287_gb300 import ibm, synth

pytestmark = pytest.mark.gpu


def _case(nx, ny, nz):
    # cells of about one width (a strongly anisotropic grid converges slowly)
    h = 0.09
    x, y, z = (h * (np.arange(n + 1) - 0.5 * n) for n in (nx, ny, nz))
    # widths that grow along x: unequal metrics in every quad
    x = x + 0.1 * x * x / x[-1]
    if nz == 1:
        v, e = synth.ellipse_polyline(0.5, 0.3, 0.4, 200)
        return synth.Case("ellipse", 2, x, y, np.array([0.0, 1.0]), v, e, 100.0, 2e-3, 1)
    v, e = synth.icosphere(2, 0.27)
    return synth.Case("sphere", 3, x, y, z, v, e, 100.0, 2e-3, 1)


def _solver(case, **opts):
    s = ibm.Solver(case, **({"precision": opts["precision"]} if "precision" in opts else {}))
    s.set_opts(**opts)
    s.set_body(case.verts, case.elems)
    s.classify()
    return s


# quads per packed row 3, 5, 9 and 30 and 31 quads to a warp; rows off the boxes' 8, 4 and 32
SHAPES = [(24, 17, 13), (40, 25, 30), (72, 33, 11), (240, 24, 10), (248, 26, 9), (104, 65, 1), (136, 33, 1)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_split_passes_equal_cell_ordered(shape):
    case = _case(*shape)
    out = []
    for fs in (1, 0):
        s = _solver(case, precision=ibm.IBM_MIXED, fine_split=fs, poisson_hist=0)
        assert s.step(2)["status"] == ibm.IBM_OK
        out.append((s.get("u"), s.get("p")))
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


# rows of a multiple of four cells take the box form of the FP32 product, 42 the general one
@pytest.mark.parametrize("shape", SHAPES + [(44, 17, 13), (42, 17, 13)], ids=lambda s: "x".join(map(str, s)))
def test_mixed_solve_equals_fp64(shape):
    case = _case(*shape)
    rng = np.random.default_rng(3)
    res = {}
    for prec in (ibm.IBM_FP64, ibm.IBM_MIXED):
        s = _solver(case, precision=prec, max_outer=400)
        rhs = torch.from_numpy(rng.uniform(-1, 1, s.N) if not res else res["rhs"]).cuda()
        phi = torch.zeros_like(rhs)
        st = s.poisson_solve(rhs, phi, rtol=1e-12, maxit=400)
        assert st["status"] == ibm.IBM_OK, st
        res.setdefault("rhs", rhs.cpu().numpy())
        res[prec] = (phi.cpu().numpy(), st)
        s.close()
    a, b = res[ibm.IBM_FP64], res[ibm.IBM_MIXED]
    # two solutions with residual 1e-12 of the right-hand side, condition below 1e5
    assert np.abs(a[0] - b[0]).max() <= 1e-7 * np.abs(a[0]).max()
    # a wrong FP32 product would be paid in refinements: each gains 1e-4 or so
    assert b[1]["outer_iters"] <= 2 * a[1]["outer_iters"] + 8, (a[1], b[1])


def test_solution_update_on_an_odd_address():
    case = _case(40, 25, 30)
    s = _solver(case, precision=ibm.IBM_FP64)
    rng = np.random.default_rng(5)
    rhs = torch.from_numpy(rng.uniform(-1, 1, s.N)).cuda()
    out = []
    for off in (0, 1):
        buf = torch.zeros(s.N + 1, dtype=torch.float64, device="cuda")
        phi = buf[off:off + s.N]
        assert s.poisson_solve(rhs, phi, rtol=1e-12, maxit=200)["status"] == ibm.IBM_OK
        out.append(phi.cpu().numpy())
    assert np.array_equal(out[0], out[1])
    s.close()


# coarse rows of a multiple of the access width and not, planes 1 and odd
@pytest.mark.parametrize("precision", [ibm.IBM_FP64, ibm.IBM_MIXED])
@pytest.mark.parametrize("shape", [(104, 70, 34), (84, 61, 47), (90, 66, 38), (300, 129, 1), (328, 130, 1)],
                         ids=lambda s: "x".join(map(str, s)))
def test_restriction_by_columns_equals_the_tail(shape, precision):
    """The restriction's column walk against the tail's cell-by-cell one."""
    case = _case(*shape)
    out = []
    for tail in (0, 1 << 20):
        s = _solver(case, precision=precision, tail_cells=tail, poisson_hist=0)
        assert s.step(2)["status"] == ibm.IBM_OK
        out.append((s.get("u"), s.get("p")))
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
