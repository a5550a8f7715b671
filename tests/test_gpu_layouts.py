"""The solve kernels' shapes: the layout flags of the factor step change the shape
they name and not the solution, and teams of every size (one, two, four and eight
warps per block or element, three-stage block solves) meet the single solve of
the same grid (whole block inverses)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1601_03432_gb300 import Batch, Grid, inputs
from paper_1601_03432_gb300 import _binding as B

BOUND = {0: 1e-9, 1: 1e-8}  # both solves stop at 1e-11 of |P b_S|


@pytest.fixture(scope="module")
def built():
    from paper_1601_03432_gb300.build import build
    build()
    assert torch.cuda.is_available()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def layout(g, precision):
    names = ("ctas", "warps", "res_T", "res_G", "table", "basis", "whole", "strips", "fp64")
    return dict(zip(names, (int(v) for v in g.host_factor("solve_layout32" if precision else "solve_layout"))))


@pytest.mark.parametrize("mx,my,n", [(5, 4, 7), (20, 18, 5), (3, 3, 32)])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_layout_flags(built, mx, my, n, precision):
    g = Grid(mx, my, n)
    f = dev(inputs.white_noise(g.r, 11))
    out, shape = {}, {}
    for flags in (0, B.FLAG_WARP_ELEMS, B.FLAG_STREAM_MATRICES, B.FLAG_NO_SMEM_RESIDENCY):
        g.factor(tol=1e-11, precision=precision, flags=flags)
        shape[flags] = layout(g, precision)
        u = torch.empty_like(f)
        assert g.solve(f, u)[0]["converged"] == 1
        out[flags] = u
    assert shape[0]["warps"] > 1 and shape[0]["res_T"] > 0
    assert shape[B.FLAG_WARP_ELEMS]["warps"] == 1
    s = shape[B.FLAG_STREAM_MATRICES]
    assert s["res_T"] == s["res_G"] == 0 and s["table"] == 1
    s = shape[B.FLAG_NO_SMEM_RESIDENCY]
    assert s["res_T"] == s["res_G"] == s["table"] == s["basis"] == 0
    for u in out.values():
        assert (u - out[0]).norm() <= BOUND[precision] * out[0].norm()


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("team", [152, 38, 19, 12, 4])
def test_team_sizes_meet_the_single_solve(built, precision, team):
    """76 black blocks: 1, 2, 4, 7 and 19 per CTA, so 8, 4, 2, 1 and 1 warps each."""
    g = Grid(19, 8, 7)
    g.factor(tol=1e-11, precision=precision)
    assert layout(g, precision)["whole"] == 1
    f = dev(inputs.white_noise(g.r, 13))
    u, ub = torch.empty_like(f), torch.empty_like(f)
    one = g.solve(f, u)[0]
    b = Batch([g], [1], team_size=team)
    rep = b.solve(f, ub)[0]
    b.close()
    assert (u - ub).norm() <= BOUND[precision] * u.norm()
    assert abs(rep["iterations"] - one["iterations"]) <= (1 if precision == 0 else 3)


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_lockstep_groups_with_long_cycles(built, precision):
    """Restart 190 with 14 columns of the largest order: the least squares' state leaves
    no room for a group's digits, so the columns run in smaller groups."""
    g = Grid(3, 2, 32)
    g.factor(tol=1e-11, precision=precision, restart=190, maxit=400)
    f = dev(np.stack([inputs.white_noise(g.r, 60 + k) for k in range(14)]))
    u, one = torch.empty_like(f), torch.empty_like(f[0])
    reps = g.solve(f, u, nrhs=14)
    for k in range(14):
        assert reps[k]["converged"] == 1
        if k % 4 == 0:
            g.solve(f[k].contiguous(), one)
            assert (one - u[k]).norm() <= BOUND[precision] * one.norm()
