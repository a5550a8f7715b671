"""Products in digits are cut relative to the largest entry of their vector, so
what has no part in a result must not set that scale, and small results keep
their own accuracy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1601_03432_gb300 import Batch, Grid, inputs


@pytest.fixture(scope="module")
def built():
    from paper_1601_03432_gb300.build import build
    build()
    assert torch.cuda.is_available()


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_batch_groups_are_independent_of_what_ran_before(built, precision):
    """Two grids of different shapes, several columns each, one team: the second
    problem's right-hand sides are 1e-12 of the first's, and restarts apply S to
    its small iterates in the workspace that the first one used.  Each column
    meets the single solve of the same right-hand side."""
    sizes = [(11, 9, 7), (6, 10, 5)]
    grids = [Grid(*s) for s in sizes]
    for g in grids:
        g.factor(tol=1e-11, precision=precision, restart=7, maxit=400)
    R, scale = 5, (1.0, 1e-12)
    fs = [scale[i] * np.stack([inputs.white_noise(g.r, 31 * i + k) for k in range(R)]) for i, g in enumerate(grids)]
    b = Batch(grids, [R, R], team_size=152)
    u = torch.zeros(sum(f.size for f in fs), dtype=torch.float64, device="cuda")
    f = dev(np.concatenate([f.ravel() for f in fs]))
    for _ in range(2):  # the second call starts on the workspace of the first
        reps = b.solve(f, u)
        assert all(r["converged"] == 1 for r in reps)
        out = torch.split(u, [x.size for x in fs])
        for i, g in enumerate(grids):
            one = torch.empty(g.r, dtype=torch.float64, device="cuda")
            for k in range(R):
                ref = g.solve(dev(fs[i][k]), one)[0]
                got = out[i].view(R, g.r)[k]
                # both stop at 1e-11 of |P b_S|
                assert (got - one).norm() <= 1e-8 * one.norm(), (i, k)
                assert abs(reps[i * R + k]["iterations"] - ref["iterations"]) <= (1 + ref["iterations"] // 7
                                                                                   if precision == 0 else 12)
    b.close()
