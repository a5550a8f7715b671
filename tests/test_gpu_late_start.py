"""Solves while other streams hold part of the SMs: the CTAs of a cooperative
launch then start at different times, and each barrier of a solve has to count
from zero in every one of them, however late it starts.  Single, mixed-precision,
lockstep and adjoint solves give the results and iteration counts they give
alone."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1601_03432_gb300 import Grid, inputs
from paper_1601_03432_gb300._binding import FLAG_ADJOINT


@pytest.fixture(scope="module")
def built():
    from paper_1601_03432_gb300.build import build
    build()
    assert torch.cuda.is_available()


# grids of one CTA per SM, of fewer CTAs than SMs, and with strips (two more barriers)
@pytest.mark.parametrize("mx,my,n", [(20, 18, 6), (9, 7, 8), (32, 32, 4)])
@pytest.mark.parametrize("precision,nrhs", [(0, 1), (1, 1), (0, 3), (1, 3)])
def test_solves_beside_other_streams(built, mx, my, n, precision, nrhs):
    g = Grid(mx, my, n)
    g.factor(precision=precision, flags=FLAG_ADJOINT if precision == 0 else 0)
    x, y = g.node_coords()
    f = torch.stack([torch.as_tensor(inputs.fourier_rhs(x, y, seed=90 + k)[0], device="cuda") for k in range(nrhs)])
    alone, beside = torch.empty_like(f), torch.empty_like(f)
    want = g.solve(f, alone, nrhs=nrhs)
    # FP64 products whose CTAs hold their SMs for about a millisecond each,
    # fewer of them than SMs or more
    side = torch.cuda.Stream()
    mats = [torch.randn(s, s, dtype=torch.float64, device="cuda") for s in (512, 768, 1536)]
    torch.cuda.synchronize()
    for rep in range(6):
        with torch.cuda.stream(side):
            for _ in range(3):
                mats[rep % 3] @ mats[rep % 3]
        got = g.solve(f, beside, nrhs=nrhs)
        if precision == 0 and nrhs == 1:
            gf = torch.empty_like(f[0])
            g.solve_adjoint(f[0].contiguous(), gf)
        # both runs stop at the solve's tolerance, 1e-10 of |P b_S|; the order of their
        # atomic sums differs
        assert (beside - alone).norm() <= 1e-8 * alone.norm()
        for a, b in zip(got, want):
            assert a["converged"] == 1 and abs(a["iterations"] - b["iterations"]) <= (1 if precision == 0 else 3)
    torch.cuda.synchronize()
