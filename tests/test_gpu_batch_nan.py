"""A NaN or Inf in one right-hand side of a batch is reported as ENAN, by single
columns and lockstep groups in both precisions, and the next solve is unaffected."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1601_03432_gb300 import Batch, Grid, SmpmError, inputs
from paper_1601_03432_gb300 import _binding as B


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_batch_reports_enan(precision, nrhs, bad):
    grids = [Grid(4, 3, 6), Grid(5, 4, 5)]
    for g in grids:
        g.factor(tol=1e-11, precision=precision)
    b = Batch(grids, [nrhs, nrhs], team_size=8)
    f = np.concatenate([inputs.white_noise(g.r, 10 * i + k) for i, g in enumerate(grids) for k in range(nrhs)])
    fd = torch.as_tensor(f, device="cuda")
    u = torch.zeros_like(fd)
    poisoned = fd.clone()
    poisoned[grids[0].r * nrhs + 7] = bad  # the second problem's first column
    with pytest.raises(SmpmError) as ei:
        b.solve(poisoned, u)
    assert ei.value.status == B.SMPM_ENAN
    assert all(r["converged"] == 1 for r in b.solve(fd, u))
    assert torch.isfinite(u).all()
    b.close()
