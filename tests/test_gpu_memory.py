"""Device memory of a factored grid: the dense coarse inverse is held once,
whatever d is modulo the 16 bytes that the kernels read it by."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1601_03432_gb300 import Grid
from paper_1601_03432_gb300._binding import FLAG_ADJOINT


def used_by_factor(mx, my, n, flags):
    g = Grid(mx, my, n)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    g.factor(flags=flags)
    torch.cuda.synchronize()
    used = free0 - torch.cuda.mem_get_info()[0]
    d = g.d
    del g
    return d, used


@pytest.mark.parametrize("flags", [0, FLAG_ADJOINT])
def test_coarse_inverse_is_held_once(flags):
    used_by_factor(32, 32, 4, flags)  # the context and the kernels' code
    d0, used0 = used_by_factor(32, 32, 4, flags)
    assert d0 % 4 == 0
    for mx, my in ((33, 31), (35, 30)):
        d, used = used_by_factor(mx, my, 4, flags)
        assert d % 4 != 0 and abs(d / d0 - 1) < 0.05
        # 31 MB per dense inverse; the rest of the factors, 14 MB, follows the grid's
        # size and the strips' height
        assert abs(used - used0) < 0.6 * 8 * d * d, (d, used, used0)


def test_failed_allocation_leaves_nothing_behind():
    """A factor step that finds no device memory reports ENOMEM, and the next solve of
    another handle on the same device is unaffected."""
    from paper_1601_03432_gb300 import SmpmError, inputs
    from paper_1601_03432_gb300 import _binding as B
    g, big = Grid(6, 5, 6), Grid(40, 40, 12)
    g.factor(tol=1e-11)
    f = torch.as_tensor(inputs.white_noise(g.r, 1), device="cuda")
    u, u2 = torch.empty_like(f), torch.empty_like(f)
    g.solve(f, u)
    torch.cuda.synchronize()
    room = 64 << 20  # the factors of the larger grid take 78 MB for one d x d matrix alone
    hold = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(SmpmError) as ei:
            big.factor(tol=1e-11)
        assert ei.value.status == B.SMPM_ENOMEM
        assert g.solve(f, u2)[0]["converged"] == 1
    finally:
        del hold
        torch.cuda.empty_cache()
    assert (u2 - u).norm() <= 1e-9 * u.norm()
