"""Products in digits are cut relative to the largest entry of their vector, so
what has no part in a result must not set that scale, and small results keep
their own accuracy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1601_03432_gb300 import Batch, Grid, inputs
from paper_1601_03432_gb300 import _binding as B


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


def applied(g, kind, v):
    g.set_apply_kernel(kind)
    y = torch.full_like(v, -7.0)
    (g.apply_schur if v.dtype == torch.float64 else g.apply_schur32)(v, y)
    torch.cuda.synchronize()
    return y.double().cpu().numpy()


# n: part of a tile, a tile and a remainder, whole tiles
@pytest.mark.parametrize("mx,my,n", [(7, 5, 3), (5, 6, 9), (6, 6, 16)])
@pytest.mark.parametrize("big", [1e12, 1e100])
def test_apply_is_blind_to_boundary_slots(built, mx, my, n, big):
    """Large values on physical-boundary slots (T_e's columns there are zero) leave
    every other entry of S v as it is, and stay where they are themselves."""
    g = Grid(mx, my, n)
    g.factor(precision=1)
    face = np.ones((my, mx, 4, n), bool)
    face[:, 0, 0], face[:, -1, 1], face[0, :, 2], face[-1, :, 3] = False, False, False, False
    face = face.ravel()
    v = np.random.default_rng(n).standard_normal(face.size)
    for dtype in (torch.float64, torch.float32):
        b = min(big, 1e30) if dtype == torch.float32 else big
        for kind in (B.APPLY_AUTO, B.APPLY_CLASS, B.APPLY_WARP):
            plain = applied(g, kind, dev(np.where(face, v, 0.0), dtype))
            got = applied(g, kind, dev(np.where(face, v, b * v), dtype))
            assert np.array_equal(got[face], plain[face]), kind
            assert np.array_equal(got[~face], dev(b * v, dtype).double().cpu().numpy()[~face])


def own_bound(T, v, mx, my, n, u):
    """(M + 2) u sum |T_e||v_e|, the error of a chain of M FMAs and the addition to
    v, at the facing slots that the products are pushed to."""
    M, e = 4 * n, np.arange(mx * my)
    own = (M + 2) * u * np.einsum("erk,ek->er", np.abs(T), np.abs(v))
    out = np.zeros_like(own)
    ix, iy = e % mx, e // mx
    for F, (dx, dy) in enumerate(((-1, 0), (1, 0), (0, -1), (0, 1))):
        ok = (0 <= ix + dx) & (ix + dx < mx) & (0 <= iy + dy) & (iy + dy < my)
        f2 = (F ^ 1) * n
        out[(e + dx + mx * dy)[ok], f2:f2 + n] = own[e[ok], F * n:(F + 1) * n]
    return out


def exact_apply(T, v, mx, my, n):
    """S v in extended precision (np.longdouble where it is longer than a double)."""
    L = np.longdouble
    M, e = 4 * n, np.arange(mx * my)
    z = np.einsum("erk,ek->er", T.astype(L), v.astype(L))
    y = v.astype(L).copy()
    ix, iy = e % mx, e // mx
    for F, (dx, dy) in enumerate(((-1, 0), (1, 0), (0, -1), (0, 1))):
        ok = (0 <= ix + dx) & (ix + dx < mx) & (0 <= iy + dy) & (iy + dy < my)
        f2 = (F ^ 1) * n
        y[(e + dx + mx * dy)[ok], f2:f2 + n] += z[e[ok], F * n:(F + 1) * n]
    return y


# square and stretched elements (rows of T_e spanning up to 2^38, where the digits
# no longer hold it), n up to the largest, three k tiles and six and eight
@pytest.mark.parametrize("mx,my,n,Lx", [(4, 5, 5, 1.0), (4, 4, 11, 1.0), (5, 4, 16, 1.0), (4, 4, 24, 1.0), (3, 4, 32, 1.0),
                                        (4, 4, 16, 8.0), (4, 4, 24, 8.0)])
def test_apply_keeps_every_entry(built, mx, my, n, Lx):
    """Every entry of S v within the rounding error of a chain of FMAs, relative to its
    own sum of magnitudes: for a unit value on one slot of each element, and for
    entries that span 2^40."""
    g = Grid(mx, my, n, Lx, 1.0)
    g.factor(precision=1)
    M, nel = 4 * n, mx * my
    T = g.host_factor("T").reshape(nel, M, M)
    rng = np.random.default_rng(n)
    vs = []
    for k in range(0, M, 1 if n <= 16 else 5):
        v = np.zeros((nel, M))
        v[:, k] = 1.0
        vs.append(v)
    for _ in range(8):
        vs.append(rng.choice([-1.0, 1.0], (nel, M)) * np.exp2(rng.uniform(-40, 0, (nel, M))))
    for dtype, u in ((torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)):
        for kind in (B.APPLY_AUTO, B.APPLY_CLASS):
            for v in vs:
                vt = dev(v.ravel(), dtype)
                vr = vt.double().cpu().numpy().reshape(nel, M)
                got = applied(g, kind, vt).reshape(nel, M)
                ref = exact_apply(T, vr, mx, my, n)
                bound = own_bound(T, vr, mx, my, n, u) + u * np.abs(ref).astype(float) + 1e-44 * (u > 1e-10)
                err = np.abs(got - ref).astype(float)
                assert np.all(err <= bound), (kind, dtype, float(np.max(err / np.maximum(bound, 1e-300))))


@pytest.mark.parametrize("mx,my,n,fp64", [(4, 3, 6, 1), (16, 16, 5, 1), (24, 20, 4, 0)])
def test_mixed_solves_of_small_grids_keep_the_fp64_coarse_inverse(built, mx, my, n, fp64):
    """Up to 2^17 entries of c_hat times CTAs the FP32 inner solves apply C^+ in FP64,
    beyond it its FP32 copy; the solution is the FP64 solve's."""
    g = Grid(mx, my, n)
    g.factor(tol=1e-11)
    f = dev(inputs.white_noise(g.r, 3))
    u, um = torch.empty_like(f), torch.empty_like(f)
    g.solve(f, u)
    g.factor(tol=1e-11, precision=1)
    ctas, coarse64 = (int(g.host_factor("solve_layout32")[i]) for i in (0, 8))
    assert coarse64 == fp64 == int(g.d * ctas <= 1 << 17)
    assert g.solve(f, um)[0]["converged"] == 1
    assert (u - um).norm() <= 1e-8 * u.norm()


# four elements per SM and one more, rows below and above 32, more than 96
@pytest.mark.parametrize("mx,my,n", [(19, 32, 8), (29, 21, 8), (38, 32, 11), (35, 35, 11), (35, 35, 6), (29, 21, 27)])
def test_default_apply_on_both_sides_of_its_lines(built, mx, my, n):
    """What AUTO takes agrees with the class and per-element kernels entry by entry."""
    g = Grid(mx, my, n, float(mx), float(my))
    g.factor(precision=1, flags=B.FLAG_OPERATOR_ONLY)
    M, nel = 4 * n, mx * my
    h = Grid(3, 3, n, 3.0, 3.0)
    h.factor_host_only()
    T9 = h.host_factor("T").reshape(9, M, M)
    ix, iy = np.arange(nel) % mx, np.arange(nel) // mx
    side = lambda i, m: np.where(i == 0, 0, np.where(i == m - 1, 2, 1))  # noqa: E731
    T = T9[3 * side(iy, my) + side(ix, mx)]
    v = np.random.default_rng(n).standard_normal((nel, M))
    for dtype, u in ((torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)):
        vt = dev(v.ravel(), dtype)
        vr = vt.double().cpu().numpy().reshape(nel, M)
        bound = 2 * own_bound(T, vr, mx, my, n, u)  # either side's rounding
        outs = [applied(g, k, vt).reshape(nel, M) for k in (B.APPLY_AUTO, B.APPLY_CLASS, B.APPLY_STREAM)]
        for o in outs[1:]:
            assert np.all(np.abs(o - outs[0]) <= bound + 2 * u * np.abs(o))
