"""The kernels that multiply in fixed-point digits, at the sizes where tiles and
weights end: the class apply (what AUTO takes) against the per-element products,
wide ranges of magnitude, Inf and NaN; solves with whole block inverses of up to
256 columns; the residual norm at short restarts; batches with teams of their
own choice and column counts just past a lockstep group."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1601_03432_gb300 import Batch, Grid, inputs
from paper_1601_03432_gb300 import _binding as B
from oracle.smpm import SMPMGrid
from oracle.schur import SchurSystem
from oracle import methods


@pytest.fixture(scope="module")
def built():
    from paper_1601_03432_gb300.build import build
    build()
    assert torch.cuda.is_available()


def rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def apply(g, kind, v):
    g.set_apply_kernel(kind)
    out = torch.full_like(v, -7.0)
    (g.apply_schur if v.dtype == torch.float64 else g.apply_schur32)(v, out)
    torch.cuda.synchronize()
    return out.double().cpu().numpy()


# 4n = 8 ... 128: less than a tile, remainders of 4, 8 and 12 rows, full tiles;
# element counts that leave class tiles of one and of seven
@pytest.mark.parametrize("mx,my,n", [(9, 5, 2), (3, 11, 3), (8, 8, 4), (6, 7, 5), (5, 13, 11), (12, 4, 16), (4, 9, 23),
                                     (10, 3, 25), (3, 3, 31), (4, 5, 32)])
def test_class_apply_against_per_element_products(built, mx, my, n):
    g = Grid(mx, my, n)
    g.factor(precision=1)
    M, nel = 4 * n, mx * my
    T = np.abs(g.host_factor("T").reshape(nel, M, M))
    rng = np.random.default_rng(n)
    general = B.APPLY_WARP if M <= 96 else B.APPLY_STREAM
    scales = {"plain": np.ones(nel), "elements": 10.0 ** rng.integers(-150, 150, nel), "tiny": np.full(nel, 1e-290)}
    for name, s in scales.items():
        v = rng.standard_normal((nel, M)) * s[:, None]
        if name == "plain":
            v *= 2.0 ** rng.integers(-8, 9, (nel, M))
        ref = apply(g, general, dev(v.ravel()))
        for kind in (B.APPLY_CLASS, B.APPLY_AUTO):
            got = apply(g, kind, dev(v.ravel()))
            # entry of the facing slot: an FP64 chain of M products on one side,
            # on the other digits cut at 2^-62 of the largest entries of row and vector,
            # without the products of weight below 256^7 (7 2^14 256^6 2^-124 < 2^-59 each)
            e = np.arange(nel)
            bound = np.zeros((nel, M))
            chain = (M + 2) * 2.0 ** -53 * np.einsum("erk,ek->er", T, np.abs(v))
            cut = M * 2.0 ** -58 * T.max(axis=2) * np.abs(v).max(axis=1)[:, None]
            own = chain + cut
            ix, iy = e % mx, e // mx
            for F, (dx, dy) in enumerate(((-1, 0), (1, 0), (0, -1), (0, 1))):
                ok = (0 <= ix + dx) & (ix + dx < mx) & (0 <= iy + dy) & (iy + dy < my)
                e2 = (e + dx + mx * dy)[ok]
                f2 = (F ^ 1) * n
                bound[e2, f2:f2 + n] = own[e[ok], F * n:(F + 1) * n]
            err = np.abs(got - ref).reshape(nel, M)
            assert np.all(err <= bound + 2.0 ** -52 * np.abs(ref).reshape(nel, M) + 1e-307), (name, kind, np.max(err - bound))
    v = rng.standard_normal(nel * M)
    a, b = (apply(g, k, dev(v, torch.float32)) for k in (general, B.APPLY_CLASS))
    assert rel(b, a) < 4 * M * 2.0 ** -24


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_class_apply_inf_and_nan_reach_the_same_entries(built, bad):
    g = Grid(7, 6, 6)
    g.factor(precision=1)
    v = np.random.default_rng(3).standard_normal(7 * 6 * 24)
    v[17 * 24 + 5] = bad
    for dtype in (torch.float64, torch.float32):
        a, b = (apply(g, k, dev(v, dtype)) for k in (B.APPLY_WARP, B.APPLY_CLASS))
        fin = np.isfinite(a)
        assert np.array_equal(fin, np.isfinite(b)) and not fin.all()
        assert np.array_equal(np.isnan(a), np.isnan(b))
        assert np.array_equal(np.sign(a[np.isinf(a)]), np.sign(b[np.isinf(a)]))
        assert rel(b[fin], a[fin]) < (1e-13 if dtype == torch.float64 else 1e-5)


# whole block inverses of 2 * 4n columns: 24 (a tile and a half), 88, 256 (the
# accumulators' limit), and blocks of several classes per CTA
@pytest.mark.parametrize("mx,my,n,graded", [(3, 2, 3, False), (4, 3, 11, True), (3, 3, 32, False), (19, 17, 4, False)])
@pytest.mark.parametrize("restart", [3, 8, 50])
def test_solve_block_inverse_and_short_restarts(built, mx, my, n, graded, restart):
    kw = {}
    if graded:
        kw = dict(xs=inputs.clustered_edges(mx, 1.0, 1.5), ys=inputs.clustered_edges(my, 1.0, 1.5))
    og = SMPMGrid(mx, my, n, **kw)
    osys = SchurSystem(og)
    f, gn = inputs.white_noise(og.r, 5), np.random.default_rng(6).standard_normal(og.kp)
    b = og.rhs(f, gn)
    ref = methods.direct_solve(og, og.assemble_L(), osys.u_L, b)
    lg = Grid(mx, my, n, **kw)
    lg.factor(tol=1e-11, restart=restart, maxit=2000)
    u = torch.zeros(og.r, dtype=torch.float64, device="cuda")
    rep = lg.solve(dev(f), u, g=dev(gn), allow_notconv=True)[0]
    _, info = methods.algorithm3(osys, b, tol=1e-11, restart=restart, maxit=2000)
    assert rep["converged"] == info["converged"]
    if rep["converged"]:
        assert rel(u.cpu().numpy(), ref) < 1e-9
    # restarted iterations are counted to within one per cycle
    assert abs(rep["iterations"] - info["iterations"]) <= 1 + (info["iterations"] // restart if restart < 50 else 0)


# one column, a lockstep group, one past a group; both precisions
@pytest.mark.parametrize("precision,bound", [(0, 1e-9), (1, 1e-8)], ids=["fp64", "mixed"])
def test_batch_default_teams_match_one_team(built, precision, bound):
    probs = [(16, 14, 8, 17), (2, 2, 4, 1), (3, 9, 6, 2), (20, 6, 5, 1), (7, 7, 9, 3)]
    grids = [Grid(mx, my, n) for mx, my, n, _ in probs]
    for g in grids:
        g.factor(tol=1e-11, precision=precision)
    nrhs = [p[3] for p in probs]
    f = dev(np.concatenate([inputs.white_noise(mx * my * n * n, 10 * i + c) for i, (mx, my, n, k) in enumerate(probs)
                            for c in range(k)]))
    out = []
    for team in (0, 152, 8):
        b = Batch(grids, nrhs, team_size=team)
        u = torch.zeros_like(f)
        reps = b.solve(f, u)
        assert all(r["converged"] == 1 for r in reps)
        teams = b.task_times()[0]
        assert len(teams) == sum(nrhs) and max(teams) < b.info()["nteams"]
        out.append((u.cpu().numpy(), [r["iterations"] for r in reps]))
        b.close()
    for u, its in out[1:]:
        assert rel(out[0][0], u) < bound
        assert max(abs(a - b) for a, b in zip(its, out[0][1])) <= (1 if precision == 0 else 3)
