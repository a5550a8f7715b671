"""C^+ by strips of element rows: the host factors solve the coarse system, with
the kernels' row ranges and staging followed CTA by CTA (CPU); solves that take
the strips agree with the oracle and with the dense form (GPU)."""
import numpy as np
import pytest

from paper_1601_03432_gb300 import Grid, inputs
from paper_1601_03432_gb300._binding import FLAG_ADJOINT

GRIDS = [(16, 16, 4, 0.0), (8, 25, 6, 0.0), (25, 9, 3, 0.0), (12, 20, 4, 2.0), (7, 31, 3, 0.0)]


def _grid(mx, my, n, stretch):
    if not stretch:
        return Grid(mx, my, n)
    return Grid(mx, my, n, xs=inputs.clustered_edges(mx, 1.0, stretch), ys=inputs.clustered_edges(my, 1.0, stretch))


def _strips_apply(g, pre, c, G):
    """The three phases of the kernels, CTA by CTA; every index is checked
    against the length of what it reads."""
    h, p, m, ns, ldn, lds, ldw = (int(v) for v in g.host_factor(pre + "_shape"))
    N, Hs, W, z = (g.host_factor("%s_%s" % (pre, k)) for k in ("N", "Hs", "W", "z"))
    d, mx, row = g.d, g.mx, 2 * g.mx - 1
    srow, RS = h * row, m + 2 * mx
    assert N.size == p * RS * ldn and Hs.size == (ns + 1) * lds and W.size == p * m * ldw and z.size == p * m
    gsep, chat, V = np.zeros(2 * p * mx + 1), np.full(d, np.nan), 2

    def dot(a, base, ld, x, at, length):
        pad = -(-length // V) * V
        assert pad <= ld and base % V == 0 and 0 <= at and at + pad <= x.size
        return a[base:base + pad] @ x[at:at + pad]

    def rows(n, rank):
        per = -(-n // G)
        return min(n, rank * per), min(n, min(n, rank * per) + per)

    for rank in range(G):
        r0, r1 = rows(p * RS, rank)
        if r0 < r1:
            b0, b1 = (r0 // RS) * srow, min(d, ((r1 - 1) // RS + 1) * srow)
            xs = np.concatenate([c[b0:b1], np.zeros(V)])
            assert xs.size <= d + 3
            for r in range(r0, r1):
                i, l = r // RS, r % RS
                mi = min(m, d - i * srow)
                if not (l < mi if l < m else (i > 0 if l < m + mx else i < p - 1)):
                    continue
                s = dot(N, r * ldn, ldn, xs, i * srow - b0, mi)
                if l < m:
                    chat[i * srow + l] = s
                else:
                    gsep[2 * i * mx + l - m] = s
    j = np.arange(ns)
    nat = (j // mx + 1) * srow - mx + j % mx
    s = c[nat] - gsep[(2 * (j // mx) + 1) * mx + j % mx] - gsep[(2 * (j // mx) + 2) * mx + j % mx]
    xs = np.concatenate([s, np.zeros(V)])
    assert xs.size <= d + 3
    for rank in range(G):
        for r in range(*rows(ns + 1, rank)):
            v = dot(Hs, r * lds, lds, xs, 0, ns)
            if r == ns:
                gsep[-1] = v
            else:
                chat[nat[r]] = v
    for rank in range(G):
        r0, r1 = rows(p * m, rank)
        if r0 < r1:
            i0, i1 = r0 // m, (r1 - 1) // m
            q = np.arange((i1 - i0 + 2) * mx + V)
            sp = i0 - 1 + q // mx
            ok = (sp >= 0) & (sp < p - 1) & (sp <= i1)
            xs = np.zeros(q.size)
            xs[ok] = chat[(sp[ok] + 1) * srow - mx + q[ok] % mx]
            assert xs.size <= d + 3
            for r in range(r0, r1):
                i, l = r // m, r % m
                if l < min(m, d - i * srow):
                    chat[i * srow + l] -= gsep[-1] * z[r] + dot(W, r * ldw, ldw, xs, (i - i0) * mx, 2 * mx)
    return chat


@pytest.mark.parametrize("mx,my,n,stretch", GRIDS)
@pytest.mark.parametrize("G", [1, 8, 152])
def test_strips_solve_the_coarse_system(mx, my, n, stretch, G):
    g = _grid(mx, my, n, stretch)
    g.factor_host_only(flags=FLAG_ADJOINT)
    C, uC = g.host_factor("C").reshape(g.d, g.d), g.host_factor("uC")
    c0 = g.host_factor("c0")
    c0 = c0 / np.linalg.norm(c0)
    rng = np.random.Generator(np.random.PCG64(3))
    for pre, A, u, nul in (("strips", C, uC, c0), ("stripsa", C.T, c0, uC)):
        r = A @ rng.standard_normal(g.d) + 0.1 * u  # a consistent part and a share of the left null vector
        x = _strips_apply(g, pre, r, G)
        want = r - u * (u @ r)
        # C's entries are of order n, its smallest nonzero singular values of order
        # 1/(mx my): products and sums lose a few digits of 2^-53
        assert np.linalg.norm(A @ x - want) <= 1e-12 * np.linalg.norm(want)
        H = g.host_factor("H" if pre == "strips" else "Ha").reshape(g.d, g.d)
        diff = x - H @ r
        diff -= nul * (nul @ diff)  # the two forms differ by the null vector only
        assert np.linalg.norm(diff) <= 1e-10 * np.linalg.norm(H @ r)


@pytest.mark.gpu
@pytest.mark.parametrize("mx,my,n,stretch", [(16, 16, 4, 0.0), (8, 25, 6, 0.0), (12, 20, 4, 2.0)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("team,nrhs", [(1, 1), (8, 1), (8, 3), (4, 16)])
def test_strips_in_team_solves(mx, my, n, stretch, precision, team, nrhs):
    """Small teams take the strips, the single solve of the same grid the fused or dense form."""
    import torch
    from paper_1601_03432_gb300 import Batch
    g = _grid(mx, my, n, stretch)
    g.factor(precision=precision)
    x, y = g.node_coords()
    f = torch.as_tensor(np.stack([inputs.fourier_rhs(x, y, seed=50 + k)[0] for k in range(nrhs)]), device="cuda")
    u, ub = torch.empty_like(f), torch.empty_like(f)
    ref = [g.solve(f[k].contiguous(), u[k])[0] for k in range(nrhs)]
    b = Batch([g], [nrhs], team_size=team)
    reps = b.solve(f.reshape(-1), ub.view(-1))
    torch.cuda.synchronize()
    # both stop at 1e-10 (of |P b_S|): FP64 iterates agree to round-off, mixed ones to the tolerance
    err = ((u - ub).norm(dim=1) / u.norm(dim=1)).max().item()
    assert err <= (1e-10 if precision == 0 else 1e-9)
    assert all(abs(a["iterations"] - r["iterations"]) <= 1 for a, r in zip(reps, ref)) or precision == 1


@pytest.mark.gpu
@pytest.mark.parametrize("mx,my,nrhs", [(32, 32, 1), (26, 33, 2), (26, 33, 7)])
def test_strips_in_grid_solves(mx, my, nrhs):
    """Grids whose single and lockstep solves take the strips: the interface residual meets tol, and
    the adjoint satisfies <gbar, u(f)> = <dl/df, f>."""
    import torch
    g = Grid(mx, my, 4)
    g.factor(flags=FLAG_ADJOINT, tol=1e-11)
    x, y = g.node_coords()
    f = torch.as_tensor(np.stack([inputs.fourier_rhs(x, y, seed=70 + k)[0] for k in range(nrhs)]), device="cuda")
    u = torch.empty_like(f)
    reps = g.solve(f, u, nrhs=nrhs)
    one = torch.empty_like(f[0])
    for k in range(nrhs):
        assert reps[k]["converged"] == 1 and reps[k]["schur_relres"] <= 1e-8
        g.solve(f[k].contiguous(), one)
        assert (one - u[k]).norm() <= 1e-10 * u[k].norm()
    gbar, gf = torch.randn_like(f[0]), torch.empty_like(f[0])
    g.solve_adjoint(gbar, gf)
    lhs, rhs = (gbar * u[0]).sum().item(), (gf * f[0]).sum().item()
    assert abs(lhs - rhs) <= 1e-8 * gbar.norm().item() * u[0].norm().item()
