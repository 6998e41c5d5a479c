"""The separable solve of the projection (kernels_sep.cu) where its tiles and its closed form change:
row counts around the 16- and 32-row groups, unequal grids along x and y, wavenumbers next to a
mode's cutoff (hyperbolic and trigonometric form) and grids so coarse that modes alternate in sign,
single columns, column ranges across the sides, and every receiver row. Bar: the oracle's, 1e-10 of
a column's largest value."""
import numpy as np
import pytest

import workloads as W
from oracle.projection import APSystem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


def rel_col_err(got, ref):
    return float((np.abs(got - ref).max(axis=1) / np.abs(ref).max(axis=1)).max())


def box(nx, ny, k, ap, n_modes, dx=0.0):
    """A rectangle of equal cells with margins of about a tenth (dx more on the left)."""
    h = 1.2 / (nx - 1)
    height = h * (ny - 1) / 1.2
    return W.Subdomain(0.0, 1.0, 0.0, height, -0.1 - dx, -0.1 * height, h, nx + int(round(dx / h)), ny, k, ap, n_modes)


def near_cutoff(n, q, shift, ap):
    """The wavenumber at which mode q's interior rows have e = b + 2a = shift k^2 (cutoff: 0)."""
    h = 1.2 / (n - 1)
    lam = -4 * np.sin(np.pi * q / (2 * (n - 1))) ** 2
    return float(np.sqrt(-(lam / h**2) / ((1 + lam / 12) - shift)))


CASES = [(f"n{n}", W.small_subdomain(n, 9.0, W.AP_DIRX_SOMMY, 2)) for n in (15, 17, 38, 40, 41, 42, 59, 60, 61)]
CASES += [("wide", box(65, 33, 8.0, W.AP_DIRX_SOMMY, 2)), ("tall", box(33, 97, 8.0, W.AP_DIRX_SOMMY, 3)),
          ("tall_dir4", box(33, 90, 8.0, W.AP_DIRICHLET4, 2)), ("off_centre", box(49, 49, 9.0, W.AP_DIRX_SOMMY_PAPER, 2, dx=0.1)),
          ("coarse_k", W.small_subdomain(17, 24.0, W.AP_DIRX_SOMMY, 2)), ("coarse_k40", W.small_subdomain(17, 40.0, W.AP_DIRX_SOMMY, 1))]
CASES += [(f"cutoff_{shift:g}", W.small_subdomain(65, near_cutoff(65, 3, shift, 1), W.AP_DIRX_SOMMY, 2))
          for shift in (0.0, 1e-14, 1e-9, -1e-9, 1e-4, -1e-4, -1e-2)]


@pytest.mark.parametrize("user", [False, True])
@pytest.mark.parametrize("name,sub", CASES, ids=[c[0] for c in CASES])
def test_columns_match_the_oracle(mdp, name, sub, user):
    plan = mdp.Plan([sub])
    G, nc, _, _ = plan.layout(0)
    xi = W.random_complex((nc, G), seed=5) if user else None
    got = plan.project(xi=None if xi is None else torch.from_numpy(xi.ravel()).cuda(), kind="P").cpu().numpy().reshape(nc, G)
    plan.status()
    assert rel_col_err(got, APSystem(sub).columns(xi=xi, kind="P")) < TOL


@pytest.mark.parametrize("fp64", [False, True])
def test_column_ranges_and_tiles_give_the_same_columns(mdp, fp64):
    """Any range of columns (single ones, ranges across the sides) and any tile width: bit for bit
    the columns of the whole call."""
    sub = W.small_subdomain(45, 9.0, W.AP_DIRX_SOMMY, 5)
    plan = mdp.Plan([sub], fp64_cols=fp64)
    G, nc, _, _ = plan.layout(0)
    ref = plan.project().view(nc, G)
    for c0, n in ((0, 1), (9, 1), (10, 1), (3, 14), (8, 5), (19, 2), (29, 11), (0, 40)):
        assert torch.equal(plan.project_columns(0, c0, n).view(n, G), ref[c0:c0 + n])
    assert torch.equal(mdp.Plan([sub], fp64_cols=fp64, tile_cols=7).project().view(nc, G), ref)


@pytest.mark.parametrize("off", [0.0, 0.1])
def test_every_receiver_row(mdp, off):
    sub = box(37, 33, 9.0, W.AP_DIRX_SOMMY, 1, dx=off)
    plan = mdp.Plan([sub])
    G, nc, _, nm = plan.layout(0)
    S = APSystem(sub)
    xi = plan.basis_densities(0)
    pot = plan.potential(0, xi).cpu().numpy()
    nlo, nhi = nm[:, 0].min() + 1, nm[:, 0].max() - 1
    for row in range(nlo + 1, nhi):
        plan.set_receivers([row])
        _, m0, cnt, _ = plan.receiver_layout(0)
        out, rec = plan.project(out_rec=True)
        ref = pot[:, row, m0:m0 + cnt]
        assert rel_col_err(rec[:nc * cnt].cpu().numpy().reshape(nc, cnt), ref) < TOL, row
    assert rel_col_err(out.cpu().numpy().reshape(nc, G), S.columns()) < TOL


@pytest.mark.parametrize("name,sub", CASES, ids=[c[0] for c in CASES])
def test_full_grid_solves_match_the_oracle(mdp, name, sub):
    """Whole-grid solves: data on every node, on the rows next to the ends, and none at all."""
    plan = mdp.Plan([sub])
    g = W.random_complex((3, sub.ny, sub.nx), seed=9)
    g[1, 3:-3] = 0
    g[2] = 0
    got = plan.solve(0, torch.from_numpy(g).cuda()).cpu().numpy()
    plan.status()
    S = APSystem(sub)
    ref = np.stack([S.solve(x) for x in g[:2]])
    assert rel_col_err(got[:2].reshape(2, -1), ref.reshape(2, -1)) < TOL
    assert not got[2].any()


def test_full_grid_solves_in_passes(mdp):
    """More right-hand sides than the workspace takes at once: bit for bit those of single calls, also in
    place."""
    sub = W.small_subdomain(65, 9.0, W.AP_DIRX_SOMMY, 2)
    plan = mdp.Plan([sub], workspace_bytes=1 << 20)
    g = torch.from_numpy(W.random_complex((40, 65, 65), seed=10)).cuda()
    one = torch.cat([plan.solve(0, g[i:i + 1]) for i in range(40)])
    assert torch.equal(plan.solve(0, g), one)
    plan.solve(0, g, out=g)
    assert torch.equal(g, one)


def tall(ny, low=False):
    """A grid of 33 x ny nodes; the subdomain takes ten twelfths of its height, or (low) half."""
    h = 1.2 / 32
    height = h * (ny - 1)
    y0, y1 = (0.25, 0.75) if low else (0.1, 0.9)
    return W.Subdomain(0.0, 1.0, 0.0, (y1 - y0) * height, -0.1, -y0 * height, h, 33, ny, 8.0, W.AP_DIRX_SOMMY, 1)


@pytest.mark.parametrize("sub", [tall(2561), tall(2564), tall(2600), tall(3480, True), tall(3600, True)],
                         ids=["n2561", "n2564", "n2600", "low3480", "low3600"])
def test_tall_grids_around_the_limits_of_the_separable_solve(mdp, sub):
    """The operand masks hold 256 groups of 16 rows and columns, the solve along y some 3500 rows: on either
    side of both limits the columns and the full-grid solves are those of the sweeps. Bar: the sweeps'
    own error at 3600 rows (1e-12 to 1e-11 at 1025), 1e-9."""
    plan, ref = mdp.Plan([sub]), mdp.Plan([sub], fp64_cols=True)
    G, nc, _, _ = plan.layout(0)
    a, b = (p.project().view(nc, G).cpu().numpy() for p in (plan, ref))
    plan.status()
    assert rel_col_err(a, b) < 1e-9
    g = torch.from_numpy(W.random_complex((2, sub.ny, sub.nx), seed=11)).cuda()
    a, b = (p.solve(0, g).view(2, -1).cpu().numpy() for p in (plan, ref))
    plan.status()
    assert rel_col_err(a, b) < 1e-9


@pytest.mark.parametrize("name,sub", CASES, ids=[c[0] for c in CASES])
@pytest.mark.parametrize("user,rec,kind", [(False, False, "P"), (True, False, "Q"), (False, True, "Q"), (True, True, "P")])
def test_gradient_is_that_of_the_sweeps(mdp, name, sub, user, rec, kind):
    """The gradient pass by the separable solve against the recurrences: basis and user densities, with a
    receiver row's cotangent, both kinds; the second pass (after a change of k) on rebuilt tables. Bar:
    1e-10 for the gradients by densities, 1e-9 for the one by k (the oracle's bars)."""
    plan, ref = mdp.Plan([sub]), mdp.Plan([sub], fp64_cols=True)
    G, nc, _, nm = plan.layout(0)
    row = int(nm[:, 0].min() + 2 + (np.ptp(nm[:, 0]) - 4) // 3)
    cot = torch.from_numpy(W.random_complex(nc * G, seed=12)).cuda()
    xi = torch.from_numpy(W.random_complex(nc * G, seed=13)).cuda() if user else None
    cr = None
    if rec:
        for p in (plan, ref):
            p.set_receivers([row])
        cr = torch.from_numpy(W.random_complex(nc * plan.receiver_layout(0)[2], seed=14)).cuda()
    for k in (None, sub.k * 1.01):
        if k is not None:
            for p in (plan, ref):
                p.update_k([k])
        (ga, ka), (gb, kb) = (p.adjoint(cot, xi=xi, kind=kind, grad_xi=user, cot_rec=cr) for p in (plan, ref))
        plan.status()
        if user:
            assert rel_col_err(ga.view(nc, G).cpu().numpy(), gb.view(nc, G).cpu().numpy()) < 1e-10
        assert abs(ka.item() - kb.item()) < 1e-9 * abs(kb.item())


def test_captured_gradient_follows_the_wavenumbers(mdp):
    """A first gradient call inside a stream capture (its tables are allocated and made there), replayed after a
    change of k, and plain calls afterwards: bit for bit those of a plan that never captured."""
    sub = W.small_subdomain(65, 9.0, W.AP_DIRX_SOMMY, 2)
    plan, ref = mdp.Plan([sub]), mdp.Plan([sub])
    cot = torch.from_numpy(W.random_complex(plan.output_size, seed=15)).cuda()
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        g.capture_begin()
        gx, gk = plan.adjoint(cot)
        g.capture_end()
    for k in (9.0, 9.4):
        for p in (plan, ref):
            p.update_k([k])
        g.replay()
        torch.cuda.synchronize()
        for p, out in ((ref, (gx, gk)), (plan, (gx, gk))):
            rx, rk = p.adjoint(cot)
            assert torch.equal(out[0], rx) and torch.equal(out[1], rk)
    plan.status()


@pytest.mark.parametrize("rows", [(-1, 16, 16), (9, 20, 9), (20, -1, 14)])
@pytest.mark.parametrize("off", [0.0, 0.1])
def test_deduplicated_subdomains_have_receiver_rows_of_their_own(mdp, rows, off):
    """Three copies of a subdomain on one set of tables, with receiver rows that differ from the first one's, in
    both orders of setting them: columns, receiver values and gradients (with and without the receivers' cotangent)
    of the plain plan. Bar: 1e-12, the same sums on placements that differ in their last bits."""
    from dataclasses import replace
    b = box(37, 33, 9.0, W.AP_DIRX_SOMMY, 2, dx=off)
    subs = [replace(b, x0=b.x0 + i, x1=b.x1 + i, ax0=b.ax0 + i) for i in range(3)]
    dd, plain = mdp.Plan(subs, dedupe=True), mdp.Plan(subs)
    assert dd.leaders() == [0, 0, 0]
    dd.set_receivers(rows[::-1])
    cot = torch.from_numpy(W.random_complex(plain.output_size, seed=16)).cuda()
    xi = torch.from_numpy(W.random_complex(plain.output_size, seed=17)).cuda()
    for p in (dd, plain):
        p.set_receivers(rows)
    cr = torch.from_numpy(W.random_complex(plain.receiver_size, seed=18)).cuda()
    for k in (None, 9.3):
        got = []
        for p in (dd, plain):
            if k is not None:
                p.update_k([k] * 3)
            res = list(p.project(out_rec=True)) + list(p.project(xi=xi, out_rec=True))
            for c in (cr, None):
                for x in (xi, None):
                    res += p.adjoint(cot, xi=x, cot_rec=c)
            p.status()
            got.append(res)
        for a, r in zip(*got):
            assert (a - r).abs().max() <= 1e-12 * r.abs().max()


@pytest.mark.parametrize("fp64", [False, True])
def test_captured_calls_without_receivers_outlive_a_change_of_the_rows(mdp, fp64):
    """Projection and gradient captured without receivers, replayed after set_receivers: bit for bit the values
    before, as are plain calls without receiver arguments."""
    subs = [W.unit_subdomain(i, 0, n, 7.0 + i, W.AP_DIRX_SOMMY, 3) for i, n in enumerate((33, 45, 33))]
    plan = mdp.Plan(subs, fp64_cols=fp64)
    cot = torch.from_numpy(W.random_complex(plan.output_size, seed=19)).cuda()
    ref = [plan.project().clone(), *plan.adjoint(cot)]
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(s):
        g.capture_begin()
        out = [plan.project(), *plan.adjoint(cot)]
        g.capture_end()
    for rows in ([-1, 20, -1], [16, 20, 16], [-1, -1, -1]):
        plan.set_receivers(rows)
        for t in out:
            t.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        for a, b, r in zip(out, [plan.project(), *plan.adjoint(cot)], ref):
            assert torch.equal(a, r) and torch.equal(b, r)
    plan.status()


@pytest.mark.parametrize("n,q,p", [(65, 1, 61), (65, 61, 1), (129, 1, 1), (129, 51, 121), (129, 81, 121), (129, 101, 111),
                                   (257, 1, 1), (257, 43, 253), (257, 190, 22), (257, 253, 1)])
def test_update_refuses_the_wavenumbers_that_plan_creation_refuses(mdp, n, q, p):
    """Discrete Dirichlet eigenvalues whose eigenvector is small at the ends: the pivots of the full factors
    stay above the tolerance, those of the system without the rows above the ring do not."""
    from paper_2103_12172_gb300 import MdpError
    lq, lp = (-4 * np.sin(np.pi * m / (2 * (n - 1))) ** 2 for m in (q, p))
    k = float(np.sqrt(-((lq + lp * (1 + lq / 6)) / (1.2 / (n - 1)) ** 2) / (1 + lq / 12 + lp / 12)))
    sub = W.small_subdomain(n, 9.0, W.AP_DIRICHLET4, 1)
    for plan in (mdp.Plan([sub]), mdp.Plan([sub], fp64_cols=True)):
        with pytest.raises(MdpError) as e:
            plan.update_k([k])
        assert e.value.code == 4   # MDP_ERR_SINGULAR
        plan.update_k([9.0])
    with pytest.raises(MdpError) as e:
        mdp.Plan([sub.with_k(k)], host_only=True)
    assert e.value.code == 4


@pytest.mark.parametrize("power", [-1000, -1020, 960])
@pytest.mark.parametrize("off", [0.0, 0.1])
def test_densities_near_the_ends_of_the_exponents_range(mdp, power, off):
    """Densities, cotangents and right-hand sides times a power of two that leaves the largest values in range: the
    same results times that power. Bar: the rounding of what falls below 2^-1074, some hundred terms of it, and 1e-14
    of a column's largest value."""
    sub = box(49, 45, 9.0, W.AP_DIRX_SOMMY, 2, dx=off)
    plan = mdp.Plan([sub])
    G, nc, _, _ = plan.layout(0)
    s = 2.0 ** power
    xi = torch.from_numpy(W.random_complex(nc * G, seed=20)).cuda()
    g = torch.from_numpy(W.random_complex((2, sub.ny, sub.nx), seed=21)).cuda()

    half = 2.0 ** (-power // 2)        # back in two steps

    def scaled(t):
        return torch.view_as_complex(torch.view_as_real(t) * s)

    for f, x, n in ((lambda x: plan.project(xi=x, kind="P"), xi, nc), (lambda x: plan.adjoint(x, grad_k=False)[0], xi, nc),
                    (lambda x: plan.solve(0, x.view(2, sub.ny, sub.nx)), g, 2)):
        ref, got = f(x).reshape(n, -1), f(scaled(x)).reshape(n, -1)
        plan.status()
        err = (torch.view_as_real(got) * half * half - torch.view_as_real(ref)).abs()
        tiny = 200 * 2.0 ** (-1074 - power) / sub.h**2
        assert (err.amax(dim=(1, 2)) <= 1e-14 * ref.abs().amax(dim=1) + tiny).all()


def column(py, dx=0):
    """py rows and 25 (dx cells off centre) columns of M+ in a grid of margins of 19 and 4 cells."""
    h = 1.0 / 25
    return W.Subdomain(0.0, 1.0, 0.0, py * h, -(4.5 + dx) * h, -19.5 * h, h, 35 + dx, py + 40, 7.0, W.AP_DIRX_SOMMY, 1)


@pytest.mark.parametrize("py,dx", [(2049, 0), (2050, 0), (2051, 0), (3300, 0), (1026, 3), (1027, 3)])
def test_columns_of_tall_grids_are_those_of_the_pivoted_factors(mdp, py, dx):
    """On either side of the limits the projection's columns are the traces of the basis densities' potentials
    solved by the pivoted factors of every mode (the sweeps' plan), which share no closed form with
    them. Bar: the factors' own error at these heights, 1e-9."""
    sub = column(py, dx)
    plan, ref = mdp.Plan([sub]), mdp.Plan([sub], fp64_cols=True)
    info = plan.sub_info(0)
    assert (info["Py"], info["xsym"]) == (py, int(dx == 0))
    G, nc, _, nm = plan.layout(0)
    u = ref.potential(0, ref.basis_densities(0)).cpu().numpy()
    plan.status()
    for p in (plan, ref):
        assert rel_col_err(p.project(kind="P").view(nc, G).cpu().numpy(), u[:, nm[:, 0], nm[:, 1]]) < 1e-9


def test_subdomains_beyond_the_limits_beside_others(mdp):
    """One plan with subdomains of the sweeps and of the separable solve, centred and not: projection and
    gradients bit for bit those of plans of their own."""
    subs = [column(2051), W.small_subdomain(33, 8.0, W.AP_DIRICHLET4, 1), column(1027, 3), box(37, 33, 9.0, W.AP_DIRX_SOMMY, 1, dx=0.1)]
    plan = mdp.Plan(subs)
    cot = torch.from_numpy(W.random_complex(plan.output_size, seed=22)).cuda()
    xi = torch.from_numpy(W.random_complex(plan.output_size, seed=23)).cuda()
    got = [plan.blocks(plan.project()), plan.blocks(plan.project(xi=xi))] + [plan.adjoint(cot, xi=x) for x in (None, xi)]
    plan.status()
    for i, sub in enumerate(subs):
        one = mdp.Plan([sub])
        x, c = plan.blocks(xi)[i].reshape(-1), plan.blocks(cot)[i].reshape(-1)
        assert torch.equal(got[0][i].reshape(-1), one.project()) and torch.equal(got[1][i].reshape(-1), one.project(xi=x))
        for (gx, gk), d in zip(got[2:], (None, x)):
            rx, rk = one.adjoint(c, xi=d)
            assert torch.equal(plan.blocks(gx)[i].reshape(-1), rx) and gk[i] == rk[0]
