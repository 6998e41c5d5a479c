"""The coupled solve of a layout in a few launches (mdp_couple_solve, mdp_couple_grad) against the same
system by single tensor operations and the dense least squares (LayeredStrip._dense_coefficients): a strip and
a block of 2 x 2, Robin sides with wavenumber-dependent and constant data, Dirichlet sides, grids of
different sizes. Bar: receivers and gradients to 1e-8 (rounding, 1e-16 with a few hundred terms, in systems of
condition 1e7)."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LAYOUTS = {"one": ([(0, 0)], [33]), "strip3": ([(0, 0), (1, 0), (2, 0)], [33, 41, 33]),
           "block": ([(0, 0), (1, 0), (0, 1), (1, 1)], [33, 45, 45, 33])}


def bc(j, side, kj, x, y):
    u = torch.exp(1j * (kj * x * 0.8 + 2.0 * y))
    if side == 1:                                   # Dirichlet
        return 1.0 + 0.0 * kj, 0.0, u
    if side == 2:                                   # constants
        return 2.0 + 1j, 0.5, u * (1.0 + x)
    return 1j * kj, 1.0 + 0.1 * kj, (1j * kj + 0.3) * u


@pytest.mark.parametrize("M", [5, 8])
@pytest.mark.parametrize("name", list(LAYOUTS))
def test_coupled_solve_and_gradient_are_those_of_the_dense_path(mdp, name, M):
    from paper_2103_12172_gb300.strip import LayeredStrip
    pos, grids = LAYOUTS[name]
    ks = [4.0 + 0.7 * j for j in range(len(pos))]
    subs = [W.unit_subdomain(i, jj, n, k, W.AP_DIRX_SOMMY, M) for (i, jj), n, k in zip(pos, grids, ks)]
    got = []
    for dense in (False, True):
        lay = LayeredStrip(subs, bc, [s.ny // 2 for s in subs], positions=pos)
        k = torch.tensor(ks, dtype=torch.float64, device="cuda", requires_grad=True)
        if dense:
            lay.receivers(k.detach())
            systems = lay._st["systems"]
            assert all(cs.ok for cs in systems.values())
            for cs in systems.values():
                cs.ok = False
        u = lay.receivers(k)
        w = [torch.linspace(0.2, 1.0, v.numel(), device="cuda") for v in u]
        loss = sum(((v - 0.3j).abs().square() * t).sum() for v, t in zip(u, w))
        (g,) = torch.autograd.grad(loss, k)
        got.append((torch.cat(u).detach(), g, torch.cat([c for c in lay.coefficients(k.detach())[0]])))
    for a, b in zip(*got):
        assert (a - b).abs().max() < 1e-8 * b.abs().max()


@pytest.mark.parametrize("form", ["one", "per_coefficient", "mixed"])
def test_boundary_coefficients_of_one_element_and_per_coefficient(mdp, form):
    """alpha (and the divisor of a Robin side) as a tensor of one element, alpha as one value per Chebyshev
    coefficient: with equal values the solution and the gradient are those of the numbers."""
    from paper_2103_12172_gb300.strip import LayeredStrip
    pos, grids = LAYOUTS["strip3"]
    M, ks = 5, [4.0, 4.7, 5.4]
    subs = [W.unit_subdomain(i, jj, n, k, W.AP_DIRX_SOMMY, M) for (i, jj), n, k in zip(pos, grids, ks)]

    def shaped(j, side, kj, x, y):
        alpha, beta, phi = bc(j, side, kj, x, y)
        alpha = torch.as_tensor(alpha, dtype=torch.complex128, device="cuda")
        if form == "one" or (form == "mixed" and side == 2):
            return alpha.reshape(1), beta if side in (1, 2) else beta.reshape(1), phi
        return alpha.expand(M) if side != 2 or form == "per_coefficient" else alpha, beta, phi

    got = []
    for cond in (bc, shaped):
        lay = LayeredStrip(subs, cond, [s.ny // 2 for s in subs], positions=pos)
        k = torch.tensor(ks, dtype=torch.float64, device="cuda", requires_grad=True)
        u = torch.cat(lay.receivers(k))
        (g,) = torch.autograd.grad((u - 0.3j).abs().square().sum(), k)
        got.append((u.detach(), g))
    for a, b in zip(*got):
        assert (a - b).abs().max() < 1e-8 * b.abs().max()


def test_layout_without_receivers_gives_empty_values(mdp):
    """No receiver row anywhere: every layer's values are empty, and so is their gradient (zero)."""
    from paper_2103_12172_gb300.strip import LayeredStrip, incident_impedance_bc
    subs = [W.unit_subdomain(j, 0, 33, 4.0 + j, W.AP_DIRX_SOMMY, 4) for j in range(2)]
    lay = LayeredStrip(subs, incident_impedance_bc(0.3), [-1, -1])
    k = torch.tensor([4.0, 5.0], dtype=torch.float64, device="cuda", requires_grad=True)
    u = lay.receivers(k)
    assert [v.numel() for v in u] == [0, 0]
    (g,) = torch.autograd.grad(sum(v.abs().sum() for v in u), k)
    assert torch.equal(g, torch.zeros_like(g))


def test_gradient_of_a_layout_with_1120_shared_unknowns(mdp):
    """8 x 8 subdomains, 10 unknowns per interface: the triangle of the shared unknowns and the vector take more
    shared memory than a kernel has without opting in. The dense path's values, 1e-8 (as above)."""
    from paper_2103_12172_gb300.strip import LayeredStrip, incident_impedance_bc
    pos = [(i, j) for j in range(8) for i in range(8)]
    ks = [4.0 + 0.02 * j for j in range(64)]
    subs = [W.unit_subdomain(i, jj, 33, k, W.AP_DIRX_SOMMY, 5) for (i, jj), k in zip(pos, ks)]
    got = []
    for dense in (False, True):
        lay = LayeredStrip(subs, incident_impedance_bc(0.3), [16] * 64, positions=pos)
        k = torch.tensor(ks, dtype=torch.float64, device="cuda", requires_grad=True)
        if dense:
            lay.receivers(k.detach())
            for cs in lay._st["systems"].values():
                assert cs.ok and cs.c.n_shared == 1120
                cs.ok = False
        u = torch.cat(lay.receivers(k))
        (g,) = torch.autograd.grad((u - 0.3j).abs().square().sum(), k)
        got.append((u.detach(), g))
    for a, b in zip(*got):
        assert (a - b).abs().max() < 1e-8 * b.abs().max()


def test_coefficients_may_be_changed_in_place(mdp):
    """The layers' coefficients are tensors of their own: an in-place change of one is differentiated and leaves the
    others as they are."""
    from paper_2103_12172_gb300.strip import LayeredStrip, incident_impedance_bc
    subs = [W.unit_subdomain(j, 0, 33, 4.0 + j, W.AP_DIRX_SOMMY, 4) for j in range(2)]
    lay = LayeredStrip(subs, incident_impedance_bc(0.3), [16, 16])
    k = torch.tensor([4.0, 5.0], dtype=torch.float64, device="cuda", requires_grad=True)
    c, _ = lay.coefficients(k)
    ref = [v.detach().clone() for v in c]
    c[0].mul_(2.0)
    assert torch.equal(c[0].detach(), 2.0 * ref[0]) and torch.equal(c[1].detach(), ref[1])
    (g,) = torch.autograd.grad(c[0].abs().square().sum(), k)
    (h,) = torch.autograd.grad(lay.coefficients(k)[0][0].abs().square().sum(), k)
    assert (g - 4.0 * h).abs().max() <= 1e-12 * h.abs().max()


def test_receivers_take_a_subclass_s_coefficients(mdp):
    from paper_2103_12172_gb300.strip import LayeredStrip, incident_impedance_bc

    class Twice(LayeredStrip):
        def coefficients(self, k):
            c, rec = super().coefficients(k)
            return [2.0 * v for v in c], rec

    subs = [W.unit_subdomain(j, 0, 33, 4.0 + j, W.AP_DIRX_SOMMY, 4) for j in range(2)]
    k = torch.tensor([4.0, 5.0], dtype=torch.float64, device="cuda", requires_grad=True)
    got = []
    for cls in (LayeredStrip, Twice):
        u = torch.cat(cls(subs, incident_impedance_bc(0.3), [16, 16]).receivers(k))
        got.append((u.detach(), torch.autograd.grad(u.abs().square().sum(), k)[0]))
    assert torch.equal(got[1][0], 2.0 * got[0][0])
    assert (got[1][1] - 4.0 * got[0][1]).abs().max() <= 1e-12 * got[1][1].abs().max()
