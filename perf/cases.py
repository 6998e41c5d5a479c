"""Timed cases: what a user of this framework has it do, through its public entry points.

A case is a dict of plain values. "call" names the entry point:

  project    Plan.project: the projection columns of every subdomain (basis, or user densities)
  sweep_k    Plan.update_k followed by Plan.project: one step of an outer loop over wavenumbers
  adjoint    Plan.adjoint: grad_xi and dLoss/dk of a loss on those columns
  solve      Plan.solve: full-grid auxiliary-problem solves
  potential  Plan.potential: difference potentials on the whole grid
  strip      LayeredStrip.receivers: the coupled layered solve (projection, assembly, least squares)
  strip_grad the squared misfit of that solve at the receivers and its wavenumber gradient

The subdomains of a case are unit squares in square auxiliary grids: "grids" and "ks" list nodes
per side and wavenumbers, "ap" the auxiliary problem (0 Dirichlet, 1 Dirichlet-x / Sommerfeld-y,
2 the Sommerfeld rows as printed), "modes" the Chebyshev modes per side, "offset" the extra margin
below and left of the square (0: centred). The wavenumbers of a state are those of the case
within 1 %, by the seed; densities, cotangents and right-hand sides are complex normal.
"""
import math

import numpy as np
import torch

from paper_2103_12172_gb300 import Plan
from paper_2103_12172_gb300.strip import LayeredStrip, incident_impedance_bc, receiver_row


class Sub:
    """A subdomain with the fields that Plan reads: the open square [i, i+1] x [0, 1] with a
    margin of 0.1 on every side, and `offset` more to the left and below."""

    def __init__(self, i, n, k, ap, modes, offset):
        self.x0, self.x1, self.y0, self.y1 = float(i), float(i + 1), 0.0, 1.0
        self.ax0, self.ay0 = i - 0.1 - offset, -0.1 - offset
        self.h = (1.2 + offset) / (n - 1)
        self.nx = self.ny = n
        self.k, self.ap_bc, self.n_modes = float(k), ap, modes


def case(name, call, grids, ks, ap=1, modes=32, offset=0.0, kind="Q", density="basis", rhs=0):
    c = {"call": call, "grids": " ".join(str(n) for n in grids), "ks": " ".join(repr(float(k)) for k in ks),
         "ap": ap, "modes": modes, "offset": offset, "kind": kind, "density": density, "rhs": rhs}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest workload: one subdomain, 128 columns, launches and latency count
        case("project_single_129", "project", [129], [10], ap=0, modes=16),
        # the 2 x 2 decomposition: four equal subdomains, 1024 columns
        case("project_dd2x2_257", "project", [257] * 4, [30] * 4),
        # the checkerboard of coarse and fine subdomains, 1536 columns
        case("project_checker_129_513", "project", [129, 513, 513, 129], [10, 100, 100, 10], modes=48),
        # one row of the 8 x 8 decomposition with its mixed grids, 4096 columns
        case("project_row8_257_1025", "project", [513, 1025, 1025, 513, 513, 1025, 257, 1025],
             [57.5, 73.8, 66.5, 33.5, 38.0, 72.4, 20.3, 69.3], modes=64),
        # user densities on off-centre subdomains whose grids have no power of two, P columns
        case("project_user_offcentre", "project", [201, 330], [24, 45], modes=20, offset=0.07, kind="P",
             density="user"),
        # one step of an outer loop over the wavenumbers: refactor, then all columns
        case("sweep_k_dd2x2_257", "sweep_k", [257] * 4, [30] * 4),
        # the gradient pass of the 2 x 2 decomposition
        case("adjoint_dd2x2_257", "adjoint", [257] * 4, [30] * 4),
        # the gradient pass for user densities on unequal grids
        case("adjoint_user_257_513", "adjoint", [257, 513], [30, 55], modes=24, kind="P", density="user"),
        # full-grid solves of many right-hand sides
        case("solve_257_rhs32", "solve", [257], [30], rhs=32),
        # the reconstruction of a few solutions on a fine grid
        case("potential_513_rhs4", "potential", [513], [60], rhs=4),
        # the layered strip: the whole coupled solve to the receivers
        case("strip_4x129", "strip", [129] * 4, [40, 43, 37, 46], modes=24),
        # and one step of its inversion: misfit and wavenumber gradient
        case("strip_gradient_4x129", "strip_grad", [129] * 4, [40, 43, 37, 46], modes=24),
    ]


def draw(rng):
    call = rng.choice(["project"] * 5 + ["sweep_k"] + ["adjoint"] * 3 + ["solve", "potential", "strip", "strip_grad"])
    ap = rng.choice([0, 1, 1, 1, 2])

    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        if rng.random() < 0.5:   # 2^p cells, the usual choice
            n = 2 ** max(6, min(int(math.log2(hi - 1)), int(round(math.log2(n))))) + 1
        return n

    def wave(n):
        return 10.0 * rng.uniform(0.9, 1.1) if ap == 0 else round((n - 1) * rng.uniform(0.06, 0.2), 2)

    if call in ("strip", "strip_grad"):
        n = size(97, 200)
        return case(None, call, [n] * rng.randint(2, 4), [wave(n)] * 4, ap=1, modes=rng.randint(12, 24))
    offset = rng.choice([0.0, 0.0, 0.05, 0.11])
    if call in ("solve", "potential"):
        n = size(65, 513)
        return case(None, call, [n], [wave(n)], ap=ap, modes=8, offset=offset, rhs=rng.randint(1, 16))
    grids = [size(65, 1025 if call == "project" else 513) for _ in range(rng.randint(1, 4))]
    return case(None, call, grids, [wave(n) for n in grids], ap=ap, modes=rng.randint(8, 16 if min(grids) < 129 else 40),
                offset=offset, kind=rng.choice(["Q", "Q", "P"]), density=rng.choice(["basis", "basis", "user"]))


def wavenumbers(case, seed):
    ks = [float(k) for k in case["ks"].split()]
    return [k * float(u) for k, u in zip(ks, np.random.default_rng(seed).uniform(0.99, 1.01, len(ks)))]


def subdomains(case, ks):
    return [Sub(i, int(n), k, case["ap"], case["modes"], case["offset"])
            for i, (n, k) in enumerate(zip(case["grids"].split(), ks))]


def normal(n, seed):
    """n complex normal values on the GPU, the same for every caller of the seed."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(n, 2, dtype=torch.float64, device="cuda", generator=g))


def strip_k(case, seed):
    return torch.tensor(wavenumbers(case, seed), dtype=torch.float64, device="cuda")


def prepare(case, seed):
    ks = wavenumbers(case, seed)
    subs = subdomains(case, ks)
    call = case["call"]
    s = {"case": case, "ks": ks}
    if call in ("strip", "strip_grad"):
        s["strip"] = LayeredStrip(subs, incident_impedance_bc(0.3), [receiver_row(sub) for sub in subs])
        s["k"] = strip_k(case, seed)[:len(subs)].requires_grad_(call == "strip_grad")
        s["data"] = [normal(cnt, 1000 + seed + j) for j, (_, _, cnt, _) in enumerate(s["strip"].rlayout)]
        return s
    plan = s["plan"] = Plan(subs)
    n = plan.output_size
    if case["density"] == "user":
        s["xi"] = normal(n, 2 * seed)
    if call == "adjoint":
        s["cot"] = normal(n, 2 * seed + 1)
    if call == "solve":
        s["g"] = normal(case["rhs"] * subs[0].nx * subs[0].ny, seed)
    if call == "potential":
        s["xi"] = normal(case["rhs"] * plan.layout(0)[0], seed)
    return s


def run(s):
    c = s["case"]
    call = c["call"]
    if call == "project":
        return s["plan"].project(xi=s.get("xi"), kind=c["kind"])
    if call == "sweep_k":
        s["plan"].update_k(s["ks"])
        return s["plan"].project(xi=s.get("xi"), kind=c["kind"])
    if call == "adjoint":
        grad_xi, grad_k = s["plan"].adjoint(s["cot"], xi=s.get("xi"), kind=c["kind"])
        return {"grad_xi": grad_xi, "grad_k": grad_k}
    if call == "solve":
        return s["plan"].solve(0, s["g"])
    if call == "potential":
        return s["plan"].potential(0, s["xi"])
    if call == "strip":
        return s["strip"].receivers(s["k"])
    u = s["strip"].receivers(s["k"])
    loss = sum((v - d).abs().square().sum() for v, d in zip(u, s["data"]))
    (grad,) = torch.autograd.grad(loss, s["k"])
    return {"loss": loss.detach(), "grad_k": grad}


# ---- what a pass cannot do without

def gamma_size(sub):
    x, y, w = inside(sub)
    return 4 * ((x[1] - x[0] + 1) + (y[1] - y[0] + 1))


def work(case):
    """Bytes: each input read once, each output written once. Flops: the ring stencil (18 per
    node), the sine transforms of the 8 dense rows next to the square (forward 4, inverse 4) for
    columns, of every row and back for grids, and one tridiagonal solve per mode and grid."""
    subs = subdomains(case, [float(k) for k in case["ks"].split()])
    call = case["call"]
    nbytes = flops = 0
    for s in subs:
        N = s.nx - 1
        dst = 2.5 * N * math.log2(N)
        G = gamma_size(s)
        if call in ("solve", "potential"):
            nbytes += 16 * case["rhs"] * (s.nx * s.ny + (s.nx * s.ny if call == "solve" else G))
            flops += case["rhs"] * (4 * dst * s.ny + 22 * N * s.ny)
            continue
        cols = 8 * s.n_modes
        passes = {"adjoint": 2, "strip_grad": 3}.get(call, 1)
        user = 1 if case["density"] == "user" else 0
        out = {"project": 1, "sweep_k": 1, "adjoint": 2}.get(call, 0)
        nbytes += 16 * G * cols * (out + user) + 16 * N
        flops += passes * cols * (18 * G + 8 * dst * (1 + user))
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---- the same results by dense linear algebra in 64 bits

def inside(sub):
    """First and last node of the grid strictly inside the square along x and y, and their mask."""
    x = sub.ax0 + np.arange(sub.nx) * sub.h
    y = sub.ay0 + np.arange(sub.ny) * sub.h
    ix = np.nonzero((sub.x0 < x) & (x < sub.x1))[0]
    iy = np.nonzero((sub.y0 < y) & (y < sub.y1))[0]
    return (ix[0], ix[-1]), (iy[0], iy[-1]), (x, y)


def gamma_nodes(sub):
    """(n, m) of the 2-node ring around the inside nodes, row by row."""
    (a, b), (c, d), _ = inside(sub)
    n, m = np.meshgrid(np.arange(c - 1, d + 2), np.arange(a - 1, b + 2), indexing="ij")
    on = (n <= c) | (n >= d) | (m <= a) | (m >= b)
    return n[on], m[on]


def dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def tensor(v):
    return torch.as_tensor(np.ascontiguousarray(v), device=dev())


def chebyshev(s, M):
    """T_j, T_j'', T_j'''' at s, j < M, by the recurrences of the polynomials and derivatives."""
    T = np.zeros((5, M, s.size))
    T[0, 0] = 1.0
    if M > 1:
        T[0, 1], T[1, 1] = s, 1.0
    for j in range(2, M):
        for p in range(5):
            T[p, j] = 2 * s * T[p, j - 1] - T[p, j - 2] + (2 * p * T[p - 1, j - 1] if p else 0.0)
    return T[0], T[2], T[4]


def basis(sub):
    """The extended basis densities [8 M, |gamma|]: Taylor terms through rho^4 from the side that
    is nearest, with normal derivatives from the Helmholtz equation."""
    n, m = gamma_nodes(sub)
    _, _, (x, y) = inside(sub)
    gx, gy = x[m], y[n]
    rho = np.stack([sub.y0 - gy, gy - sub.y1, sub.x0 - gx, gx - sub.x1])
    near = np.abs(rho) <= np.abs(rho).min(axis=0) + 1e-9 * sub.h
    own = np.argmax(near, axis=0)
    r = rho[own, np.arange(own.size)]
    t = np.where(own <= 1, 2 * (gx - sub.x0) - 1, 2 * (gy - sub.y0) - 1)
    M, k2 = sub.n_modes, sub.k ** 2
    f, f2, f4 = chebyshev(t, M)
    f2, f4 = 4 * f2, 16 * f4
    u2 = -f2 - k2 * f
    dirichlet = f + r ** 2 / 2 * u2 + r ** 4 / 24 * (f4 + 2 * k2 * f2 + k2 ** 2 * f)
    neumann = r * f + r ** 3 / 6 * u2
    out = np.zeros((8 * M, own.size))
    for side in range(4):
        at = own == side
        out[side * M:(side + 1) * M, at] = dirichlet[:, at]
        out[(4 + side) * M:(5 + side) * M, at] = neumann[:, at]
    return tensor(out.astype(complex))


def mode_matrices(sub):
    """[modes, rows, rows]: the auxiliary problem along y for every sine mode along x, and its
    first row's node."""
    N, h, k2 = sub.nx - 1, sub.h, sub.k ** 2
    q = np.arange(1, N)
    lam = -4 * np.sin(np.pi * q / (2 * N)) ** 2
    a = 1 / h ** 2 + lam / (6 * h ** 2) + k2 / 12
    b = -2 * a + lam / h ** 2 + k2 + k2 * lam / 12
    first, rows = (1, sub.ny - 2) if sub.ap_bc == 0 else (0, sub.ny)
    T = np.zeros((N - 1, rows, rows), dtype=complex)
    i = np.arange(rows)
    T[:, i, i] = b[:, None]
    T[:, i[1:], i[:-1]] = T[:, i[:-1], i[1:]] = a[:, None]
    if sub.ap_bc:
        printed = sub.ap_bc == 2
        alpha = (1 - k2 * h * h / 24 - lam / 6 if printed else 1 + k2 * h * h / 24 + lam / 24) / h ** 2
        beta = 1j * sub.k * (1 + k2 * h * h / 8 + lam / (2 if printed else 8)) / h
        for end, other in ((0, 1), (-1, -2)):
            T[:, end, :] = 0
            T[:, end, end] = alpha + beta / 2
            T[:, end, other] = -alpha + beta / 2
    return tensor(T), first


def ap_solve(sub, g, hermitian=False):
    """G g (or its conjugate transpose on g) for g [columns, ny, nx], zero on the outermost nodes."""
    N = sub.nx - 1
    q = torch.arange(1, N, dtype=torch.float64, device=dev())
    S = torch.sin(math.pi / N * torch.remainder(torch.outer(q, q), 2 * N)).to(torch.complex128)
    T, first = mode_matrices(sub)
    rows = T.shape[1]
    ghat = torch.einsum("qm,cnm->qnc", S, g[:, first:first + rows, 1:N])
    uhat = torch.linalg.solve(T.mH if hermitian else T, ghat)
    u = torch.zeros_like(g)
    u[:, first:first + rows, 1:N] = torch.einsum("qm,qnc->cnm", S, uhat) * (2 / N)
    return u


def stencil(sub, w):
    """L w on the nodes inside the square, zero elsewhere (the operator is real and symmetric)."""
    (a, b), (c, d), _ = inside(sub)
    h2, k2 = sub.h ** 2, sub.k ** 2
    coef = {0: -4 / h2 + 4 / (6 * h2) + 8 * k2 / 12, 1: 1 / h2 - 2 / (6 * h2) + k2 / 12, 2: 1 / (6 * h2)}
    r = torch.zeros_like(w)
    for i in (-1, 0, 1):
        for j in (-1, 0, 1):
            r[:, c:d + 1, a:b + 1] += coef[abs(i) + abs(j)] * w[:, c + i:d + 1 + i, a + j:b + 1 + j]
    return r


def stencil_transposed(sub, v):
    """The transpose of stencil(): takes v on the inside nodes."""
    (a, b), (c, d), _ = inside(sub)
    h2, k2 = sub.h ** 2, sub.k ** 2
    coef = {0: -4 / h2 + 4 / (6 * h2) + 8 * k2 / 12, 1: 1 / h2 - 2 / (6 * h2) + k2 / 12, 2: 1 / (6 * h2)}
    w = torch.zeros_like(v)
    for i in (-1, 0, 1):
        for j in (-1, 0, 1):
            w[:, c + i:d + 1 + i, a + j:b + 1 + j] += coef[abs(i) + abs(j)] * v[:, c:d + 1, a:b + 1]
    return w


def exact(case, seed):
    call = case["call"]
    if call in ("strip", "strip_grad") or max(int(n) for n in case["grids"].split()) > 540:
        return None
    subs = subdomains(case, wavenumbers(case, seed))
    if call == "solve":
        s = subs[0]
        g = normal(case["rhs"] * s.nx * s.ny, seed).view(-1, s.ny, s.nx).clone()
        g[:, 0] = g[:, -1] = 0
        return ap_solve(s, g)
    sizes = [(8 * s.n_modes if call != "potential" else case["rhs"], gamma_nodes(s)[0].size) for s in subs]
    total = sum(c * G for c, G in sizes)
    user = normal(total, 2 * seed if call != "potential" else seed) if case["density"] == "user" or call == "potential" else None
    cot = normal(total, 2 * seed + 1) if call == "adjoint" else None
    at, out = 0, []
    for s, (cols, G) in zip(subs, sizes):
        n, m = (torch.as_tensor(v, device=dev()) for v in gamma_nodes(s))
        w = torch.zeros(cols, s.ny, s.nx, dtype=torch.complex128, device=dev())
        if call == "adjoint":
            c = cot[at:at + cols * G].view(cols, G)
            w[:, n, m] = c
            res = -stencil_transposed(s, ap_solve(s, w, hermitian=True))[:, n, m]
            if case["kind"] == "P":
                res = res + c
        else:
            xi = basis(s) if user is None else user[at:at + cols * G].view(cols, G)
            w[:, n, m] = xi
            u = ap_solve(s, stencil(s, w))
            if call == "potential":
                return w - u
            res = -u[:, n, m] + (xi if case["kind"] == "P" else 0)
        out.append(res.reshape(-1))
        at += cols * G
    out = torch.cat(out)
    return {"grad_xi": out, "grad_k": None} if call == "adjoint" else out
