"""Layered strip: domain-decomposition coupling on top of the batched projection columns, and
its gradient with respect to the per-layer wavenumbers.

Subdomains Omega_j = [j, j+1] x [0, 1] (a duct, Section 4) with wavenumbers k_j. Per layer the
library computes Q_j = (P_gamma - I) Ex Psi (Section 3.2.5) and the difference potential of
every basis column at a receiver row (Eq. potential_solution_homo) in one batched pass. The
coupling follows Sections 3.3-3.5: outer sides carry alpha u + beta du/dn = phi expanded in the
Chebyshev basis (Eq. BC_coefficients), interfaces carry c^(0) continuous and c^(1) opposite
(Section 3.3.2); the BC and interface equations are eliminated (Section 3.3.3) and the stacked
system is solved in the least-squares sense by QR (steps 2(b)-(c)). The loss is the squared
misfit of the reconstructed solution at the receivers.

The coupling is small dense linear algebra (hundreds of unknowns) written with torch so that
autograd carries the chain rule; the AP solves, the projection columns, the receiver values and
their wavenumber derivatives run in libmdp (forward: mdp_project_batch_rec; backward:
mdp_ap_adjoint_rec).
"""
from __future__ import annotations

import ctypes as C
import math

import torch

from . import Plan, _lib, linalg


class ProjectWithReceivers(torch.autograd.Function):
    """(Q, receiver values) of the basis columns of every subdomain as functions of k."""

    @staticmethod
    def forward(ctx, k, plan):
        ks = [float(v) for v in k.detach().cpu().tolist()]
        if getattr(plan, "_k_current", None) != ks:
            plan.update_k(ks)
            plan._k_current = ks
        out, rec = plan.project(out_rec=True)
        ctx.plan, ctx.ks = plan, ks
        ctx.k_meta = (k.dtype, k.device)
        return out, rec

    @staticmethod
    def backward(ctx, g_out, g_rec):
        plan = ctx.plan
        if getattr(plan, "_k_current", None) != ctx.ks:
            plan.update_k(ctx.ks)
            plan._k_current = ctx.ks
        g_out = torch.zeros(plan.output_size, dtype=torch.complex128, device="cuda") if g_out is None else g_out
        g_rec = None if g_rec is None else g_rec.contiguous()
        _, gk = plan.adjoint(g_out.contiguous(), grad_xi=False, cot_rec=g_rec)
        dtype, device = ctx.k_meta
        return gk.to(dtype=dtype, device=device), None


def least_squares_grads(A, b, x, w, mm):
    """Gradients of the least-squares minimiser x of ||A x - b|| for the incoming gradient g,
    given w = (A^H A)^{-1} g: with r = b - A x, grad_b = A w and grad_A = r w^H - (A w) x^H.
    mm: the matrix-vector product to use."""
    Aw = mm(A, w)
    r = b - mm(A, x)
    grad_A = torch.outer(r, w.conj()) - torch.outer(Aw, x.conj())
    return grad_A, Aw


class LeastSquares(torch.autograd.Function):
    """x = argmin ||A x - b|| for a full-column-rank CUDA matrix A (m >= n) by Householder QR of
    the column-equilibrated A D (Section 3.5, steps 2(b)-(c); the scaling leaves the minimiser
    unchanged and improves the conditioning of R), all on libmdp's kernels: the QR
    (mdp_householder_qr, or the two-stage structured form when the row blocks are given), the
    triangular solves (mdp_triangular_solve) and the products (mdp_complex_matmul). The backward
    pass uses the closed form of the minimiser's derivative instead of differentiating the
    factorisation: w = (A^H A)^{-1} g = D R^{-1} R^{-H} D g for the incoming gradient g, then
    least_squares_grads."""

    @staticmethod
    def forward(ctx, A, b, blocks=None):
        if not A.is_cuda:
            raise TypeError("LeastSquares runs on libmdp's CUDA kernels: A must be a CUDA tensor")
        linalg.check_pending()                         # status words of earlier solves that have completed
        D = 1.0 / torch.linalg.vector_norm(A, dim=0)
        if blocks is not None:
            fac = linalg.structured_qr(A * D, b, *blocks)   # per-subdomain QRs, then the shared unknowns
        else:
            fac = linalg.householder_qr(A * D, b)
        linalg.defer_check(fac)                        # checked later, without stalling the stream
        x = D * fac.lstsq()
        ctx.fac = fac
        ctx.save_for_backward(A, b, x, D)
        return x

    @staticmethod
    def backward(ctx, g):
        A, b, x, D = ctx.saved_tensors
        w = D * ctx.fac.gram_solve((D * g).to(torch.complex128))
        grad_A, grad_b = least_squares_grads(A, b, x, w, linalg.matmul)
        return grad_A, grad_b, None


def _ptr(t):
    return None if t is None else t.data_ptr()


class _Blocks:
    """Blocks [cols][len_j] of one tensor and the ranges of a stacked vector they act on, with the index
    tensors on the device."""

    def __init__(self, cols, lens, offs, device):
        self.n, self.cols, self.lens = len(lens), cols, list(lens)
        self.starts = [sum(lens[:j]) for j in range(len(lens))]
        self.total, self.max = sum(lens), max(max(lens), 1)
        self.ints = torch.tensor(self.lens + self.starts, dtype=torch.int32).to(device)
        self.offs = torch.tensor(list(offs), dtype=torch.int64).to(device)
        self.args = (self.n, self.cols, self.max, self.ints.data_ptr(), self.ints.data_ptr() + 4 * self.n,
                     self.offs.data_ptr())


class BlockValues(torch.autograd.Function):
    """y_j = B_j v_j for every block of a _Blocks layout: B flat, v [blocks, cols], y stacked."""

    @staticmethod
    def forward(ctx, B, v, blocks):
        v = v.contiguous()
        y = torch.empty(max(blocks.total, 1), dtype=torch.complex128, device=B.device)[:blocks.total]
        if blocks.total:
            _lib.check(_lib.lib().mdp_block_values(*blocks.args, _ptr(B), _ptr(v), _ptr(y), linalg._stream()),
                       "mdp_block_values")
        ctx.save_for_backward(B, v)
        ctx.blocks = blocks
        return y

    @staticmethod
    def backward(ctx, gy):
        B, v = ctx.saved_tensors
        if not ctx.blocks.total:   # no receiver anywhere
            return torch.zeros_like(B), torch.zeros_like(v), None
        gy = gy.resolve_conj().contiguous()
        gB = torch.empty_like(B) if ctx.needs_input_grad[0] else None
        gv = torch.empty_like(v) if ctx.needs_input_grad[1] else None
        _lib.check(_lib.lib().mdp_block_values_grad(*ctx.blocks.args, _ptr(B), _ptr(v), _ptr(gy), _ptr(gB), _ptr(gv),
                                                    linalg._stream()), "mdp_block_values_grad")
        return gB, gv, None


class CoupledSystem:
    """The index tables of mdp_couple for a structure of unknowns (LayeredStrip._structure) whose outer
    sides have the given kinds ("robin", "dirichlet"), on the device; ok: the library takes the system."""

    def __init__(self, st, kinds, M, rows, offs, device):
        N, n, cols = len(rows), st["n"], st["col_sets"]
        count = {}
        for cj in cols:
            for c in cj:
                count[c] = count.get(c, 0) + 1
        shared = sorted(c for c, v in count.items() if v > 1)
        order = [[c for c in cj if count[c] == 1] + [c for c in cj if count[c] > 1] for cj in cols]
        private = [sum(count[c] == 1 for c in cj) for cj in cols]
        pos = {c: i for i, c in enumerate(shared)}
        nmax, mmax = max(len(o) for o in order), max(rows)
        s0 = [sum(len(order[i]) - private[i] for i in range(j)) for j in range(N)]
        ms = sum(len(o) - p for o, p in zip(order, private))
        per_col = [[[0] * nmax for _ in range(N)] for _ in range(6)]   # unk, slot0, neg0, slot1, rho, sidx
        per_coef = [[[v] * (8 * M) for _ in range(N)] for v in (-1, 0, -1)]   # su, sf, se
        touch = [[] for _ in range(n)]
        sides = []                                                     # qj, qe, qr, qu
        q = 0
        for j in range(N):
            entry = {}                                                 # unknown -> (slot0, neg0, slot1, q)
            for side, spec in enumerate(st["sides"][j]):
                z, o = side * M, (4 + side) * M
                c = spec[1]
                for m in range(M):
                    if spec[0] == "if":
                        entry[c + m] = (z + m, 0, -1, 0)
                        entry[c + M + m] = (o + m, int(spec[2] < 0), -1, 0)
                        links = [(z + m, c + m, 0), (o + m, c + M + m, int(spec[2] < 0))]
                    elif kinds[q] == "robin":
                        entry[c + m] = (z + m, 0, o + m, q)
                        links = [(z + m, c + m, 0), (o + m, c + m, 2 + q)]
                        per_coef[2][j][o + m] = q * M + m
                    else:
                        entry[c + m] = (o + m, 0, -1, 0)
                        links = [(o + m, c + m, 0)]
                        per_coef[2][j][z + m] = q * M + m
                    for slot, u, f in links:
                        per_coef[0][j][slot], per_coef[1][j][slot] = u, f
                if spec[0] != "if":
                    sides.append((j, o if kinds[q] == "robin" else z, o if kinds[q] == "robin" else -1, c))
                    q += 1
            for p, u in enumerate(order[j]):
                for t, v in zip(per_col, (u,) + entry[u] + (pos.get(u, 0),)):
                    t[j][p] = v
                touch[u].append(j * nmax + p)
        flat = [rows, [len(o) for o in order], private, s0, [sum(rows[:j]) for j in range(N)]]
        flat += [r for t in per_col + per_coef for r in t]
        flat += [(t + [-1, -1])[:2] for t in touch] + [shared] + [[s[i] for s in sides] for i in range(4)]
        self.ints = torch.tensor([v for r in flat for v in r], dtype=torch.int32).to(device)
        self.offs = torch.tensor(list(offs), dtype=torch.int64).to(device)
        self.c = _lib.mdp_couple(N, M, n, len(shared), ms, mmax, nmax, q, sum(rows), self.ints.data_ptr(),
                                 self.offs.data_ptr())
        L = _lib.lib()
        self.buffer, self.grad_buffer = L.mdp_couple_buffer(self.c), L.mdp_couple_grad_buffer(self.c)
        self.work_ints = L.mdp_couple_work_ints(self.c)
        self.ok = self.buffer > 0 and all(len(t) in (1, 2) for t in touch)
        self.status = [N] + ([int(L.mdp_householder_qr_work_ints(N)) + 1] if shared else [])


class CoupledSolve(torch.autograd.Function):
    """The coefficients [N, 8 M] of every subdomain's boundary data from the projection columns `out`, the
    outer sides' rho [sides] and eps [sides, M] and the sources' F [rows] or None, by mdp_couple_solve: the
    least squares of LeastSquares on the structured system, assembled, solved and differentiated in a
    few launches."""

    @staticmethod
    def forward(ctx, out, rho, eps, src, cs):
        linalg.check_pending()                         # status words of earlier solves that have completed
        dev = out.device
        rho, eps = rho.resolve_conj().contiguous(), eps.resolve_conj().contiguous()
        buf = torch.empty(cs.buffer, dtype=torch.complex128, device=dev)
        work = torch.empty(cs.work_ints, dtype=torch.int32, device=dev)
        x = torch.empty(cs.c.n, dtype=torch.complex128, device=dev)
        coef = torch.empty((cs.c.n_blocks, 8 * cs.c.n_modes), dtype=torch.complex128, device=dev)
        _lib.check(_lib.lib().mdp_couple_solve(cs.c, _ptr(out), _ptr(rho), _ptr(eps), _ptr(src), _ptr(buf), _ptr(work),
                                               _ptr(x), _ptr(coef), linalg._stream()), "mdp_couple_solve")
        linalg.defer_status(work, cs.status)           # checked later, without stalling the stream
        ctx.save_for_backward(out, rho, src, buf, x, coef)
        ctx.cs = cs
        return coef

    @staticmethod
    def backward(ctx, g):
        out, rho, src, buf, x, coef = ctx.saved_tensors
        cs = ctx.cs
        g = g.resolve_conj().contiguous()
        tmp = torch.empty(cs.grad_buffer, dtype=torch.complex128, device=out.device)
        gout = torch.empty_like(out) if ctx.needs_input_grad[0] else None
        grho = torch.empty_like(rho)
        geps = torch.empty((cs.c.n_outer, cs.c.n_modes), dtype=torch.complex128, device=out.device)
        _lib.check(_lib.lib().mdp_couple_grad(cs.c, _ptr(out), _ptr(rho), _ptr(src), _ptr(buf), _ptr(x), _ptr(coef),
                                              _ptr(g), _ptr(tmp), _ptr(gout), _ptr(grho), _ptr(geps), linalg._stream()),
                   "mdp_couple_grad")
        return gout, grho, geps, None, None


def cheb_coeffs(fvals, n):
    """Chebyshev coefficients of the degree n-1 interpolant from values at the n first-kind
    Chebyshev points x_i = cos(pi (i + 1/2) / n) (i = 0..n-1): c_m = (2/n) sum_i f(x_i) T_m(x_i),
    c_0 halved. fvals [n] complex (CUDA; the product runs on mdp_complex_matmul)."""
    i = torch.arange(n, dtype=torch.float64, device=fvals.device)
    m = torch.arange(n, dtype=torch.float64, device=fvals.device)
    T = torch.cos(m[:, None] * math.pi * (i[None, :] + 0.5) / n)   # T_m(x_i)
    c = (2.0 / n) * linalg.matmul(T, fvals)
    c[0] = c[0] / 2
    return c


def cheb_points(n, device):
    i = torch.arange(n, dtype=torch.float64, device=device)
    return torch.cos(math.pi * (i + 0.5) / n)


def _sides_at_once(bc):
    """bc.sides_at_once where it stands for bc itself: defined with or below the class's __call__ (a subclass
    that overrides __call__ alone is asked side by side)."""
    for c in type(bc).__mro__:
        if "sides_at_once" in vars(c):
            break
        if "__call__" in vars(c):
            return None
    return getattr(bc, "sides_at_once", None)


class LayeredStrip:
    """A rectangular layout of square subdomains that share whole sides (default: a strip
    along x; `positions[j]` = cell (i, j) of subdomain j otherwise, Section 3.4) with outer
    boundary data bc(j, side, k_j, x, y) -> (alpha, beta, phi values) (torch, differentiable in
    k_j), a receiver row per subdomain and optionally a source per subdomain."""

    def __init__(self, subdomains, bc, receiver_rows, tile_cols=0, source=None, positions=None):
        self.subs = list(subdomains)
        self.N = len(self.subs)
        self.M = self.subs[0].n_modes
        self.bc = bc
        self.source = source        # source(j) -> fun(x, y) -> (f, f_x, f_y, f_xx, f_yy), or None
        self._src_cache = {}
        self.pos = [tuple(p) for p in positions] if positions is not None else [(j, 0) for j in range(self.N)]
        self.at = {p: j for j, p in enumerate(self.pos)}
        self.plan = Plan(self.subs, tile_cols=tile_cols)
        self.plan.set_receivers(receiver_rows)
        self.layout = [self.plan.layout(j) for j in range(self.N)]
        self.rlayout = [self.plan.receiver_layout(j) for j in range(self.N)]
        self._rec_blocks = None
        self._consts = {}

    def neighbour(self, j, side):
        i, jj = self.pos[j]
        di, dj = {1: (0, -1), 2: (0, 1), 3: (-1, 0), 4: (1, 0)}[side]
        return self.at.get((i + di, jj + dj))

    def outer(self, j, side):
        return self.neighbour(j, side) is None

    def iface(self, j, side):
        """(key, sign) of an interface: named by the left/bottom subdomain's side 4 or 2; c^(1)
        enters with + there and - on the neighbour (opposite outward normals)."""
        if side in (4, 2):
            return (j, side), 1.0
        return (self.neighbour(j, side), 4 if side == 3 else 2), -1.0

    def _side_xy(self, j, side, s):
        sb = self.subs[j]
        if side in (1, 2):
            return sb.x0 + (s + 1) / 2 * (sb.x1 - sb.x0), torch.full_like(s, sb.y0 if side == 1 else sb.y1)
        return torch.full_like(s, sb.x0 if side == 3 else sb.x1), sb.y0 + (s + 1) / 2 * (sb.y1 - sb.y0)

    def source_terms(self, j, kj):
        """(F_j, u_j) of layer j's source at wavenumber kj (None without a source), cached per k."""
        if self.source is None or self.source(j) is None:
            return None
        key = (j, float(kj))
        if key not in self._src_cache:
            fgrid, src4 = self.plan.source_foot_data(j, self.source(j))
            self._src_cache = {kk: v for kk, v in self._src_cache.items() if kk[0] != j}
            self._src_cache[key] = self.plan.source_terms(j, torch.from_numpy(fgrid).cuda(),
                                                          torch.from_numpy(src4).cuda())
        return self._src_cache[key]

    def receivers(self, k):
        """Solution at the receivers of every layer (list of complex tensors), differentiable in k
        (without a source; the source terms are not differentiated)."""
        if self.source is not None and k.requires_grad:
            raise NotImplementedError("the k-gradient of the source terms is not implemented")
        if getattr(self.coefficients, "__func__", None) is LayeredStrip.coefficients:
            coef, rec = self._coefficients(k)
        else:                              # a subclass's own coefficients
            cvecs, rec = self.coefficients(k)
            coef = torch.stack(list(cvecs)).to(torch.complex128)
        if self._rec_blocks is None:
            self._rec_blocks = _Blocks(self.layout[0][1], [r[2] for r in self.rlayout], [r[3] for r in self.rlayout],
                                       rec.device)
        vals = BlockValues.apply(rec, coef, self._rec_blocks)
        res = []
        for j, val in enumerate(vals.split(self._rec_blocks.lens)):
            row, m0, cnt, _ = self.rlayout[j]
            st = self.source_terms(j, self.plan_k(j))
            if st is not None:
                val = val + st[1][row, m0:m0 + cnt]
            res.append(val)
        return res

    def plan_k(self, j):
        """The wavenumber the plan is factored for in layer j."""
        ks = getattr(self.plan, "_k_current", None)
        return ks[j] if ks is not None else self.subs[j].k

    def field(self, k):
        """The solution on the whole grid of every layer, [ny, nx] complex tensors (the difference
        potential of the layer's boundary density, Eq. potential_solution_homo; meaningful on
        N+). Not differentiable."""
        with torch.no_grad():
            cvecs, _ = self.coefficients(k)
            out = []
            for j in range(self.N):
                dens = self.plan.basis_densities(j)                      # [8M, |gamma|]
                xi = linalg.matmul(dens.transpose(0, 1), cvecs[j])[None, :].contiguous()
                u = self.plan.potential(j, xi)[0]
                st = self.source_terms(j, self.plan_k(j))
                out.append(u if st is None else u + st[1])
            return out

    def _structure(self, device):
        """What the coupled system's shape depends on, built once: the unknowns (one block of M
        per outer side, two per interface), each subdomain's sides as ("outer", c) or
        ("if", c, sign), the unknowns each subdomain's rows touch, the Chebyshev points of every
        outer side, and the Chebyshev analysis matrix."""
        if getattr(self, "_st", None) is not None and self._st["device"] == device:
            return self._st
        M, N = self.M, self.N
        idx, n = {}, 0
        for j in range(N):
            for side in (1, 2, 3, 4):
                if self.outer(j, side):
                    idx[(j, side)] = n
                    n += M
            for side in (4, 2):
                if not self.outer(j, side):
                    idx[("if", j, side)] = n
                    n += 2 * M
        s = cheb_points(M, device)
        sides, col_sets, pts = [], [], {}
        for j in range(N):
            spec, used = [], []
            for side in (1, 2, 3, 4):
                if self.outer(j, side):
                    c = idx[(j, side)]
                    spec.append(("outer", c))
                    used.extend(range(c, c + M))
                    pts[(j, side)] = self._side_xy(j, side, s)
                else:
                    key, sgn = self.iface(j, side)
                    c = idx[("if",) + key]
                    spec.append(("if", c, sgn))
                    used.extend(range(c, c + 2 * M))
            sides.append(spec)
            col_sets.append(sorted(set(used)))
        i_ = torch.arange(M, dtype=torch.float64, device=device)
        T = torch.cos(i_[:, None] * math.pi * (i_[None, :] + 0.5) / M)   # T_m(x_i)
        w = torch.full((M,), 2.0 / M, dtype=torch.float64, device=device)
        w[0] = 1.0 / M
        self._st = {"device": device, "n": n, "sides": sides, "col_sets": col_sets, "pts": pts,
                    "cheb": (T.transpose(0, 1).to(torch.complex128).contiguous(), w), "systems": {}, "layer": {},
                    "outer": list(pts), "xy": [torch.stack(t) for t in zip(*pts.values())]}
        return self._st

    def _scalars(self, vals, device):
        """The values (numbers, tensors of one element) as one complex tensor: numbers that are no tensors are put
        on the device once."""
        if not any(isinstance(v, torch.Tensor) for v in vals):
            key = (str(device),) + tuple(complex(v) for v in vals)
            t = self._consts.get(key)
            if t is None:
                t = torch.tensor(key[1:], dtype=torch.complex128).to(device)
                if len(self._consts) < 16:
                    self._consts[key] = t
            return t
        ts = [v.reshape(()).to(torch.complex128) if isinstance(v, torch.Tensor)
              else torch.tensor(complex(v), dtype=torch.complex128) for v in vals]
        if len({t.device for t in ts}) > 1:
            ts = [t.to(device) for t in ts]
        return torch.stack(ts).to(device)

    def coefficients(self, k):
        """The Chebyshev coefficients [c^(0) sides 1..4, c^(1) sides 1..4] of every layer's boundary
        data from the coupled least-squares solve, and the receiver output of the projection."""
        coef, rec = self._coefficients(k)
        return [c.clone() for c in coef.unbind(0)], rec   # tensors of their own, as the caller may change them in place

    def _coefficients(self, k):
        """coefficients() as one tensor [N, 8 M].
        Outer side of unknown block u: alpha c0 + beta c1 = d (d the Chebyshev coefficients of
        the data); with beta != 0 the unknown is c0 and the side's rows read Q0 - (alpha/beta) Q1
        against u and -Q1 d / beta on the right; with beta = 0 the unknown is c1 (rows Q1) and
        the right-hand side -Q0 d / alpha. Interfaces: c0 shared, c1 with opposite signs."""
        M, N = self.M, self.N
        out, rec = ProjectWithReceivers.apply(k, self.plan)
        st = self._structure(out.device)
        # boundary data of every outer side, analysed into Chebyshev coefficients in one product
        alphas = bcs = phi = None
        at_once = _sides_at_once(self.bc)
        if at_once is not None and st["outer"]:
            layer = st["layer"].get(str(k.device))
            if layer is None:
                layer = st["layer"][str(k.device)] = torch.tensor([j for j, _ in st["outer"]]).to(k.device)
            alphas, betas, phi = at_once(k.index_select(0, layer), [s for _, s in st["outer"]], *st["xy"])
            if any(beta == 0 for beta in betas):
                alphas, bcs = None, list(zip(alphas.unbind(0), betas))
        else:
            bcs, phis = [], []
            for j in range(N):
                kj = None
                for side, spec in zip((1, 2, 3, 4), st["sides"][j]):
                    if spec[0] == "outer":
                        kj = k[j] if kj is None else kj
                        x, y = st["pts"][(j, side)]
                        alpha, beta, ph = self.bc(j, side, kj, x, y)
                        bcs.append((alpha, beta))
                        phis.append(ph.to(torch.complex128))
            betas = [beta for _, beta in bcs]
            phi = torch.stack(phis) if phis else None
        Tt, w = st["cheb"]
        d_all = linalg.matmul(phi, Tt) * w if phi is not None else None   # [outer sides, M]
        kinds = tuple("robin" if beta != 0 else "dirichlet" for beta in betas)
        cs = st["systems"].get(kinds)
        if cs is None:
            cs = st["systems"][kinds] = CoupledSystem(st, kinds, M, [lay[0] for lay in self.layout],
                                                      [lay[2] for lay in self.layout], out.device)
        # CoupledSolve takes one alpha and one beta per side; a side may also have one per coefficient
        single = bcs is None or all(not isinstance(v, torch.Tensor) or v.dim() == 0 or v.shape == (1,) for ab in bcs for v in ab)
        if not (cs.ok and single):
            bcs = list(zip(alphas.unbind(0), betas)) if bcs is None else bcs
            return torch.stack(self._dense_coefficients(out, bcs, d_all, st)), rec
        if not betas:
            rho = eps = torch.empty(0, dtype=torch.complex128, device=out.device)
        else:
            if bcs is None:
                div = self._scalars(betas, out.device)
            else:
                div = self._scalars([b if kd == "robin" else a for (a, b), kd in zip(bcs, kinds)], out.device)
                alphas = self._scalars([a if kd == "robin" else 0.0 for (a, b), kd in zip(bcs, kinds)], out.device)
            rho = -alphas / div
            eps = d_all / div[:, None]
        src = [self.source_terms(j, self.plan_k(j)) for j in range(N)]
        if any(t is not None for t in src):
            src = torch.cat([torch.zeros(lay[0], dtype=torch.complex128, device=out.device) if t is None else t[0].reshape(-1)
                             for t, lay in zip(src, self.layout)])
        else:
            src = None
        return CoupledSolve.apply(out, rho, eps, src, cs), rec

    def _dense_coefficients(self, out, bcs, d_all, st):
        """The coefficients by single tensor operations and LeastSquares, for systems CoupledSolve does not
        take (a layer with fewer gamma nodes than unknowns, triangles beyond a CTA's shared memory, or sides with an
        alpha per coefficient)."""
        M, N, n = self.M, self.N, st["n"]
        A_rows, b_rows, coef = [], [], []
        q = 0
        for j in range(N):
            G, nc, off, _ = self.layout[j]
            Q = out[off:off + G * nc].view(nc, G).transpose(0, 1)          # [G, 8M]
            A = torch.zeros(G, n, dtype=torch.complex128, device=out.device)
            e = []                      # Q e is minus the right-hand side
            cj = []
            for side, spec in zip((1, 2, 3, 4), st["sides"][j]):
                Q0 = Q[:, (side - 1) * M: side * M]
                Q1 = Q[:, 4 * M + (side - 1) * M: 4 * M + side * M]
                if spec[0] == "outer":
                    c = spec[1]
                    alpha, beta = bcs[q]
                    d = d_all[q]
                    q += 1
                    if beta != 0:
                        A[:, c:c + M] = Q0 - (alpha / beta) * Q1
                        e.append((4 * M + (side - 1) * M, d / beta))
                        cj.append(("robin", c, d, alpha, beta))
                    else:
                        A[:, c:c + M] = Q1
                        e.append(((side - 1) * M, d / alpha))
                        cj.append(("dirichlet", c, d, alpha, beta))
                else:
                    _, c, sgn = spec
                    A[:, c:c + M] = Q0
                    A[:, c + M:c + 2 * M] = sgn * Q1
                    cj.append(("if", c, sgn))
            if e:
                ev = torch.zeros(8 * M, dtype=torch.complex128, device=out.device)
                for r, val in e:
                    ev[r:r + M] = val
                b = -linalg.matmul(Q, ev)
            else:
                b = torch.zeros(G, dtype=torch.complex128, device=out.device)
            src = self.source_terms(j, self.plan_k(j))
            if src is not None:
                b = b + src[0]
            A_rows.append(A)
            b_rows.append(b)
            coef.append(cj)
        A = torch.cat(A_rows)
        b = torch.cat(b_rows)
        xsol = LeastSquares.apply(A, b, ([r.shape[0] for r in A_rows], st["col_sets"]))
        cvecs = []
        for j in range(N):
            parts0, parts1 = [], []
            for spec in coef[j]:
                if spec[0] == "robin":
                    _, c, d, alpha, beta = spec
                    u0 = xsol[c:c + M]
                    parts0.append(u0)
                    parts1.append((d - alpha * u0) / beta)
                elif spec[0] == "dirichlet":
                    _, c, d, alpha, beta = spec
                    parts0.append(d / alpha)
                    parts1.append(xsol[c:c + M])
                else:
                    _, c, sgn = spec
                    parts0.append(xsol[c:c + M])
                    parts1.append(sgn * xsol[c + M:c + 2 * M])
            cvecs.append(torch.cat(parts0 + parts1))
        return cvecs


class incident_impedance_bc:
    """Outer data of config `strip4x1`: impedance sides du/dn + i k_j u = phi with phi from the
    plane wave exp(i k_j (x cos theta + y sin theta)) of the layer's own wavenumber. sides_at_once() gives the data of
    many sides at once: their layers' wavenumbers [S], side numbers, points x, y [S, M] -> alpha [S],
    the numbers beta, phi [S, M]; LayeredStrip takes it where a boundary condition has it."""

    def __init__(self, theta):
        self.ct, self.sn = math.cos(theta), math.sin(theta)
        self.dirs = {1: -self.sn, 2: self.sn, 3: -self.ct, 4: self.ct}   # outward normal times direction
        self._factors = {}

    def __call__(self, j, side, kj, x, y):
        ik = 1j * kj
        return ik, 1.0, torch.exp(ik * (x * self.ct + y * self.sn)) * (ik * (1.0 + self.dirs[side]))

    def sides_at_once(self, ks, side, x, y):
        ik = 1j * ks.to(x.device)
        dirs = tuple(self.dirs[s] for s in side)
        key = (dirs, x.dtype, x.device)
        n = self._factors.get(key)   # of these directions, on the device once
        if n is None:
            n = torch.tensor([1.0 + v for v in dirs], dtype=x.dtype).to(x.device)
            if len(self._factors) < 16:
                self._factors[key] = n
        return ik, [1.0] * len(side), torch.exp(ik[:, None] * torch.add(x * self.ct, y, alpha=self.sn)) * (ik * n)[:, None]


def receiver_row(sub, y_target=0.9):
    """Grid row whose y is nearest y_target (within M+)."""
    import numpy as np
    y = sub.ay0 + np.arange(sub.ny) * sub.h
    return int(np.argmin(np.abs(y - y_target)))
