// Full-grid solves u = G^(h) g (Section 3.2.1) for subdomains with the separable tables: sine transforms
// along x as digit contractions on the tensor cores (digit_gemm.cuh: every row of the grid against the
// sines, odd and even modes on folded columns), and per mode the closed form of T_q^{-1} along y,
//   x_n = sum_j kappa(|n - j|) g_j + phi(n)^T R M,   M_b = sum_j phi_b(j) g_j
// (kernels_sep.cu), by first-order recurrences over segments of rows that run in parallel.
//
// Four kernels a pass: k_full_cut, k_full_gemm (forward), k_full_y, then cut and gemm again (inverse) and
// k_full_out. They replaced direct O(N^2) sums on the FP64 pipe and one thread per mode sweeping an
// uncoalesced column: 257^2, 32 right-hand sides 3.85 ms -> 312 us; 513^2, 4 right-hand sides with the
// potential's ring and correction 4.25 ms -> 250 us. k_full_y is half of it, FP64-bound.
#include "sep_modes.cuh"

#include <algorithm>

#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace mdp {

// per mode: kind, lambda (with its sign), kappa(0) = c, c (1 - lambda^2), sign, R11, R12, R22, F, and of the
// rotation of kinds 0, 1: -+s^2 (s = sin or sinh theta), C(1), C and S at row 0;
// 1 / lambda, 1 / c, log2 |lambda|
enum { MX_KIND = 0, MX_LAM, MX_C, MX_C1, MX_SG, MX_R = 6, MX_F = 12, MX_SS, MX_CS1, MX_CS0,   // CS0: 2
       MX_LI = 17, MX_CI, MX_L2 };

// The table of the solve along y, over all rows 0 .. N: evanescent modes phi = (lambda^n, lambda^(N-n)),
// the others C and S about the middle row.
__global__ void k_full_modes(const SubDesc *subs, int s0, unsigned char *sep) {
  const int si = s0 + blockIdx.y;
  const SubDesc &d = subs[si];
  const int q = blockIdx.x * 32 + threadIdx.x + 1;
  if (d.leader != si || q > d.Nq) return;
  double *T = reinterpret_cast<double *>(sep + d.sep_mx) + (long long)(q - 1) * SEP_MXW;
  const ModeShape m = mode_shape(d, q, reinterpret_cast<const double *>(sep + d.sep_ab) + 2 * (q - 1));
  const int N = d.ny - 1;
  const double lam = m.sg * exp(-m.th), c = m.kind == 2 ? -1.0 / (2.0 * m.a * sinh(m.th)) : 0.0;
  cplx R11, R12, R22;
  if (m.kind < 2) reflect_cs(m, N, 0.5 * N, R11, R12, R22);
  else {
    reflect_exp(m, N, 0, N, c, R11, R12, R22);
    // phi_2 = lambda^(N-n) carries the sign sg^N more than (-1)^n e^{-theta (N - n)}
    if (m.sg < 0.0 && (N & 1)) R12 = cmk(-R12.re, -R12.im);
  }
  const double sth = m.kind == 0 ? sin(m.th) : m.kind == 1 ? sinh(m.th) : 0.0;
  T[MX_SS] = m.kind == 0 ? -sth * sth : sth * sth;
  T[MX_CS1] = m.kind < 2 ? sep_c(m.kind, m.th, 1.0) : 0.0;
  T[MX_CS0] = m.kind < 2 ? sep_c(m.kind, m.th, -0.5 * N) : 0.0;
  T[MX_CS0 + 1] = m.kind < 2 ? sep_s(m.kind, m.th, -0.5 * N) : 0.0;
  T[MX_KIND] = m.kind; T[MX_LAM] = lam; T[MX_C] = c;
  T[MX_C1] = -c * expm1(-2.0 * m.th);
  T[MX_SG] = m.sg;
  T[MX_LI] = m.sg * exp(m.th);
  T[MX_CI] = -2.0 * m.a * sinh(m.th);
  T[MX_L2] = -m.th * 1.4426950408889634;
  T[MX_R] = R11.re; T[MX_R + 1] = R11.im; T[MX_R + 2] = R12.re; T[MX_R + 3] = R12.im;
  T[MX_R + 4] = R22.re; T[MX_R + 5] = R22.im;
  T[MX_F] = 1.0 / (2.0 * m.a);
}

namespace {

// What every kernel of a pass reads, as a kernel argument: the first loads of a block would otherwise be a
// chain of dependent reads of the descriptor.
struct FullArg {
  SubDesc d;
  SepGeo g;
  FullWs w;
  int nr;
  const unsigned char *sep;
  double *ws;
  long long ws_n, sep_n;   // doubles of the workspace, bytes of the tables; for the bounds-checked build
};
// bounds-checked build: the slices of this pass are those of its right-hand sides and lie in the workspace, and
// so do the tables
static __device__ __noinline__ bool full_in_bounds(const FullArg &p) {
  const FullWs r = full_ws(p.d, p.nr);
  bool ok = p.nr >= 1 && r.total <= p.ws_n && p.w.rows == r.rows && p.w.R == r.R && p.w.ldf == r.ldf && p.w.ldu == r.ldu &&
            p.w.a == r.a && p.w.ex == r.ex && p.w.mask == r.mask && p.w.f == r.f && p.w.u == r.u;
  sep_tables(p.d, [&](const long long &o, long long n, int) { ok = ok && o >= 0 && o + n <= p.sep_n; });
  if (!ok) flag_bounds(p.d.dstatus);
  return ok;
}
#define MDP_CHECK_FULL(p)                                   \
  do {                                                      \
    if (MDP_CHECKED && !full_in_bounds(p)) return;          \
  } while (0)

// A: the grid's rows on folded columns (INV false: g(m) +- g(Nx - m)) or the modes (INV), cut into digits.
// Row order (right-hand side, unknown row, part): a block's 8 rows are 4 grid rows, complex parts in turn.
template <bool INV>
__global__ void __launch_bounds__(256) k_full_cut(const __grid_constant__ FullArg p, const double2 *g) {
  pdl_wait();
  MDP_CHECK_FULL(p);
  const SubDesc &d = p.d;
  const SepGeo &geo = p.g;
  const FullWs &w = p.w;
  double *ws = p.ws;
  const int e = blockIdx.y, row = blockIdx.x * 8 + (threadIdx.x & 7), kl = threadIdx.x >> 3;
  const int nk = INV ? geo.nqh / 16 : geo.nkx, part = row & 1;
  const int n = (row >> 1) % d.Nt + d.nfirst, N = d.Nx;
  const bool live = row < w.rows && (INV || (n >= 1 && n <= d.ny - 2));   // the rows at the ends take no data
  const double *src = INV ? ws + w.f + (long long)row * w.ldf + e * geo.nqh
                          : reinterpret_cast<const double *>(g + ((long long)((row >> 1) / d.Nt) * d.ny + n) * d.nx) + part;
  auto value = [&](int k) -> double {
    if (!live) return 0.0;
    if (INV) return src[k];
    const int m = 1 + k;
    if (2 * m > N) return 0.0;
    const double a = src[2 * m], b = 2 * m == N ? 0.0 : src[2 * (N - m)];
    return e == 0 ? a + b : a - b;
  };
  __shared__ int emax[8];
  __shared__ unsigned smask[SEP_MASK];
  if (threadIdx.x < 8) { emax[threadIdx.x] = 0; smask[threadIdx.x] = 0; }
  __syncthreads();
  double x[8];   // the first 256 values of K stay in registers between the two passes
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = kl < 2 * nk ? value(8 * kl + j) : 0.0;
  int m = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) m = max(m, (__double2hiint(x[j]) >> 20) & 0x7ff);
  for (int k8 = kl + 32; k8 < 2 * nk; k8 += 32)
#pragma unroll
    for (int j = 0; j < 8; ++j) m = max(m, (__double2hiint(value(8 * k8 + j)) >> 20) & 0x7ff);
  for (int off = 16; off >= 8; off >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) < 8) atomicMax(&emax[threadIdx.x & 7], m);
  __syncthreads();
  const int E = max(emax[threadIdx.x & 7], 1), t = e * (w.R / 128) + row / 128;
  if (kl == 0) reinterpret_cast<int *>(ws + w.ex)[e * w.R + row] = E;
  unsigned char *A = reinterpret_cast<unsigned char *>(ws + w.a) + (long long)t * nk * SEP_ABLK;
  const int r = row & 127, off0 = (r >> 3) * 256 + (r & 7) * 16;
  for (int k8 = kl; k8 < 2 * nk; k8 += 32) {
    long long V[8], any = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      V[j] = fixed_of(k8 == kl ? x[j] : value(8 * k8 + j), E);
      any |= V[j];
    }
    if (any) atomicOr(&smask[k8 >> 6], 1u << ((k8 >> 1) & 31));
    store_digits(A + (long long)(k8 >> 1) * SEP_ABLK + off0 + (k8 & 1) * 128, 4096, V);
  }
  __syncthreads();
  unsigned *mask = reinterpret_cast<unsigned *>(ws + w.mask) + (INV ? 2 * (w.R / 128) * SEP_MASK : 0) + t * SEP_MASK;
  if (threadIdx.x < SEP_MASK && smask[threadIdx.x]) atomicOr(mask + threadIdx.x, smask[threadIdx.x]);
}

template <bool INV>
struct FullSrc {
  const FullArg &p;
  struct Tile : DigitTile {
    int e, mt, nt;
  };
  __device__ __forceinline__ int total() const { return 2 * (p.w.R / 128) * (INV ? p.g.ntx : p.g.nqh / 32); }
  __device__ __forceinline__ bool tile(int v, Tile &t) const {
    const int nt = INV ? p.g.ntx : p.g.nqh / 32, nk = INV ? p.g.nqh / 16 : p.g.nkx, tr = v / nt, nm = p.w.R / 128;
    t.nt = v % nt;
    t.e = tr / nm;
    t.mt = tr % nm;
    t.A = reinterpret_cast<const unsigned char *>(p.ws + p.w.a) + (long long)tr * nk * SEP_ABLK;
    t.B = p.sep + (INV ? p.d.sep_xi : p.d.sep_xf) + ((long long)t.e * nt + t.nt) * nk * SEP_BBLK;
    t.nkj = t.ND = t.ti = 0;
    t.eb = INV ? inv_exp(p.d) : 0;
    t.masks(reinterpret_cast<const unsigned *>(p.ws + p.w.mask) + ((INV ? 2 * nm : 0) + tr) * SEP_MASK, nullptr);
    t.ex = reinterpret_cast<const int *>(p.ws + p.w.ex) + tr * 128;
    return !MDP_CHECKED || t.in_bounds(p.ws, p.ws_n, p.sep, p.sep_n, p.sep, p.sep_n, nk, p.d.dstatus);
  }
  __device__ __forceinline__ const double *out() const { return p.ws; }
  __device__ __forceinline__ long long out_n() const { return p.ws_n; }
  __device__ __forceinline__ void dest(const Tile &t, int r, int o, double *&dst, long long &step, int &cnt) const {
    const int row = t.mt * 128 + r, o0 = t.nt * 32 + o;
    step = 1;
    cnt = row < p.w.rows ? 8 : 0;
    dst = INV ? p.ws + p.w.u + ((long long)t.e * p.w.R + row) * p.w.ldu + o0
              : p.ws + p.w.f + (long long)row * p.w.ldf + t.e * (p.w.ldf / 2) + o0;
  }
};

template <bool INV>
__global__ void __launch_bounds__(SG_THREADS, 1) k_full_gemm(const __grid_constant__ FullArg p, int *status) {
  pdl_wait();
  MDP_CHECK_FULL(p);
  const FullSrc<INV> src{p};
  digit_gemm(src, status);
}

// x = T_q^{-1} g along y, in place on f: a block takes 16 modes of one right-hand side (lanes 0..15 their real,
// 16..31 their imaginary parts), warp s the rows of segment s. Evanescent modes: y_n = lambda y_{n-1} + g_n
// upwards, x_n = lambda x_{n+1} + c (1 - lambda^2) y_n downwards (their composition is c sum_j
// lambda^|n-j| g_j), each with the carry of the other segments, then R's part. The others: x_n =
// phi_1 (A + F (M_2 - 2 P_2(n))) + phi_2 (B + F (2 P_1(n) - M_1)) with the running moments P_b. The
// segments of a block are spread over a cluster of 4 SMs, their rows in shared memory: the warps that hold
// the propagating modes take 3 times the others' FP64 instructions, and a warp's FP64 instruction holds
// its SM's pipe for 19 cycles (a block on one SM: 207 us for 513^2, 4 right-hand sides, 24 % of the pipe).
__device__ __forceinline__ double ipow(double x, int n) {
  double r = 1.0;
  for (; n; n >>= 1, x *= x)
    if (n & 1) r *= x;
  return r;
}
constexpr int FULL_Y_CTAS = 4, FULL_Y_WARPS = 8;   // CTAs of a cluster, most warps of one
__global__ void __cluster_dims__(1, 1, FULL_Y_CTAS) __launch_bounds__(32 * FULL_Y_WARPS) k_full_y(const __grid_constant__ FullArg p) {
  pdl_wait();
  MDP_CHECK_FULL(p);
  extern __shared__ double ysh[];   // [2][warps][32] of this CTA, [2][all warps][32], then this CTA's rows [rows][32]
  const cg::cluster_group cl = cg::this_cluster();
  const SubDesc &d = p.d;
  const SepGeo &g = p.g;
  const FullWs &w = p.w;
  double *ws = p.ws;
  const int lane = threadIdx.x, nw = blockDim.y, NW = nw * FULL_Y_CTAS, s = blockIdx.z * nw + threadIdx.y;
  const int Nt = d.Nt, N = d.ny - 1;
  const int ci = blockIdx.x * 16 + (lane & 15), im = lane >> 4, e = ci / g.nqh, q = sep_parity_mode(e, ci - e * g.nqh);
  const bool live = q <= d.Nq;
  const int seg = (Nt + NW - 1) / NW, i0 = min(Nt, s * seg), i1 = min(Nt, i0 + seg);
  const long long gstep = 2LL * w.ldf;
  double *fg = ws + w.f + (long long)blockIdx.y * Nt * gstep + im * w.ldf + ci;
  double *f = ysh + (2 * nw + 2 * NW) * 32 + lane - 32LL * blockIdx.z * nw * seg;   // row i: f[32 i]
#pragma unroll 8
  for (int i = i0; i < i1; ++i) f[32 * i] = fg[i * gstep];   // a thread reads only what it writes
  const double *T = reinterpret_cast<const double *>(p.sep + d.sep_mx) + (long long)(live ? q - 1 : 0) * SEP_MXW;
  const int kind = (int)T[MX_KIND];
  const double lam = T[MX_LAM], sg = T[MX_SG];
  // what every segment has to say, gathered from the cluster's CTAs after each exchange
  double *mine0 = ysh, *mine1 = ysh + nw * 32, *sh0 = ysh + 2 * nw * 32, *sh1 = sh0 + NW * 32;
  const int me = threadIdx.y * 32 + lane;
  auto exchange = [&](double a, double b) {
    mine0[me] = a;
    mine1[me] = b;
    cl.sync();
    for (int k = threadIdx.y; k < NW; k += nw) {
      const double *r0 = cl.map_shared_rank(mine0, k / nw), *r1 = cl.map_shared_rank(mine1, k / nw);
      sh0[k * 32 + lane] = r0[(k % nw) * 32 + lane];
      sh1[k * 32 + lane] = r1[(k % nw) * 32 + lane];
    }
    cl.sync();   // the values may be overwritten, and the CTA may end
  };
  // the other part of a lane's mode: (re, im) of a value that this lane holds one part of
  auto both = [&](double v) { const double o = __shfl_xor_sync(0xffffffffu, v, 16); return im ? cmk(o, v) : cmk(v, o); };
  auto part = [&](cplx v) { return im ? v.im : v.re; };
  // rotation state of kinds 0, 1 at the segment's first row
  double ss = 0.0, c1 = 0.0, C0 = 0.0, S0 = 0.0, w0 = 1.0, a = 0.0, b = 0.0;
  if (live && kind < 2) {
    ss = T[MX_SS];
    c1 = T[MX_CS1];
    C0 = T[MX_CS0];
    S0 = T[MX_CS0 + 1];
    double Cp = c1, Sp = 1.0;   // the rotation by 1, 2, 4, ... rows
    for (int m = i0 + d.nfirst; m; m >>= 1) {
      if (m & 1) { const double Cn = fma(S0 * ss, Sp, C0 * Cp); S0 = fma(S0, Cp, C0 * Sp); C0 = Cn; }
      const double Cq = fma(Sp * ss, Sp, Cp * Cp);
      Sp = 2.0 * Sp * Cp;
      Cp = Cq;
    }
    w0 = sg < 0.0 && ((i0 + d.nfirst) & 1) ? -1.0 : 1.0;
    double C = C0, S = S0, v = w0;
    for (int i = i0; i < i1; ++i) {
      const double gv = v * f[32 * i];
      a = fma(C, gv, a);
      b = fma(S, gv, b);
      const double Cn = fma(S, ss, C * c1);
      S = fma(S, c1, C);
      C = Cn;
      v *= sg;
    }
  } else if (live) {
#pragma unroll 4
    for (int i = i0; i < i1; ++i) a = fma(lam, a, f[32 * i]);
  }
  exchange(a, b);
  const double ll = kind == 2 ? ipow(lam, seg) : 0.0;   // lambda^seg
  double ytop = 0.0, m1 = 0.0, m2 = 0.0, p1 = 0.0, p2 = 0.0;
  if (live && kind == 2) {
    double y = 0.0;
    for (int k = 0; k < s; ++k) y = fma(ll, y, sh0[k * 32 + lane]);
#pragma unroll 4
    for (int i = i0; i < i1; ++i) {   // upwards
      y = fma(lam, y, f[32 * i]);
      f[32 * i] = y;
    }
    ytop = y;
    a = 0.0;                          // the segment's part of the downward sum, sum lambda^(i - i0) y_i
#pragma unroll 4
    for (int i = i1 - 1; i >= i0; --i) a = fma(lam, a, f[32 * i]);
  } else if (live) {
    for (int k = 0; k < NW; ++k) {
      const double u = sh0[k * 32 + lane], v = sh1[k * 32 + lane];
      if (k < s) { p1 += u; p2 += v; }
      m1 += u;
      m2 += v;
    }
  }
  const cplx R11 = ld2(T + MX_R), R12 = ld2(T + MX_R + 2), R22 = ld2(T + MX_R + 4);
  {   // every lane takes part in the exchange; kind 2 has no moments yet
    const cplx M1 = both(m1), M2 = both(m2);
    if (live && kind < 2) {
      const double F = T[MX_F];
      const double A = fma(F, m2, part(cadd(cmul(R11, M1), cmul(R12, M2)))), B = fma(-F, m1, part(cadd(cmul(R12, M1), cmul(R22, M2))));
      double C = C0, S = S0, v = w0;
      for (int i = i0; i < i1; ++i) {
        const double gv = v * f[32 * i];
        p1 = fma(C, gv, p1);
        p2 = fma(S, gv, p2);
        f[32 * i] = v * fma(C, fma(-2.0 * F, p2, A), S * fma(2.0 * F, p1, B));
        const double Cn = fma(S, ss, C * c1);
        S = fma(S, c1, C);
        C = Cn;
        v *= sg;
      }
    }
  }
  const double c = T[MX_C], cc = T[MX_C1];
  exchange(cc * a, ytop);
  // the top row takes x = c y there: as if the row above held c lambda y. Empty last segments pass on.
  const int last = (Nt - 1) / seg;
  const double yt = sh1[last * 32 + lane];
  double x = c * lam * yt, mine = x;   // x just above segment k
  for (int k = last; k >= 0; --k) {
    if (k == s) mine = x;
    const int len = min(seg, Nt - k * seg);
    x = fma(len == seg ? ll : ipow(lam, len), x, sh0[k * 32 + lane]);
  }
  // moments of phi = (lambda^n, lambda^(N-n)) from the two ends: c M_1 is x continued to row 0, M_2 is y at row N
  const double e1 = d.nfirst ? lam : 1.0;
  const cplx M1 = both(kind == 2 ? e1 * x * T[MX_CI] : 0.0), M2 = both(e1 * yt);
  if (live && kind == 2) {
    const double A = part(cadd(cmul(R11, M1), cmul(R12, M2))), B = part(cadd(cmul(R12, M1), cmul(R22, M2)));
    const int nt = i1 - 1 + d.nfirst;   // grid row of the segment's last row
    const float l2 = (float)T[MX_L2];
    x = mine;
    // 2^-90 of the reflected waves is zero to working precision: the rows far from both ends
    if (__all_sync(__activemask(), l2 * (i0 + d.nfirst) < -90.0f && l2 * (N - nt) < -90.0f)) {
#pragma unroll 4
      for (int i = i1 - 1; i >= i0; --i) {
        x = fma(lam, x, cc * f[32 * i]);
        fg[i * gstep] = x;
      }
    } else {
      const double li = T[MX_LI];
      double pa = i1 > i0 ? ipow(lam, nt) : 0.0, pb = i1 > i0 ? ipow(lam, N - nt) : 0.0;
#pragma unroll 4
      for (int i = i1 - 1; i >= i0; --i) {
        x = fma(lam, x, cc * f[32 * i]);
        fg[i * gstep] = fma(pa, A, fma(pb, B, x));
        pa *= li;
        pb *= lam;
      }
    }
  } else if (live) {
    for (int i = i0; i < i1; ++i) fg[i * gstep] = f[32 * i];
  }
}

// u(m) = U_0 + U_1, u(Nx - m) = U_0 - U_1 on the unknown rows, 0 on the Dirichlet ends.
__global__ void __launch_bounds__(256) k_full_out(const __grid_constant__ FullArg p, double2 *u) {
  pdl_wait();
  MDP_CHECK_FULL(p);
  const SubDesc &d = p.d;
  const FullWs &w = p.w;
  const double *ws = p.ws;
  const int m = blockIdx.x * blockDim.x + threadIdx.x, n = blockIdx.y, rl = blockIdx.z, i = n - d.nfirst, N = d.Nx;
  if (2 * m > N) return;
  double2 up = make_double2(0.0, 0.0), um = up;
  if (m >= 1 && i >= 0 && i < d.Nt) {
    const double *U = ws + w.u + (2LL * (rl * (long long)d.Nt + i)) * w.ldu + m - 1;
    const long long other = (long long)w.R * w.ldu;
    const double a = U[0], b = U[other], ai = U[w.ldu], bi = U[other + w.ldu];
    up = make_double2(a + b, ai + bi);
    um = make_double2(a - b, ai - bi);
  }
  double2 *row = u + ((long long)rl * d.ny + n) * d.nx;
  row[m] = up;
  if (2 * m != N) row[N - m] = um;
}

}  // namespace

static constexpr int FULL_Y_SMEM = 227 * 1024;

cudaError_t set_full_kernel_attributes() {
  cudaError_t e = cudaFuncSetAttribute(k_full_gemm<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_full_gemm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_full_y, cudaFuncAttributeMaxDynamicSharedMemorySize, FULL_Y_SMEM);
  return e;
}

// k_full_y keeps a quarter of the rows of 32 columns in a CTA's shared memory (157 KB at 2459 rows); above some
// 3500 rows they do not fit and the solve goes by the factors.
static int full_y_smem(int nw, int seg) { return ((2 + 2 * FULL_Y_CTAS) * nw + nw * seg) * 256; }
bool full_solve_fits(const SubDesc &d) {
  const int nw = FULL_Y_WARPS;   // the widest segments' and the most warps' need
  return full_y_smem(nw, (d.Nt + nw * FULL_Y_CTAS - 1) / (nw * FULL_Y_CTAS) + 1) <= FULL_Y_SMEM;
}

cudaError_t launch_full_solve(const mdp_plan *p, int sub, int nrhs, const double2 *g, double2 *u, cudaStream_t st) {
  const SubDesc &d = p->subs[sub].d;
  const SepGeo geo = sep_geo(d);
  // right-hand sides per pass: as many as the workspace and a grid's z limit take
  int chunk = (int)std::min<long long>(std::min(nrhs, 32768), std::max<long long>(1, p->ws_doubles / full_ws(d, 1).total));
  while (chunk > 1 && full_ws(d, chunk).total > p->ws_doubles) --chunk;
  if (full_ws(d, chunk).total > p->ws_doubles) return cudaErrorMemoryAllocation;

  for (int r0 = 0; r0 < nrhs; r0 += chunk) {
    const int nr = std::min(chunk, nrhs - r0);
    const FullWs w = full_ws(d, nr);
    // segments along y, a multiple of the cluster's 4: of about 64 rows where the blocks fill the chip (each
    // segment has a fixed cost of some 60 FP64 instructions), else of 16
    const int rows = nr * (w.ldf / 16) >= 2 * p->n_sm ? 64 : 16;
    const int nw = std::min(FULL_Y_WARPS, std::max(1, (d.Nt + rows * FULL_Y_CTAS - 1) / (rows * FULL_Y_CTAS)));
    const int seg = (d.Nt + nw * FULL_Y_CTAS - 1) / (nw * FULL_Y_CTAS);
    const int ysm = full_y_smem(nw, seg);
    const double2 *gc = g + (long long)r0 * d.nx * d.ny;
    double2 *uc = u + (long long)r0 * d.nx * d.ny;
    auto gemm_grid = [&](int nt) { return dim3((unsigned)std::min(p->n_sm, 2 * (w.R / 128) * nt)); };
    cudaError_t e = cudaMemsetAsync(p->d_ws + w.mask, 0, 2LL * (w.R / 128) * SEP_MASK * 8, st);
    if (e != cudaSuccess) return e;
    FullArg a{d, geo, w, nr, p->d_sep, p->d_ws, p->ws_doubles, p->sep_bytes};
#if MDP_CHECKED
    const char *fault = std::getenv("MDP_FAULT_INJECT");   // "full": the mode space past the workspace's end
    if (fault && !std::strcmp(fault, "full")) a.w.f = p->ws_doubles;
#endif
    pdl(k_full_cut<false>, dim3(w.R / 8, 2), dim3(256), 0, st, a, gc);
    pdl(k_full_gemm<false>, dim3(gemm_grid(geo.nqh / 32)), dim3(SG_THREADS), SG_SMEM, st, a, p->d_status);
    pdl(k_full_y, dim3(w.ldf / 16, nr, FULL_Y_CTAS), dim3(32, nw), ysm, st, a);
    pdl(k_full_cut<true>, dim3(w.R / 8, 2), dim3(256), 0, st, a, gc);
    pdl(k_full_gemm<true>, dim3(gemm_grid(geo.ntx)), dim3(SG_THREADS), SG_SMEM, st, a, p->d_status);
    const int nm = d.Nx / 2 + 1, tm = std::min(256, (nm + 31) / 32 * 32);
    pdl(k_full_out, dim3((nm + tm - 1) / tm, d.ny, nr), dim3(tm), 0, st, a, uc);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace mdp
