// Full-grid solves u = G^(h) g (Section 3.2.1) for subdomains with the separable tables: sine transforms
// along x as digit contractions on the tensor cores (digit_gemm.cuh: every row of the grid against the
// sines, odd and even modes on folded columns), and per mode the closed form of T_q^{-1} along y,
//   x_n = sum_j kappa(|n - j|) g_j + phi(n)^T R M,   M_b = sum_j phi_b(j) g_j
// (kernels_sep.cu), by first-order recurrences over segments of rows that run in parallel.
//
// Four kernels a pass: k_full_cut, k_full_gemm (forward), k_full_y, then cut and gemm again (inverse) and
// k_full_out. They replaced direct O(N^2) sums on the FP64 pipe and one thread per mode sweeping an
// uncoalesced column: 257^2, 32 right-hand sides 3.85 ms, 513^2, 4 right-hand sides 4.2 ms.
#include "sep_modes.cuh"

#include <algorithm>

namespace mdp {

// per mode: kind, theta, lambda (with its sign), kappa(0) = c, c (1 - lambda^2), sign, R11, R12, R22, F
enum { MX_KIND = 0, MX_TH, MX_LAM, MX_C, MX_C1, MX_SG, MX_R = 6, MX_F = 12 };

// The table of the solve along y, over all rows 0 .. N: evanescent modes phi = (lambda^n, lambda^(N-n)),
// the others C and S about the middle row.
__global__ void k_full_modes(const SubDesc *subs, int s0, unsigned char *sep) {
  const int si = s0 + blockIdx.y;
  const SubDesc &d = subs[si];
  const int q = blockIdx.x * 128 + threadIdx.x + 1;
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
  T[MX_KIND] = m.kind; T[MX_TH] = m.th; T[MX_LAM] = lam; T[MX_C] = c;
  T[MX_C1] = -c * expm1(-2.0 * m.th);
  T[MX_SG] = m.sg;
  T[MX_R] = R11.re; T[MX_R + 1] = R11.im; T[MX_R + 2] = R12.re; T[MX_R + 3] = R12.im;
  T[MX_R + 4] = R22.re; T[MX_R + 5] = R22.im;
  T[MX_F] = 1.0 / (2.0 * m.a);
}

namespace {

// A: the grid's rows on folded columns (INV false: g(m) +- g(Nx - m)) or the modes (INV), cut into digits.
// Row order (right-hand side, unknown row, part): a block's 8 rows are 4 grid rows, complex parts in turn.
template <bool INV>
__global__ void __launch_bounds__(256) k_full_cut(const SubDesc *subs, int sub, const double2 *g, double *ws, int nr) {
  const SubDesc &d = subs[sub];
  const SepGeo geo = sep_geo(d);
  const FullWs w = full_ws(d, nr);
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
  const int E = max(emax[threadIdx.x & 7], 53), t = e * (w.R / 128) + row / 128;
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
  const SubDesc *subs;
  int sub, nr;
  const unsigned char *sep;
  double *ws;
  struct Tile : DigitTile {
    int e, mt, nt;
  };
  __device__ __forceinline__ int total() const {
    const SubDesc &d = subs[sub];
    const SepGeo g = sep_geo(d);
    return 2 * (full_ws(d, nr).R / 128) * (INV ? g.ntx : g.nqh / 32);
  }
  __device__ __forceinline__ bool tile(int v, Tile &t) const {
    const SubDesc &d = subs[sub];
    const SepGeo g = sep_geo(d);
    const FullWs w = full_ws(d, nr);
    const int nt = INV ? g.ntx : g.nqh / 32, nk = INV ? g.nqh / 16 : g.nkx, tr = v / nt;
    t.nt = v % nt;
    t.e = tr / (w.R / 128);
    t.mt = tr % (w.R / 128);
    t.A = reinterpret_cast<const unsigned char *>(ws + w.a) + (long long)tr * nk * SEP_ABLK;
    t.B = sep + (INV ? d.sep_xi : d.sep_xf) + ((long long)t.e * nt + t.nt) * nk * SEP_BBLK;
    t.nkj = t.ND = t.ti = t.eb = 0;
    t.ma = reinterpret_cast<const unsigned *>(ws + w.mask) + ((INV ? 2 * (w.R / 128) : 0) + tr) * SEP_MASK;
    t.mb = nullptr;
    t.ex = reinterpret_cast<const int *>(ws + w.ex) + tr * 128;
    return true;
  }
  __device__ __forceinline__ void dest(const Tile &t, int r, int o, double *&dst, long long &step, int &cnt) const {
    const SubDesc &d = subs[sub];
    const FullWs w = full_ws(d, nr);
    const int row = t.mt * 128 + r, o0 = t.nt * 32 + o;
    step = 1;
    cnt = row < w.rows ? 16 : 0;
    dst = INV ? ws + w.u + ((long long)t.e * w.R + row) * w.ldu + o0
              : ws + w.f + (long long)row * w.ldf + t.e * (w.ldf / 2) + o0;
  }
};

template <bool INV>
__global__ void __launch_bounds__(SG_THREADS, 1)
    k_full_gemm(const SubDesc *subs, int sub, int nr, const unsigned char *sep, double *ws, int *status) {
  const FullSrc<INV> src{subs, sub, nr, sep, ws};
  digit_gemm(src, status);
}

// x = T_q^{-1} g along y, in place on f: a block takes 32 modes of one right-hand side, warp s the rows of
// segment s. Evanescent modes: y_n = lambda y_{n-1} + g_n upwards, x_n = lambda x_{n+1} + c (1 - lambda^2) y_n
// downwards (their composition is c sum_j lambda^|n-j| g_j), each with the carry of the other segments,
// then R's part. The others: x_n = phi_1 (A + F (M_2 - 2 P_2(n))) + phi_2 (B + F (2 P_1(n) - M_1)) with the running
// moments P_b. Bound by the chain of dependent FP64 operations of a segment (3 passes of its rows) and
// by reading f three times, mostly from L2.
__global__ void __launch_bounds__(768) k_full_y(const SubDesc *subs, int sub, const unsigned char *sep, double *ws, int nr) {
  extern __shared__ double ysh[];   // [4][warps][32]
  const SubDesc &d = subs[sub];
  const SepGeo g = sep_geo(d);
  const FullWs w = full_ws(d, nr);
  const int lane = threadIdx.x, s = threadIdx.y, NW = blockDim.y, Nt = d.Nt, N = d.ny - 1;
  const int ci = blockIdx.x * 32 + lane, e = ci / g.nqh, q = sep_parity_mode(e, ci - e * g.nqh);
  const bool live = q <= d.Nq;
  const int seg = (Nt + NW - 1) / NW, i0 = min(Nt, s * seg), i1 = min(Nt, i0 + seg);
  const long long step = 2LL * w.ldf;
  double *f = ws + w.f + (long long)blockIdx.y * Nt * step + ci;   // row i: f[i step], its imaginary part ldf on
  const double *T = reinterpret_cast<const double *>(sep + d.sep_mx) + (long long)(live ? q - 1 : 0) * SEP_MXW;
  const int kind = (int)T[MX_KIND];
  const double th = T[MX_TH], lam = T[MX_LAM], sg = T[MX_SG];
  double *sh[4];
  for (int k = 0; k < 4; ++k) sh[k] = ysh + (k * NW) * 32;
  const int me = s * 32 + lane;
  // rotation state of kinds 0, 1 at the segment's first row
  const double sth = kind == 0 ? sin(th) : sinh(th), ss = kind == 0 ? -sth * sth : sth * sth;
  const double c1 = kind < 2 ? sep_c(kind, th, 1.0) : 0.0;
  double C0 = 0.0, S0 = 0.0, w0 = 1.0;
  cplx a = cmk(0.0, 0.0), b = a;
  if (live) {
    if (kind == 2) {
      for (int i = i0; i < i1; ++i) {
        a.re = fma(lam, a.re, f[i * step]);
        a.im = fma(lam, a.im, f[i * step + w.ldf]);
      }
    } else {
      const double x = i0 + d.nfirst - 0.5 * N;
      C0 = sep_c(kind, th, x); S0 = sep_s(kind, th, x);
      w0 = sg < 0.0 && ((i0 + d.nfirst) & 1) ? -1.0 : 1.0;
      double C = C0, S = S0, v = w0;
      for (int i = i0; i < i1; ++i) {
        const double gr = v * f[i * step], gi = v * f[i * step + w.ldf];
        a = cmk(fma(C, gr, a.re), fma(C, gi, a.im));
        b = cmk(fma(S, gr, b.re), fma(S, gi, b.im));
        const double Cn = fma(S, ss, C * c1);
        S = fma(S, c1, C);
        C = Cn;
        v *= sg;
      }
    }
  }
  sh[0][me] = a.re; sh[1][me] = a.im; sh[2][me] = b.re; sh[3][me] = b.im;
  __syncthreads();
  const double ll = kind == 2 ? exp(-th * seg) * (sg < 0.0 && (seg & 1) ? -1.0 : 1.0) : 0.0;   // lambda^seg
  cplx ytop = cmk(0.0, 0.0);
  if (live && kind == 2) {
    cplx y = cmk(0.0, 0.0);
    for (int k = 0; k < s; ++k) { y.re = fma(ll, y.re, sh[0][k * 32 + lane]); y.im = fma(ll, y.im, sh[1][k * 32 + lane]); }
    // upwards; on the way the segment's part of the downward sum, a = sum lambda^(i - i0) y_i
    double pw = 1.0;
    a = cmk(0.0, 0.0);
    for (int i = i0; i < i1; ++i) {
      y.re = fma(lam, y.re, f[i * step]);
      y.im = fma(lam, y.im, f[i * step + w.ldf]);
      f[i * step] = y.re;
      f[i * step + w.ldf] = y.im;
      a.re = fma(pw, y.re, a.re);
      a.im = fma(pw, y.im, a.im);
      pw *= lam;
    }
    ytop = y;
  } else if (live) {
    cplx m1 = cmk(0.0, 0.0), m2 = m1, p1 = m1, p2 = m1;
    for (int k = 0; k < NW; ++k) {
      const cplx u = cmk(sh[0][k * 32 + lane], sh[1][k * 32 + lane]), v = cmk(sh[2][k * 32 + lane], sh[3][k * 32 + lane]);
      if (k < s) { p1 = cadd(p1, u); p2 = cadd(p2, v); }
      m1 = cadd(m1, u);
      m2 = cadd(m2, v);
    }
    const cplx R11 = ld2(T + MX_R), R12 = ld2(T + MX_R + 2), R22 = ld2(T + MX_R + 4);
    const double F = T[MX_F];
    const cplx A = caxpy(F, m2, cadd(cmul(R11, m1), cmul(R12, m2))), B = caxpy(-F, m1, cadd(cmul(R12, m1), cmul(R22, m2)));
    double C = C0, S = S0, v = w0;
    for (int i = i0; i < i1; ++i) {
      const double gr = v * f[i * step], gi = v * f[i * step + w.ldf];
      p1 = cmk(fma(C, gr, p1.re), fma(C, gi, p1.im));
      p2 = cmk(fma(S, gr, p2.re), fma(S, gi, p2.im));
      f[i * step] = v * fma(C, fma(-2.0 * F, p2.re, A.re), S * fma(2.0 * F, p1.re, B.re));
      f[i * step + w.ldf] = v * fma(C, fma(-2.0 * F, p2.im, A.im), S * fma(2.0 * F, p1.im, B.im));
      const double Cn = fma(S, ss, C * c1);
      S = fma(S, c1, C);
      C = Cn;
      v *= sg;
    }
  }
  __syncthreads();
  sh[0][me] = a.re; sh[1][me] = a.im; sh[2][me] = ytop.re; sh[3][me] = ytop.im;
  __syncthreads();
  if (!live || kind != 2) return;
  const double c = T[MX_C], cc = T[MX_C1];
  // the top row takes x = c y there: as if the row above held c lambda y. Empty last segments pass on.
  const int last = (Nt - 1) / seg;
  const cplx yt = cmk(sh[2][last * 32 + lane], sh[3][last * 32 + lane]);
  cplx x = cmk(c * lam * yt.re, c * lam * yt.im), mine = x;   // x just above segment k
  for (int k = last; k >= 0; --k) {
    if (k == s) mine = x;
    const int len = min(seg, Nt - k * seg);
    const double l = len == seg ? ll : exp(-th * len) * (sg < 0.0 && (len & 1) ? -1.0 : 1.0);
    x.re = fma(l, x.re, cc * sh[0][k * 32 + lane]);
    x.im = fma(l, x.im, cc * sh[1][k * 32 + lane]);
  }
  if (i0 >= i1) return;
  // moments of phi = (lambda^n, lambda^(N-n)) from the two ends: c M_1 is x continued to row 0, M_2 is y at row N
  const double e1 = d.nfirst ? lam : 1.0;
  const cplx m1 = cmk(e1 * x.re / c, e1 * x.im / c), m2 = cmk(e1 * yt.re, e1 * yt.im);
  const cplx R11 = ld2(T + MX_R), R12 = ld2(T + MX_R + 2), R22 = ld2(T + MX_R + 4);
  const cplx A = cadd(cmul(R11, m1), cmul(R12, m2)), B = cadd(cmul(R12, m1), cmul(R22, m2));
  const int nt = i1 - 1 + d.nfirst;   // grid row of the segment's last row
  double pa = exp(-th * nt) * (sg < 0.0 && (nt & 1) ? -1.0 : 1.0), pb = exp(-th * (N - nt)) * (sg < 0.0 && ((N - nt) & 1) ? -1.0 : 1.0);
  const double li = 1.0 / lam;
  x = mine;
  for (int i = i1 - 1; i >= i0; --i) {
    x.re = fma(lam, x.re, cc * f[i * step]);
    x.im = fma(lam, x.im, cc * f[i * step + w.ldf]);
    f[i * step] = fma(pa, A.re, fma(pb, B.re, x.re));
    f[i * step + w.ldf] = fma(pa, A.im, fma(pb, B.im, x.im));
    pa *= li;
    pb *= lam;
  }
}

// u(m) = (2/Nx) (U_0 + U_1), u(Nx - m) = (2/Nx) (U_0 - U_1) on the unknown rows, 0 on the Dirichlet ends.
__global__ void __launch_bounds__(128) k_full_out(const SubDesc *subs, int sub, const double *ws, double2 *u, int nr) {
  const SubDesc &d = subs[sub];
  const FullWs w = full_ws(d, nr);
  const int m = blockIdx.x * 128 + threadIdx.x, n = blockIdx.y, rl = blockIdx.z, i = n - d.nfirst, N = d.Nx;
  if (2 * m > N) return;
  double2 p = make_double2(0.0, 0.0), q = p;
  if (m >= 1 && i >= 0 && i < d.Nt) {
    const double *U = ws + w.u + (2LL * (rl * (long long)d.Nt + i)) * w.ldu + m - 1;
    const long long other = (long long)w.R * w.ldu;
    const double sc = 2.0 / N, a = U[0], b = U[other], ai = U[w.ldu], bi = U[other + w.ldu];
    p = make_double2(sc * (a + b), sc * (ai + bi));
    q = make_double2(sc * (a - b), sc * (ai - bi));
  }
  double2 *row = u + ((long long)rl * d.ny + n) * d.nx;
  row[m] = p;
  if (2 * m != N) row[N - m] = q;
}

}  // namespace

cudaError_t set_full_kernel_attributes() {
  cudaError_t e = cudaFuncSetAttribute(k_full_gemm<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_full_gemm<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM);
  return e;
}

cudaError_t launch_full_solve(const mdp_plan *p, int sub, int nrhs, const double2 *g, double2 *u, cudaStream_t st) {
  const SubDesc &d = p->subs[sub].d;
  const SepGeo geo = sep_geo(d);
  // right-hand sides per pass: as many as the workspace and a grid's z limit take
  int chunk = (int)std::min<long long>(std::min(nrhs, 32768), std::max<long long>(1, p->ws_doubles / full_ws(d, 1).total));
  while (chunk > 1 && full_ws(d, chunk).total > p->ws_doubles) --chunk;
  if (full_ws(d, chunk).total > p->ws_doubles) return cudaErrorMemoryAllocation;
  // segments of about 16 rows along y, at most 24 (768 threads of 80 registers)
  const int nw = std::min(24, (d.Nt + 15) / 16);
  for (int r0 = 0; r0 < nrhs; r0 += chunk) {
    const int nr = std::min(chunk, nrhs - r0);
    const FullWs w = full_ws(d, nr);
    const double2 *gc = g + (long long)r0 * d.nx * d.ny;
    double2 *uc = u + (long long)r0 * d.nx * d.ny;
    auto gemm_grid = [&](int nt) { return dim3((unsigned)std::min(p->n_sm, 2 * (w.R / 128) * nt)); };
    cudaError_t e = cudaMemsetAsync(p->d_ws + w.mask, 0, 2LL * (w.R / 128) * SEP_MASK * 8, st);
    if (e != cudaSuccess) return e;
    k_full_cut<false><<<dim3(w.R / 8, 2), 256, 0, st>>>(p->d_subs, sub, gc, p->d_ws, nr);
    k_full_gemm<false><<<gemm_grid(geo.nqh / 32), SG_THREADS, SG_SMEM, st>>>(p->d_subs, sub, nr, p->d_sep, p->d_ws, p->d_status);
    k_full_y<<<dim3(w.ldf / 32, nr), dim3(32, nw), 4 * nw * 32 * sizeof(double), st>>>(p->d_subs, sub, p->d_sep, p->d_ws, nr);
    k_full_cut<true><<<dim3(w.R / 8, 2), 256, 0, st>>>(p->d_subs, sub, gc, p->d_ws, nr);
    k_full_gemm<true><<<gemm_grid(geo.ntx), SG_THREADS, SG_SMEM, st>>>(p->d_subs, sub, nr, p->d_sep, p->d_ws, p->d_status);
    k_full_out<<<dim3((d.Nx / 2 + 128) / 128, d.ny, nr), 128, 0, st>>>(p->d_subs, sub, p->d_ws, uc, nr);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace mdp
