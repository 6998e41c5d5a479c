// The coupled system of a layout of subdomains (Sections 3.3-3.5): from the projection columns Q_j to the
// Chebyshev coefficients of every subdomain's boundary data, and the gradient of that map.
//
// Per subdomain the coefficients are c_j = S_j x + e_j: x the unknowns (a block of M per outer side, two per
// interface), S_j with entries 1, -1 or rho = -alpha/beta of a side, e_j the boundary data eps = d/beta (or
// d/alpha on a Dirichlet side). The least-squares system min sum_j ||Q_j c_j - f_j||^2 has block columns that
// one or two subdomains touch, and is solved by QR in the nested order of linalg.structured_qr: every
// subdomain's rows on its own columns (those no other touches first), then the stacked R_ss of the shared ones.
// Its gradient needs no factor but R: with g the gradient of the coefficients, w = (A^H A)^{-1} S^H g and
// r = f - Q c,  grad Q_j = r_j (S_j w)^H - (Q_j S_j w) c_j^H,  and with h = g - Q^H Q S w, z = Q^H r:
// grad e = h,  grad S = h x^H + z w^H.
//
// A pass is some 25 kernels where the assembly, the permutations and their gradients as single tensor
// operations were 260 (750 with the gradient), bound by their launches: 4 layers of 129^2, 24 modes per side,
// 7.4 -> 4.2 ms to the receivers, 21.7 -> 6.1 ms with the gradient by the wavenumbers (3.3 and 4.5 with the
// boundary data of all sides at once and a shorter QR). Each kernel is a stream
// over Q (10 MB there, in L2) with an FP64 product or two per element, 5 to 15 us; the triangular solves take
// the two levels' triangles, so that the chain is the shared unknowns and one subdomain's own ones instead of
// all (195 us for 144 + 72, 309 us for all 384 in one CTA).
#include "trsv.cuh"

#include "mdp.h"

namespace mdp {
namespace {

// the int tables of mdp_couple, in the order of mdp.h
struct Cp {
  int N, M, C, n, ns, ms, mmax, nmax, no, rows;
  const int *G, *nj, *pj, *s0, *r0;                       // [N]
  const int *unk, *slot0, *neg0, *slot1, *rho, *sidx;     // [N][nmax]
  const int *su, *sf, *se;                                // [N][C]
  const int *touch;                                       // [n][2]
  const int *shu;                                         // [ns]
  const int *qj, *qe, *qr, *qu;                           // [no]
  const long long *off;                                   // [N]
};
Cp unpack(const mdp_couple *c) {
  Cp p;
  p.N = c->n_blocks; p.M = c->n_modes; p.C = 8 * c->n_modes; p.n = c->n; p.ns = c->n_shared; p.ms = c->shared_rows;
  p.mmax = c->max_rows; p.nmax = c->max_cols; p.no = c->n_outer; p.rows = c->rows;
  const int *t = c->tables;
  auto take = [&](long long k) { const int *q = t; t += k; return q; };
  p.G = take(p.N); p.nj = take(p.N); p.pj = take(p.N); p.s0 = take(p.N); p.r0 = take(p.N);
  const long long nn = (long long)p.N * p.nmax, nc = (long long)p.N * p.C;
  p.unk = take(nn); p.slot0 = take(nn); p.neg0 = take(nn); p.slot1 = take(nn); p.rho = take(nn); p.sidx = take(nn);
  p.su = take(nc); p.sf = take(nc); p.se = take(nc);
  p.touch = take(2LL * p.n);
  p.shu = take(p.ns);
  p.qj = take(p.no); p.qe = take(p.no); p.qr = take(p.no); p.qu = take(p.no);
  p.off = c->offsets;
  return p;
}

__device__ __forceinline__ double2 c2add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 c2fma(double2 a, double2 b, double2 c) {   // a b + c
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
__device__ __forceinline__ double2 c2cfma(double2 a, double2 b, double2 c) {   // conj(a) b + c
  return make_double2(fma(a.x, b.x, fma(a.y, b.y, c.x)), fma(a.x, b.y, fma(-a.y, b.x, c.y)));
}
__device__ __forceinline__ double2 zero2() { return make_double2(0.0, 0.0); }

// cv = S x + eps (either may be null: left out)
__global__ void __launch_bounds__(128) k_cp_vec(Cp p, const double2 *x, const double2 *rho, const double2 *eps, double2 *cv) {
  pdl_wait();
  const int i = blockIdx.x * 128 + threadIdx.x;
  if (i >= p.N * p.C) return;
  double2 v = zero2();
  if (x && p.su[i] >= 0) {
    const double2 a = x[p.su[i]];
    const int f = p.sf[i];
    v = f == 0 ? a : f == 1 ? make_double2(-a.x, -a.y) : c2mul(rho[f - 2], a);
  }
  if (eps && p.se[i] >= 0) v = c2add(v, eps[p.se[i]]);
  cv[i] = v;
}

// y_t(rows of block j) = sg_t B_j v_t (+ add for t = 0), B_j stored [C][len_j] from off_j. A block takes 32 rows;
// its 16 warps split the columns, summed in order.
template <int T>
__global__ void __launch_bounds__(512) k_cp_gemv(const double2 *B, const long long *off, const int *len, const int *yoff, int C,
                                                 const double2 *v, long long vs, double2 *y, long long ys, double sg0,
                                                 double sg1, const double2 *add) {
  pdl_wait();
  __shared__ double2 sh[T][16][32];
  const int j = blockIdx.y, L = len[j], g = blockIdx.x * 32 + threadIdx.x;
  if (blockIdx.x * 32 >= L) return;
  const double2 *b = B + off[j] + g, *vj = v + (long long)j * C;
  double2 acc[T];
#pragma unroll
  for (int t = 0; t < T; ++t) acc[t] = zero2();
  if (g < L)
#pragma unroll 4
    for (int c = threadIdx.y; c < C; c += 16) {
      const double2 a = b[(long long)c * L];
#pragma unroll
      for (int t = 0; t < T; ++t) acc[t] = c2fma(a, vj[t * vs + c], acc[t]);
    }
#pragma unroll
  for (int t = 0; t < T; ++t) sh[t][threadIdx.y][threadIdx.x] = acc[t];
  __syncthreads();
  if (threadIdx.y >= T || g >= L) return;
  const int t = threadIdx.y;
  double2 s = sh[t][0][threadIdx.x];
  for (int w = 1; w < 16; ++w) s = c2add(s, sh[t][w][threadIdx.x]);
  const double sg = t == 0 ? sg0 : sg1;
  s = make_double2(sg * s.x, sg * s.y);
  const long long o = yoff[j] + g;
  if (t == 0 && add) s = c2add(s, add[o]);
  y[t * ys + o] = s;
}

// block totals of T complex values per thread (128 threads), returned to thread 0
template <int T>
__device__ __forceinline__ void block_total(double2 (&a)[T]) {
  __shared__ double2 sh[4][T];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    for (int o = 16; o > 0; o >>= 1) {
      a[t].x += __shfl_xor_sync(0xffffffffu, a[t].x, o);
      a[t].y += __shfl_xor_sync(0xffffffffu, a[t].y, o);
    }
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][t] = a[t];
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < T; ++t) a[t] = c2add(c2add(sh[0][t], sh[1][t]), c2add(sh[2][t], sh[3][t]));
}

// z_t = B_j^H u_t: one block per column
template <int T>
__global__ void __launch_bounds__(128) k_cp_dots(const double2 *B, const long long *off, const int *len, const int *yoff, int C,
                                                 const double2 *u, long long us, double2 *z, long long zs) {
  pdl_wait();
  const int c = blockIdx.x, j = blockIdx.y, L = len[j];
  const double2 *b = B + off[j] + (long long)c * L, *uj = u + yoff[j];
  double2 acc[T];
#pragma unroll
  for (int t = 0; t < T; ++t) acc[t] = zero2();
#pragma unroll 4
  for (int g = threadIdx.x; g < L; g += 128) {
    const double2 a = b[g];
#pragma unroll
    for (int t = 0; t < T; ++t) acc[t] = c2cfma(a, uj[t * us + g], acc[t]);
  }
  block_total(acc);
  if (threadIdx.x == 0)
#pragma unroll
    for (int t = 0; t < T; ++t) z[t * zs + (long long)j * C + c] = acc[t];
}

// grad B_j = u_0 a^H - u_1 b^H (T = 1: the first term)
template <int T>
__global__ void __launch_bounds__(128) k_cp_outer(const long long *off, const int *len, const int *yoff, int C, const double2 *u,
                                                  long long us, const double2 *a, const double2 *b, double2 *gB) {
  pdl_wait();
  const int c = blockIdx.y, j = blockIdx.z, L = len[j], g = blockIdx.x * 128 + threadIdx.x;
  if (g >= L) return;
  const double2 ac = a[(long long)j * C + c], u0 = u[yoff[j] + g];
  double2 v = c2cfma(ac, u0, zero2());
  if (T == 2) {
    const double2 bc = b[(long long)j * C + c], u1 = u[us + yoff[j] + g];
    v = c2cfma(make_double2(-bc.x, -bc.y), u1, v);
  }
  gB[off[j] + (long long)c * L + g] = v;
}

// the column of A of local column p of block j, at row g
__device__ __forceinline__ double2 a_entry(const Cp &p, const double2 *Q, const double2 *rho, long long jp, long long o, int L, int g) {
  double2 v = Q[o + (long long)p.slot0[jp] * L + g];
  if (p.neg0[jp]) v = make_double2(-v.x, -v.y);
  const int s1 = p.slot1[jp];
  return s1 < 0 ? v : c2fma(rho[p.rho[jp]], Q[o + (long long)s1 * L + g], v);
}

// D = 1 / the norms of A's columns: one block per unknown
__global__ void __launch_bounds__(128) k_cp_norm(Cp p, const double2 *Q, const double2 *rho, double *D) {
  pdl_wait();
  const int u = blockIdx.x;
  double2 acc[1] = {zero2()};
  for (int t = 0; t < 2; ++t) {
    const int jp = p.touch[2 * u + t];
    if (jp < 0) continue;
    const int j = jp / p.nmax, L = p.G[j];
    for (int g = threadIdx.x; g < L; g += 128) {
      const double2 a = a_entry(p, Q, rho, jp, p.off[j], L, g);
      acc[0].x = fma(a.x, a.x, fma(a.y, a.y, acc[0].x));
    }
  }
  block_total(acc);
  if (threadIdx.x == 0) D[u] = 1.0 / sqrt(acc[0].x);
}

// the subdomains' matrices [A_j D | b_j], column-major, padded with zeros to nmax + 1 columns of mmax rows
__global__ void __launch_bounds__(128) k_cp_build(Cp p, const double2 *Q, const double2 *rho, const double *D, const double2 *b,
                                                  double2 *Mx) {
  pdl_wait();
  const int g = blockIdx.x * 128 + threadIdx.x, c = blockIdx.y, j = blockIdx.z, L = p.G[j];
  if (g >= p.mmax) return;
  double2 v = zero2();
  if (g < L) {
    if (c == p.nmax) v = b[p.r0[j] + g];
    else if (c < p.nj[j]) {
      const long long jp = (long long)j * p.nmax + c;
      const double s = D[p.unk[jp]];
      v = a_entry(p, Q, rho, jp, p.off[j], L, g);
      v = make_double2(s * v.x, s * v.y);
    }
  }
  Mx[((long long)j * (p.nmax + 1) + c) * p.mmax + g] = v;
}

// [S | q_s]: the stacked R_ss of the subdomains in the shared columns
__global__ void __launch_bounds__(128) k_cp_gather(Cp p, const double2 *Mx, double2 *S) {
  pdl_wait();
  const int r = blockIdx.x * 128 + threadIdx.x, c = blockIdx.y;
  if (r >= p.ms) return;
  int j = 0;
  while (j + 1 < p.N && p.s0[j + 1] <= r) ++j;
  const int i = r - p.s0[j], pj = p.pj[j];
  const double2 *Mj = Mx + (long long)j * (p.nmax + 1) * p.mmax;
  double2 v = zero2();
  if (c == p.ns) v = Mj[(long long)p.nmax * p.mmax + pj + i];
  else
    for (int t = 0; t < 2; ++t) {
      const int jp = p.touch[2 * p.shu[c] + t];
      if (jp < 0 || jp / p.nmax != j) continue;
      const int lc = jp % p.nmax;
      if (pj + i <= lc) v = Mj[(long long)lc * p.mmax + pj + i];
    }
  S[(long long)c * p.ms + r] = v;
}

// the shared unknowns: ys = R_s^{-1} rhs, or (GRAM) R_s^{-1} R_s^{-H} (gx - the subdomains' parts)
template <bool GRAM>
__global__ void __launch_bounds__(kTrThreads) k_cp_shared(Cp p, const double2 *S, const double *D, const double2 *gx,
                                                          const double2 *part, double2 *ys, double2 *x) {
  pdl_wait();
  __shared__ TrBlock T;
  extern __shared__ __align__(16) double2 xs[];
  for (int c = threadIdx.x; c < p.ns; c += kTrThreads) {
    if (!GRAM) { xs[c] = S[(long long)p.ns * p.ms + c]; continue; }
    double2 v = gx[p.shu[c]];
    for (int t = 0; t < 2; ++t) {
      const int jp = p.touch[2 * p.shu[c] + t];
      if (jp < 0) continue;
      const double2 q = part[jp];
      v.x -= q.x;
      v.y -= q.y;
    }
    xs[c] = v;
  }
  if (GRAM) trsv_body<true>(p.ns, S, p.ms, xs, T);
  trsv_body<false>(p.ns, S, p.ms, xs, T);
  for (int c = threadIdx.x; c < p.ns; c += kTrThreads) {
    const double s = D[p.shu[c]];
    ys[c] = xs[c];
    x[p.shu[c]] = make_double2(s * xs[c].x, s * xs[c].y);
  }
}

// a subdomain's own unknowns: x_p = R_pp^{-1} (rhs - R_ps x_s), rhs from the QR's last column or (yp) given
__global__ void __launch_bounds__(kTrThreads) k_cp_private(Cp p, const double2 *Mx, const double *D, const double2 *ys,
                                                           const double2 *yp, double2 *x) {
  pdl_wait();
  __shared__ TrBlock T;
  extern __shared__ __align__(16) double2 xs[];   // [pj], then [8][pj] partial sums
  const int j = blockIdx.x, pj = p.pj[j], sj = p.nj[j] - pj, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double2 *Mj = Mx + (long long)j * (p.nmax + 1) * p.mmax;
  double2 *ps = xs + pj;
  for (int i = lane; i < pj; i += 32) {
    double2 s = zero2();
#pragma unroll 4
    for (int c = warp; c < sj; c += 8)
      s = c2fma(Mj[(long long)(pj + c) * p.mmax + i], ys[p.sidx[(long long)j * p.nmax + pj + c]], s);
    ps[warp * pj + i] = s;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < pj; i += kTrThreads) {
    double2 v = yp ? yp[(long long)j * p.nmax + i] : Mj[(long long)p.nmax * p.mmax + i];
    for (int w = 0; w < 8; ++w) { v.x -= ps[w * pj + i].x; v.y -= ps[w * pj + i].y; }
    xs[i] = v;
  }
  trsv_body<false>(pj, Mj, p.mmax, xs, T);
  for (int i = threadIdx.x; i < pj; i += kTrThreads) {
    const int u = p.unk[(long long)j * p.nmax + i];
    x[u] = make_double2(D[u] * xs[i].x, D[u] * xs[i].y);
  }
}

// yp = R_pp^{-H} gx_p and the subdomain's part R_ps^H yp of the shared right-hand side
__global__ void __launch_bounds__(kTrThreads) k_cp_private_h(Cp p, const double2 *Mx, const double2 *gx, double2 *yp, double2 *part) {
  pdl_wait();
  __shared__ TrBlock T;
  extern __shared__ __align__(16) double2 xs[];
  const int j = blockIdx.x, pj = p.pj[j], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double2 *Mj = Mx + (long long)j * (p.nmax + 1) * p.mmax;
  const long long jp = (long long)j * p.nmax;
  for (int i = threadIdx.x; i < pj; i += kTrThreads) xs[i] = gx[p.unk[jp + i]];
  trsv_body<true>(pj, Mj, p.mmax, xs, T);
  for (int i = threadIdx.x; i < pj; i += kTrThreads) yp[jp + i] = xs[i];
  for (int c = pj + warp; c < p.nj[j]; c += 8) {
    double2 s = zero2();
    for (int i = lane; i < pj; i += 32) s = c2cfma(Mj[(long long)c * p.mmax + i], xs[i], s);
    for (int o = 16; o > 0; o >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    if (lane == 0) part[jp + c] = s;
  }
}

// gx = D S^H g
__global__ void __launch_bounds__(128) k_cp_gx(Cp p, const double2 *g, const double2 *rho, const double *D, double2 *gx) {
  pdl_wait();
  const int u = blockIdx.x * 128 + threadIdx.x;
  if (u >= p.n) return;
  double2 v = zero2();
  for (int t = 0; t < 2; ++t) {
    const int jp = p.touch[2 * u + t];
    if (jp < 0) continue;
    const double2 *gj = g + (long long)(jp / p.nmax) * p.C;
    const double2 a = gj[p.slot0[jp]];
    v = p.neg0[jp] ? make_double2(v.x - a.x, v.y - a.y) : c2add(v, a);
    if (p.slot1[jp] >= 0) v = c2cfma(rho[p.rho[jp]], gj[p.slot1[jp]], v);
  }
  gx[u] = make_double2(D[u] * v.x, D[u] * v.y);
}

// gradients by the boundary data of an outer side: grad eps = h, grad rho = h x^H + z w^H; one block per side
__global__ void __launch_bounds__(128) k_cp_sides(Cp p, const double2 *g, const double2 *z, const double2 *x, const double2 *w,
                                                  double2 *grho, double2 *geps) {
  pdl_wait();
  const int q = blockIdx.x;
  const long long o = (long long)p.qj[q] * p.C, zs = (long long)p.N * p.C;
  const int e = p.qe[q], r = p.qr[q], u = p.qu[q];
  double2 acc[1] = {zero2()};
  for (int m = threadIdx.x; m < p.M; m += 128) {
    const double2 a = g[o + e + m], b = z[zs + o + e + m];
    geps[(long long)q * p.M + m] = make_double2(a.x - b.x, a.y - b.y);
    if (r >= 0) {
      const double2 c = g[o + r + m], d = z[zs + o + r + m];
      acc[0] = c2cfma(x[u + m], make_double2(c.x - d.x, c.y - d.y), acc[0]);
      acc[0] = c2cfma(w[u + m], z[o + r + m], acc[0]);
    }
  }
  block_total(acc);
  if (threadIdx.x == 0) grho[q] = acc[0];
}

// the buffer kept for the gradient: matrices, shared matrix, column scales; then scratch
struct CpBuf {
  long long M, S, D, tau, b, cv, ys, total;
};
CpBuf cp_buf(const Cp &p) {
  CpBuf w;
  long long o = 0;
  auto take = [&](long long k) { const long long q = o; o += (k + 15) & ~15LL; return q; };
  w.M = take((long long)p.N * (p.nmax + 1) * p.mmax);
  w.S = take((long long)(p.ns + 1) * p.ms);
  w.D = take((p.n + 1) / 2);
  w.tau = take((long long)p.N * p.nmax + p.ns);
  w.b = take(p.rows);
  w.cv = take((long long)p.N * p.C);
  w.ys = take(p.ns);
  w.total = o;
  return w;
}
struct CpGrad {
  long long gx, yp, part, ys, w, sw, u, z, total;
};
CpGrad cp_grad(const Cp &p) {
  CpGrad w;
  long long o = 0;
  auto take = [&](long long k) { const long long q = o; o += (k + 15) & ~15LL; return q; };
  w.gx = take(p.n);
  w.yp = take((long long)p.N * p.nmax);
  w.part = take((long long)p.N * p.nmax);
  w.ys = take(p.ns);
  w.w = take(p.n);
  w.sw = take(2LL * p.N * p.C);   // c, S w
  w.u = take(2LL * p.rows);       // r, A w
  w.z = take(2LL * p.N * p.C);
  w.total = o;
  return w;
}

bool valid(const mdp_couple *c) {
  return c && c->n_blocks >= 1 && c->n_blocks <= 65535 && c->n_modes >= 1 && c->n >= 1 && c->n_shared >= 0 &&
         c->n_shared <= c->n && c->shared_rows >= c->n_shared && c->max_cols >= 1 && c->max_rows >= c->max_cols &&
         c->max_cols < 65535 && c->n_outer >= 0 && c->rows >= 1 && c->tables && c->offsets && 8 * c->n_modes <= 65535 &&
         c->n_shared < 65535 && (size_t)c->n_shared * 16 <= 200 * 1024 && (size_t)c->max_cols * 9 * 16 <= 200 * 1024;
}
// dynamic shared memory beside the static 16.5 KiB of trsv_body; valid() keeps the sum below 217 KiB
template <class K>
bool smem_ok(K *k, size_t bytes) {
  return bytes <= 24 * 1024 || cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

}  // namespace
}  // namespace mdp

using namespace mdp;

extern "C" long long mdp_couple_buffer(const mdp_couple *c) { return valid(c) ? cp_buf(unpack(c)).total : 0; }
extern "C" long long mdp_couple_grad_buffer(const mdp_couple *c) { return valid(c) ? cp_grad(unpack(c)).total : 0; }
extern "C" long long mdp_couple_work_ints(const mdp_couple *c) {
  return valid(c) ? mdp_householder_qr_work_ints(c->n_blocks) + mdp_householder_qr_work_ints(1) : 0;
}

extern "C" mdp_status mdp_couple_solve(const mdp_couple *c, const mdp_c64 *Q_, const mdp_c64 *rho_, const mdp_c64 *eps_,
                                       const mdp_c64 *src_, mdp_c64 *buf_, int *work, mdp_c64 *x_, mdp_c64 *coef_,
                                       void *cuda_stream) {
  if (!valid(c) || !Q_ || !buf_ || !work || !x_ || !coef_ || (c->n_outer > 0 && (!rho_ || !eps_))) return MDP_ERR_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const Cp p = unpack(c);
  const CpBuf w = cp_buf(p);
  const double2 *Q = (const double2 *)Q_, *rho = (const double2 *)rho_, *eps = (const double2 *)eps_, *src = (const double2 *)src_;
  double2 *buf = (double2 *)buf_, *x = (double2 *)x_, *coef = (double2 *)coef_;
  double *D = (double *)(buf + w.D);
  const size_t sms = (size_t)p.ns * 16, smp = (size_t)p.nmax * 9 * 16;
  if (!smem_ok(k_cp_shared<false>, sms) || !smem_ok(k_cp_private, smp)) return MDP_ERR_CUDA;
  const unsigned nv = (unsigned)((p.N * p.C + 127) / 128);
  pdl(k_cp_vec, dim3(nv), dim3(128), 0, st, p, nullptr, rho, eps, buf + w.cv);
  pdl(k_cp_gemv<1>, dim3((p.mmax + 31) / 32, p.N), dim3(32, 16), 0, st, Q, p.off, p.G, p.r0, p.C, buf + w.cv, 0, buf + w.b, 0, -1.0, 0.0, src);
  pdl(k_cp_norm, dim3(p.n), dim3(128), 0, st, p, Q, rho, D);
  pdl(k_cp_build, dim3((p.mmax + 127) / 128, p.nmax + 1, p.N), dim3(128), 0, st, p, Q, rho, D, buf + w.b, buf + w.M);
  if (cudaGetLastError() != cudaSuccess) return MDP_ERR_CUDA;
  mdp_status s = mdp_householder_qr_batched(p.N, p.mmax, p.nmax, 1, (mdp_c64 *)(buf + w.M), p.mmax, (long long)(p.nmax + 1) * p.mmax,
                                            (mdp_c64 *)(buf + w.tau), work, st);
  if (s != MDP_OK) return s;
  if (p.ns > 0) {
    pdl(k_cp_gather, dim3((p.ms + 127) / 128, p.ns + 1), dim3(128), 0, st, p, buf + w.M, buf + w.S);
    if (cudaGetLastError() != cudaSuccess) return MDP_ERR_CUDA;
    s = mdp_householder_qr_batched(1, p.ms, p.ns, 1, (mdp_c64 *)(buf + w.S), p.ms, 0, (mdp_c64 *)(buf + w.tau + (long long)p.N * p.nmax),
                                   work + mdp_householder_qr_work_ints(p.N), st);
    if (s != MDP_OK) return s;
    pdl(k_cp_shared<false>, dim3(1), dim3(kTrThreads), sms, st, p, buf + w.S, D, nullptr, nullptr, buf + w.ys, x);
  }
  pdl(k_cp_private, dim3(p.N), dim3(kTrThreads), smp, st, p, buf + w.M, D, buf + w.ys, nullptr, x);
  pdl(k_cp_vec, dim3(nv), dim3(128), 0, st, p, x, rho, eps, coef);
  return cudaGetLastError() == cudaSuccess ? MDP_OK : MDP_ERR_CUDA;
}

extern "C" mdp_status mdp_couple_grad(const mdp_couple *c, const mdp_c64 *Q_, const mdp_c64 *rho_, const mdp_c64 *src_,
                                      const mdp_c64 *buf_, const mdp_c64 *x_, const mdp_c64 *coef_, const mdp_c64 *g_,
                                      mdp_c64 *tmp_, mdp_c64 *gQ_, mdp_c64 *grho_, mdp_c64 *geps_, void *cuda_stream) {
  if (!valid(c) || !Q_ || !buf_ || !x_ || !coef_ || !g_ || !tmp_ || (c->n_outer > 0 && (!rho_ || !grho_ || !geps_)))
    return MDP_ERR_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const Cp p = unpack(c);
  const CpBuf w = cp_buf(p);
  const CpGrad t = cp_grad(p);
  const double2 *Q = (const double2 *)Q_, *rho = (const double2 *)rho_, *src = (const double2 *)src_, *buf = (const double2 *)buf_;
  const double2 *x = (const double2 *)x_, *coef = (const double2 *)coef_, *g = (const double2 *)g_;
  double2 *tmp = (double2 *)tmp_, *gQ = (double2 *)gQ_;
  const double *D = (const double *)(buf + w.D);
  const size_t sms = (size_t)p.ns * 16, smp = (size_t)p.nmax * 9 * 16;
  if (!smem_ok(k_cp_shared<true>, sms) || !smem_ok(k_cp_private, smp) || !smem_ok(k_cp_private_h, smp)) return MDP_ERR_CUDA;
  const long long nc = (long long)p.N * p.C;
  pdl(k_cp_gx, dim3((p.n + 127) / 128), dim3(128), 0, st, p, g, rho, D, tmp + t.gx);
  pdl(k_cp_private_h, dim3(p.N), dim3(kTrThreads), smp, st, p, buf + w.M, tmp + t.gx, tmp + t.yp, tmp + t.part);
  if (p.ns > 0) pdl(k_cp_shared<true>, dim3(1), dim3(kTrThreads), sms, st, p, buf + w.S, D, tmp + t.gx, tmp + t.part, tmp + t.ys, tmp + t.w);
  pdl(k_cp_private, dim3(p.N), dim3(kTrThreads), smp, st, p, buf + w.M, D, tmp + t.ys, tmp + t.yp, tmp + t.w);
  if (cudaMemcpyAsync(tmp + t.sw, coef, sizeof(double2) * (size_t)nc, cudaMemcpyDeviceToDevice, st) != cudaSuccess) return MDP_ERR_CUDA;
  pdl(k_cp_vec, dim3((unsigned)((nc + 127) / 128)), dim3(128), 0, st, p, tmp + t.w, rho, nullptr, tmp + t.sw + nc);
  pdl(k_cp_gemv<2>, dim3((p.mmax + 31) / 32, p.N), dim3(32, 16), 0, st, Q, p.off, p.G, p.r0, p.C, tmp + t.sw, nc, tmp + t.u, p.rows, -1.0, 1.0, src);
  if (gQ)
    pdl(k_cp_outer<2>, dim3((p.mmax + 127) / 128, p.C, p.N), dim3(128), 0, st, p.off, p.G, p.r0, p.C, tmp + t.u, p.rows, tmp + t.sw + nc, coef, gQ);
  if (p.no > 0) {
    pdl(k_cp_dots<2>, dim3(p.C, p.N), dim3(128), 0, st, Q, p.off, p.G, p.r0, p.C, tmp + t.u, p.rows, tmp + t.z, nc);
    pdl(k_cp_sides, dim3(p.no), dim3(128), 0, st, p, g, tmp + t.z, x, tmp + t.w, (double2 *)grho_, (double2 *)geps_);
  }
  return cudaGetLastError() == cudaSuccess ? MDP_OK : MDP_ERR_CUDA;
}

extern "C" mdp_status mdp_block_values(int n_blocks, int cols, int max_len, const int *len, const int *yoff, const long long *off,
                                       const mdp_c64 *B, const mdp_c64 *v, mdp_c64 *y, void *cuda_stream) {
  if (n_blocks < 1 || n_blocks > 65535 || cols < 1 || max_len < 1 || !len || !yoff || !off || !B || !v || !y) return MDP_ERR_ARG;
  pdl(k_cp_gemv<1>, dim3((max_len + 31) / 32, n_blocks), dim3(32, 16), 0, (cudaStream_t)cuda_stream, 
      (const double2 *)B, off, len, yoff, cols, (const double2 *)v, 0, (double2 *)y, 0, 1.0, 0.0, nullptr);
  return cudaGetLastError() == cudaSuccess ? MDP_OK : MDP_ERR_CUDA;
}

extern "C" mdp_status mdp_block_values_grad(int n_blocks, int cols, int max_len, const int *len, const int *yoff, const long long *off,
                                            const mdp_c64 *B, const mdp_c64 *v, const mdp_c64 *gy, mdp_c64 *gB, mdp_c64 *gv,
                                            void *cuda_stream) {
  if (n_blocks < 1 || n_blocks > 65535 || cols < 1 || cols > 65535 || max_len < 1 || !len || !yoff || !off || !B || !v || !gy)
    return MDP_ERR_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const double2 *u = (const double2 *)gy;
  if (gB)
    pdl(k_cp_outer<1>, dim3((max_len + 127) / 128, cols, n_blocks), dim3(128), 0, st, off, len, yoff, cols, u, 0, (const double2 *)v, nullptr, (double2 *)gB);
  if (gv)
    pdl(k_cp_dots<1>, dim3(cols, n_blocks), dim3(128), 0, st, (const double2 *)B, off, len, yoff, cols, u, 0, (double2 *)gv, 0);
  return cudaGetLastError() == cudaSuccess ? MDP_OK : MDP_ERR_CUDA;
}
