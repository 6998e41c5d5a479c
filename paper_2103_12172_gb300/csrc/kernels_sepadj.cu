// The gradient pass through the separable Green's function (kernels_sep.cu): with mu = A^{-H} Tr^T c,
//   grad_xi = -L^T mu on gamma (+ c for P columns),
//   dLoss/dk = -Re <c, Tr G' r> - Re <mu, s>,   s = dL/dk w + L dw/dk on the ring,  G' = dG/dk.
// On the rows in question G is symmetric, so mu = conj(G conj(c)): the projection with gamma and the ring
// exchanged. The stages are those of kernels_sep.cu: A_MID and A_FWD cut the conjugate cotangent against the
// transposed K, the moment tables and the sines; k_adj_modes applies the transpose of the modes' matrix;
// A_SYN and A_INV give mu on the ring.
//
// <c, Tr G' r> needs no field: T_q^{-1} = kappa + phi^T R phi, so its k-derivative is a bilinear form of
// what the two passes have at hand. Per mode, with F the cotangent's inputs (moments, transforms of the gamma
// rows) and in the residual's (transforms of the dense rows, moments): F^T dMAT/dk in, plus the moments
// against d phi/dk (extra outputs of the stage 1 contractions) times the other side's coefficients; and
// sum conj(c) (dK/dk r) on the middle rows, one more Toeplitz product of the residual. The recomputed field
// of every mode and row and its adjoint, most of the pass by the recurrences, are gone: 4 x 257^2 with 1024
// basis columns takes 586 us (4418 by the recurrences), 257^2 and 513^2 with user densities 663 us (4536).
// A first pass after a change of the wavenumbers makes the tables too, 400 us more.
#include "sep_modes.cuh"

#include <algorithm>

namespace mdp {
namespace {

// ---------------------------------------------------------------- k-derivatives of the modes
// value and k-derivative
struct Du { double v, d; };
__device__ __forceinline__ Du du(double v, double d = 0.0) { return {v, d}; }
__device__ __forceinline__ Du operator+(Du a, Du b) { return {a.v + b.v, a.d + b.d}; }
__device__ __forceinline__ Du operator-(Du a, Du b) { return {a.v - b.v, a.d - b.d}; }
__device__ __forceinline__ Du operator-(Du a) { return {-a.v, -a.d}; }
__device__ __forceinline__ Du operator*(Du a, Du b) { return {a.v * b.v, fma(a.v, b.d, a.d * b.v)}; }
__device__ __forceinline__ Du operator*(double a, Du b) { return {a * b.v, a * b.d}; }
__device__ __forceinline__ Du operator/(Du a, Du b) {
  const double i = 1.0 / b.v, q = a.v * i;
  return {q, (a.d - q * b.d) * i};
}
struct Dc { Du re, im; };
__device__ __forceinline__ Dc operator+(Dc a, Dc b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ Dc operator-(Dc a, Dc b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ Dc operator*(Dc a, Dc b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ Dc operator*(Du a, Dc b) { return {a * b.re, a * b.im}; }
__device__ __forceinline__ Dc operator/(Dc a, Dc b) {
  const Du n = du(1.0) / (b.re * b.re + b.im * b.im);
  return {(a.re * b.re + a.im * b.im) * n, (a.im * b.re - a.re * b.im) * n};
}

enum {
  MD_MAT = 0,     // d MT_MAT / dk
  MD_P1D = 36,    // d phi / dk at the dense rows and the gamma rows
  MD_P2D = 40,
  MD_P1G = 44,
  MD_P2G = 48,
  MD_RI = 52,     // d Im(R11, R12, R22) / dk
  MD_T1 = 55,     // d T1 / dk, d T2 / dk
  MD_T2 = 56,
  MD_RHO1 = 57,   // scales (powers of two) of d phi/dk in the moment tables
  MD_RHO2 = 58,
  MD_RFD = 59,    // scale of d kappa/dk in a receiver row's moment table
  MD_TC = 62,     // d theta/dk (kind 2), d cosh theta or cos theta / dk (kinds 0, 1)
  MD_COS = 63,    // cos or cosh theta, -4 t (1 - t) = cos^2 - 1, t
  MD_SS = 64,
  MD_T = 65,
};
static_assert(MD_T < ADJ_MDW, "derivative table width");

// dS/dc of S(x) = sin(x theta) / sin theta (sinh), c = cos theta (cosh), ss = c^2 - 1, t = (1 - c) / 2. Where x theta
// is small the quotient cancels: S = x 2F1(1 - x, 1 + x; 3/2; t), so dS/dc = x (x^2 - 1)/3 2F1(2 - x, 2 + x; 5/2; t),
// whose terms fall by a factor of at least 16 for |t| max(x, 1)^2 < 1/16.
__device__ __forceinline__ double ds_dc(double x, double th, double c, double t, double iss, double C, double S) {
  if (th * fmax(fabs(x), 1.0) >= 0.5) return fma(x, C, -c * S) * iss;
  const double y = x * x;
  double term = 1.0, sum = 1.0;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    term *= ((double)((k + 2) * (k + 2)) - y) * (t * (1.0 / ((k + 2.5) * (k + 1.0))));
    sum += term;
  }
  return x * (y - 1.0) * (1.0 / 3.0) * sum;
}
// the inverse of a power of two
__device__ __forceinline__ double inv2(double r) { return __hiloint2double(0x7fe00000 - __double2hiint(r), 0); }

__global__ void __launch_bounds__(32) k_adj_mode_tab(const SubDesc *subs, int s0, const unsigned char *sep, unsigned char *adj) {
  const int si = s0 + blockIdx.y;
  const SubDesc &d = subs[si];
  const int q = blockIdx.x * 32 + threadIdx.x + 1;
  if (!d.tc_cols || d.leader != si || q > d.Nq) return;
  const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
  double *D = reinterpret_cast<double *>(adj + d.adj_md) + (long long)(q - 1) * ADJ_MDW;
  const double *ab = reinterpret_cast<const double *>(sep + d.sep_ab) + 2 * (q - 1);
  const double h = d.h, h2 = h * h, k = d.k, k2 = k * k;
  const double sq = sin(M_PI * q / (2.0 * d.Nx)), lam = -4.0 * sq * sq;
  const int kind = (int)T[MT_KIND], N = d.ny - 1, J0 = d.nlo - 1, J1 = d.nhi + 1, L = d.nhi - d.nlo;
  const double sg = T[MT_SG], thv = T[MT_TH], n1 = T[MT_N1], n2 = T[MT_N2];
  const double mid = 0.5 * (J0 + J1), Lh = 0.5 * (J1 - J0);
  Du a = du(ab[0], k / 6.0);
  const Du b = du(ab[1], -2.0 * (k / 6.0) + 2.0 * k + 2.0 * k * lam / 12.0);
  Du t = (b + 2.0 * a) / (4.0 * a);
  if (sg < 0.0) { t = du(1.0) - t; a = -a; }
  Du c = du(1.0) - 2.0 * t;                  // cos theta or cosh theta
  const double ss = -4.0 * t.v * (1.0 - t.v), iss = thv > 0.0 ? 1.0 / ss : 0.0;   // c^2 - 1
  Dc al0 = {du(1.0), du(0.0)}, al1 = {du(0.0), du(0.0)};
  if (d.cplx) {
    const bool paper = d.ap_bc == MDP_AP_DIRX_SOMMY_PAPER;
    const Du alpha = du(paper ? (1.0 - k2 * h2 / 24.0 - lam / 6.0) / h2 : (1.0 + k2 * h2 / 24.0 + lam / 24.0) / h2,
                        paper ? -k / 12.0 : k / 12.0);
    const Du beta = du(k * (1.0 + k2 * h2 / 8.0 + lam / (paper ? 2.0 : 8.0)) / h,
                       (1.0 + 3.0 * k2 * h2 / 8.0 + lam / (paper ? 2.0 : 8.0)) / h);
    al0 = {alpha, 0.5 * beta};
    al1 = {(-sg) * alpha, (0.5 * sg) * beta};
  }
  Du lo1[3], lo2[3], hi1[3], hi2[3], kv[6], T1, T2 = du(0.0), el[3] = {du(0.0), du(0.0), du(0.0)};
  Dc R11, R12, R22;
  double rho1, rho2, kb;
  if (kind < 2) {
    const Du i2a = du(1.0) / (2.0 * a);
    // C and S at x, derivatives through c: dC/dc = x S
    const double isth = thv > 0.0 ? 1.0 / (kind == 0 ? sin(thv) : sinh(thv)) : 0.0;
    auto cs = [&](double x, Du &C, Du &S) {
      double cv = 1.0, sv = x;
      if (thv > 0.0) {
        if (kind == 0) sincos(x * thv, &sv, &cv);
        else { cv = cosh(x * thv); sv = sinh(x * thv); }
        sv *= isth;
      }
      C = du(cv, x * sv * c.d);
      S = du(sv, c.d * ds_dc(x, thv, c.v, t.v, iss, cv, sv));
    };
    auto end = [&](double x0, double x1, Dc &e1, Dc &e2) {   // al0 z(x0) + al1 z(x1)
      Du C0, S0, C1, S1;
      cs(x0, C0, S0);
      cs(x1, C1, S1);
      e1 = {al0.re * C0 + al1.re * C1, al0.im * C0 + al1.im * C1};
      e2 = {al0.re * S0 + al1.re * S1, al0.im * S0 + al1.im * S1};
    };
    Dc b1, b2, t1, t2;
    end(0.0 - mid, 1.0 - mid, b1, b2);
    end(N - mid, N - 1 - mid, t1, t2);
    const Dc ad = a * (b1 * t2 - b2 * t1);
    R11 = du(1.0 / (n1 * n1)) * ((b2 * t2) / ad);
    R22 = du(1.0 / (n2 * n2)) * ((b1 * t1) / ad);
    R12 = du(-0.5 / (n1 * n2)) * ((b1 * t2 + b2 * t1) / ad);
    Du Ce, Se, C, S;
    for (int j = 0; j < 3; ++j) {
      cs(Lh - j, C, S);
      if (j == 0) { Ce = C; Se = S; }
      lo1[j] = hi1[j] = n1 * C;
      hi2[j] = n2 * S;
      lo2[j] = -hi2[j];
    }
    kv[0] = du(0.0);
    kv[1] = i2a;
    kv[2] = 2.0 * (c * i2a);
    for (int j = 3; j < 6; ++j) { cs(L - 4 + j, C, S); kv[j] = S * i2a; }
    T1 = (1.0 / n1) * (Se * i2a);
    T2 = (1.0 / n2) * (Ce * i2a);
    // bounds of d phi/dk and d kappa/dk over the rows: |S| <= min(x, 1/sin theta) (its own value, growing, next to
    // the cutoff), |dC/dc| = x |S|, |dS/dc| <= max(1, x^2) times the bound of S
    const double x2 = fmax(1.0, Lh * Lh), sm = kind == 0 ? fmin(fmax(Lh, 1.0), fabs(isth)) : fmax(fabs(Se.v), 1.0);
    const double s2 = kind == 0 ? 2.0 * sm : 2.0 * sm * Ce.v;   // S up to distance 2 Lh
    rho1 = n1 * fabs(c.d) * Lh * sm;
    rho2 = n2 * fabs(c.d) * x2 * sm;
    kb = s2 * fma(fabs(i2a.v) * fabs(c.d), 4.0 * x2, fabs(i2a.d));
  } else {
    const Du th = du(thv, c.d / sinh(thv));
    const Du em = du(exp(-thv), -th.d * exp(-thv)), ep = du(exp(thv), th.d * exp(thv));
    auto ex = [&](double m) { const double v = exp(-thv * m); return du(v, -m * th.d * v); };   // e^{-theta m}
    const Du fl = ex(L - 1), c0 = du(-1.0) / (a * (ep - em));
    const Dc num = {al0.re + al1.re * ep, al0.im + al1.im * ep}, den = {al0.re + al1.re * em, al0.im + al1.im * em};
    const Dc ref = num / den, rb = (-ex(2.0 * J0)) * ref, rt = (-ex(2.0 * (N - J1))) * ref, rr = rb * rt;
    const Du dl = ex(J1 - J0), dl2 = dl * dl;
    const Dc Dn = {du(1.0) - rr.re * dl2, -(rr.im * dl2)};
    R11 = (c0 * rb) / Dn;
    R22 = (c0 * rt) / Dn;
    R12 = (c0 * dl) * rr / Dn;
    const Du e2 = em * em;
    lo1[0] = hi2[0] = du(1.0); lo1[1] = hi2[1] = em; lo1[2] = hi2[2] = e2;
    hi1[0] = lo2[0] = fl * e2 * em; hi1[1] = lo2[1] = fl * e2; hi1[2] = lo2[2] = fl * em;
    kv[0] = c0; kv[1] = c0 * em; kv[2] = c0 * e2; kv[3] = c0 * fl; kv[4] = c0 * fl * em; kv[5] = c0 * fl * e2;
    el[0] = c0; el[1] = c0 * ep; el[2] = c0 * ep * ep;
    T1 = c0;
    // max over x of x e^{-theta x}: 1 / (e theta), or its value at x = 1 when theta > 1
    rho1 = rho2 = fabs(th.d) * (thv > 1.0 ? exp(-thv) : 0.36788 / thv);
    kb = fabs(c0.d) + fabs(c0.v) * rho1;
    D[MD_TC] = th.d;
  }
  if (kind < 2) D[MD_TC] = c.d;
  D[MD_COS] = c.v; D[MD_SS] = ss; D[MD_T] = t.v;
  auto sgn = [&](int i) { return (sg < 0.0 && (i & 1)) ? -1.0 : 1.0; };
  auto p1 = [&](int i) { return sgn(i - J0) * (i - J0 < 3 ? lo1[i - J0] : hi1[J1 - i]); };
  auto p2 = [&](int i) { return sgn(i - J0) * (i - J0 < 3 ? lo2[i - J0] : hi2[J1 - i]); };
  auto kap = [&](int x) { return sgn(x) * (x < 3 ? kv[x] : kv[x - L + 4]); };
  const Du f = (1.0 / (n1 * n2)) * (du(1.0) / (2.0 * a));
  const int rows_d[4] = {d.nlo, d.nlo + 1, d.nhi - 1, d.nhi}, rows_g[4] = {d.nlo - 1, d.nlo, d.nhi, d.nhi + 1};
  for (int r = 0; r < 4; ++r) {
    D[MD_P1D + r] = p1(rows_d[r]).d; D[MD_P2D + r] = p2(rows_d[r]).d;
    D[MD_P1G + r] = p1(rows_g[r]).d; D[MD_P2G + r] = p2(rows_g[r]).d;
  }
  for (int i = 0; i < 6; ++i) {   // as the modes' matrix in k_sep_mode_tab
    const Du f1 = i < 4 ? p1(rows_d[i]) : du(i == 4 ? 1.0 : 0.0), f2 = i < 4 ? p2(rows_d[i]) : du(i == 5 ? 1.0 : 0.0);
    const Du A = R11.re * f1 + R12.re * f2, B = R12.re * f1 + R22.re * f2;
    Du E1 = du(0.0), E2 = du(0.0);
    if (i < 4) {
      const int j = rows_d[i];
      const double up = i < 2 ? 1.0 : -1.0;
      if (kind < 2) { E1 = (-up) * (f * f2); E2 = up * (f * f1); }
      else if (i < 2) E1 = sgn(j - J0) * el[j - J0];
      else E2 = sgn(j - J0) * el[J1 - j];
    }
    D[MD_MAT + i] = (A + E1).d;
    D[MD_MAT + 6 + i] = (B + E2).d;
    for (int r = 0; r < 4; ++r) {
      const int n = rows_g[r];
      Du w;
      if (i < 4) w = kap(abs(n - rows_d[i]));
      else {
        const double up = r < 2 ? 1.0 : -1.0;
        if (kind < 2) w = i == 4 ? (-up) * (f * p2(n)) : up * (f * p1(n));
        else if (i == 4) w = r < 2 ? sgn(n - J0) * el[n - J0] : du(0.0);
        else w = r < 2 ? du(0.0) : sgn(n - J0) * el[J1 - n];
      }
      D[MD_MAT + 6 * (2 + r) + i] = (p1(n) * A + p2(n) * B + w).d;
    }
  }
  D[MD_RI] = R11.im.d; D[MD_RI + 1] = R12.im.d; D[MD_RI + 2] = R22.im.d;
  D[MD_T1] = T1.d; D[MD_T2] = T2.d;
  auto scale = [](double bound) { return bound > 0.0 ? pow2i(-(ilogb(bound) + 1)) : 1.0; };
  D[MD_RHO1] = scale(rho1); D[MD_RHO2] = scale(rho2); D[MD_RFD] = scale(kb);
}

// d phi/dk at a subdomain's receiver row
__global__ void __launch_bounds__(32) k_adj_rec(const SubDesc *subs, int s0, const unsigned char *sep, unsigned char *adj) {
  const SubDesc &d = subs[s0 + blockIdx.y];
  const int q = blockIdx.x * 32 + threadIdx.x + 1;
  if (!d.tc_cols || d.nrec < 0 || q > d.Nq) return;
  const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
  const double *D = reinterpret_cast<const double *>(adj + d.adj_md) + (long long)(q - 1) * ADJ_MDW;
  double *Q = reinterpret_cast<double *>(adj + d.adj_rp) + q - 1;
  const int kind = (int)T[MT_KIND], J0 = d.nlo - 1, J1 = d.nhi + 1;
  const double th = T[MT_TH], tc = D[MD_TC], sr = T[MT_SG] < 0.0 && ((d.nrec - J0) & 1) ? -1.0 : 1.0;
  if (kind == 2) {
    Q[0] = sr * (-(d.nrec - J0) * tc * exp(-th * (d.nrec - J0)));
    Q[d.Nq] = sr * (-(J1 - d.nrec) * tc * exp(-th * (J1 - d.nrec)));
    return;
  }
  const double x = d.nrec - 0.5 * (J0 + J1), iss = th > 0.0 ? 1.0 / D[MD_SS] : 0.0;
  double C = 1.0, S = x;
  if (th > 0.0) {
    if (kind == 0) sincos(x * th, &S, &C);
    else { C = cosh(x * th); S = sinh(x * th); }
    S *= 1.0 / (kind == 0 ? sin(th) : sinh(th));
  }
  Q[0] = sr * (T[MT_N1] * (x * S * tc));
  Q[d.Nq] = sr * (T[MT_N2] * (tc * ds_dc(x, th, D[MD_COS], D[MD_T], iss, C, S)));
}

// d phi/dk on the rows J0 .. J1, [2][Py + 2][Nq], from phi
__global__ void __launch_bounds__(128) k_adj_phid(const SubDesc *subs, int s0, const unsigned char *sep, unsigned char *adj) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  const int q = blockIdx.x * 128 + threadIdx.x + 1, rows = d.Py + 2, i0 = blockIdx.y * 8;
  if (!d.tc_cols || d.leader != si || q > d.Nq || i0 >= rows) return;
  const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
  const double *D = reinterpret_cast<const double *>(adj + d.adj_md) + (long long)(q - 1) * ADJ_MDW;
  const double *P1 = reinterpret_cast<const double *>(sep + d.sep_phi) + (q - 1), *P2 = P1 + (long long)rows * d.Nq;
  double *Q1 = reinterpret_cast<double *>(adj + d.adj_phid) + (q - 1), *Q2 = Q1 + (long long)rows * d.Nq;
  const double tc = D[MD_TC], c = D[MD_COS], th = T[MT_TH];
  const int kind = (int)T[MT_KIND], i1 = min(rows, i0 + 8);
  const double n2 = T[MT_N2], r12 = T[MT_N1] * inv2(n2), r21 = inv2(r12), iss = kind < 2 && th > 0.0 ? 1.0 / D[MD_SS] : 0.0;
  for (int i = i0; i < i1; ++i) {
    const long long o = (long long)i * d.Nq;
    if (kind == 2) {
      Q1[o] = -tc * i * P1[o];
      Q2[o] = -tc * (rows - 1 - i) * P2[o];
      continue;
    }
    const double x = i - 0.5 * (rows - 1), s = P2[o];   // n2 S with the row's sign
    const double w = T[MT_SG] < 0.0 && (i & 1) ? -n2 : n2;
    Q1[o] = tc * x * r12 * s;
    Q2[o] = tc * w * ds_dc(x, th, c, D[MD_T], iss, P1[o] * r21 * inv2(n2) * (w == n2 ? 1.0 : -1.0), s * inv2(n2) * (w == n2 ? 1.0 : -1.0));
  }
}

// d kappa/dk at row distance `dist` of mode q
__device__ __forceinline__ double kappa_d(const SubDesc &d, const double *T, const double *D, const double *P, const double *Q,
                                          int q, int dist) {
  const long long o = (long long)dist * d.Nq + q - 1, o2 = o + (long long)(d.Py + 2) * d.Nq;
  return fma(D[MD_T1], P[o], fma(D[MD_T2], P[o2], fma(T[MT_T1], Q[o], T[MT_T2] * Q[o2])));
}

// dK_sc/dk (d): as k_sep_kd
__global__ void __launch_bounds__(128) k_adj_kd(const SubDesc *subs, int s0, const double *tab, const unsigned char *sep,
                                                unsigned char *adj) {
  const int si = s0 + blockIdx.y;
  const SubDesc &d = subs[si];
  const int dist = blockIdx.x;
  if (!d.tc_cols || d.leader != si || dist >= d.Py) return;
  const SepGeo g = sep_geo(d);
  const double *S = tab + d.sin_off, *P = reinterpret_cast<const double *>(sep + d.sep_phi);
  const double *Q = reinterpret_cast<const double *>(adj + d.adj_phid);
  const int N2 = 2 * d.Nx;
  double acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = 0.0;
  for (int q = threadIdx.x + 1; q <= d.Nq; q += 128) {
    const double kq = kappa_d(d, reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW,
                              reinterpret_cast<const double *>(adj + d.adj_md) + (long long)(q - 1) * ADJ_MDW, P, Q, q, dist);
    double so[4], sc[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      so[s] = s < g.nS ? S[(int)(((long long)q * sep_out_col(d, s)) % N2)] * kq : 0.0;
      sc[s] = s < g.nS ? S[(int)(((long long)q * sep_src_col(d, s)) % N2)] : 0.0;
    }
    if (d.xsym) {
#pragma unroll
      for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) acc[s * 2 + cc] = fma(so[s], sc[cc], acc[s * 2 + cc]);
    } else {
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) acc[s * 4 + cc] = fma(so[s], sc[cc], acc[s * 4 + cc]);
    }
  }
  __shared__ double sh[4][2][16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    for (int off = 16; off >= 2; off >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], off);
    if (lane < 2) sh[warp][lane][i] = acc[i];
  }
  __syncthreads();
  if ((int)threadIdx.x < g.ncls * g.nS * g.nS) {
    double v = 0.0;
    for (int w = 0; w < 4; ++w)
      v += d.xsym ? sh[w][threadIdx.x >> 2][threadIdx.x & 3] : sh[w][0][threadIdx.x] + sh[w][1][threadIdx.x];
    reinterpret_cast<double *>(adj + d.adj_kdd)[(long long)threadIdx.x * d.Py + dist] = v * (2.0 / d.Nx);
  }
}

// Toeplitz blocks: K with gamma and the ring exchanged (dK false), or dK/dk for the residual (dK true)
__global__ void __launch_bounds__(256) k_adj_tb(const SubDesc *subs, int s0, const unsigned char *sep, unsigned char *adj, int dK) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  if (!d.tc_cols || d.leader != si) return;
  const SepGeo g = sep_geo(d);
  const AdjGeo a = adj_geo(d, g);
  const int ND = dK ? g.ND : a.ND, nkj = dK ? g.nkj : a.nkj;
  const int eo = blockIdx.y / g.nS, src = blockIdx.y % g.nS, blk0 = blockIdx.x * 4;   // (class, output), source
  if (eo >= g.ncls * g.nS || blk0 >= ND) return;
  const int e = eo / g.nS, out = eo % g.nS;
  const double *K = reinterpret_cast<const double *>(dK ? adj + d.adj_kdd : sep + d.sep_kd) + (long long)e * g.nS * g.nS * d.Py;
  auto pair = [&](int c) { return K + (long long)(dK ? out * g.nS + c : c * g.nS + out) * d.Py; };
  __shared__ int emax;
  if (threadIdx.x == 0) emax = 0;
  __syncthreads();
  int m = 0;
  for (int i = threadIdx.x; i < g.nS * d.Py; i += 256) m = max(m, (__double2hiint(pair(i / d.Py)[i % d.Py]) >> 20) & 0x7ff);
  for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(&emax, m);
  __syncthreads();
  const int ex = min(max(emax - 1022, -900), 900);
  if (threadIdx.x == 0 && blockIdx.x == 0 && src == 0)
    reinterpret_cast<int *>(adj + d.adj_kde)[(dK ? g.ncls * g.nS : 0) + eo] = ex;
  const int blk = blk0 + (threadIdx.x >> 6), o = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1;
  if (blk >= ND) return;
  const double sc = pow2i(54 - ex);
  const double *Kc = pair(src);
  long long V[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {   // output row minus source row: -1 (residual to gamma), +1 (gamma to the ring)
    const int dist = abs(16 * (blk - (nkj - 1)) + o - (8 * half + j) + (dK ? -1 : 1));
    V[j] = dist < d.Py ? __double2ll_rn(Kc[dist] * sc) : 0;
  }
  unsigned char *B = adj + (dK ? d.adj_dtb : d.adj_tb) + (((long long)eo * g.nS + src) * ND + blk) * SEP_BBLK;
  store_digits(B + (o >> 3) * 256 + half * 128 + (o & 7) * 16, 1024, V);
}

__device__ __forceinline__ void mark_tile(unsigned *mask, int kb, const long long *V) {
  long long any = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) any |= V[j];
  if (__any_sync(0xffffffffu, any != 0) && (threadIdx.x & 31) == 0) atomicOr(mask + (kb >> 5), 1u << (kb & 31));
}

// Moment tables: of the cotangent (res false: phi_1, phi_2 and their k-derivatives at the gamma columns), or
// of the residual (res true: the k-derivatives of phi_1, phi_2 and, per subdomain, of kappa at its receiver row).
__global__ void __launch_bounds__(256) k_adj_mb(const SubDesc *subs, int s0, const double *tab, const unsigned char *sep,
                                                unsigned char *adj, int res) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  if (!d.tc_cols) return;
  const SepGeo g = sep_geo(d);
  const AdjGeo a = adj_geo(d, g);
  // the receiver row's groups come last: a launch captured without any makes the others all the same
  const int n = g.nqp / 32, nto = (res ? 2 : ADJ_MOM) * n, nk = res ? g.nk1 : a.nk1, nkj = res ? g.nkj : a.nkj;
  int e = blockIdx.y / nto, to = blockIdx.y % nto;
  const int kb = blockIdx.x * 4 + (threadIdx.x >> 6);
  if (res && e >= g.ncls && d.nrec >= 0) {
    const int y = blockIdx.y - g.ncls * nto;
    e = y / n;
    to = nto + y % n;
  }
  if (e >= g.ncls || kb >= nk) return;
  const int o = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1;
  const int b = to * 32 / g.nqp, q = sep_mode(d, e, to * 32 % g.nqp + o);
  if (!(res && b == 2) && d.leader != si) return;
  const int c = kb / nkj, j0 = (kb % nkj) * 16 + 8 * half;
  long long V[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) V[j] = 0;
  if (q <= d.Nq) {
    const double sn = tab[d.sin_off + (int)(((long long)q * (res ? sep_src_col(d, c) : sep_out_col(d, c))) % (2 * d.Nx))];
    const double *P = reinterpret_cast<const double *>(sep + d.sep_phi), *Q = reinterpret_cast<const double *>(adj + d.adj_phid);
    const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
    const double *D = reinterpret_cast<const double *>(adj + d.adj_md) + (long long)(q - 1) * ADJ_MDW;
    const long long p2 = (long long)(d.Py + 2) * d.Nq;
    const bool der = res ? b < 2 : b >= 2;
    const int bb = der && !res ? b - 2 : b;
    const double rho = der ? D[MD_RHO1 + bb] : 1.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j0 + j >= (res ? g.Pj : g.Pi)) continue;
      const int row = (res ? 3 : 2) + j0 + j;          // counted from J0 = nlo - 1
      double v;
      if (res && b == 2) v = kappa_d(d, T, D, P, Q, q, abs(d.nrec - (d.nlo - 1) - row)) * D[MD_RFD];
      else v = (der ? Q : P)[(bb ? p2 : 0) + (long long)row * d.Nq + q - 1] * rho;
      V[j] = fix54(v * sn);
    }
  }
  const SepMoment m = res ? adj_dmoment(d, g, e, to)
                          : SepMoment{d.adj_mb + ((long long)e * nto + to) * nk * SEP_BBLK, d.adj_zm + 4LL * SEP_MASK * (e * nto + to)};
  mark_tile(reinterpret_cast<unsigned *>(adj + m.mask), kb, V);
  unsigned char *B = adj + m.blocks + (long long)kb * SEP_BBLK;
  store_digits(B + (o >> 3) * 256 + half * 128 + (o & 7) * 16, 1024, V);
}

// The synthesis on the ring columns: output (c, j), K index (b, q): (2/Nx) sin(pi q m_c/Nx) times phi_b(j), or
// (b = 2, per subdomain) kappa_q(|rec - j|) scaled to below 1.
__global__ void __launch_bounds__(256) k_adj_b3(const SubDesc *subs, int s0, const double *tab, const unsigned char *sep,
                                                unsigned char *adj) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  if (!d.tc_cols) return;
  const SepGeo g = sep_geo(d);
  const AdjGeo a = adj_geo(d, g);
  const int e = blockIdx.y / a.nt3, to = blockIdx.y % a.nt3, kb = blockIdx.x * 4 + (threadIdx.x >> 6);
  if (e >= g.ncls || kb >= a.nk3) return;
  const int o = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1;
  const int c = to / a.nti, i = (to % a.nti) * 32 + o, m = sep_src_col(d, c);
  const int k2 = 2 * g.nqp / 16, b = kb * 16 / g.nqp;
  if (b < 2 && d.leader != si) return;
  const int q0 = kb * 16 % g.nqp + 8 * half, row = 3 + i;
  const double *S = tab + d.sin_off, *P = reinterpret_cast<const double *>(sep + d.sep_phi), sc = inv_scale(d);
  const long long p2 = (long long)(d.Py + 2) * d.Nq;
  long long V[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int q = sep_mode(d, e, q0 + j);
    V[j] = 0;
    if (i >= g.Pj || q > d.Nq) continue;
    double v;
    if (b < 2) v = P[b * p2 + (long long)row * d.Nq + q - 1];
    else {
      const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
      const long long od = (long long)abs(d.nrec - (d.nlo - 1) - row) * d.Nq + q - 1;
      v = fma(T[MT_T1], P[od], T[MT_T2] * P[p2 + od]) * T[MT_RF];
    }
    V[j] = fix54(v * (sc * S[(int)(((long long)q * m) % (2 * d.Nx))]));
  }
  const long long t = (long long)e * a.nt3 + to;
  mark_tile(reinterpret_cast<unsigned *>(adj + (b < 2 ? d.adj_z3 : d.adj_r3z)) + t * SEP_MASK, kb, V);
  unsigned char *B = adj + (b < 2 ? d.adj_b3 + (t * k2 + kb) * SEP_BBLK : d.adj_r3 + (t * (k2 / 2) + kb - k2) * SEP_BBLK);
  store_digits(B + (o >> 3) * 256 + half * 128 + (o & 7) * 16, 1024, V);
}

// sines of the gamma rows' transforms (inv false) and, times 2/Nx, of the dense ring rows' inverse ones
__global__ void __launch_bounds__(256) k_adj_sines(const SubDesc *subs, int s0, const double *tab, unsigned char *adj, int inv) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  if (!d.tc_cols || d.leader != si) return;
  const SepGeo g = sep_geo(d);
  const AdjGeo a = adj_geo(d, g);
  const int nto = inv ? a.ntr : g.nqh / 32, nk = inv ? g.nqh / 16 : a.nkf, m0 = inv ? g.mf : g.mg;
  const int e = blockIdx.y / nto, to = blockIdx.y % nto, kb = blockIdx.x * 4 + (threadIdx.x >> 6);
  if (e >= 2 || kb >= nk) return;
  const int o = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1;
  const double *S = tab + d.sin_off, sc = inv ? inv_scale(d) : 1.0;
  long long V[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int ko = to * 32 + o, kk = kb * 16 + 8 * half + j;
    const int q = sep_parity_mode(e, inv ? kk : ko), m = m0 + (inv ? ko : kk);
    V[j] = q <= d.Nq && 2 * m <= d.Nx ? fix54(sc * S[(int)(((long long)q * m) % (2 * d.Nx))]) : 0;
  }
  unsigned char *B = adj + (inv ? d.adj_bi : d.adj_bf) + (((long long)e * nto + to) * nk + kb) * SEP_BBLK;
  store_digits(B + (o >> 3) * 256 + half * 128 + (o & 7) * 16, 1024, V);
}

// ---------------------------------------------------------------- operands
__global__ void __launch_bounds__(256) k_adj_clear(Batch bt, const SubDesc *subs, double *ws) {
  pdl_wait();
  Item it; int local;
  locate(bt, blockIdx.x, it, local);
  MDP_CHECK_ITEM(bt, subs, it, local, F_ACLR);
  const SubDesc &d = subs[it.sub];
  unsigned *m0 = reinterpret_cast<unsigned *>(ws + it.a_off + sep_ws(d, it.ncols).mask);
  unsigned *m1 = reinterpret_cast<unsigned *>(ws + it.a_off + adj_ws(d, it.ncols).mask);
  const int n0 = sep_mask_words(it.ncols), n1 = adj_mask_words(it.ncols);
  for (int i = threadIdx.x; i < n0; i += 256) m0[i] = 0;
  for (int i = threadIdx.x; i < n1; i += 256) m1[i] = 0;
}

// as k_sep_cut: A_MID the cotangent at the gamma columns (gathered by k_adj_cols), A_FWD at the gamma rows
// and the receiver row, A_SYN the coefficients, A_INV the field of the dense ring rows; the cotangent conjugated
template <int JOB>
__device__ __forceinline__ void adj_cut_body(const Item &it, const SubDesc &d, double *ws, const double2 *cot,
                                             const double2 *cot_rec, int local) {
  const SepGeo g = sep_geo(d);
  const AdjGeo a = adj_geo(d, g);
  const AdjWs w = adj_ws(d, it.ncols);
  const int R = adj_rows(d, JOB, it.ncols);
  const int e = local / (R / 8), row = (local % (R / 8)) * 8 + (threadIdx.x & 7), kl = threadIdx.x >> 3;
  const int cp = sep_pad128(it.ncols), nk = adj_nk(a, JOB);
  const long long nc = it.ncols;
  const int col = row % cp, part = (row / cp) & 1, rr = row / (2 * cp);
  bool live = col < it.ncols;
  const double *src = nullptr;
  int m0 = 0, m1 = -1;   // A_FWD: the row's columns
  if (JOB == A_MID) src = ws + it.r_off;
  else if (JOB == A_SYN) src = ws + it.a_off + w.aeff + (long long)e * 3 * g.nqp * R + row;
  else if (JOB == A_INV) src = ws + it.y_off;
  else if (rr < 4) {
    const int W = d.Px + 2, M4 = 4 * (d.Py - 2);
    m0 = d.mlo - 1;
    m1 = d.mhi + 1;
    src = reinterpret_cast<const double *>(cot + it.io_off + (long long)col * d.G + (rr == 0 ? 0 : rr == 1 ? W : rr == 2 ? 2 * W + M4 : 3 * W + M4)) + part;
  } else if (cot_rec) {
    m0 = d.mlo + 1;
    m1 = d.mhi - 1;
    src = reinterpret_cast<const double *>(cot_rec + d.rec_off + (long long)(it.col0 + col) * (d.Px - 2)) + part;
  } else live = false;
  const double cj = (JOB == A_MID || JOB == A_FWD) && part ? -1.0 : 1.0;
  auto value = [&](int k) -> double {
    if (!live) return 0.0;
    if (JOB == A_MID) {
      const int s = k / (16 * a.nkj), i = k - s * 16 * a.nkj;
      if (i >= g.Pi) return 0.0;
      return src[2 * ((4LL * i + (d.xsym ? 2 * s + e : s)) * nc + col) + part];
    }
    if (JOB == A_FWD) {
      const int m = g.mg + k, mm = d.Nx - m;
      if (k >= g.Ng) return 0.0;
      const double x = m >= m0 && m <= m1 ? src[2 * (m - m0)] : 0.0;
      const double y = mm != m && mm >= m0 && mm <= m1 ? src[2 * (mm - m0)] : 0.0;
      return e == 0 ? x + y : x - y;
    }
    if (JOB == A_SYN) return sep_mode(d, e, k % g.nqp) <= d.Nq ? src[(long long)k * R] : 0.0;
    const int q = sep_parity_mode(e, k);
    return q <= d.Nq ? src[2 * (((long long)(q - 1) * 5 + rr) * nc + col) + part] : 0.0;
  };
  __shared__ int emax[8];
  __shared__ unsigned smask[SEP_MASK];
  if (threadIdx.x < 8) { emax[threadIdx.x] = 0; smask[threadIdx.x] = 0; }
  __syncthreads();
  double x[8];
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
  const int E = max(emax[threadIdx.x & 7], 1), tr = e * (R / 128) + row / 128;
  if (kl == 0) reinterpret_cast<int *>(ws + it.a_off + w.ex[JOB])[e * R + row] = E;
  unsigned char *A = reinterpret_cast<unsigned char *>(ws + it.a_off + w.a[JOB]) + (long long)tr * nk * SEP_ABLK;
  const int r = row & 127, off0 = (r >> 3) * 256 + (r & 7) * 16;
  for (int k8 = kl; k8 < 2 * nk; k8 += 32) {
    long long V[8], any = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      V[j] = fixed_of(k8 == kl ? x[j] : value(8 * k8 + j), E);
      if (cj < 0.0) V[j] = -V[j];
      any |= V[j];
    }
    if (any) atomicOr(&smask[k8 >> 6], 1u << ((k8 >> 1) & 31));
    store_digits(A + (long long)(k8 >> 1) * SEP_ABLK + off0 + (k8 & 1) * 128, 4096, V);
  }
  __syncthreads();
  if (threadIdx.x < SEP_MASK && smask[threadIdx.x])
    atomicOr(reinterpret_cast<unsigned *>(ws + it.a_off + w.mask) + adj_mask_of(JOB, it.ncols) + tr * SEP_MASK + threadIdx.x,
             smask[threadIdx.x]);
}
template <int STAGE>
__global__ void __launch_bounds__(256) k_adj_cut(Batch bt, const SubDesc *subs, double *ws, const double2 *cot,
                                                 const double2 *cot_rec) {
  pdl_wait();
  Item it; int local;
  locate(bt, blockIdx.x, it, local);
  MDP_CHECK_ITEM(bt, subs, it, local, STAGE == 1 ? F_AC1 : F_AC3);
  const SubDesc &d = subs[it.sub];
  constexpr int J0 = STAGE == 1 ? A_MID : A_SYN, J1 = STAGE == 1 ? A_FWD : A_INV;
  const int n0 = adj_cut_blocks(d, adj_geo(d, sep_geo(d)), J0, it.ncols);
  if (local < n0) adj_cut_body<J0>(it, d, ws, cot, cot_rec, local);
  else adj_cut_body<J1>(it, d, ws, cot, cot_rec, local - n0);
}

// ---------------------------------------------------------------- contractions
// the residual's: dK/dk, moments, their k-derivatives, dense rows (operands of k_sep_cut, stage 1)
struct GradSrc {
  Batch bt;
  const SubDesc *subs;
  const unsigned char *sep, *adj;
  double *ws;
  int user, fam;
  struct Tile : DigitTile {
    Item it;
    int e, mt, nt, R, fwd;
  };
  __device__ __forceinline__ int total() const { return bt.total_blocks; }
  __device__ __forceinline__ bool tile(int v, Tile &t) const {
    int local;
    locate(bt, v, t.it, local);
    const Item &it = t.it;
    if (MDP_CHECKED && !item_in_bounds(bt, subs, it, local, fam, true)) return false;
    const SubDesc &d = subs[it.sub];
    const SepGeo g = sep_geo(d);
    const SepWs w = sep_ws(d, it.ncols);
    const int Rm = sep_rows(d, J_MID, it.ncols, it.col0, user), n0 = g.ncls * (Rm / 128) * grad_mid_tiles(d, g);
    t.fwd = local >= n0;
    if (t.fwd) local -= n0;
    const int job = t.fwd ? J_FWD : J_MID;
    t.R = t.fwd ? sep_rows(d, J_FWD, it.ncols, it.col0, user) : Rm;
    const int nk = sep_nk(g, job), nt = t.fwd ? g.nqh / 32 : grad_mid_tiles(d, g), per = (t.R / 128) * nt;
    t.e = local / per;
    t.mt = (local % per) / nt;
    t.nt = local % nt;
    const int tr = t.e * (t.R / 128) + t.mt;
    t.A = reinterpret_cast<const unsigned char *>(ws + it.a_off + w.a[job]) + (long long)tr * nk * SEP_ABLK;
    t.ex = reinterpret_cast<const int *>(ws + it.a_off + w.ex[job]) + tr * 128;
    const unsigned *ma = reinterpret_cast<const unsigned *>(ws + it.a_off + w.mask) + sep_mask_of(job, it.ncols) + tr * SEP_MASK;
    const unsigned *mb = nullptr;
    t.eb = t.nkj = t.ND = t.ti = 0;
    const int nm = 2 * g.nqp / 32;   // tiles of the moments
    if (t.fwd) t.B = sep + d.sep_bf + ((long long)t.e * (g.nqh / 32) + t.nt) * nk * SEP_BBLK;
    else if (t.nt < g.nt3) {
      const int es = t.e * g.nS + t.nt / g.nti;
      t.B = adj + d.adj_dtb + (long long)es * g.nS * g.ND * SEP_BBLK;
      t.nkj = g.nkj; t.ND = g.ND; t.ti = t.nt % g.nti;
      t.eb = reinterpret_cast<const int *>(adj + d.adj_kde)[g.ncls * g.nS + es];
    } else if (t.nt < g.nt3 + nm) {
      const SepMoment m = sep_moment(d, g, t.e, t.nt - g.nt3);
      t.B = sep + m.blocks;
      mb = reinterpret_cast<const unsigned *>(sep + m.mask);
    } else {
      const SepMoment m = adj_dmoment(d, g, t.e, t.nt - g.nt3 - nm);
      t.B = adj + m.blocks;
      mb = reinterpret_cast<const unsigned *>(adj + m.mask);
    }
    t.masks(ma, mb);
    return !MDP_CHECKED || t.in_bounds(ws, bt.ws_n, sep, bt.sep_n, adj, bt.adj_n, nk, bt.status);
  }
  __device__ __forceinline__ const double *out() const { return ws; }
  __device__ __forceinline__ long long out_n() const { return bt.ws_n; }
  __device__ __forceinline__ void dest(const Tile &t, int r, int o, double *&dst, long long &step, int &cnt) const {
    const Item &it = t.it;
    const SubDesc &d = subs[it.sub];
    const SepGeo g = sep_geo(d);
    const SepWs w = sep_ws(d, it.ncols);
    const int row = t.mt * 128 + r, o0 = t.nt * 32 + o, nm = 2 * g.nqp / 32;
    step = t.R;
    cnt = 8;
    if (t.fwd) {
      const int cp = sep_pad128(it.ncols), parts = user ? 2 : 1;
      int col = row % cp;
      cnt = col < it.ncols && 2 * o0 + 1 + t.e <= d.Nq ? (d.Nq - (1 + t.e) - 2 * o0) / 2 + 1 : 0;
      if (!user && cnt > 0) col = sep_col_of(d, it.col0, it.ncols, col);
      step = 2LL * it.ncols * parts;
      dst = ws + it.gr_off + (((long long)(row / (cp * parts)) * d.Nq + 2 * o0 + t.e) * it.ncols + col) * parts + (row / cp) % parts;
    } else if (t.nt < g.nt3) {
      const int i0 = (t.nt % g.nti) * 32 + o;
      cnt = g.Pi - i0;
      dst = ws + it.a_off + w.u1 + ((long long)(t.e * g.nS + t.nt / g.nti) * g.Pi + i0) * t.R + row;
    } else if (t.nt < g.nt3 + nm) {
      dst = ws + it.a_off + w.mom + ((long long)t.e * 3 * g.nqp + o0 - 32 * g.nt3) * t.R + row;
    } else {
      dst = ws + it.a_off + adj_ws(d, it.ncols).dmom + ((long long)t.e * ADJ_DMOM * g.nqp + o0 - 32 * (g.nt3 + nm)) * t.R + row;
    }
  }
};
// the cotangent's
template <int STAGE>
struct AdjSrc {
  Batch bt;
  const SubDesc *subs;
  const unsigned char *adj;
  double *ws;
  struct Tile : DigitTile {
    Item it;
    int job, e, mt, nt, R;
  };
  __device__ __forceinline__ int total() const { return bt.total_blocks; }
  __device__ __forceinline__ bool tile(int v, Tile &t) const {
    int local;
    locate(bt, v, t.it, local);
    const Item &it = t.it;
    if (MDP_CHECKED && !item_in_bounds(bt, subs, it, local, STAGE == 1 ? F_AG1 : F_ATCOLS, true)) return false;
    const SubDesc &d = subs[it.sub];
    const SepGeo g = sep_geo(d);
    const AdjGeo a = adj_geo(d, g);
    const AdjWs w = adj_ws(d, it.ncols);
    t.job = STAGE == 1 ? A_MID : A_SYN;
    const int n0 = adj_tiles(d, a, t.job, it.ncols);
    if (local >= n0) { ++t.job; local -= n0; }
    t.R = adj_rows(d, t.job, it.ncols);
    const int nk = adj_nk(a, t.job), nt = adj_nt(a, t.job), per = (t.R / 128) * nt;
    t.e = local / per;
    t.mt = (local % per) / nt;
    t.nt = local % nt;
    const int tr = t.e * (t.R / 128) + t.mt;
    t.A = reinterpret_cast<const unsigned char *>(ws + it.a_off + w.a[t.job]) + (long long)tr * nk * SEP_ABLK;
    t.ex = reinterpret_cast<const int *>(ws + it.a_off + w.ex[t.job]) + tr * 128;
    const unsigned *ma = reinterpret_cast<const unsigned *>(ws + it.a_off + w.mask) + adj_mask_of(t.job, it.ncols) + tr * SEP_MASK;
    const unsigned *mb = nullptr, *mb2 = nullptr;
    t.eb = t.nkj = t.ND = t.ti = 0;
    if (t.job == A_SYN) {
      const long long v3 = (long long)t.e * a.nt3 + t.nt;
      const int k2 = 2 * g.nqp / 16;
      t.B = adj + d.adj_b3 + v3 * k2 * SEP_BBLK;
      mb = reinterpret_cast<const unsigned *>(adj + d.adj_z3) + v3 * SEP_MASK;
      if (a.nb == 3) {
        t.k2 = k2;
        t.B2 = adj + d.adj_r3 + v3 * (k2 / 2) * SEP_BBLK;
        mb2 = reinterpret_cast<const unsigned *>(adj + d.adj_r3z) + v3 * SEP_MASK;
      }
      t.eb = inv_exp(d);
    } else if (t.job == A_INV) {
      t.B = adj + d.adj_bi + ((long long)t.e * a.ntr + t.nt) * nk * SEP_BBLK;
      t.eb = inv_exp(d);
    } else if (t.job == A_FWD) {
      t.B = adj + d.adj_bf + ((long long)t.e * (g.nqh / 32) + t.nt) * nk * SEP_BBLK;
    } else if (t.nt < a.nt3) {
      const int ec = t.e * g.nS + t.nt / a.nti;
      t.B = adj + d.adj_tb + (long long)ec * g.nS * a.ND * SEP_BBLK;
      t.nkj = a.nkj; t.ND = a.ND; t.ti = t.nt % a.nti;
      t.eb = reinterpret_cast<const int *>(adj + d.adj_kde)[ec];
    } else {
      const int m = t.e * (ADJ_MOM * g.nqp / 32) + t.nt - a.nt3;
      t.B = adj + d.adj_mb + (long long)m * nk * SEP_BBLK;
      mb = reinterpret_cast<const unsigned *>(adj + d.adj_zm) + m * SEP_MASK;
    }
    t.masks(ma, mb, mb2);
    return !MDP_CHECKED || t.in_bounds(ws, bt.ws_n, adj, bt.adj_n, adj, bt.adj_n, nk, bt.status);
  }
  __device__ __forceinline__ const double *out() const { return ws; }
  __device__ __forceinline__ long long out_n() const { return bt.ws_n; }
  __device__ __forceinline__ void dest(const Tile &t, int r, int o, double *&dst, long long &step, int &cnt) const {
    const Item &it = t.it;
    const SubDesc &d = subs[it.sub];
    const SepGeo g = sep_geo(d);
    const AdjGeo a = adj_geo(d, g);
    const AdjWs w = adj_ws(d, it.ncols);
    const int row = t.mt * 128 + r, o0 = t.nt * 32 + o;
    step = t.R;
    cnt = 8;
    if (t.job == A_SYN || t.nkj > 0) {
      const int j0 = (t.nt % a.nti) * 32 + o;
      cnt = g.Pj - j0;
      dst = ws + it.a_off + (t.nkj > 0 ? w.u1 : w.u3) + ((long long)(t.e * g.nS + t.nt / a.nti) * g.Pj + j0) * t.R + row;
    } else if (t.job == A_MID) {
      dst = ws + it.a_off + w.mom + ((long long)t.e * ADJ_MOM * g.nqp + o0 - 32 * a.nt3) * t.R + row;
    } else if (t.job == A_INV) {
      cnt = g.Kf - o0;
      dst = ws + it.a_off + w.ui + ((long long)t.e * g.Kf + o0) * t.R + row;
    } else {
      const int cp = sep_pad128(it.ncols), col = row % cp;
      cnt = col < it.ncols && 2 * o0 + 1 + t.e <= d.Nq ? (d.Nq - (1 + t.e) - 2 * o0) / 2 + 1 : 0;
      step = 4LL * it.ncols;
      dst = ws + it.a_off + w.ga + (((long long)(row / (2 * cp)) * d.Nq + 2 * o0 + t.e) * it.ncols + col) * 2 + ((row / cp) & 1);
    }
  }
};
__global__ void __launch_bounds__(SG_THREADS, 1)
    k_grad_gemm(Batch bt, const SubDesc *subs, const unsigned char *sep, const unsigned char *adj, double *ws, int user, int fam,
                int *status) {
  pdl_wait();
  const GradSrc src{bt, subs, sep, adj, ws, user, fam};
  digit_gemm(src, status);
}
template <int STAGE>
__global__ void __launch_bounds__(SG_THREADS, 1)
    k_adj_gemm(Batch bt, const SubDesc *subs, const unsigned char *adj, double *ws, int *status) {
  pdl_wait();
  const AdjSrc<STAGE> src{bt, subs, adj, ws};
  digit_gemm(src, status);
}

// ---------------------------------------------------------------- modes
// FP64-bound: some 200 instructions per mode and 32 columns with both ends (100 in two 3 x 3 blocks where they do
// not see each other, as for most modes; a body each, so that the table's loads are not behind branches: 93 us
// for 4 x 257^2 with 1024 columns, 116 by the full matrix, 152 with the branches inside).
// Per (mode, column): the transpose of the projection's modes' matrix on the cotangent's moments and gamma
// rows (F): A_b for the middle ring rows, the field at the 4 dense ring rows. With DK the mode's part of
// <c, Tr G' r>, returned.
// far: the two ends do not see each other, two 3 x 3 blocks of the matrix
template <bool CIN, bool DK, bool far>
__device__ __forceinline__ double adj_modes_body(const Item &it, const SubDesc &d, const SepGeo &g, const SepWs &sw, const AdjWs &w,
                                                 const unsigned char *sep, const unsigned char *adj, double *ws, bool rec, int b,
                                                 int row1, int q) {
  const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
  const double *D = reinterpret_cast<const double *>(adj + d.adj_md) + (long long)(q - 1) * ADJ_MDW;
  const int e = d.xsym ? ((q & 1) ? 0 : 1) : 0, qi = d.xsym ? (q - 1) >> 1 : q - 1;
  const int cp = sep_pad128(it.ncols), R = 2 * cp;
  const long long nc = it.ncols;
  const double *ga = ws + it.a_off + w.ga;
  const double *prec = reinterpret_cast<const double *>(sep + d.sep_rp) + q - 1;   // phi at the receiver row
  const double *mom = ws + it.a_off + w.mom + ((long long)e * ADJ_MOM * g.nqp + qi) * R + b;
  cplx F[6], dM[2], f4 = cmk(0.0, 0.0);   // moments, gamma rows; derivative moments; receiver row
#pragma unroll
  for (int r = 0; r < 4; ++r) F[2 + r] = ld2(ga + 2 * (((long long)r * d.Nq + (q - 1)) * nc + b));
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double *p = mom + (long long)k * g.nqp * R, *pd = mom + (long long)(2 + k) * g.nqp * R;
    F[k] = cmk(p[0], p[cp]);
    if (DK) { const double ir = inv2(D[MD_RHO1 + k]); dM[k] = cmk(pd[0] * ir, pd[cp] * ir); }
  }
  if (rec) {
    f4 = ld2(ga + 2 * ((4LL * d.Nq + (q - 1)) * nc + b));
    F[0] = caxpy(prec[0], f4, F[0]);
    F[1] = caxpy(prec[d.Nq], f4, F[1]);
  }
  const bool imag = T[MT_IMAG] != 0.0;
  cplx m1 = F[0], m2 = F[1], iA = cmk(0.0, 0.0), iB = iA;   // moments of all rows; i Im R times them
  if (imag) {
#pragma unroll
    for (int r = 0; r < 4; ++r) { m1 = caxpy(T[MT_P1G + r], F[2 + r], m1); m2 = caxpy(T[MT_P2G + r], F[2 + r], m2); }
    const cplx u = cadd(cmk(T[MT_R + 1] * m1.re, T[MT_R + 1] * m1.im), cmk(T[MT_R + 3] * m2.re, T[MT_R + 3] * m2.im));
    const cplx v = cadd(cmk(T[MT_R + 3] * m1.re, T[MT_R + 3] * m1.im), cmk(T[MT_R + 5] * m2.re, T[MT_R + 5] * m2.im));
    iA = cmk(-u.im, u.re);
    iB = cmk(-v.im, v.re);
  }
  auto column = [&](int k, cplx v) {   // F^T times column k of the matrix, added to v
    if (far) {
      const int e_ = k < 4 ? k >> 1 : k - 4;
      v = caxpy(T[MT_MAT + 6 * e_ + k], F[e_], v);
      v = caxpy(T[MT_MAT + 6 * (2 + 2 * e_) + k], F[2 + 2 * e_], v);
      return caxpy(T[MT_MAT + 6 * (3 + 2 * e_) + k], F[3 + 2 * e_], v);
    }
#pragma unroll
    for (int o = 0; o < 6; ++o) v = caxpy(T[MT_MAT + 6 * o + k], F[o], v);
    return v;
  };
  // coefficients on the middle rows (columns 4, 5 of the matrix)
  cplx A[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) A[k] = column(4 + k, k == 0 ? iA : iB);
  double *ae = ws + it.a_off + w.aeff + ((long long)e * 3 * g.nqp + qi) * R + b;
#pragma unroll
  for (int k = 0; k < 2; ++k) { ae[(long long)k * g.nqp * R] = A[k].re; ae[(long long)k * g.nqp * R + cp] = A[k].im; }
  if (d.nrec >= 0) {
    const double s = T[MT_RFI];
    ae[2LL * g.nqp * R] = s * f4.re;
    ae[2LL * g.nqp * R + cp] = s * f4.im;
  }
  double *y = ws + it.y_off;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    cplx v = imag ? caxpy(T[MT_P1D + r], iA, cmk(T[MT_P2D + r] * iB.re, T[MT_P2D + r] * iB.im)) : cmk(0.0, 0.0);
    v = column(r, v);
    st2(y + 2 * (((long long)(q - 1) * 5 + r) * nc + b), v);
  }
  if (!DK) return 0.0;
  // ---- the residual's side
  const int R1 = sep_rows(d, J_MID, it.ncols, it.col0, CIN);
  const double *gr = ws + it.gr_off;
  const double *rm = ws + it.a_off + sw.mom + ((long long)e * 3 * g.nqp + qi) * R1 + row1;
  const double *rd = ws + it.a_off + w.dmom + ((long long)e * ADJ_DMOM * g.nqp + qi) * R1 + row1;
  const cplx zero = cmk(0.0, 0.0);
  auto at = [&](const double *p, int slot, double s) {
    if (row1 < 0) return zero;
    const double *v = p + (long long)slot * g.nqp * R1;
    return cmk(s * v[0], CIN ? s * v[cp] : 0.0);
  };
  auto axpy = [&](double s, cplx x, cplx y_) { return CIN ? caxpy(s, x, y_) : cmk(fma(s, x.re, y_.re), 0.0); };
  cplx in[6], dm[2];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const long long o = ((long long)r * d.Nq + (q - 1)) * nc + b;
    in[r] = CIN ? ld2(gr + 2 * o) : cmk(gr[o], 0.0);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) { in[4 + k] = at(rm, k, 1.0); dm[k] = at(rd, k, inv2(D[MD_RHO1 + k])); }
  auto redot = [&](cplx x, cplx z) { return CIN ? fma(x.re, z.re, -x.im * z.im) : x.re * z.re; };   // Re x z
  auto row = [&](const double *M, int o) {   // row o of a matrix times the residual's inputs
    cplx v = zero;
    if (far) {
      const int e_ = o < 2 ? o : (o - 2) >> 1;
      v = axpy(M[6 * o + 2 * e_], in[2 * e_], v);
      v = axpy(M[6 * o + 2 * e_ + 1], in[2 * e_ + 1], v);
      return axpy(M[6 * o + 4 + e_], in[4 + e_], v);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) v = axpy(M[6 * o + k], in[k], v);
    return v;
  };
  double s = 0.0;
#pragma unroll
  for (int o = 0; o < 6; ++o) s += redot(F[o], row(D + MD_MAT, o));
#pragma unroll
  for (int k = 0; k < 2; ++k) s += redot(A[k], dm[k]);
  // forward coefficients against the cotangent's derivative moments, with i Im R and its derivative
  cplx a0 = row(T + MT_MAT, 0), a1 = row(T + MT_MAT, 1);
  if (imag) {
    cplx r1 = in[4], r2 = in[5], e1 = zero, e2 = zero, h1 = zero, h2 = zero;   // moments of all rows; d phi/dk parts of the full rows
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      r1 = axpy(T[MT_P1D + r], in[r], r1);
      r2 = axpy(T[MT_P2D + r], in[r], r2);
      e1 = axpy(D[MD_P1D + r], in[r], e1);
      e2 = axpy(D[MD_P2D + r], in[r], e2);
      h1 = caxpy(D[MD_P1G + r], F[2 + r], h1);
      h2 = caxpy(D[MD_P2G + r], F[2 + r], h2);
    }
    const double I11 = T[MT_R + 1], I12 = T[MT_R + 3], I22 = T[MT_R + 5];
    const double J11 = D[MD_RI], J12 = D[MD_RI + 1], J22 = D[MD_RI + 2];
    auto imdot = [&](cplx x, cplx z) { return CIN ? fma(x.re, z.im, x.im * z.re) : x.im * z.re; };   // Im x z
    const cplx u1 = axpy(I11, r1, axpy(I12, r2, zero)), u2 = axpy(I12, r1, axpy(I22, r2, zero));
    const cplx v1 = axpy(I11, e1, axpy(I12, e2, zero)), v2 = axpy(I12, e1, axpy(I22, e2, zero));
    const cplx w1 = axpy(J11, r1, axpy(J12, r2, zero)), w2 = axpy(J12, r1, axpy(J22, r2, zero));
    // Re (i x z) = -Im x z
    s -= imdot(m1, w1) + imdot(m2, w2) + imdot(m1, v1) + imdot(m2, v2) + imdot(h1, u1) + imdot(h2, u2);
    a0 = cadd(a0, cmk(-u1.im, u1.re));
    a1 = cadd(a1, cmk(-u2.im, u2.re));
  }
  auto redotc = [&](cplx x, cplx z) { return fma(x.re, z.re, -x.im * z.im); };
  s += redotc(dM[0], a0) + redotc(dM[1], a1);
  if (rec) {
    const cplx m3 = at(rd, 2, inv2(D[MD_RFD]));
    const double *dp = reinterpret_cast<const double *>(adj + d.adj_rp) + q - 1;
    s += redotc(f4, cadd(caxpy(dp[0], a0, caxpy(dp[d.Nq], a1, zero)), m3));
  }
  return s;
}
template <bool CIN, bool DK>
__global__ void __launch_bounds__(128) k_adj_modes(Batch bt, const SubDesc *subs, const unsigned char *sep, const unsigned char *adj,
                                                   double *ws, int has_rec) {
  pdl_wait();
  __shared__ double sh[128];
  Item it; int local;
  locate(bt, blockIdx.x, it, local);
  MDP_CHECK_ITEM(bt, subs, it, local, F_AMODE);
  const SubDesc &d = subs[it.sub];
  const int cb = (it.ncols + 31) >> 5;
  const int per = sep_modes_per_block(d, it.ncols);
  const int b = (local % cb) * 32 + threadIdx.x, q0 = (local / cb) * per + threadIdx.y + 1;
  double s = 0.0;
  if (b < it.ncols) {
    const SepGeo g = sep_geo(d);
    const SepWs sw = sep_ws(d, it.ncols);
    const AdjWs w = adj_ws(d, it.ncols);
    const int row1 = CIN ? b : sep_row_of(d, it.col0, it.ncols, b) - sep_first34(d, it.col0, it.ncols);
    for (int q = q0; q < q0 + per - (int)threadIdx.y && q <= d.Nq; q += 4)
      s += reinterpret_cast<const double *>(sep + d.sep_mt)[(long long)(q - 1) * SEP_MTW + MT_FAR] != 0.0
               ? adj_modes_body<CIN, DK, true>(it, d, g, sw, w, sep, adj, ws, has_rec && d.nrec >= 0, b, row1, q)
               : adj_modes_body<CIN, DK, false>(it, d, g, sw, w, sep, adj, ws, has_rec && d.nrec >= 0, b, row1, q);
  }
  if (DK) {
    s = block_sum<128>(s, sh);
    if (threadIdx.x == 0 && threadIdx.y == 0) ws[it.red_off + local] = -(2.0 / d.Nx) * s;
  }
}

// ---------------------------------------------------------------- mu on the ring
// mu = conj of the sums, into the ring rows that k_adj_gamma reads ([ring node][column], complex); with DK the
// k-gradient's parts -Re <mu, s> and, of the middle rows, -Re <c, (dK/dk r)>.
template <bool CIN, bool DK>
__global__ void __launch_bounds__(256) k_adj_out(Batch bt, const SubDesc *subs, double *ws, const double2 *cot) {
  pdl_wait();
  __shared__ double sh[256];
  Item it; int local;
  locate(bt, blockIdx.x, it, local);
  MDP_CHECK_ITEM(bt, subs, it, local, F_AOUT);
  const SubDesc &d = subs[it.sub];
  const SepGeo g = sep_geo(d);
  const AdjWs w = adj_ws(d, it.ncols);
  const int cb = (it.ncols + 31) >> 5, cp = sep_pad128(it.ncols), R = 2 * cp;
  const int n0 = cb * ((g.Pj + 7) / 8), n1 = cb * ((4 * g.Kf + 7) / 8);
  const long long nc = it.ncols;
  const int part = local < n0 ? 0 : local < n0 + n1 ? 1 : 2, l = part == 0 ? local : part == 1 ? local - n0 : local - n0 - n1;
  const int b = (l % cb) * 32 + threadIdx.x, u = (l / cb) * 8 + threadIdx.y;
  double dk = 0.0;
  auto put = [&](int ri, cplx v, bool support) {   // v = conj(mu); s of basis columns (k_ring): real, on its support
    st2(ws + it.r_off + 2 * ((long long)ri * nc + b), cmk(v.re, -v.im));
    if (DK && CIN) {
      const cplx s = ld2(ws + it.s_off + 2 * ((long long)ri * nc + b));
      dk -= fma(v.re, s.re, -v.im * s.im);   // Re conj(mu) s
    } else if (DK && support) {
      dk = fma(-v.re, ws[it.s_off + (long long)ri * nc + b], dk);
    }
  };
  const int side = CIN || b >= it.ncols ? 0 : col_side(d, it.col0 + b);
  if (b < it.ncols && part == 0 && u < g.Pj) {
    cplx v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {   // (class, column) or column
      const long long o = ((long long)k * g.Pj + u) * R + b;
      const double *p1 = ws + it.a_off + w.u1 + o, *p3 = ws + it.a_off + w.u3 + o;
      v[k] = cmk(p1[0] + p3[0], p1[cp] + p3[cp]);
    }
    const int r0 = 2 * d.Px + 4 * u;
    const bool l = side == 3, r = side == 4;
    if (d.xsym) { put(r0, cadd(v[0], v[2]), l); put(r0 + 1, cadd(v[1], v[3]), l); put(r0 + 2, csub(v[1], v[3]), r); put(r0 + 3, csub(v[0], v[2]), r); }
    else { put(r0, v[0], l); put(r0 + 1, v[1], l); put(r0 + 2, v[2], r); put(r0 + 3, v[3], r); }
  } else if (b < it.ncols && part == 1 && u < 4 * g.Kf) {
    const int rr = u / g.Kf, k = u % g.Kf, m = g.mf + k, m2 = d.Nx - m, Ri = adj_rows(d, A_INV, it.ncols);
    const double *p0 = ws + it.a_off + w.ui + (long long)k * Ri + rr * R + b, *p1 = p0 + (long long)g.Kf * Ri;
    const cplx x = cmk(p0[0], p0[cp]), y = cmk(p1[0], p1[cp]);
    const int base = rr * d.Px + (rr < 2 ? 0 : 4 * (d.Py - 4)) - d.mlo;
    auto support = [&](int mm) {
      return side == 1 ? rr < 2 : side == 2 ? rr >= 2 : side == 3 ? mm <= d.mlo + 1 : mm >= d.mhi - 1;
    };
    if (m >= d.mlo && m <= d.mhi) put(base + m, cadd(x, y), support(m));
    if (m2 != m && m2 >= d.mlo && m2 <= d.mhi) put(base + m2, csub(x, y), support(m2));
  } else if (DK && b < it.ncols && part == 2 && u < g.Pi) {
    const int row1 = CIN ? b : sep_row_of(d, it.col0, it.ncols, b) - sep_first34(d, it.col0, it.ncols);
    if (row1 >= 0) {
      const int R1 = sep_rows(d, J_MID, it.ncols, it.col0, CIN);
      const double *ud = ws + it.a_off + sep_ws(d, it.ncols).u1;
      cplx v[4], z[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const double *p = ud + ((long long)k * g.Pi + u) * R1 + row1;
        v[k] = cmk(p[0], CIN ? p[cp] : 0.0);
      }
      if (d.xsym) { z[0] = cadd(v[0], v[2]); z[1] = cadd(v[1], v[3]); z[2] = csub(v[1], v[3]); z[3] = csub(v[0], v[2]); }
      else { z[0] = v[0]; z[1] = v[1]; z[2] = v[2]; z[3] = v[3]; }
      const double2 *c = cot + it.io_off + (long long)b * d.G + 2 * (d.Px + 2) + 4 * u;
#pragma unroll
      for (int s = 0; s < 4; ++s) dk -= CIN ? fma(c[s].x, z[s].re, c[s].y * z[s].im) : c[s].x * z[s].re;
    }
  }
  if (DK) {
    int base[5];
    red_slots(d, it.ncols, base);
    const double s = block_sum<256>(dk, sh);
    if (threadIdx.x == 0 && threadIdx.y == 0) ws[it.red_off + base[1] + local] = s;
  }
}

}  // namespace

// ---------------------------------------------------------------- launchers
cudaError_t set_sepadj_kernel_attributes() {
  cudaError_t e = cudaFuncSetAttribute(k_grad_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_adj_gemm<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_adj_gemm<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM);
  return e;
}

cudaError_t launch_adj_sines(const mdp_plan *p, cudaStream_t st) {
  int k[2] = {0, 0}, t[2] = {0, 0};
  for (size_t i = 0; i < p->subs.size(); ++i) {
    const SubDesc &d = p->subs[i].d;
    if (!d.tc_cols || d.leader != (int)i) continue;
    const SepGeo g = sep_geo(d);
    const AdjGeo a = adj_geo(d, g);
    k[0] = std::max(k[0], (a.nkf + 3) / 4);
    k[1] = std::max(k[1], (g.nqh / 16 + 3) / 4);
    t[0] = std::max(t[0], 2 * g.nqh / 32);
    t[1] = std::max(t[1], 2 * a.ntr);
  }
  const int ns = (int)p->subs.size();
  if (t[0] == 0) return cudaSuccess;
  for (int s0 = 0; s0 < ns; s0 += 65535)
    for (int inv = 0; inv < 2; ++inv)
      k_adj_sines<<<dim3(k[inv], t[inv], (unsigned)std::min(65535, ns - s0)), 256, 0, st>>>(p->d_subs, s0, p->d_tables, p->d_adj, inv);
  return cudaGetLastError();
}

cudaError_t launch_adj_tables(const mdp_plan *p, cudaStream_t st) {
  int mq = 0, mrow = 0, mdist = 0, mes = 0, mtb[2] = {0, 0}, mk[2] = {0, 0}, mt[2] = {0, 0}, m3 = 0, m3k = 0, mrec = 0;
  for (size_t i = 0; i < p->subs.size(); ++i) {
    const SubDesc &d = p->subs[i].d;
    if (!d.tc_cols || (d.leader != (int)i && d.nrec < 0)) continue;   // a duplicate has its receiver row's tables
    const SepGeo g = sep_geo(d);
    const AdjGeo a = adj_geo(d, g);
    if (d.nrec >= 0) mrec = std::max(mrec, (d.Nq + 31) / 32);
    mq = std::max(mq, (d.Nq + 127) / 128);
    mrow = std::max(mrow, (d.Py + 2 + 7) / 8);
    mdist = std::max(mdist, d.Py);
    mes = std::max(mes, g.ncls * g.nS * g.nS);
    mtb[0] = std::max(mtb[0], (a.ND + 3) / 4);
    mtb[1] = std::max(mtb[1], (g.ND + 3) / 4);
    mk[0] = std::max(mk[0], (a.nk1 + 3) / 4);
    mk[1] = std::max(mk[1], (g.nk1 + 3) / 4);
    mt[0] = std::max(mt[0], g.ncls * ADJ_MOM * g.nqp / 32);
    mt[1] = std::max(mt[1], g.ncls * g.nb * g.nqp / 32);
    m3 = std::max(m3, g.ncls * a.nt3);
    m3k = std::max(m3k, (a.nk3 + 3) / 4);
  }
  if (mq == 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(p->d_adj, 0, (size_t)p->adj_masks, st);
  if (e != cudaSuccess) return e;
  const SubDesc *ds = p->d_subs;
  const double *tab = p->d_tables;
  const int ns = (int)p->subs.size();
  for (int s0 = 0; s0 < ns; s0 += 65535) {
    const unsigned n = (unsigned)std::min(65535, ns - s0);
    k_adj_mode_tab<<<dim3(4 * mq, n), 32, 0, st>>>(ds, s0, p->d_sep, p->d_adj);
    if (mrec > 0) k_adj_rec<<<dim3(mrec, n), 32, 0, st>>>(ds, s0, p->d_sep, p->d_adj);
    k_adj_phid<<<dim3(mq, mrow, n), 128, 0, st>>>(ds, s0, p->d_sep, p->d_adj);
    k_adj_kd<<<dim3(mdist, n), 128, 0, st>>>(ds, s0, tab, p->d_sep, p->d_adj);
    for (int w = 0; w < 2; ++w) {
      k_adj_tb<<<dim3(mtb[w], mes, n), 256, 0, st>>>(ds, s0, p->d_sep, p->d_adj, w);
      k_adj_mb<<<dim3(mk[w], mt[w], n), 256, 0, st>>>(ds, s0, tab, p->d_sep, p->d_adj, w);
    }
    k_adj_b3<<<dim3(m3k, m3, n), 256, 0, st>>>(ds, s0, tab, p->d_sep, p->d_adj);
  }
  return cudaGetLastError();
}

// the residual's side (with the k-gradient), before the cotangent takes the ring buffer
cudaError_t launch_sep_adj_residual(mdp_plan *p, const Batch *fb, bool user, bool rec, cudaStream_t st) {
  const int fc = user ? F_C1U : F_C1B, fg = user ? F_GG1U : F_GG1B;
  if (fb[fc].total_blocks == 0) return cudaSuccess;
  prof_begin(p, F_C1B, st);
  cudaError_t e = launch_sep_cut1(fb[fc], subs_of(p, rec), p->d_ws, user, fc, st);
  prof_end(p, F_C1B, st);
  if (e != cudaSuccess) return e;
  prof_begin(p, F_GG1B, st);
  pdl(k_grad_gemm, dim3(std::min(fb[fg].total_blocks, p->n_sm)), dim3(SG_THREADS), SG_SMEM, st, fb[fg], subs_of(p, rec), p->d_sep,
      p->d_adj, p->d_ws, user, fg, p->d_status);
  prof_end(p, F_GG1B, st);
  return cudaGetLastError();
}

// the cotangent's side, after k_adj_cols
cudaError_t launch_sep_adjoint(mdp_plan *p, const Batch *fb, bool user, bool dk, const double2 *cot, const double2 *cot_rec,
                               cudaStream_t st) {
  if (fb[F_AMODE].total_blocks == 0) return cudaSuccess;
  const SubDesc *ds = subs_of(p, cot_rec != nullptr);
  double *ws = p->d_ws;
  const int hr = cot_rec ? 1 : 0;
  const dim3 b4(32, 4), b8(32, 8);
  auto gemm_grid = [&](int f) { return dim3((unsigned)std::min(fb[f].total_blocks, p->n_sm)); };
#define ADJ_LAUNCH(f, kern, grid, block, smem, ...)                                  \
  do {                                                                               \
    prof_begin(p, f, st);                                                            \
    pdl(kern, dim3(grid), dim3(block), smem, st, fb[f], ds, __VA_ARGS__);            \
    prof_end(p, f, st);                                                              \
  } while (0)
  ADJ_LAUNCH(F_AC1, k_adj_cut<1>, fb[F_AC1].total_blocks, 256, 0, ws, cot, cot_rec);
  ADJ_LAUNCH(F_AG1, k_adj_gemm<1>, gemm_grid(F_AG1), SG_THREADS, SG_SMEM, p->d_adj, ws, p->d_status);
  if (!dk) ADJ_LAUNCH(F_AMODE, (k_adj_modes<true, false>), fb[F_AMODE].total_blocks, b4, 0, p->d_sep, p->d_adj, ws, hr);
  else if (user) ADJ_LAUNCH(F_AMODE, (k_adj_modes<true, true>), fb[F_AMODE].total_blocks, b4, 0, p->d_sep, p->d_adj, ws, hr);
  else ADJ_LAUNCH(F_AMODE, (k_adj_modes<false, true>), fb[F_AMODE].total_blocks, b4, 0, p->d_sep, p->d_adj, ws, hr);
  ADJ_LAUNCH(F_AC3, k_adj_cut<3>, fb[F_AC3].total_blocks, 256, 0, ws, cot, cot_rec);
  ADJ_LAUNCH(F_ATCOLS, k_adj_gemm<3>, gemm_grid(F_ATCOLS), SG_THREADS, SG_SMEM, p->d_adj, ws, p->d_status);
  if (!dk) ADJ_LAUNCH(F_AOUT, (k_adj_out<true, false>), fb[F_AOUT].total_blocks, b8, 0, ws, cot);
  else if (user) ADJ_LAUNCH(F_AOUT, (k_adj_out<true, true>), fb[F_AOUT].total_blocks, b8, 0, ws, cot);
  else ADJ_LAUNCH(F_AOUT, (k_adj_out<false, true>), fb[F_AOUT].total_blocks, b8, 0, ws, cot);
#undef ADJ_LAUNCH
  return cudaGetLastError();
}

// the operand masks of a wave's items, before anything is cut into them
cudaError_t launch_adj_clear(mdp_plan *p, const Batch *fb, bool rec, cudaStream_t st) {
  if (fb[F_ACLR].total_blocks == 0) return cudaSuccess;
  pdl(k_adj_clear, dim3(fb[F_ACLR].total_blocks), dim3(256), 0, st, fb[F_ACLR], subs_of(p, rec), p->d_ws);
  return cudaGetLastError();
}

}  // namespace mdp
