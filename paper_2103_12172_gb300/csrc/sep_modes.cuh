// The interior recurrence of a sine mode and the reflections at its ends (kernels_sep.cu, kernels_full.cu).
#pragma once
#include "digit_gemm.cuh"

namespace mdp {

__device__ __forceinline__ cplx cdivd(cplx a, cplx b) {
  const double n = 1.0 / fma(b.re, b.re, b.im * b.im);
  return {fma(a.re, b.re, a.im * b.im) * n, fma(a.im, b.re, -a.re * b.im) * n};
}
// the two homogeneous solutions at distance x from the middle row (kinds 0 and 1)
__device__ __forceinline__ double sep_c(int kind, double th, double x) { return kind == 0 ? cos(x * th) : cosh(x * th); }
__device__ __forceinline__ double sep_s(int kind, double th, double x) {
  if (th == 0.0) return x;
  return kind == 0 ? sin(x * th) / sin(th) : sinh(x * th) / sinh(th);
}

// Rows (a, b, a) of mode q between its ends: cosh or cos theta = -b / (2 a). On coarse grids (t > 1/2)
// x_i = (-1)^i z_i turns (a, b, a) into (-a, b, -a): sg = -1 and the signed a belong to z. Kind 0:
// propagating, 1: evanescent next to the cutoff (theta N < 4), 2: evanescent. The rows at the ends, for z:
// al0 z_0 + al1 z_1 = 0 and its mirror image.
struct ModeShape {
  double a, sg, th;
  int kind;
  cplx al0, al1;
};
// ab: the interior entries (a, b) of T_q as the factorisation of the same tables rounded them (the host's
// at plan creation, else this device's): b + 2 a is exact, and an error of b moves theta by its half over
// theta^2, so both forms of the solve are to start from the same b
__device__ __forceinline__ ModeShape mode_shape(const SubDesc &d, int q, const double *ab) {
  ModeShape m;
  const double h = d.h, h2 = h * h, k = d.k, k2 = k * k;
  const double sq = sin(M_PI * q / (2.0 * d.Nx)), lam = -4.0 * sq * sq;
  m.a = ab[0];
  double t = (ab[1] + 2.0 * m.a) / (4.0 * m.a);         // sin^2(theta/2), or -sinh^2(theta/2)
  m.sg = 1.0;
  if (t > 0.5) { m.sg = -1.0; t = 1.0 - t; m.a = -m.a; }
  m.th = t > 0.0 ? 2.0 * asin(sqrt(t)) : 2.0 * asinh(sqrt(-t));
  m.kind = t > 0.0 ? 0 : m.th * (d.ny - 1) < 4.0 ? 1 : 2;
  m.al0 = cmk(1.0, 0.0);
  m.al1 = cmk(0.0, 0.0);
  if (d.cplx) {
    const bool paper = d.ap_bc == MDP_AP_DIRX_SOMMY_PAPER;
    const double alpha = paper ? (1.0 - k2 * h2 / 24.0 - lam / 6.0) / h2 : (1.0 + k2 * h2 / 24.0 + lam / 24.0) / h2;
    const double beta = k * (1.0 + k2 * h2 / 8.0 + lam / (paper ? 2.0 : 8.0)) / h;
    m.al0 = cmk(alpha, 0.5 * beta);
    m.al1 = cmk(-m.sg * alpha, 0.5 * m.sg * beta);
  }
  return m;
}
// kinds 0, 1: R for phi = (C(x), S(x)) about the row mid (not normalised), ends at 0 and N
__device__ __forceinline__ void reflect_cs(const ModeShape &m, int N, double mid, cplx &R11, cplx &R12, cplx &R22) {
  auto lin = [&](double x, double y) { return cmk(fma(m.al0.re, x, m.al1.re * y), fma(m.al0.im, x, m.al1.im * y)); };
  const cplx b1 = lin(sep_c(m.kind, m.th, 0.0 - mid), sep_c(m.kind, m.th, 1.0 - mid));
  const cplx b2 = lin(sep_s(m.kind, m.th, 0.0 - mid), sep_s(m.kind, m.th, 1.0 - mid));
  const cplx t1 = lin(sep_c(m.kind, m.th, N - mid), sep_c(m.kind, m.th, N - 1 - mid));
  const cplx t2 = lin(sep_s(m.kind, m.th, N - mid), sep_s(m.kind, m.th, N - 1 - mid));
  const cplx det = csub(cmul(b1, t2), cmul(b2, t1)), ad = cmk(m.a * det.re, m.a * det.im);
  R11 = cdivd(cmul(b2, t2), ad);
  R22 = cdivd(cmul(b1, t1), ad);
  R12 = cdivd(cadd(cmul(b1, t2), cmul(b2, t1)), cmk(-2.0 * ad.re, -2.0 * ad.im));
}
// kind 2: R for phi = (e^{-theta (i - J0)}, e^{-theta (J1 - i)}), kappa(0) = c
__device__ __forceinline__ void reflect_exp(const ModeShape &m, int N, int J0, int J1, double c, cplx &R11, cplx &R12,
                                            cplx &R22) {
  const double ep = exp(m.th), em = exp(-m.th);
  const cplx num = cmk(fma(m.al1.re, ep, m.al0.re), fma(m.al1.im, ep, m.al0.im));
  const cplx den = cmk(fma(m.al1.re, em, m.al0.re), fma(m.al1.im, em, m.al0.im));
  const cplx ref = cdivd(num, den);
  const double wb = -exp(-2.0 * m.th * J0), wt = -exp(-2.0 * m.th * (N - J1)), dl = exp(-m.th * (J1 - J0));
  const cplx rb = cmk(wb * ref.re, wb * ref.im), rt = cmk(wt * ref.re, wt * ref.im), rr = cmul(rb, rt);
  const cplx D = cmk(1.0 - rr.re * dl * dl, -rr.im * dl * dl);
  R11 = cdivd(cmk(c * rb.re, c * rb.im), D);
  R22 = cdivd(cmk(c * rt.re, c * rt.im), D);
  R12 = cdivd(cmk(c * dl * rr.re, c * dl * rr.im), D);
}

}  // namespace mdp
