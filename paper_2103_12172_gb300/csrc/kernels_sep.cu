// The projection's solves by the separable Green's function of the per-mode systems, with every
// long sum on the tensor cores.
//
// Away from the two ends the rows of T_q (sine mode q along x, Section 3.2.1) have constant
// coefficients (a, b, a), and the ring that carries r = L^(h) w lies strictly between the ends. On
// those rows the inverse is therefore
//   T_q^{-1}(i, j) = kappa_q(|i - j|) + sum_{a,b} phi_a(i) R_ab phi_b(j):
// kappa_q is a fundamental solution of the constant-coefficient recurrence (cosh theta = -b/2a:
// the decaying exponential for an evanescent mode, sin(|d| theta) / (2 a sin theta) for a
// propagating one, its hyperbolic form next to the cutoff, where the exponential would cancel),
// phi_1, phi_2 two homogeneous solutions (decaying away from either end, or cosine and sine about
// the middle row), and the symmetric 2 x 2 matrix R follows from the rows at the two ends (the
// Dirichlet or Sommerfeld conditions). Summed over q with the sine factors of the ring's columns
// m_c and the trace's columns m_s, the middle rows need
//   u(s, i) = sum_{c,j} K_sc(|i - j|) r_c(j) + sum_{q,b} (2/Nx) sin(pi q m_s/Nx) phi_b(i) A_b(q),
//   K_sc(d) = (2/Nx) sum_q sin(pi q m_s/Nx) sin(pi q m_c/Nx) kappa_q(d),
// where A_1, A_2 combine, per mode, the moments sum_{c,j} sin(pi q m_c/Nx) phi_b(j) r_c(j) and the
// transforms of the 4 dense ring rows. So two contractions (k_sep_gemm) replace the recurrences:
//   stage 1: r times [K | moment tables], K dimension (c, j); the dense rows times sines;
//   stage 2 (k_sep_modes): per (mode, column) A_1, A_2 and the 4 gamma rows of the field;
//   stage 3: A times [sines x phi], K dimension (b, q); the gamma rows' field times sines.
// The sine transforms of the 8 full rows are direct sums too: at up to 1025^2 the tensor cores take
// less time for N^2/2 exact products (odd and even modes on folded columns) than the FP64 pipe for a
// length-N FFT, on any N (257^2, 1024 columns: 58 + 117 us by FFT, 4 x 257^2).
// On x-centred subdomains odd and even modes separate (sums and differences of the mirrored
// columns), which halves both dimensions: two classes with 2 columns each, else one with 4.
//
// Both contractions are to FP64 accuracy on the fp16 tensor cores (digit_gemm.cuh). 4 x 257^2, 1024 columns:
// 209 us where the sweeps took 1392; 257^2 to 1025^2 x 8: 2.09 ms (41.2), of it k_sep_gemm 1.22, k_sep_cut 0.41,
// k_sep_out 0.19, k_sep_modes 0.14.
// Against 64-bit sums over the closed form in extended precision (k = 10 on 129^2, k = 30 on
// 257^2) the result is off by 1e-15 to 8e-15 (2-norm), plain FP64 sums by 4e-15 to 5e-14 and the
// pivoted recurrences by 4e-14 to 2.5e-13.
#include "sep_modes.cuh"

#include <algorithm>

namespace mdp {
namespace {

// ---------------------------------------------------------------- mode table
__global__ void __launch_bounds__(32) k_sep_mode_tab(const SubDesc *subs, int s0, unsigned char *sep, int entries) {
  const int si = s0 + blockIdx.y;
  const SubDesc &d = subs[si];
  const int q = blockIdx.x * 32 + threadIdx.x + 1;   // one warp per block: the FP64 pipe is an SM's
  if (d.leader != si || q > d.Nq) return;
  double *T = reinterpret_cast<double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
  double *ab = reinterpret_cast<double *>(sep + d.sep_ab) + 2 * (q - 1);
  if (entries) {   // as mode_rows of factor.cu
    const double h2 = d.h * d.h, k2 = d.k * d.k;
    const double sq = sin(M_PI * q / (2.0 * d.Nx)), lam = -4.0 * sq * sq;
    ab[0] = 1.0 / h2 + lam / (6.0 * h2) + k2 / 12.0;
    ab[1] = -2.0 * ab[0] + lam / h2 + k2 + k2 * lam / 12.0;
  }
  const ModeShape ms = mode_shape(d, q, ab);
  const double a = ms.a, sg = ms.sg, th = ms.th;
  const int kind = ms.kind, N = d.ny - 1, J0 = d.nlo - 1, J1 = d.nhi + 1;
  const double mid = 0.5 * (J0 + J1), Lh = 0.5 * (J1 - J0);
  double n1 = 1.0, n2 = 1.0, c = 0.0, rf;
  cplx R11, R12, R22;
  const int rows_d[4] = {d.nlo, d.nlo + 1, d.nhi - 1, d.nhi}, rows_g[4] = {d.nlo - 1, d.nlo, d.nhi, d.nhi + 1};
  const int L = d.nhi - d.nlo;   // J1 - J0 - 2
  // phi_1, phi_2 at the 3 rows from either end (J0 + k, J1 - k), kappa at 0, 1, 2, L-1, L, L+1 without the sign
  // sg^i; kappa(d) = T1 phi_1(J0 + d) + T2 phi_2(J0 + d). An FP64 instruction takes this thread's warp 64
  // cycles whatever its lanes do, a transcendental function some 50 of them: the neighbouring rows
  // follow by one rotation or one factor.
  double lo1[3], lo2[3], hi1[3], hi2[3], kv[6], T1, T2 = 0.0, el[3] = {0.0, 0.0, 0.0};
  if (kind < 2) {
    const double sth = kind == 0 ? sin(th) : sinh(th), c1 = sep_c(kind, th, 1.0), ss = kind == 0 ? -sth * sth : sth * sth;
    auto cs = [&](double x, double &C, double &S) {
      if (th == 0.0) { C = 1.0; S = x; return; }
      if (kind == 0) { sincos(x * th, &S, &C); S /= sth; }
      else { C = cosh(x * th); S = sinh(x * th) / sth; }
    };
    auto up = [&](double &C, double &S) { const double Cn = fma(S, ss, C * c1); S = fma(S, c1, C); C = Cn; };
    double CL, SL, Ch, Sh, C2, S2;
    cs(Lh, Ch, Sh);              // the end rows: C even, S odd about the middle
    cs(L - 1, CL, SL);
    cs(J1 - J0, C2, S2);
    double bound = kind == 0 ? fmin(fmax(Lh, 1.0), 1.0 / sth) : Sh;
    n2 = pow2i(-(ilogb(fmax(bound, 1.0)) + 1));
    if (kind == 1) n1 = 0.25;
    reflect_cs(ms, N, mid, R11, R12, R22);
    const double s1 = 1.0 / n1, s2 = 1.0 / n2;   // powers of two
    R11 = cmk(R11.re * s1 * s1, R11.im * s1 * s1);
    R12 = cmk(R12.re * s1 * s2, R12.im * s1 * s2);
    R22 = cmk(R22.re * s2 * s2, R22.im * s2 * s2);
    double C = Ch, S = -Sh;
    for (int k = 0; k < 3; ++k) {
      lo1[k] = hi1[k] = n1 * C;
      lo2[k] = n2 * S;
      hi2[k] = -n2 * S;
      up(C, S);
    }
    const double ia = 1.0 / (2.0 * a);
    kv[0] = 0.0; kv[1] = ia; kv[2] = 2.0 * c1 * ia;
    for (int k = 3; k < 6; ++k) { kv[k] = SL * ia; up(CL, SL); }
    T1 = Sh * ia / n1;
    T2 = Ch * ia / n2;
    const double kb = kind == 0 ? fmin((double)(J1 - J0), 1.0 / sth) : S2;
    rf = pow2i(-(ilogb(fmax(kb, 1.0) / (2.0 * fabs(a))) + 1));
  } else {
    const double em = exp(-th), ep = exp(th), fl = exp(-th * (L - 1));
    c = -1.0 / (a * (ep - em));
    reflect_exp(ms, N, J0, J1, c, R11, R12, R22);
    const double far = fl * em * em * em;   // J1 - J0 = L + 2
    lo1[0] = hi2[0] = 1.0; lo1[1] = hi2[1] = em; lo1[2] = hi2[2] = em * em;
    hi1[0] = lo2[0] = far; hi1[1] = lo2[1] = fl * em * em; hi1[2] = lo2[2] = fl * em;
    kv[0] = c; kv[1] = c * em; kv[2] = c * em * em;
    kv[3] = c * fl; kv[4] = c * fl * em; kv[5] = c * fl * em * em;
    el[0] = c; el[1] = c * ep; el[2] = c * ep * ep;   // kappa as a wave from J0: c e^{theta k} at the sources J0 + k
    T1 = c;
    rf = pow2i(-(ilogb(fabs(c)) + 1));
  }
  auto sgn = [&](int i) { return (sg < 0.0 && (i & 1)) ? -1.0 : 1.0; };   // sg^i
  auto p1 = [&](int i) { return sgn(i - J0) * (i - J0 < 3 ? lo1[i - J0] : hi1[J1 - i]); };
  auto p2 = [&](int i) { return sgn(i - J0) * (i - J0 < 3 ? lo2[i - J0] : hi2[J1 - i]); };
  auto kap = [&](int x) { return sgn(x) * (x < 3 ? kv[x] : kv[x - L + 4]); };
  const double f = 1.0 / (2.0 * a * n1 * n2);
  // an imaginary part below 2^-62 of kappa's scale is zero to working precision
  const bool imag = kind < 2 ? d.cplx : fmax(fmax(fabs(R11.im), fabs(R12.im)), fabs(R22.im)) > 0x1p-62 * fabs(c);
  double *mat = T + MT_MAT;
  for (int r = 0; r < 4; ++r) {
    T[MT_P1D + r] = p1(rows_d[r]); T[MT_P2D + r] = p2(rows_d[r]);
    T[MT_P1G + r] = p1(rows_g[r]); T[MT_P2G + r] = p2(rows_g[r]);
  }
  for (int k = 0; k < 6; ++k) {   // inputs: dense rows, moments
    const double f1 = k < 4 ? T[MT_P1D + k] : k == 4 ? 1.0 : 0.0, f2 = k < 4 ? T[MT_P2D + k] : k == 5 ? 1.0 : 0.0;
    const double A = fma(R11.re, f1, R12.re * f2), B = fma(R12.re, f1, R22.re * f2);
    double E1 = 0.0, E2 = 0.0;    // a dense row through kappa, on the middle rows
    if (k < 4) {
      const int j = rows_d[k];
      const double up = k < 2 ? 1.0 : -1.0;   // dense rows 0, 1 lie below the middle rows
      if (kind < 2) { E1 = -up * f * f2; E2 = up * f * f1; }
      else if (k < 2) E1 = el[j - J0] * sgn(j - J0);
      else E2 = el[J1 - j] * sgn(j - J0);
    }
    mat[k] = A + E1;
    mat[6 + k] = B + E2;
    for (int r = 0; r < 4; ++r) {
      const int n = rows_g[r];
      double w;                   // the input's field at gamma row n through kappa
      if (k < 4) w = kap(abs(n - rows_d[k]));
      else {
        const double up = r < 2 ? 1.0 : -1.0;   // gamma rows 0, 1 lie below the middle rows
        if (kind < 2) w = k == 4 ? -up * f * T[MT_P2G + r] : up * f * T[MT_P1G + r];
        else if (k == 4) w = r < 2 ? el[n - J0] * sgn(n - J0) : 0.0;
        else w = r < 2 ? 0.0 : el[J1 - n] * sgn(n - J0);
      }
      mat[6 * (2 + r) + k] = fma(T[MT_P1G + r], A, fma(T[MT_P2G + r], B, w));
    }
  }
  T[MT_R + 0] = R11.re; T[MT_R + 1] = R11.im; T[MT_R + 2] = R12.re; T[MT_R + 3] = R12.im;
  T[MT_R + 4] = R22.re; T[MT_R + 5] = R22.im;
  T[MT_IMAG] = imag ? 1.0 : 0.0;
  T[MT_FAR] = kind == 2 && lo2[0] < 0x1p-90 ? 1.0 : 0.0;   // 2^-90 of the other end is zero to working precision
  T[MT_RFI] = 1.0 / rf;
  T[MT_T1] = T1;
  T[MT_T2] = T2;
  T[MT_RF] = rf;
  T[MT_F] = f;
  T[MT_TH] = th; T[MT_KIND] = kind; T[MT_SG] = sg; T[MT_N1] = n1; T[MT_N2] = n2;
}

// phi_1, phi_2 at a subdomain's receiver row
__global__ void __launch_bounds__(32) k_sep_rec(const SubDesc *subs, int s0, unsigned char *sep) {
  const SubDesc &d = subs[s0 + blockIdx.y];
  const int q = blockIdx.x * 32 + threadIdx.x + 1;
  if (!d.tc_cols || d.nrec < 0 || q > d.Nq) return;
  const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
  double *P = reinterpret_cast<double *>(sep + d.sep_rp) + q - 1;
  const int kind = (int)T[MT_KIND], J0 = d.nlo - 1, J1 = d.nhi + 1;
  const double th = T[MT_TH], sr = T[MT_SG] < 0.0 && ((d.nrec - J0) & 1) ? -1.0 : 1.0, x = d.nrec - 0.5 * (J0 + J1);
  P[0] = sr * (kind == 2 ? exp(-th * (d.nrec - J0)) : T[MT_N1] * sep_c(kind, th, x));
  P[d.Nq] = sr * (kind == 2 ? exp(-th * (J1 - d.nrec)) : T[MT_N2] * sep_s(kind, th, x));
}

// phi_1, phi_2 on the rows J0 .. J1, [2][Py + 2][Nq]: a thread takes one mode and 8 rows, the
// first by exp / sincos, the others by multiplying on (a rotation or a decay: 8 roundings).
constexpr int PHI_ROWS = 8;
__global__ void __launch_bounds__(128) k_sep_phi(const SubDesc *subs, int s0, unsigned char *sep) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  const int q = blockIdx.x * 128 + threadIdx.x + 1, rows = d.Py + 2, i0 = blockIdx.y * PHI_ROWS;
  if (d.leader != si || q > d.Nq || i0 >= rows) return;
  const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
  double *P1 = reinterpret_cast<double *>(sep + d.sep_phi) + (q - 1), *P2 = P1 + (long long)rows * d.Nq;
  const double th = T[MT_TH], sg = T[MT_SG];
  const int kind = (int)T[MT_KIND], i1 = min(rows, i0 + PHI_ROWS);
  const double sg0 = (sg < 0.0 && (i0 & 1)) ? -1.0 : 1.0;
  if (kind == 2) {
    const double lam = sg * exp(-th);
    double v = sg0 * exp(-th * i0);
    for (int i = i0; i < i1; ++i) { P1[(long long)i * d.Nq] = v; v *= lam; }
    v = ((sg < 0.0 && ((i1 - 1) & 1)) ? -1.0 : 1.0) * exp(-th * (rows - i1));
    for (int i = i1 - 1; i >= i0; --i) { P2[(long long)i * d.Nq] = v; v *= lam; }
    return;
  }
  const double x = i0 - 0.5 * (rows - 1), n1 = sg0 * T[MT_N1], n2 = sg0 * T[MT_N2];
  // C(x+1) = C(x) C(1) -/+ S(x) s^2, S(x+1) = S(x) C(1) + C(x) (s = sin theta or sinh theta)
  const double c1 = sep_c(kind, th, 1.0), s = kind == 0 ? sin(th) : sinh(th), ss = kind == 0 ? -s * s : s * s;
  double C = sep_c(kind, th, x), S = sep_s(kind, th, x), w = 1.0;
  for (int i = i0; i < i1; ++i) {
    P1[(long long)i * d.Nq] = w * n1 * C;
    P2[(long long)i * d.Nq] = w * n2 * S;
    const double Cn = fma(S, ss, C * c1);
    S = fma(S, c1, C);
    C = Cn;
    w *= sg;
  }
}

// K_sc(d) for every class, output and source column: one block per distance d, sums over the modes.
__global__ void __launch_bounds__(128) k_sep_kd(const SubDesc *subs, int s0, const double *tab, unsigned char *sep) {
  const int si = s0 + blockIdx.y;
  const SubDesc &d = subs[si];
  const int dist = blockIdx.x;
  if (!d.tc_cols || d.leader != si || dist >= d.Py) return;
  const SepGeo g = sep_geo(d);
  const double *S = tab + d.sin_off, *T = reinterpret_cast<const double *>(sep + d.sep_mt);
  const double *P1 = reinterpret_cast<const double *>(sep + d.sep_phi) + (long long)dist * d.Nq;
  const double *P2 = P1 + (long long)(d.Py + 2) * d.Nq;
  const int N2 = 2 * d.Nx;
  double acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = 0.0;
  for (int q = threadIdx.x + 1; q <= d.Nq; q += 128) {
    const double *t = T + (long long)(q - 1) * SEP_MTW;
    const double kq = fma(t[MT_T1], P1[q - 1], t[MT_T2] * P2[q - 1]);
    double so[4], sc[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      so[s] = s < g.nS ? S[(int)(((long long)q * sep_out_col(d, s)) % N2)] * kq : 0.0;
      sc[s] = s < g.nS ? S[(int)(((long long)q * sep_src_col(d, s)) % N2)] : 0.0;
    }
    if (d.xsym) {
      // acc[(class, s, c)]; 128 is even, so a thread's modes all have its own parity
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
  // fixed-order sums: over the lanes of one parity (x-centred) or all lanes, then the 4 warps
  __shared__ double sh[4][2][16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    for (int off = 16; off >= 2; off >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], off);
    if (lane < 2) sh[warp][lane][i] = acc[i];
  }
  __syncthreads();
  const int ns = g.ncls * g.nS * g.nS;
  if ((int)threadIdx.x < ns) {
    double v = 0.0;
    if (d.xsym) {   // class 0: odd q, which lanes of even index hold
      const int e = threadIdx.x >> 2, i = threadIdx.x & 3;
      for (int w = 0; w < 4; ++w) v += sh[w][e][i];
    } else {
      for (int w = 0; w < 4; ++w) v += sh[w][0][threadIdx.x] + sh[w][1][threadIdx.x];
    }
    reinterpret_cast<double *>(sep + d.sep_kd)[(long long)threadIdx.x * d.Py + dist] = v * (2.0 / d.Nx);
  }
}

// set bit kb of a tile's mask if the warp (32 outputs, one half of the 16 values of K) has a nonzero digit
__device__ __forceinline__ void mark_group(unsigned *mask, int kb, const long long *V) {
  long long any = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) any |= V[j];
  if (__any_sync(0xffffffffu, any != 0) && (threadIdx.x & 31) == 0) atomicOr(mask + (kb >> 5), 1u << (kb & 31));
}
// The Toeplitz blocks of K (32 outputs x 16 sources, by the offset of the two groups) on the scale of
// the largest |K_sc| of the output column: 64 threads (32 outputs x 2 K halves) per block.
__global__ void __launch_bounds__(256) k_sep_tb(const SubDesc *subs, int s0, unsigned char *sep) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  if (!d.tc_cols || d.leader != si) return;
  const SepGeo g = sep_geo(d);
  const int es = blockIdx.y / g.nS, c = blockIdx.y % g.nS;   // (class, output), source
  const int blk0 = blockIdx.x * 4;
  if (es >= g.ncls * g.nS || blk0 >= g.ND) return;
  const double *K = reinterpret_cast<const double *>(sep + d.sep_kd) + (long long)es * g.nS * d.Py;
  __shared__ int emax;
  if (threadIdx.x == 0) emax = 0;
  __syncthreads();
  int m = 0;
  for (int i = threadIdx.x; i < g.nS * d.Py; i += 256) m = max(m, (__double2hiint(K[i]) >> 20) & 0x7ff);
  for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(&emax, m);
  __syncthreads();
  const int e = min(max(emax - 1022, -900), 900);   // |K| <= 2^e
  if (threadIdx.x == 0 && blockIdx.x == 0 && c == 0) reinterpret_cast<int *>(sep + d.sep_kde)[es] = e;
  const int blk = blk0 + (threadIdx.x >> 6), o = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1;
  if (blk >= g.ND) return;
  const double sc = pow2i(54 - e);
  const double *Kc = K + (long long)c * d.Py;
  long long V[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    // row distance of output i = 32 ti + o (row nlo+1+i) and source 16 kj + k (row nlo+2+j)
    const int dist = abs(16 * (blk - (g.nkj - 1)) + o - (8 * half + j) - 1);
    V[j] = dist < d.Py ? __double2ll_rn(Kc[dist] * sc) : 0;
  }
  unsigned char *B = sep + d.sep_tb + (((long long)es * g.nS + c) * g.ND + blk) * SEP_BBLK;
  store_digits(B + (o >> 3) * 256 + half * 128 + (o & 7) * 16, 1024, V);
}

// The moment tables, B of stage 1 beyond K: output (b, q), K index (c, j): sin(pi q m_c/Nx) phi_b(j),
// and (b = 2, with a receiver row) sin(pi q m_c/Nx) kappa_q(|rec - j|) scaled to below 1: subdomains that
// share their leader's tables may each have a row of their own, so b = 2 is made and kept per subdomain.
__global__ void __launch_bounds__(256) k_sep_mb(const SubDesc *subs, int s0, const double *tab, unsigned char *sep) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  if (!d.tc_cols) return;
  const SepGeo g = sep_geo(d);
  const int nto = g.nb * g.nqp / 32;
  const int e = blockIdx.y / nto, to = blockIdx.y % nto;
  const int kb = blockIdx.x * 4 + (threadIdx.x >> 6);
  if (e >= g.ncls || kb >= g.nk1) return;
  const int o = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1;
  const int b = to * 32 / g.nqp;
  if (b < 2 && d.leader != si) return;
  const int qi = to * 32 % g.nqp + o, q = sep_mode(d, e, qi);
  const int c = kb / g.nkj, j0 = (kb % g.nkj) * 16 + 8 * half;
  long long V[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) V[j] = 0;
  if (q <= d.Nq) {
    const double sc = tab[d.sin_off + (int)(((long long)q * sep_src_col(d, c)) % (2 * d.Nx))];
    const double *P = reinterpret_cast<const double *>(sep + d.sep_phi) + (q - 1);
    const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
    const long long p2 = (long long)(d.Py + 2) * d.Nq;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j0 + j >= g.Pj) continue;
      const int row = 3 + j0 + j;                      // grid row nlo + 2 + j, counted from J0 = nlo - 1
      double v;
      if (b < 2) v = P[b * p2 + (long long)row * d.Nq];
      else {
        const int dist = abs(d.nrec - (d.nlo - 1) - row);
        v = fma(T[MT_T1], P[(long long)dist * d.Nq], T[MT_T2] * P[p2 + (long long)dist * d.Nq]) * T[MT_RF];
      }
      V[j] = fix54(v * sc);
    }
  }
  const SepMoment m = sep_moment(d, g, e, to);
  mark_group(reinterpret_cast<unsigned *>(sep + m.mask), kb, V);
  unsigned char *B = sep + m.blocks + (long long)kb * SEP_BBLK;
  store_digits(B + (o >> 3) * 256 + half * 128 + (o & 7) * 16, 1024, V);
}

// The synthesis table, B of stage 3: output (s, i), K index (b, q): (2/Nx) sin(pi q m_s/Nx) phi_b(i).
__global__ void __launch_bounds__(256) k_sep_b3(const SubDesc *subs, int s0, const double *tab, unsigned char *sep) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  if (!d.tc_cols || d.leader != si) return;
  const SepGeo g = sep_geo(d);
  const int e = blockIdx.y / g.nt3, to = blockIdx.y % g.nt3;
  const int kb = blockIdx.x * 4 + (threadIdx.x >> 6);
  if (e >= g.ncls || kb >= g.nk3) return;
  const int o = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1;
  const int s = to / g.nti, i = (to % g.nti) * 32 + o;
  const int b = kb * 16 / g.nqp, q0 = kb * 16 % g.nqp + 8 * half;
  const int m = sep_out_col(d, s), N2 = 2 * d.Nx;
  const double *S = tab + d.sin_off, sc = inv_scale(d);
  const double *P = reinterpret_cast<const double *>(sep + d.sep_phi) + ((long long)b * (d.Py + 2) + 2 + i) * d.Nq;
  long long V[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int q = sep_mode(d, e, q0 + j);
    V[j] = (i < g.Pi && q <= d.Nq) ? fix54(P[q - 1] * (sc * S[(int)(((long long)q * m) % N2)])) : 0;
  }
  mark_group(reinterpret_cast<unsigned *>(sep + d.sep_z3) + (e * g.nt3 + to) * SEP_MASK, kb, V);
  unsigned char *B = sep + d.sep_b3 + (((long long)e * g.nt3 + to) * g.nk3 + kb) * SEP_BBLK;
  store_digits(B + (o >> 3) * 256 + half * 128 + (o & 7) * 16, 1024, V);
}

// The sine tables of the full rows' transforms (which: 0 FWD, 1 INV, 2, 3 the same over every folded column
// for full-grid solves). FWD: output q of parity e, K index m' - mf; INV: output m' - mg, K index q of
// parity e; both sin(pi q m'/Nx) over the folded columns m' <= Nx/2, the inverse times 2/Nx.
__global__ void __launch_bounds__(256) k_sep_sines(const SubDesc *subs, int s0, const double *tab, unsigned char *sep, int which) {
  const int si = s0 + blockIdx.z;
  const SubDesc &d = subs[si];
  if (!d.tc_cols || d.leader != si) return;
  const SepGeo g = sep_geo(d);
  const bool inv = which & 1, full = which & 2;
  const double sc = inv ? inv_scale(d) : 1.0;
  const int nto = inv ? (full ? g.ntx : g.ntg) : g.nqh / 32, nk = inv ? g.nqh / 16 : full ? g.nkx : g.nkf;
  const int m0 = full ? 1 : inv ? g.mg : g.mf;
  const int e = blockIdx.y / nto, to = blockIdx.y % nto;
  const int kb = blockIdx.x * 4 + (threadIdx.x >> 6);
  if (e >= 2 || kb >= nk) return;
  const int o = threadIdx.x & 31, half = (threadIdx.x >> 5) & 1;
  const double *S = tab + d.sin_off;
  long long V[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int ko = to * 32 + o, kk = kb * 16 + 8 * half + j;
    const int q = sep_parity_mode(e, inv ? kk : ko), m = m0 + (inv ? ko : kk);
    V[j] = q <= d.Nq && 2 * m <= d.Nx ? fix54(sc * S[(int)(((long long)q * m) % (2 * d.Nx))]) : 0;
  }
  unsigned char *B = sep + (full ? (inv ? d.sep_xi : d.sep_xf) : inv ? d.sep_bi : d.sep_bf) + (((long long)e * nto + to) * nk + kb) * SEP_BBLK;
  store_digits(B + (o >> 3) * 256 + half * 128 + (o & 7) * 16, 1024, V);
}

// ---------------------------------------------------------------- operand A
// Cut the rows of A into digits in the MMA's operand layout, per 128 rows and 16 values of K 7 x 4 KiB:
//   MID: ring residuals of the middle rows, FWD: of the dense rows (folded columns),
//   SYN: A_b of the modes, INV: the modes' field at the rows to transform back.
// A block takes 8 rows of one class (one core-matrix row group): their largest exponents first, then
// the digits; the values are read twice, the second time from L1/L2. Groups of 16 values of K whose
// digits are all zero in 128 rows (the imaginary parts of evanescent modes, the ring away from a
// column's side) are left out of the contraction by their bit in the tile's mask; so are those of the
// moment and synthesis tables, where phi has decayed below 2^-55 (nine tenths of them at 1025^2).
template <bool CIN, int JOB>
__device__ __forceinline__ void sep_cut_body(const Item &it, const SubDesc &d, double *ws, int local) {
  const SepGeo g = sep_geo(d);
  const SepWs w = sep_ws(d, it.ncols);
  const int R = sep_rows(d, JOB, it.ncols, it.col0, CIN);
  const int e = local / (R / 8), row = (local % (R / 8)) * 8 + (threadIdx.x & 7), kl = threadIdx.x >> 3;
  const int cp = sep_pad128(it.ncols), nk = sep_nk(g, JOB);
  const long long nc = it.ncols;
  // the row's column and part, and its values
  constexpr bool IN = JOB == J_MID || JOB == J_FWD;
  const int parts = IN ? (CIN ? 2 : 1) : (d.cplx || CIN ? 2 : 1);
  int col = row % cp, part = (row / cp) % parts;
  const int rr = row / (cp * parts);
  bool live = col < it.ncols;
  if (!CIN) {   // basis columns: the rows are ordered by side
    if (JOB == J_MID) { col = row + sep_first34(d, it.col0, it.ncols); part = 0; live = col < it.ncols; }
    col = live ? sep_col_of(d, it.col0, it.ncols, col) : 0;
  }
  const double *src = JOB == J_SYN ? ws + it.a_off + w.aeff + (long long)e * 2 * g.nqp * R + row
                      : JOB == J_INV ? ws + it.y_off : ws + it.r_off;
  // basis columns: what k_ring leaves unwritten is zero (side: 0..3)
  const int side = CIN || !live ? 0 : col_side(d, it.col0 + col) - 1;
  auto ring = [&](long long slot) { return CIN ? src[2 * (slot * nc + col) + part] : src[slot * nc + col]; };
  auto value = [&](int k) -> double {
    if (!live) return 0.0;
    if (JOB == J_MID) {
      const int c = k / (16 * g.nkj), j = k - c * 16 * g.nkj;
      if (j >= g.Pj) return 0.0;
      if (!CIN && !d.xsym && (c < 2) != (side == 2)) return 0.0;
      return ring(d.xsym ? 8LL * d.Ph + 4 * j + 2 * c + e : 2LL * d.Px + 4 * j + c);
    }
    if (JOB == J_FWD) {
      if (k >= g.Kf) return 0.0;
      if (!CIN && side < 2 && (rr < 2) != (side == 0)) return 0.0;
      if (!CIN && side >= 2 && d.xsym && k > 1) return 0.0;
      if (d.xsym) return ring((long long)rr * 2 * d.Ph + 2 * k + e);
      const long long rb = rr < 2 ? (long long)rr * d.Px : (long long)rr * d.Px + 4 * (d.Py - 4);
      const int m = g.mf + k, m2 = d.Nx - m;
      const int lo = !CIN && side == 3 ? d.mhi - 1 : d.mlo, hi = !CIN && side == 2 ? d.mlo + 1 : d.mhi;   // the row's support
      const double a = m >= lo && m <= hi ? ring(rb + m - d.mlo) : 0.0;
      const double b = m2 != m && m2 >= lo && m2 <= hi ? ring(rb + m2 - d.mlo) : 0.0;
      return e == 0 ? a + b : a - b;
    }
    if (JOB == J_SYN) return sep_mode(d, e, k % g.nqp) <= d.Nq ? src[(long long)k * R] : 0.0;
    const int q = sep_parity_mode(e, k);
    const long long o = ((long long)(q - 1) * 5 + rr) * nc + col;
    return q <= d.Nq ? (parts == 2 ? src[2 * o + part] : src[o]) : 0.0;
  };
  __shared__ int emax[8];
  __shared__ unsigned smask[SEP_MASK];
  if (threadIdx.x < 8) { emax[threadIdx.x] = 0; smask[threadIdx.x] = 0; }
  __syncthreads();
  // the first 256 values of K stay in registers between the two passes
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
  const int E = max(emax[threadIdx.x & 7], 1);
  if (kl == 0) reinterpret_cast<int *>(ws + it.a_off + w.ex[JOB])[e * R + row] = E;
  unsigned char *A = reinterpret_cast<unsigned char *>(ws + it.a_off + w.a[JOB]) +
                     ((long long)(e * (R / 128) + row / 128) * nk) * SEP_ABLK;
  const int r = row & 127, off0 = (r >> 3) * 256 + (r & 7) * 16;
  for (int k8 = kl; k8 < 2 * nk; k8 += 32) {
    long long V[8], any = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      V[j] = fixed_of(k8 == kl ? x[j] : value(8 * k8 + j), E);   // |x| < 2^(E - 1022) -> |V| <= 2^54
      any |= V[j];
    }
    if (any) atomicOr(&smask[k8 >> 6], 1u << ((k8 >> 1) & 31));
    store_digits(A + (long long)(k8 >> 1) * SEP_ABLK + off0 + (k8 & 1) * 128, 4096, V);
  }
  __syncthreads();
  if (threadIdx.x < SEP_MASK && smask[threadIdx.x])
    atomicOr(reinterpret_cast<unsigned *>(ws + it.a_off + w.mask) + sep_mask_of(JOB, it.ncols) +
                 (e * (R / 128) + row / 128) * SEP_MASK + threadIdx.x,
             smask[threadIdx.x]);
}

template <bool CIN, int STAGE>
__global__ void __launch_bounds__(256) k_sep_cut(Batch bt, const SubDesc *subs, double *ws, int fam) {
  pdl_wait();
  Item it; int local;
  locate(bt, blockIdx.x, it, local);
  MDP_CHECK_ITEM(bt, subs, it, local, fam);
  const SubDesc &d = subs[it.sub];
  constexpr int J0 = STAGE == 1 ? J_MID : J_SYN, J1 = STAGE == 1 ? J_FWD : J_INV;
  const int n0 = sep_cut_blocks(d, sep_geo(d), J0, it.ncols, it.col0, CIN);
  if (local < n0) sep_cut_body<CIN, J0>(it, d, ws, local);
  else sep_cut_body<CIN, J1>(it, d, ws, local - n0);
}

// ---------------------------------------------------------------- the contractions
template <int STAGE>
struct SepSrc {
  Batch bt;
  const SubDesc *subs;
  const unsigned char *sep;
  double *ws;
  int user, fam;
  struct Tile : DigitTile {
    Item it;
    int job, e, mt, nt, R;
  };
  __device__ __forceinline__ int total() const { return bt.total_blocks; }
  __device__ __forceinline__ bool tile(int v, Tile &t) const {
    int local;
    locate(bt, v, t.it, local);
    const Item &it = t.it;
    if (MDP_CHECKED && !item_in_bounds(bt, subs, it, local, fam, false)) return false;
    const SubDesc &d = subs[it.sub];
    const SepGeo g = sep_geo(d);
    const SepWs w = sep_ws(d, it.ncols);
    t.job = STAGE == 1 ? J_MID : J_SYN;
    const int n0 = sep_tiles(d, g, t.job, it.ncols, it.col0, user);
    if (local >= n0) { ++t.job; local -= n0; }
    t.R = sep_rows(d, t.job, it.ncols, it.col0, user);
    const int nk = sep_nk(g, t.job), nt = sep_nt(g, t.job), per = (t.R / 128) * nt;
    t.e = local / per;
    t.mt = (local % per) / nt;
    t.nt = local % nt;
    const int tr = t.e * (t.R / 128) + t.mt;   // tile row
    t.A = reinterpret_cast<const unsigned char *>(ws + it.a_off + w.a[t.job]) + (long long)tr * nk * SEP_ABLK;
    t.ex = reinterpret_cast<const int *>(ws + it.a_off + w.ex[t.job]) + tr * 128;
    const unsigned *ma = reinterpret_cast<const unsigned *>(ws + it.a_off + w.mask) + sep_mask_of(t.job, it.ncols) + tr * SEP_MASK;
    const unsigned *mb = nullptr;
    t.eb = t.nkj = t.ND = t.ti = 0;
    if (t.job == J_SYN) {
      t.B = sep + d.sep_b3 + ((long long)t.e * g.nt3 + t.nt) * nk * SEP_BBLK;
      mb = reinterpret_cast<const unsigned *>(sep + d.sep_z3) + (t.e * g.nt3 + t.nt) * SEP_MASK;
      t.eb = inv_exp(d);
    } else if (t.job == J_INV) {
      t.B = sep + d.sep_bi + ((long long)t.e * g.ntg + t.nt) * nk * SEP_BBLK;
      t.eb = inv_exp(d);
    } else if (t.job == J_FWD) {
      t.B = sep + d.sep_bf + ((long long)t.e * (g.nqh / 32) + t.nt) * nk * SEP_BBLK;
    } else if (t.nt < g.nt3) {   // K
      const int es = t.e * g.nS + t.nt / g.nti;
      t.B = sep + d.sep_tb + (long long)es * g.nS * g.ND * SEP_BBLK;
      t.nkj = g.nkj; t.ND = g.ND; t.ti = t.nt % g.nti;
      t.eb = reinterpret_cast<const int *>(sep + d.sep_kde)[es];
    } else {                     // moments
      const SepMoment m = sep_moment(d, g, t.e, t.nt - g.nt3);
      t.B = sep + m.blocks;
      mb = reinterpret_cast<const unsigned *>(sep + m.mask);
    }
    t.masks(ma, mb);
    return !MDP_CHECKED || t.in_bounds(ws, bt.ws_n, sep, bt.sep_n, sep, bt.sep_n, nk, bt.status);
  }
  __device__ __forceinline__ const double *out() const { return ws; }
  __device__ __forceinline__ long long out_n() const { return bt.ws_n; }
  __device__ __forceinline__ void dest(const Tile &t, int r, int o, double *&dst, long long &step, int &cnt) const {
    const Item &it = t.it;
    const SubDesc &d = subs[it.sub];
    const SepGeo g = sep_geo(d);
    const SepWs w = sep_ws(d, it.ncols);
    const int row = t.mt * 128 + r, o0 = t.nt * 32 + o;
    const bool direct = t.nkj > 0;
    step = t.R;
    if (t.job == J_SYN || direct) {
      const int i0 = (t.nt % g.nti) * 32 + o;
      cnt = g.Pi - i0;
      dst = ws + it.a_off + (direct ? w.u1 : w.u3) + ((long long)(t.e * g.nS + t.nt / g.nti) * g.Pi + i0) * t.R + row;
    } else if (t.job == J_MID) {
      cnt = 8;
      dst = ws + it.a_off + w.mom + ((long long)t.e * 3 * g.nqp + o0 - 32 * g.nt3) * t.R + row;
    } else if (t.job == J_INV) {
      cnt = g.Ng - o0;
      dst = ws + it.a_off + w.ui + ((long long)t.e * g.Ng + o0) * t.R + row;
    } else {                   // the dense rows' transforms: modes q = 2 (o0 + k) + 1 + e
      const int cp = sep_pad128(it.ncols), parts = user ? 2 : 1;
      int col = row % cp;
      cnt = col < it.ncols && 2 * o0 + 1 + t.e <= d.Nq ? (d.Nq - (1 + t.e) - 2 * o0) / 2 + 1 : 0;
      if (!user && cnt > 0) col = sep_col_of(d, it.col0, it.ncols, col);
      step = 2LL * it.ncols * parts;
      dst = ws + it.gr_off + (((long long)(row / (cp * parts)) * d.Nq + 2 * o0 + t.e) * it.ncols + col) * parts + (row / cp) % parts;
    }
  }
};

template <int STAGE>
__global__ void __launch_bounds__(SG_THREADS, 1)
    k_sep_gemm(Batch bt, const SubDesc *subs, const unsigned char *sep, double *ws, int user, int fam, int *status) {
  pdl_wait();
  const SepSrc<STAGE> src{bt, subs, sep, ws, user, fam};
  digit_gemm(src, status);
}

// ---------------------------------------------------------------- stage 2
// Per (mode, column): the coefficients A_1, A_2 of the homogeneous part on the middle rows and the field
// at the 4 gamma rows (+ the receiver row) from the 4 dense rows' transforms and the moments: a 6 x 6
// real matrix per mode (36 FMAs a part, 18 where the ends are far apart for the mode), and where R has an
// imaginary part 20 more. CD: complex results (Sommerfeld AP or complex data). FP64-bound: 27 us at
// 4 x 257^2, 1024 columns.
template <bool CD, bool CIN>
__device__ __forceinline__ void sep_modes_body(const Item &it, const SubDesc &d, const SepGeo &g, const SepWs &w,
                                               const unsigned char *sep, double *ws, int b, int row, int row1, int q) {
  const double *T = reinterpret_cast<const double *>(sep + d.sep_mt) + (long long)(q - 1) * SEP_MTW;
  const int e = d.xsym ? ((q & 1) ? 0 : 1) : 0, qi = d.xsym ? (q - 1) >> 1 : q - 1;
  const int cp = sep_pad128(it.ncols), R1 = sep_rows(d, J_MID, it.ncols, it.col0, CIN), R3 = (CD ? 2 : 1) * cp;
  const long long nc = it.ncols;
  const double *gr = ws + it.gr_off;
  const double *mom = ws + it.a_off + w.mom + ((long long)e * 3 * g.nqp + qi) * R1 + row1;
  constexpr int P = CIN ? 2 : 1;
  double in[P][6], out[2][6];   // [part][input], [part][output]
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const long long o = ((long long)r * d.Nq + (q - 1)) * nc + b;
    if (CIN) { const cplx v = ld2(gr + 2 * o); in[0][r] = v.re; in[P - 1][r] = v.im; }
    else in[0][r] = gr[o];
  }
#pragma unroll
  for (int p = 0; p < P; ++p) {        // row1 < 0: no source on the middle rows
    in[p][4] = row1 >= 0 ? mom[p * cp] : 0.0;
    in[p][5] = row1 >= 0 ? mom[(long long)g.nqp * R1 + p * cp] : 0.0;
  }
  if (T[MT_FAR] != 0.0) {   // the two ends do not see each other: two 3 x 3 blocks
#pragma unroll
    for (int o = 0; o < 6; ++o) {
      const int end = o < 2 ? o : (o - 2) >> 1, k0 = 2 * end;   // outputs A_1, A_2, gamma rows 0..3
#pragma unroll
      for (int p = 0; p < P; ++p)
        out[p][o] = fma(T[MT_MAT + 6 * o + k0], in[p][k0],
                        fma(T[MT_MAT + 6 * o + k0 + 1], in[p][k0 + 1], T[MT_MAT + 6 * o + 4 + end] * in[p][4 + end]));
    }
  } else {
#pragma unroll
    for (int o = 0; o < 6; ++o)
#pragma unroll
      for (int p = 0; p < P; ++p) {
        double v = T[MT_MAT + 6 * o] * in[p][0];
#pragma unroll
        for (int k = 1; k < 6; ++k) v = fma(T[MT_MAT + 6 * o + k], in[p][k], v);
        out[p][o] = v;
      }
  }
  if (CD && !CIN)
#pragma unroll
    for (int o = 0; o < 6; ++o) out[1][o] = 0.0;
  if (CD && T[MT_IMAG] != 0.0) {       // i Im R times the moments of all rows
#pragma unroll
    for (int p = 0; p < P; ++p) {
      double m1 = in[p][4], m2 = in[p][5];
#pragma unroll
      for (int r = 0; r < 4; ++r) { m1 = fma(T[MT_P1D + r], in[p][r], m1); m2 = fma(T[MT_P2D + r], in[p][r], m2); }
      double A = fma(T[MT_R + 1], m1, T[MT_R + 3] * m2), B = fma(T[MT_R + 3], m1, T[MT_R + 5] * m2);
      if (p == 1) { A = -A; B = -B; }
      out[1 - p][0] += A;
      out[1 - p][1] += B;
#pragma unroll
      for (int r = 0; r < 4; ++r) out[1 - p][2 + r] = fma(T[MT_P1G + r], A, fma(T[MT_P2G + r], B, out[1 - p][2 + r]));
    }
  }
  double *ae = ws + it.a_off + w.aeff + ((long long)e * 2 * g.nqp + qi) * R3 + row;
  ae[0] = out[0][0];
  ae[(long long)g.nqp * R3] = out[0][1];
  if (CD) { ae[cp] = out[1][0]; ae[(long long)g.nqp * R3 + cp] = out[1][1]; }
  double *y = ws + it.y_off;
  auto ystore = [&](int slot, double re, double im) {
    const long long o = ((long long)(q - 1) * 5 + slot) * nc + b;
    if (CD) st2(y + 2 * o, cmk(re, im)); else y[o] = re;
  };
#pragma unroll
  for (int r = 0; r < 4; ++r) ystore(r, out[0][2 + r], CD ? out[1][2 + r] : 0.0);
}
// The field at the subdomain's receiver row, from the coefficients that the thread has stored and the third moment: in a
// pass of its own, so that calls without receivers keep the modes' matrix to 62 and 70 registers, 8 and 7 blocks to
// an SM (72 and 94 with the row's pointers beside it: 4 x 257^2 209.5 -> 208.9 us, complex data 257.8 -> 255.7).
template <bool CD, bool CIN>
__device__ __forceinline__ void sep_rec_body(const Item &it, const SubDesc &d, const SepGeo &g, const SepWs &w,
                                             const unsigned char *sep, double *ws, int b, int row, int row1, int q) {
  const double f = reinterpret_cast<const double *>(sep + d.sep_mt)[(long long)(q - 1) * SEP_MTW + MT_RFI];
  const double *phi = reinterpret_cast<const double *>(sep + d.sep_rp) + q - 1;
  const double p1 = phi[0], p2 = phi[d.Nq];
  const int e = d.xsym ? ((q & 1) ? 0 : 1) : 0, qi = d.xsym ? (q - 1) >> 1 : q - 1;
  const int cp = sep_pad128(it.ncols), R1 = sep_rows(d, J_MID, it.ncols, it.col0, CIN), R3 = (CD ? 2 : 1) * cp;
  const double *m3 = ws + it.a_off + w.mom + ((long long)(3 * e + 2) * g.nqp + qi) * R1 + row1;
  const double *ae = ws + it.a_off + w.aeff + ((long long)e * 2 * g.nqp + qi) * R3 + row, *be = ae + (long long)g.nqp * R3;
  const double re = fma(p1, ae[0], fma(p2, be[0], row1 >= 0 ? f * m3[0] : 0.0));
  const long long o = ((long long)(q - 1) * 5 + 4) * it.ncols + b;
  double *y = ws + it.y_off;
  if (CD) st2(y + 2 * o, cmk(re, fma(p1, ae[cp], fma(p2, be[cp], CIN && row1 >= 0 ? f * m3[cp] : 0.0))));
  else y[o] = re;
}

template <bool CIN>
__global__ void __launch_bounds__(128, CIN ? 7 : 8) k_sep_modes(Batch bt, const SubDesc *subs, const unsigned char *sep, double *ws) {
  pdl_wait();
  Item it; int local;
  locate(bt, blockIdx.x, it, local);
  MDP_CHECK_ITEM(bt, subs, it, local, F_SMODE);
  const SubDesc &d = subs[it.sub];
  const int cb = (it.ncols + 31) >> 5;
  const int per = sep_modes_per_block(d, it.ncols);
  const int b = (local % cb) * 32 + threadIdx.x, q0 = (local / cb) * per + threadIdx.y + 1;
  if (b >= it.ncols) return;
  const SepGeo g = sep_geo(d);
  const SepWs w = sep_ws(d, it.ncols);
  const int row = CIN ? b : sep_row_of(d, it.col0, it.ncols, b);
  const int row1 = CIN ? b : row - sep_first34(d, it.col0, it.ncols);
  for (int q = q0; q < q0 + per - (int)threadIdx.y && q <= d.Nq; q += 4) {
    if (d.cplx || CIN) sep_modes_body<true, CIN>(it, d, g, w, sep, ws, b, row, row1, q);
    else sep_modes_body<false, CIN>(it, d, g, w, sep, ws, b, row, row1, q);
  }
  if (d.nrec < 0) return;
  for (int q = q0; q < q0 + per - (int)threadIdx.y && q <= d.Nq; q += 4) {
    if (d.cplx || CIN) sep_rec_body<true, CIN>(it, d, g, w, sep, ws, b, row, row1, q);
    else sep_rec_body<false, CIN>(it, d, g, w, sep, ws, b, row, row1, q);
  }
}

// ---------------------------------------------------------------- output columns
// u at the 4 gamma columns of a middle row from the two stages' sums; Q = -u, P = xi - u.
template <bool CD, bool CIN>
__device__ __forceinline__ void sep_out_body(const Item &it, const SubDesc &d, const double *tab, const double *ws,
                                             const double2 *xi_user, double2 *out, int kind, int b, int i) {
  const SepGeo g = sep_geo(d);
  const SepWs w = sep_ws(d, it.ncols);
  const int cp = sep_pad128(it.ncols), R1 = sep_rows(d, J_MID, it.ncols, it.col0, CIN), R3 = (CD ? 2 : 1) * cp;
  const int row = CIN ? b : sep_row_of(d, it.col0, it.ncols, b);
  const int row1 = CIN ? b : row - sep_first34(d, it.col0, it.ncols);
  cplx v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {   // (class, output) or output
    const long long t = (long long)k * g.Pi + i;
    const double *p3 = ws + it.a_off + w.u3 + t * R3 + row, *p1 = ws + it.a_off + w.u1 + t * R1 + row1;
    v[k] = cmk(p3[0], CD ? p3[cp] : 0.0);
    if (row1 >= 0) {
      v[k].re += p1[0];
      if (CIN) v[k].im += p1[cp];
    }
  }
  cplx u[4];
  if (d.xsym) { u[0] = cadd(v[0], v[2]); u[1] = cadd(v[1], v[3]); u[2] = csub(v[1], v[3]); u[3] = csub(v[0], v[2]); }
  else { u[0] = v[0]; u[1] = v[1]; u[2] = v[2]; u[3] = v[3]; }
  const int g0 = 2 * (d.Px + 2) + 4 * i;
  if (MDP_CHECKED && g0 + 3 >= d.G) { flag_bounds(d.dstatus); return; }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    cplx r = cmk(-u[s].re, CD ? -u[s].im : 0.0);
    if (kind == MDP_OUT_P) r = cadd(r, density<CIN>(d, it, ws, tab, xi_user, b, g0 + s));
    out[it.io_off + (long long)b * d.G + g0 + s] = make_double2(r.re, r.im);
  }
}

// The full gamma rows and the receiver row: u(m) = U_0(m) + U_1(m), u(Nx - m) = U_0(m) - U_1(m) from the
// two parities' sums over the folded columns. A block takes one row, 32 folded columns m and 32 basis columns, turned through shared memory so that the loads run along the columns and
// the stores along m.
template <bool CD, bool CIN>
__device__ __forceinline__ void sep_rows_out_body(const Item &it, const SubDesc &d, const double *tab, const double *ws,
                                                  const double2 *xi_user, double2 *out, double2 *out_rec, int kind, int b0,
                                                  int slot, int mt, double2 (*sh)[32][33], long long rec_n) {
  const SepGeo g = sep_geo(d);
  const int cp = sep_pad128(it.ncols), parts = CD ? 2 : 1, R = sep_rows(d, J_INV, it.ncols, it.col0, CIN);
  const double *ui = ws + it.a_off + sep_ws(d, it.ncols).ui;
  const int b = b0 + threadIdx.x;
  const int row = slot * parts * cp + (CIN || b >= it.ncols ? b : sep_row_of(d, it.col0, it.ncols, b));
  for (int k = threadIdx.y; k < 32; k += 8) {
    const int m = mt * 32 + k;
    cplx u0 = cmk(0.0, 0.0), u1 = u0;
    if (m < g.Ng && b < it.ncols) {
      const double *p0 = ui + (long long)m * R + row, *p1 = p0 + (long long)g.Ng * R;
      u0 = cmk(p0[0], CD ? p0[cp] : 0.0);
      u1 = cmk(p1[0], CD ? p1[cp] : 0.0);
    }
    const cplx s = cadd(u0, u1), t = csub(u0, u1);
    sh[0][k][threadIdx.x] = make_double2(s.re, s.im);
    sh[1][k][threadIdx.x] = make_double2(t.re, t.im);
  }
  __syncthreads();
  const int W = d.Px + 2, m1 = g.mg + mt * 32 + (int)threadIdx.x;
  if (2 * m1 > d.Nx) return;
  const int gbase = slot <= 1 ? slot * W : 2 * W + 4 * (d.Py - 2) + (slot - 2) * W;
  for (int k = threadIdx.y; k < 32 && b0 + k < it.ncols; k += 8)
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int m = side == 0 ? m1 : d.Nx - m1;
      if (side == 1 && m == m1) continue;
      const double2 v = sh[side][threadIdx.x][k];
      if (slot == 4) {
        if (out_rec && m >= d.mlo + 1 && m <= d.mhi - 1) {
          const long long o = d.rec_off + (long long)(it.col0 + b0 + k) * (d.Px - 2) + (m - d.mlo - 1);
          if (MDP_CHECKED && (o < 0 || o >= rec_n)) { flag_bounds(d.dstatus); continue; }
          out_rec[o] = make_double2(-v.x, -v.y);
        }
        continue;
      }
      if (m < d.mlo - 1 || m > d.mhi + 1) continue;
      const int gi = gbase + m - (d.mlo - 1);
      if (MDP_CHECKED && (gi < 0 || gi >= d.G)) { flag_bounds(d.dstatus); continue; }
      cplx r = cmk(-v.x, CD ? -v.y : 0.0);
      if (kind == MDP_OUT_P) r = cadd(r, density<CIN>(d, it, ws, tab, xi_user, b0 + k, gi));
      out[it.io_off + (long long)(b0 + k) * d.G + gi] = make_double2(r.re, r.im);
    }
}

template <bool CIN>
__global__ void __launch_bounds__(256) k_sep_out(Batch bt, const SubDesc *subs, const double *tab, const double *ws,
                                                 const double2 *xi_user, double2 *out, double2 *out_rec, int kind) {
  pdl_wait();
  __shared__ double2 sh[2][32][33];
  Item it; int local;
  locate(bt, blockIdx.x, it, local);
  MDP_CHECK_ITEM(bt, subs, it, local, F_SOUT);
  const SubDesc &d = subs[it.sub];
  const int cb = (it.ncols + 31) >> 5, nmid = cb * ((d.Py - 2 + 7) / 8);
  if (local >= nmid) {
    local -= nmid;
    const int t = local / cb, ntg = sep_geo(d).ntg;
    const int b0 = (local % cb) * 32;
    if (d.cplx || CIN) sep_rows_out_body<true, CIN>(it, d, tab, ws, xi_user, out, out_rec, kind, b0, t / ntg, t % ntg, sh, bt.rec_n);
    else sep_rows_out_body<false, CIN>(it, d, tab, ws, xi_user, out, out_rec, kind, b0, t / ntg, t % ntg, sh, bt.rec_n);
    return;
  }
  const int b = (local % cb) * 32 + threadIdx.x, i = (local / cb) * 8 + threadIdx.y;
  if (b >= it.ncols || i >= d.Py - 2) return;
  if (d.cplx || CIN) sep_out_body<true, CIN>(it, d, tab, ws, xi_user, out, kind, b, i);
  else sep_out_body<false, CIN>(it, d, tab, ws, xi_user, out, kind, b, i);
}

}  // namespace

// ---------------------------------------------------------------- launchers
cudaError_t set_sep_kernel_attributes() {
  cudaError_t e = cudaFuncSetAttribute(k_sep_gemm<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sep_gemm<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, SG_SMEM);
  return e;
}

cudaError_t launch_sep_tables(const mdp_plan *p, const SubDesc *ds, const double *tab, unsigned char *sep, bool entries,
                              cudaStream_t st) {
  int mq = 0, mrow = 0, mdist = 0, mtb = 0, mes = 0, mmb = 0, mmk = 0, m3 = 0, m3k = 0, mrec = 0;
  for (size_t i = 0; i < p->subs.size(); ++i) {
    const SubDesc &d = p->subs[i].d;
    if (d.tc_cols && d.nrec >= 0) mrec = std::max(mrec, (d.Nq + 31) / 32);
    if (d.tc_cols && (d.leader == (int)i || d.nrec >= 0)) {   // a duplicate has its receiver row's moments
      const SepGeo g = sep_geo(d);
      mmb = std::max(mmb, g.ncls * g.nb * g.nqp / 32);
      mmk = std::max(mmk, (g.nk1 + 3) / 4);
    }
    if (d.leader != (int)i) continue;
    mq = std::max(mq, (d.Nq + 127) / 128);
    mrow = std::max(mrow, (d.Py + 2 + PHI_ROWS - 1) / PHI_ROWS);
    if (!d.tc_cols) continue;
    const SepGeo g = sep_geo(d);
    mdist = std::max(mdist, d.Py);
    mtb = std::max(mtb, (g.ND + 3) / 4);
    mes = std::max(mes, g.ncls * g.nS * g.nS);
    m3 = std::max(m3, g.ncls * g.nt3);
    m3k = std::max(m3k, (g.nk3 + 3) / 4);
  }
  if (p->sep_masks > 0) {
    const cudaError_t e = cudaMemsetAsync(sep, 0, (size_t)p->sep_masks, st);
    if (e != cudaSuccess) return e;
  }
  const int ns = (int)p->subs.size();
  for (int s0 = 0; s0 < ns; s0 += 65535) {   // subdomains per launch: a grid's y / z limit
    const unsigned n = (unsigned)std::min(65535, ns - s0);
    k_sep_mode_tab<<<dim3(4 * mq, n), 32, 0, st>>>(ds, s0, sep, entries);
    k_full_modes<<<dim3(4 * mq, n), 32, 0, st>>>(ds, s0, sep);
    if (mrec > 0) k_sep_rec<<<dim3(mrec, n), 32, 0, st>>>(ds, s0, sep);
    k_sep_phi<<<dim3(mq, mrow, n), 128, 0, st>>>(ds, s0, sep);
    if (mdist == 0) continue;   // no subdomain on the tensor cores
    k_sep_kd<<<dim3(mdist, n), 128, 0, st>>>(ds, s0, tab, sep);
    k_sep_tb<<<dim3(mtb, mes, n), 256, 0, st>>>(ds, s0, sep);
    k_sep_mb<<<dim3(mmk, mmb, n), 256, 0, st>>>(ds, s0, tab, sep);
    k_sep_b3<<<dim3(m3k, m3, n), 256, 0, st>>>(ds, s0, tab, sep);
  }
  return cudaGetLastError();
}

cudaError_t launch_sep_sines(const mdp_plan *p, const SubDesc *ds, const double *tab, unsigned char *sep, cudaStream_t st) {
  int k[4] = {0, 0, 0, 0}, t[4] = {0, 0, 0, 0};
  for (size_t i = 0; i < p->subs.size(); ++i) {
    const SubDesc &d = p->subs[i].d;
    if (!d.tc_cols || d.leader != (int)i) continue;
    const SepGeo g = sep_geo(d);
    const int nk[4] = {g.nkf, g.nqh / 16, g.nkx, g.nqh / 16}, nt[4] = {g.nqh / 32, g.ntg, g.nqh / 32, g.ntx};
    for (int w = 0; w < 4; ++w) {
      k[w] = std::max(k[w], (nk[w] + 3) / 4);
      t[w] = std::max(t[w], 2 * nt[w]);
    }
  }
  const int ns = (int)p->subs.size();
  if (t[0] == 0) return cudaSuccess;
  for (int s0 = 0; s0 < ns; s0 += 65535)
    for (int w = 0; w < 4; ++w)
      k_sep_sines<<<dim3(k[w], t[w], (unsigned)std::min(65535, ns - s0)), 256, 0, st>>>(ds, s0, tab, sep, w);
  return cudaGetLastError();
}

cudaError_t launch_sep_cut1(const Batch &b, const SubDesc *subs, double *ws, bool user, int fam, cudaStream_t st) {
  if (user) pdl(k_sep_cut<true, 1>, b.total_blocks, dim3(256), 0, st, b, subs, ws, fam);
  else pdl(k_sep_cut<false, 1>, b.total_blocks, dim3(256), 0, st, b, subs, ws, fam);
  return cudaGetLastError();
}

cudaError_t launch_sep_project(mdp_plan *p, const Batch *fb, int out_kind, const double2 *xi_user, double2 *out,
                               double2 *out_rec, cudaStream_t st) {
  const bool user = xi_user != nullptr;
  if (fb[F_SMODE].total_blocks == 0) return cudaSuccess;
  const SubDesc *ds = subs_of(p, out_rec != nullptr);
  double *ws = p->d_ws;
  const int f1c = user ? F_C1U : F_C1B, f1 = user ? F_G1U : F_G1B, f3c = user ? F_C3U : F_C3B, f3 = user ? F_G3U : F_TCOLS;
  auto grid = [&](int f) { return dim3((unsigned)fb[f].total_blocks); };
  auto gemm_grid = [&](int f) { return dim3((unsigned)std::min(fb[f].total_blocks, p->n_sm)); };
#define SEP_LAUNCH(as, ...)   \
  do {                        \
    prof_begin(p, as, st);    \
    __VA_ARGS__;              \
    prof_end(p, as, st);      \
  } while (0)
  if (user) SEP_LAUNCH(F_C1B, pdl(k_sep_cut<true, 1>, grid(f1c), dim3(256), 0, st, fb[f1c], ds, ws, f1c));
  else SEP_LAUNCH(F_C1B, pdl(k_sep_cut<false, 1>, grid(f1c), dim3(256), 0, st, fb[f1c], ds, ws, f1c));
  SEP_LAUNCH(F_G1B, pdl(k_sep_gemm<1>, dim3(gemm_grid(f1)), dim3(SG_THREADS), SG_SMEM, st, fb[f1], ds, p->d_sep, ws, user, f1, p->d_status));
  if (user) SEP_LAUNCH(F_SMODE, pdl(k_sep_modes<true>, grid(F_SMODE), dim3(32, 4), 0, st, fb[F_SMODE], ds, p->d_sep, ws));
  else SEP_LAUNCH(F_SMODE, pdl(k_sep_modes<false>, grid(F_SMODE), dim3(32, 4), 0, st, fb[F_SMODE], ds, p->d_sep, ws));
  if (user) SEP_LAUNCH(F_C3B, pdl(k_sep_cut<true, 3>, grid(f3c), dim3(256), 0, st, fb[f3c], ds, ws, f3c));
  else SEP_LAUNCH(F_C3B, pdl(k_sep_cut<false, 3>, grid(f3c), dim3(256), 0, st, fb[f3c], ds, ws, f3c));
  SEP_LAUNCH(F_TCOLS, pdl(k_sep_gemm<3>, dim3(gemm_grid(f3)), dim3(SG_THREADS), SG_SMEM, st, fb[f3], ds, p->d_sep, ws, user, f3, p->d_status));
  if (user) SEP_LAUNCH(F_SOUT, pdl(k_sep_out<true>, grid(F_SOUT), dim3(32, 8), 0, st, fb[F_SOUT], ds, p->d_tables, ws, xi_user, out, out_rec, out_kind));
  else SEP_LAUNCH(F_SOUT, pdl(k_sep_out<false>, grid(F_SOUT), dim3(32, 8), 0, st, fb[F_SOUT], ds, p->d_tables, ws, xi_user, out, out_rec, out_kind));
#undef SEP_LAUNCH
  return cudaGetLastError();
}

}  // namespace mdp
