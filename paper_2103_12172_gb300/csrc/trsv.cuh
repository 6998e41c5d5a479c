// Triangular solves with the R of the Householder QR by one CTA (qr.cu, couple.cu).
#pragma once
#include "kernels_common.cuh"

namespace mdp {

__device__ __forceinline__ double2 c2mul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// ---- triangular solve --------------------------------------------------------------------------
// R x = b (back substitution) or R^H x = b (forward substitution), R upper triangular,
// column-major with leading dimension ldr (only i <= j is read). One CTA, the vector in
// shared memory; blocks of 32 rows: the block's 32 x 32 triangle is staged in
// shared memory by all threads (coalesced), warp 0 forms the 32 reciprocals of its diagonal at
// once and solves the block with shuffles, then all threads subtract the block's contribution
// from the rows still to solve, one row per thread (loads issued 8 at a time, no reductions).
constexpr int kTrThreads = 256;

__device__ __forceinline__ double2 crcp(double2 d) {   // 1 / d
  const double den = fma(d.x, d.x, d.y * d.y);
  return make_double2(d.x / den, -d.y / den);
}

// xs: the n values in shared memory, written by the CTA's threads before a barrier-free call; replaced by
// the solution (visible to every thread on return). Only rows <= columns of R are read.
// T: shared memory for the diagonal block, T[col][row] = R(i0 + row, i0 + col); the caller's, as a kernel that
// solves with R and R^H would hold two where the block is static here, past what a launch gets without opting in.
typedef double2 TrBlock[32][33];
template <bool CT>
__device__ __forceinline__ void trsv_body(int n, const double2 *__restrict__ R, long long ldr, double2 *xs, TrBlock &T) {
  const int nblk = (n + 31) / 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t = 0; t < nblk; ++t) {
    const int bi = CT ? t : nblk - 1 - t;
    const int i0 = bi * 32, w = min(32, n - i0);
    for (int e = threadIdx.x; e < 32 * 32; e += kTrThreads) {
      const int cc = e >> 5, rr = e & 31;   // rr fastest: a column of the block, coalesced
      T[cc][rr] = cc < w && rr <= cc ? R[(long long)(i0 + cc) * ldr + i0 + rr] : make_double2(0.0, 0.0);
    }
    __syncthreads();   // T, and the previous block's updates of xs
    if (warp == 0) {
      const int r = i0 + lane;
      double2 v = lane < w ? xs[r] : make_double2(0.0, 0.0);
      const double2 dinv = lane < w ? crcp(T[lane][lane]) : make_double2(0.0, 0.0);
      if (!CT) {
        for (int j = w - 1; j >= 0; --j) {
          if (lane == j) v = c2mul(v, dinv);
          const double2 xj = make_double2(__shfl_sync(0xffffffffu, v.x, j), __shfl_sync(0xffffffffu, v.y, j));
          if (lane < j) {
            const double2 a = T[j][lane];   // R(r, i0 + j)
            v.x -= fma(a.x, xj.x, -a.y * xj.y);
            v.y -= fma(a.x, xj.y, a.y * xj.x);
          }
        }
      } else {
        const double2 dinvc = make_double2(dinv.x, -dinv.y);   // 1 / conj(d)
        for (int j = 0; j < w; ++j) {
          if (lane == j) v = c2mul(v, dinvc);
          const double2 xj = make_double2(__shfl_sync(0xffffffffu, v.x, j), __shfl_sync(0xffffffffu, v.y, j));
          if (lane > j && lane < w) {
            const double2 a = T[lane][j];   // R(i0 + j, r); L(r, i0 + j) = conj of it
            v.x -= fma(a.x, xj.x, a.y * xj.y);
            v.y -= fma(a.x, xj.y, -a.y * xj.x);
          }
        }
      }
      if (lane < w) xs[r] = v;
    }
    __syncthreads();
    if (!CT) {   // rows above the block: thread per row, R(r, i0 + j) coalesced over r
      for (int r = threadIdx.x; r < i0; r += kTrThreads) {
        double sx = 0.0, sy = 0.0;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
          if (j < w) {
            const double2 a = R[(long long)(i0 + j) * ldr + r];
            const double2 x = xs[i0 + j];
            sx = fma(a.x, x.x, fma(-a.y, x.y, sx));
            sy = fma(a.x, x.y, fma(a.y, x.x, sy));
          }
        }
        xs[r].x -= sx;
        xs[r].y -= sy;
      }
    } else {     // rows below the block: thread per row, conj(R(i0 + j, r)) from column r of R
      for (int r = i0 + w + threadIdx.x; r < n; r += kTrThreads) {
        const double2 *rc = R + (long long)r * ldr + i0;
        double sx = 0.0, sy = 0.0;
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
          if (j < w) {
            const double2 a = rc[j];
            const double2 x = xs[i0 + j];
            sx = fma(a.x, x.x, fma(a.y, x.y, sx));
            sy = fma(a.x, x.y, fma(-a.y, x.x, sy));
          }
        }
        xs[r].x -= sx;
        xs[r].y -= sy;
      }
    }
  }
  __syncthreads();
}

}  // namespace mdp
