// Contractions on the fp16 tensor cores, to FP64 accuracy relative to the largest values of a row and of a table,
// by error-free splitting (Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012): the operands' cut
// into digits, and the kernel body that streams digit blocks, issues the MMAs and adds their exact sums
// (kernels_sep.cu, kernels_full.cu).
//
// Every operand value becomes an integer |V| <= 2^54 on one scale (a row of A: its largest value; B: a
// bound of its table) and V 7 balanced base-256 digits, exact in fp16: a value is kept to 2^-55 of the scale, so one
// 2^-30 of the row's largest has 24 bits of its own. Of the 49 digit products those of weight t + u <= 7 are kept
// (34): the five of weight 8, the largest left out, are together below 2^-59 of the product of the two
// scales for a value of K, under the operands' own rounding. Products of equal weight share one FP32 accumulator: at most 7 x 128 x 2^14
// < 2^24 between two read-backs of 128 values of K, so every sum is an exact integer.
#pragma once
#include "tc_common.cuh"

#include <climits>

namespace mdp {

__device__ __forceinline__ double pow2i(int k) {
  return k < -1022 ? 0.0 : __longlong_as_double((long long)(min(k, 1023) + 1023) << 52);
}
// the 7 digits of 8 consecutive-K values |x| 2^(54 - e) at 16 bytes each, `stride` bytes apart
__device__ __forceinline__ void store_digits(unsigned char *dst, long long stride, const long long *V) {
  unsigned hi[8], lo[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const unsigned long long w = (unsigned long long)V[j] + 0x0080808080808080ull;
    hi[j] = (unsigned)(w >> 32);
    lo[j] = (unsigned)w;
  }
#define MDP_SEP_DIGIT(T)                                                        \
  *reinterpret_cast<uint4 *>(dst + (T) * stride) =                              \
      make_uint4(digit_pair<6 - (T)>(hi[0], lo[0], hi[1], lo[1]),               \
                 digit_pair<6 - (T)>(hi[2], lo[2], hi[3], lo[3]),               \
                 digit_pair<6 - (T)>(hi[4], lo[4], hi[5], lo[5]),               \
                 digit_pair<6 - (T)>(hi[6], lo[6], hi[7], lo[7]));
  MDP_SEP_DIGIT(0) MDP_SEP_DIGIT(1) MDP_SEP_DIGIT(2) MDP_SEP_DIGIT(3) MDP_SEP_DIGIT(4) MDP_SEP_DIGIT(5) MDP_SEP_DIGIT(6)
#undef MDP_SEP_DIGIT
}
// 2/Nx = inv_scale 2^inv_exp, inv_scale in (1/2, 1]: the normalisation of the inverse transforms, in their tables
__device__ __forceinline__ int inv_exp(const SubDesc &d) { return __clz(d.Nx) - 30; }
__device__ __forceinline__ double inv_scale(const SubDesc &d) { return (double)(1 << (31 - __clz(d.Nx))) / d.Nx; }
// table value |x| <= 1 on the fixed scale 2^54
__device__ __forceinline__ long long fix54(double x) { return __double2ll_rn(x * 0x1p54); }

// round(x 2^(1076 - E)) for |x| < 2^(E - 1022), 1 <= E (nothing for E = 2047: Inf or NaN in the row), by
// integer operations: the significand (53 bits) lies e - 1075 up (e = 1 for subnormal numbers), so it moves up one
// bit for e = E and down E - e - 1 bits otherwise, rounded half up
__device__ __forceinline__ long long fixed_of(double x, int E) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned long long m = (e ? 1ULL << 52 : 0ULL) | (b & 0xfffffffffffffLL);
  const int s = min(E - (e ? e : 1), 63);          // 0: up one bit
  const long long v = (long long)(((m << 2) >> s) + 1) >> 1;
  return E < 2047 ? (b < 0 ? -v : v) : 0;
}

// A tile of 128 rows x 32 outputs: the digit blocks of its rows and outputs, consecutive in groups of 16
// values of K, except that with nkj the B block of group kb is a Toeplitz one (nkj groups per source
// column, ND blocks per column, output group ti); the mask of groups with nonzero digits; the exponents of the rows and of the table.
struct DigitTile {
  const unsigned char *A, *B, *B2 = nullptr;
  int k2 = 1 << 30;          // groups of K from k2 on have their B blocks at B2
  int nkj, ND, ti;
  unsigned m[SEP_MASK];      // groups of K with nonzero digits in the tile's rows and in its outputs
  const int *ex;
  int eb;
  // mb, mb2 may be null
  __device__ __forceinline__ void masks(const unsigned *ma, const unsigned *mb, const unsigned *mb2 = nullptr) {
    const uint4 *p = reinterpret_cast<const uint4 *>(ma);
    uint4 a = p[0], b = p[1];
    if (mb) {
      const uint4 *r = reinterpret_cast<const uint4 *>(mb);
      uint4 c = r[0], e = r[1];
      if (mb2) {             // of the groups from k2 on
        const uint4 *s = reinterpret_cast<const uint4 *>(mb2);
        const uint4 c2 = s[0], e2 = s[1];
        c.x |= c2.x; c.y |= c2.y; c.z |= c2.z; c.w |= c2.w;
        e.x |= e2.x; e.y |= e2.y; e.z |= e2.z; e.w |= e2.w;
      }
      a.x &= c.x; a.y &= c.y; a.z &= c.z; a.w &= c.w;
      b.x &= e.x; b.y &= e.y; b.z &= e.z; b.w &= e.w;
    }
    m[0] = a.x; m[1] = a.y; m[2] = a.z; m[3] = a.w; m[4] = b.x; m[5] = b.y; m[6] = b.z; m[7] = b.w;
  }
  // bounds-checked build: nk groups of K, their blocks and the exponents inside the workspace and the tables
  __device__ __noinline__ bool in_bounds(const double *ws, long long ws_n, const unsigned char *t0, long long n0,
                                         const unsigned char *t1, long long n1, int nk, int *status) const {
    auto in = [](const void *p, long long n, const void *lo, long long size) {
      const long long o = (const char *)p - (const char *)lo;
      return o >= 0 && n >= 0 && o + n <= size;
    };
    auto tab = [&](const unsigned char *p, long long n) { return in(p, n, t0, n0) || in(p, n, t1, n1); };
    const long long blocks = nkj ? (long long)((nk + nkj - 1) / nkj) * ND : min(nk, k2);
    bool ok = nk <= 32 * SEP_MASK && in(A, (long long)nk * SEP_ABLK, ws, 8 * ws_n) && in(ex, 128 * sizeof(int), ws, 8 * ws_n) &&
              tab(B, blocks * SEP_BBLK) && (nk <= k2 || tab(B2, (long long)(nk - k2) * SEP_BBLK));
#pragma unroll
    for (int wd = 0; wd < SEP_MASK; ++wd) {
      const int left = nk - 32 * wd;   // groups of this word
      ok = ok && !(left <= 0 ? m[wd] : left < 32 ? m[wd] >> left : 0u);
    }
    if (!ok) flag_bounds(status);
    return ok;
  }
  __device__ __forceinline__ int groups() const {
    int n = 0;
#pragma unroll
    for (int wd = 0; wd < SEP_MASK; ++wd) n += __popc(m[wd]);
    return n;
  }
};

// Persistent CTAs, one per SM: warp 17 streams the digit blocks of A (28 KiB) and B (7 KiB) of 16
// values of K into 5 shared-memory stages with bulk copies, one thread of warp 16 issues the MMAs,
// and after every 128 values of K hands one of two accumulator sets (8 weights x 32 outputs, FP32)
// to the 16 other warps (a quarter of the rows and 8 outputs each; 8 warps left their latencies in the
// open), which add them up as integers and at the end of a tile scale them into FP64. A tile is 128 rows x 32 outputs. One MMA (M = 128, N = 256, K = 16) per A digit t: its B
// operand starts t digits before B's first one, in 7 KiB of zeros, so that digit u meets the
// accumulator of weight t + u and every MMA of a set has the same accumulator and shape (MMAs into
// overlapping accumulators of other shapes have no defined order). The zeros are 22 of 56 digit
// pairs. What bounds it: the tensor pipe, 7 x 128 cycles per 16 values of K; the operands' way from
// L2 takes 35 KiB in that time, 39 bytes per cycle and SM.
constexpr int SG_STAGES = 5, SG_EPI = 16, SG_THREADS = 32 * (SG_EPI + 2), SG_CHUNK = 8;   // K16 steps per accumulator set
constexpr int SG_STAGE_BYTES = SEP_ABLK + SEP_BBLK;
// shared memory: the A stages, then zeros and B stages in turn, 7 KiB each, and closing zeros
constexpr int SG_B0 = SG_STAGES * SEP_ABLK;
constexpr int SG_SMEM = SG_B0 + (2 * SG_STAGES + 1) * SEP_BBLK + 1024;

// 8 consecutive FP32 columns of this warp's 32 TMEM lanes, twice (two weights in flight)
__device__ __forceinline__ void tmem_ld8x2(unsigned ta, unsigned tb, float *v) {
  unsigned r[16];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(ta)
               : "memory");
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(tb)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void bulk_load(unsigned dst, const void *src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// (hi 2^32 + lo) 2^ex, rounded to nearest, by integer operations: the FP64 pipe takes 64 cycles per warp
// instruction, and three conversions per output had taken as long as the tile's MMAs.
__device__ __forceinline__ double sum_to_double(long long hi, long long lo, int ex) {
  long long h = hi + (lo >> 32);          // |h| < 2^51
  unsigned l = (unsigned)lo;
  const bool neg = h < 0;
  if (neg) { h = ~h + (l == 0 ? 1 : 0); l = 0u - l; }
  const int lz = h ? __clzll(h) : 64 + __clz((int)l);
  // the leading 64 bits of the 96, then 53 of them rounded
  unsigned long long top = lz <= 32 ? ((unsigned long long)l << lz) >> 32 : (unsigned long long)l << ((lz - 32) & 63);
  if (lz < 64) top |= (unsigned long long)h << lz;
  const int e = 1023 + 95 - lz + ex;      // biased exponent
  unsigned long long v = ((unsigned long long)(e - 1) << 52) + (top >> 11) + ((top >> 10) & 1);
  if (e < 1) v = e < -52 ? 0 : ((top >> (11 - e)) + 1) >> 1;   // subnormal: 1 - e bits less
  if (lz == 96) v = 0;
  if (e > 2046) v = 0x7ff0000000000000ULL;
  if (ex == INT_MAX) v = 0x7ff8000000000000ULL;
  return __longlong_as_double((long long)(v | ((unsigned long long)neg << 63)));
}

// Src: total() tiles, tile(v, t) fills tile v (false: skipped by every warp), dest(t, row, o, ...) says where
// the 8 outputs from o on of a row go, inside out_n() doubles from out(). One CTA of SG_THREADS threads per SM with SG_SMEM bytes.
template <class Src>
__device__ __forceinline__ void digit_gemm(const Src &src, int *status) {
  extern __shared__ unsigned char sg_raw[];
  const int total = src.total();
  __shared__ __align__(8) unsigned long long full_bar[SG_STAGES], empty_bar[SG_STAGES], tfull_bar[2], tempty_bar[2], drain_bar;
  __shared__ unsigned tmem_slot;
  __shared__ volatile int abort_sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int s = 0; s < SG_STAGES; ++s) { mbar_init(smem_u32(&full_bar[s]), 1); mbar_init(smem_u32(&empty_bar[s]), 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(smem_u32(&tfull_bar[s]), 1); mbar_init(smem_u32(&tempty_bar[s]), 32 * SG_EPI); }
    mbar_init(smem_u32(&drain_bar), 1);
    abort_sh = 0;
  }
  if (warp == SG_EPI) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const unsigned sbase = (smem_u32(sg_raw) + 1023u) & ~1023u;
  {
    unsigned char *z = sg_raw + (sbase - smem_u32(sg_raw)) + SG_B0;
    for (int i = tid; i < (SG_STAGES + 1) * (SEP_BBLK / 16); i += SG_THREADS)
      *reinterpret_cast<uint4 *>(z + (i / (SEP_BBLK / 16)) * 2 * SEP_BBLK + (i % (SEP_BBLK / 16)) * 16) = make_uint4(0, 0, 0, 0);
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = tmem_slot;

  if (warp == SG_EPI + 1) {
    // ---------------------------------------------------------------- operand loads
    if (lane == 0) {
      unsigned gs = 0;
      for (int v = blockIdx.x; v < total && !abort_sh; v += gridDim.x) {
        typename Src::Tile t;
        if (!src.tile(v, t)) continue;   // every warp skips it
        bool ok = true;
#pragma unroll
        for (int wd = 0; wd < SEP_MASK; ++wd)
          for (unsigned bits = ok ? t.m[wd] : 0u; bits; bits &= bits - 1, ++gs) {
            const int kb = 32 * wd + __ffs(bits) - 1;
            const unsigned st = gs % SG_STAGES;
            if (gs >= SG_STAGES && !mbar_wait(smem_u32(&empty_bar[st]), (gs / SG_STAGES - 1) & 1u, &abort_sh)) { ok = false; break; }
            const unsigned bar = smem_u32(&full_bar[st]);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(SG_STAGE_BYTES) : "memory");
            bulk_load(sbase + st * SEP_ABLK, t.A + (long long)kb * SEP_ABLK, SEP_ABLK, bar);
            const long long bo = t.nkj ? (long long)(kb / t.nkj) * t.ND + 2 * t.ti - kb % t.nkj + t.nkj - 1 : kb;
            bulk_load(sbase + SG_B0 + (2 * st + 1) * SEP_BBLK, kb < t.k2 ? t.B + bo * SEP_BBLK : t.B2 + (kb - t.k2) * SEP_BBLK,
                      SEP_BBLK, bar);
          }
        if (!ok) break;
      }
      // leave only when every copy issued has landed (each wait bounded)
      for (unsigned s = gs >= SG_STAGES ? gs - SG_STAGES : 0; s < gs; ++s) {
        const long long t0 = clock64();
        while (!mbar_try(smem_u32(&full_bar[s % SG_STAGES]), (s / SG_STAGES) & 1u))
          if (clock64() - t0 > TC_WAIT_CYCLES) { abort_sh = 1; break; }
      }
    }
    __syncwarp();
  } else if (warp == SG_EPI) {
    // ---------------------------------------------------------------- MMAs
    if (lane == 0) {
      unsigned gs = 0, cc = 0;   // stages and accumulator sets used
      for (int v = blockIdx.x; v < total && !abort_sh; v += gridDim.x) {
        typename Src::Tile t;
        if (!src.tile(v, t)) continue;
        const int n = t.groups();   // steps
        bool ok = true;
        for (int s = 0; s < n && ok; ++cc) {
          const unsigned buf = cc & 1u, D = tmem + 256u * buf;
          if (cc >= 2 && !mbar_wait(smem_u32(&tempty_bar[buf]), ((cc >> 1) - 1) & 1u, &abort_sh)) { ok = false; break; }
          tc_fence_after();
          const int send = min(n, s + SG_CHUNK);
          for (bool first = true; s < send; ++s, ++gs, first = false) {
            const unsigned st = gs % SG_STAGES;
            if (!mbar_wait(smem_u32(&full_bar[st]), (gs / SG_STAGES) & 1u, &abort_sh)) { ok = false; break; }
            tc_fence_after();
            const unsigned a0 = sbase + st * SEP_ABLK, b0 = sbase + SG_B0 + (2 * st + 1) * SEP_BBLK;
#pragma unroll
            for (int dg = 0; dg < 7; ++dg)
              tc_mma(D, smem_desc(a0 + 4096 * dg, 128, 256), smem_desc(b0 - 1024 * dg, 128, 256), f16_idesc(256),
                     first && dg == 0 ? 0u : 1u);
            tc_commit(smem_u32(&empty_bar[st]));
          }
          if (ok) tc_commit(smem_u32(&tfull_bar[buf]));
        }
        if (!ok) break;
      }
      if (abort_sh) {   // no MMA in flight when the tensor memory is freed (bounded)
        tc_commit(smem_u32(&drain_bar));
        const long long t0 = clock64();
        while (!mbar_try(smem_u32(&drain_bar), 0u) && clock64() - t0 < TC_WAIT_CYCLES) {}
      }
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- sums and results
    const int quarter = warp & 3, part = warp >> 2;   // TMEM lanes of the warp, its outputs
    unsigned cc = 0;
    for (int v = blockIdx.x; v < total && !abort_sh; v += gridDim.x) {
      typename Src::Tile t;
      if (!src.tile(v, t)) continue;
      const int n = t.groups();
      // weights 0..3 and 4..7 of 8 outputs, as sums of I_w 2^(8 (3 - w)), I_w 2^(8 (7 - w))
      long long hi[8], lo[8];
#pragma unroll
      for (int o = 0; o < 8; ++o) hi[o] = lo[o] = 0;
      bool ok = true;
      for (int s = 0; s < n; s += SG_CHUNK, ++cc) {
        const unsigned buf = cc & 1u;
        if (!mbar_wait(smem_u32(&tfull_bar[buf]), (cc >> 1) & 1u, &abort_sh)) { ok = false; break; }
        tc_fence_after();
        const unsigned acc = tmem + ((unsigned)(32 * quarter) << 16) + 256u * buf + 8u * part;
#pragma unroll
        for (int wt = 0; wt < 4; ++wt) {
          float dv[16];
          tmem_ld8x2(acc + 32u * wt, acc + 32u * (wt + 4), dv);
#pragma unroll
          for (int o = 0; o < 8; ++o) {
            hi[o] += (long long)__float2int_rn(dv[o]) * (1LL << (8 * (3 - wt)));
            lo[o] += (long long)__float2int_rn(dv[8 + o]) * (1LL << (8 * (3 - wt)));
          }
        }
        tc_fence_before();
        mbar_arrive(smem_u32(&tempty_bar[buf]));
      }
      if (!ok) break;
      // value = (hi 2^32 + lo) 2^40 2^(E - 1022 - 54) 2^(eb - 54)
      const int row = 32 * quarter + lane;
      const int E = t.ex[row];
      const int ex = E < 2047 ? E - 1090 + t.eb : INT_MAX;   // Inf or NaN in the row: NaN
      double *dst;
      int cnt;                   // outputs of this thread (of 8), `step` doubles apart
      long long step;
      src.dest(t, row, 8 * part, dst, step, cnt);
      if (MDP_CHECKED && cnt > 0) {
        const long long o = dst - src.out();
        if (o < 0 || o + (min(cnt, 8) - 1) * step >= src.out_n()) { flag_bounds(status); cnt = 0; }
      }
      if (step == 1 && cnt >= 8) {
#pragma unroll
        for (int o = 0; o < 8; o += 2)
          *reinterpret_cast<double2 *>(dst + o) =
              make_double2(sum_to_double(hi[o], lo[o], ex), sum_to_double(hi[o + 1], lo[o + 1], ex));
      } else {
#pragma unroll
        for (int o = 0; o < 8; ++o)
          if (o < cnt) dst[o * step] = sum_to_double(hi[o], lo[o], ex);
      }
    }
  }
  if (abort_sh && tid == 0) atomicCAS(status, 0, (int)MDP_ERR_TIMEOUT);   // the first error sticks
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == SG_EPI)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

}  // namespace mdp
