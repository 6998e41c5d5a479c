// Internal structures shared by the host plan and the CUDA kernels.
#pragma once
#include <cstdint>
#include <vector>
#include <string>
#include <algorithm>
#include <utility>
#include <cstdlib>
#include <cmath>
#include <cstring>
#include <cuda_runtime.h>
#include "mdp.h"

// The bounds-checked build (libmdp_checked.so) is compiled with MDP_CHECKED=1: every batched
// kernel validates its block's work item and the gamma indices it writes through (first violation
// in the status word as MDP_ERR_BOUNDS, the access skipped), and MDP_FAULT_INJECT is honoured.
#ifndef MDP_CHECKED
#define MDP_CHECKED 0
#endif

namespace mdp {

// Per-subdomain geometry, coefficients and table offsets (POD; copied to the device).
//
// Grid: nodes (m, n), x_m = ax0 + m h, y_n = ay0 + n h. M+ is the node rectangle
// [mlo, mhi] x [nlo, nhi]. gamma is the 2-node ring [mlo-1, mhi+1] x [nlo-1, nhi+1]
// minus [mlo+1, mhi-1] x [nlo+1, nhi-1]; the support of r = L w|M+ ("ring") is
// [mlo, mhi] x [nlo, nhi] minus [mlo+2, mhi-2] x [nlo+2, nhi-2].
// Sine modes q = 1..Nq along x (Nq = Nx - 1, Nx = nx - 1 cells). The tridiagonal
// unknowns along y are rows n = nfirst .. nfirst + Nt - 1 (matrix row i = n - nfirst).
struct SubDesc {
  int nx, ny, Nx, Nq;
  int mlo, mhi, nlo, nhi;
  int Px, Py;       // M+ nodes along x and y
  int G, R;         // |gamma| = 4(Px + Py), |ring| = 4 Px + 4 (Py - 4)
  int nfirst, Nt;   // first y row of the tridiagonal unknowns, and their count
  int i0;           // first stored matrix row of the partial sweeps: (nlo - 1) - nfirst
  int NYf;          // stored rows of the forward (projection) sweep: Nt - i0
  int n_modes, n_cols;
  int cplx;         // 1: complex factors (Sommerfeld AP), 0: real (Dirichlet AP)
  int ap_bc;
  int xsym;         // 1: mlo + mhi == Nx (subdomain centred along x): paired ring layout
  int Ph;           // xsym: pair units per dense ring row, Nx/2 - mlo + 1
  int R2;           // ring residual slots: R, or 8 Ph + 4 (Py - 4) with xsym
  int nrec;         // receiver row (nlo+1 .. nhi-1) or -1; receivers m = mlo+1 .. mhi-1
  int rows_fft;     // inverse transform of the gamma rows by FFT (Nx a power of 2, 2Nx <= 4096)
  int fpb;          // FFTs (columns) per block of the dense-row kernels: max(1, 1024 / (2 Nx))
  int leader;       // index of the subdomain owning this one's tables (itself unless deduplicated)
  int tc_cols;      // 1: the projection, the gradient pass and the full-grid solves run through the separable
                    // Green's function (kernels_sep.cu, kernels_sepadj.cu, kernels_full.cu); 0: per-mode sweeps
  int n_prop;       // modes q = 1 .. n_prop below the cutoff (a matter of scheduling: k_factor_chain)
  double h, k;
  double x0, x1, y0, y1, ax0, ay0;
  double c0, c1, c2;  // 9-point coefficients: centre, edge, corner (Eq. FD_scheme)
  double dc0, dc1;    // their k-derivatives (the corner one is 0)
  long long fact_off;   // doubles: factor rows [Nq][Nt][FW], FW = 8 (complex) or 4 (real)
  long long piv_off;    // bytes: pivot flags [Nq][Nt]
  long long dT_off;     // doubles: dT_q/dk rows [Nq][Nt][6] (sub, diag, super; complex)
  long long sin_off;    // doubles: sin(pi j / Nx), j = 0 .. 2Nx-1, then (2/Nx) sin(pi j/Nx)
  long long geo_off;    // doubles: gamma geometry [G][4] = (owner, s, rho, side length)
  long long seg_off;    // doubles: per mode [Nq][5] = (rlo, rhi, frlo, frhi, itop): real rows of the
                        // factor table, real rows of the forward-sweep table, last swept row
  long long fs_off;     // doubles: projection forward-sweep table [Nq][NYf][FSW] (rows i0..)
  // bytes into the plan's separable tables (kernels_sep.cu), device only; without tc_cols the first three
  long long sep_zm, sep_z3;   // words: masks of the nonzero groups of K of sep_mb's and sep_b3's tiles
  long long sep_ab;     // doubles [Nq][2]: interior entries (off-diagonal, diagonal) of T_q
  long long sep_mt;     // per mode SEP_MTW doubles
  long long sep_phi;    // doubles [2][Py + 2][Nq]: phi_1, phi_2 on the rows nlo-1 .. nhi+1
  long long sep_kd;     // doubles [class][output][source][Py]: K by row distance
  long long sep_kde;    // ints [class][output]: exponent of the largest |K|
  long long sep_tb, sep_mb, sep_b3;   // digit blocks of K (Toeplitz), of the moments, of the synthesis
  long long sep_bf, sep_bi;           // of the dense rows' transform and of the gamma rows' (sines only)
  long long sep_xf, sep_xi;           // of the full-grid transforms
  // bytes into the plan's gradient tables (kernels_sepadj.cu): masks of adj_mb, adj_b3, adj_dmb (words); per mode
  // ADJ_MDW doubles; k-derivatives of phi and K; digit blocks of K with gamma and the ring exchanged, of the
  // moments, of the synthesis, of the full rows' transforms, and of dK/dk and d phi/dk for the residual
  long long adj_zm, adj_z3, adj_zd, adj_md, adj_phid, adj_kdd, adj_kde, adj_tb, adj_mb, adj_b3, adj_bf, adj_bi, adj_dtb,
      adj_dmb;
  long long sep_mx;     // per mode SEP_MXW doubles: the full-grid solve along y (kernels_full.cu)
  // what depends on the receiver row, each subdomain's own (the rest is its leader's): phi_1, phi_2 there
  // (doubles [2][Nq]), the third block of the moments and its masks; in the gradient tables d phi/dk, the
  // third block of the residual's derivative moments, and the third K block of the synthesis
  long long sep_rp, sep_rz, sep_rb, adj_rp, adj_rz, adj_rb, adj_r3z, adj_r3;
  long long out_off;    // complex elements: start of the subdomain's output block
  long long rec_off;    // complex elements: start of the receiver block [n_cols][Px - 2]
  int *dstatus;         // the plan's device status word (bounds-checked build: first error; else unused)
};

// One batch work item: columns [col0, col0 + ncols) of subdomain `sub`, with its
// workspace slices (offsets in doubles from the workspace base).
struct Item {
  int sub, col0, ncols, flags;   // flags: bit0 basis densities, bit1 real data path
  long long xi_off;   // basis densities [G][ncols] (real) / dxi/dk follows for the gradient
  long long r_off;    // ring residual [R][ncols] (real or complex)
  long long gr_off;   // forward sine transform of the 4 dense ring rows [4][Nq][ncols]
  long long y_off;    // mode-space field [Nq][NY][ncols]
  long long a_off;    // adjoint mode-space field [Nq][Nt][ncols] (gradient pass), or in the projection the
                      // operands and sums of the separable solve (SepWs)
  long long s_off;    // gradient source on the ring [R][ncols] (complex)
  long long red_off;  // per-block partial sums of the k-gradient (gradient pass)
  long long io_off;   // complex elements: column col0 of this item in xi / out / cot / grad_xi
};

enum { ITEM_BASIS = 1, ITEM_REAL = 2 };

// Launch-time view of a list of items: a device array plus, for each kernel family,
// per-item prefix sums of blocks. A single item may be passed by value instead.
struct Batch {
  const Item *items;    // device array (nullptr: use `one`)
  const int *prefix;    // device array [n_items + 1] of block prefix sums for this kernel
  const int *order;     // device array [total_blocks]: the item-major block number that launch
                        // block b runs (nullptr: b itself); the sweeps run their longest first
  int n_items;
  int total_blocks;
  Item one;
  // ranges the bounds-checked build validates every block's item against: subdomains, workspace
  // doubles, table doubles, pivot-flag bytes, and complex elements of the output / density /
  // cotangent and receiver arrays of the call; the status word that records the first violation
  int n_subs;
  int grad;             // the items are laid out for the gradient pass
  long long ws_n, tab_n, piv_n, out_n, rec_n;
  long long sep_n, adj_n;   // bytes of the separable and the gradient tables
  int *status;
};

constexpr int FSW = 24;  // doubles per forward-sweep table row

// ---- separable projection (kernels_sep.cu)
constexpr int SEP_MTW = 72;               // doubles per mode of the mode table
constexpr int SEP_MXW = 20;               // doubles per mode of the full-grid solve's table
constexpr int SEP_ABLK = 7 * 128 * 16 * 2;  // bytes of A: 7 digits x 128 rows x 16 values of K, fp16
constexpr int SEP_BBLK = 7 * 32 * 16 * 2;   // bytes of B: 7 digits x 32 outputs x 16 values of K
constexpr int SEP_MASK = 8;               // words of a K mask: at most 256 groups of 16

// The contractions (jobs) of the projection: stage 1 runs MID (ring residuals of the middle rows
// against K and the moments) and FWD (sine transform of the 4 dense ring rows), stage 3 SYN (the
// middle rows' gamma columns from the modes) and INV (inverse sine transform of the 4 gamma rows and
// the receiver row).
enum SepJob { J_MID = 0, J_FWD, J_SYN, J_INV };

// Sizes of a subdomain's contractions.
struct SepGeo {
  int ncls, nS;        // MID, SYN: classes of modes (odd, even) on x-centred subdomains, else 1; output (and
                       // source) columns. FWD, INV: always the two parities
  int nqp;             // modes per class, padded to 32
  int nqh;             // modes per parity, padded to 32 (x-centred: nqp)
  int Pi, Pj;          // output rows nlo+1 .. nhi-1, source rows nlo+2 .. nhi-2
  int nti, nkj;        // groups of 32 outputs, of 16 sources per column
  int nb;              // moments per mode: 2, or 3 with a receiver row
  int mf, Kf, nkf;     // FWD: folded columns m = mf .. Nx/2 of the dense ring rows (m with Nx - m), groups of 16
  int mg, Ng, ntg;     // INV: folded columns m = mg .. Nx/2 of the gamma rows, groups of 32
  int slots;           // INV: rows transformed back: 4 gamma rows (+ the receiver row)
  int nkx, ntx;        // full-grid transforms: folded columns m = 1 .. Nx/2 in groups of 16, of 32
  int nk1, nk3;        // K of MID (source column, row) and SYN (b, mode) in units of 16
  int nt1, nt3;        // MID, SYN: tiles of 32 outputs
  int ND;              // distinct Toeplitz blocks per (output, source) column
};
// modes below the cutoff at the subdomain's k: 4 sin^2(pi q / (2 Nx)) (1/h^2 + k^2/12) < k^2
inline int propagating_modes(const SubDesc &d) {
  const double s = 0.5 * std::sqrt(d.k * d.k / (1.0 / (d.h * d.h) + d.k * d.k / 12.0));
  return s >= 1.0 ? d.Nq : std::min(d.Nq, (int)(2.0 * d.Nx / M_PI * std::asin(s)) + 1);
}
// modes per block (4 warps) of k_sep_modes and k_adj_modes: 16, or 4 where the item has fewer blocks of 16 than a
// GB300 has SMs (a block's modes follow one another: 129^2, 128 columns: k_sep_modes 14.8 -> 6.7 us). The workspace is
// laid out by it before the device is asked, so the number is the part's; another part's runs as well, less well split.
constexpr int GB300_SMS = 152;
inline __host__ __device__ int sep_modes_per_block(const SubDesc &d, int ncols) {
  return ((ncols + 31) / 32) * ((d.Nq + 15) / 16) < GB300_SMS ? 4 : 16;
}
inline __host__ __device__ SepGeo sep_geo(const SubDesc &d) {
  SepGeo g;
  g.ncls = d.xsym ? 2 : 1;
  g.nS = d.xsym ? 2 : 4;
  g.nqh = ((d.Nq + 1) / 2 + 31) / 32 * 32;
  g.nqp = d.xsym ? g.nqh : (d.Nq + 31) / 32 * 32;
  g.Pi = d.Py - 2;
  g.Pj = d.Py - 4;
  g.nti = (g.Pi + 31) / 32;
  g.nkj = (g.Pj + 15) / 16;
  g.nb = d.nrec >= 0 ? 3 : 2;
  g.mf = d.mlo < d.Nx - d.mhi ? d.mlo : d.Nx - d.mhi;
  g.Kf = d.Nx / 2 - g.mf + 1;
  g.nkf = (g.Kf + 15) / 16;
  g.mg = g.mf - 1;
  g.Ng = g.Kf + 1;
  g.ntg = (g.Ng + 31) / 32;
  g.nkx = (d.Nx / 2 + 15) / 16;
  g.ntx = (d.Nx / 2 + 31) / 32;
  g.slots = d.nrec >= 0 ? 5 : 4;
  g.nk1 = g.nS * g.nkj;
  g.nk3 = 2 * g.nqp / 16;
  g.nt3 = g.nS * g.nti;
  g.nt1 = g.nt3 + g.nb * g.nqp / 32;
  g.ND = 2 * g.nti + g.nkj;
  return g;
}
// mode number of entry qi of class e (past Nq: padding), of entry qi of parity e (0: odd modes)
inline __host__ __device__ int sep_mode(const SubDesc &d, int e, int qi) { return d.xsym ? 2 * qi + 1 + e : qi + 1; }
inline __host__ __device__ int sep_parity_mode(int e, int qi) { return 2 * qi + 1 + e; }
// The separable tables of a subdomain: f(offset, bytes, class) for each, in a fixed order; class TAB_MASK: masks, at the
// plan's first bytes, TAB_OWN: a duplicate has its own (else its leader's).
enum { TAB_MASK = 1, TAB_OWN = 2 };
template <class D, class F>
inline __host__ __device__ void sep_tables(D &d, F f) {
  if (d.tc_cols) {
    const SepGeo g = sep_geo(d);
    const long long n = g.nqp / 32, zw = 4LL * SEP_MASK * g.ncls, pairs = (long long)g.ncls * g.nS * g.nS;
    f(d.sep_rz, zw * n, TAB_MASK | TAB_OWN);
    f(d.sep_zm, zw * 2 * n, TAB_MASK);
    f(d.sep_z3, zw * g.nt3, TAB_MASK);
    f(d.sep_rp, 16LL * d.Nq, TAB_OWN);
    f(d.sep_rb, g.ncls * n * g.nk1 * SEP_BBLK, TAB_OWN);
    f(d.sep_kd, 8 * pairs * d.Py, 0);
    f(d.sep_kde, 4LL * g.ncls * g.nS, 0);
    f(d.sep_tb, pairs * g.ND * SEP_BBLK, 0);
    f(d.sep_mb, g.ncls * 2 * n * g.nk1 * SEP_BBLK, 0);
    f(d.sep_b3, (long long)g.ncls * g.nt3 * g.nk3 * SEP_BBLK, 0);
    f(d.sep_bf, 2LL * (g.nqh / 32) * g.nkf * SEP_BBLK, 0);
    f(d.sep_bi, 2LL * g.ntg * (g.nqh / 16) * SEP_BBLK, 0);
    f(d.sep_xf, 2LL * (g.nqh / 32) * g.nkx * SEP_BBLK, 0);
    f(d.sep_xi, 2LL * g.ntx * (g.nqh / 16) * SEP_BBLK, 0);
  }
  f(d.sep_ab, 16LL * d.Nq, 0);
  f(d.sep_mt, 8LL * SEP_MTW * d.Nq, 0);
  f(d.sep_mx, 8LL * SEP_MXW * d.Nq, 0);
  f(d.sep_phi, 16LL * (d.Py + 2) * d.Nq, 0);
}
// bytes into the separable tables of the moments of 32 modes (output group `to` of class e): blocks of all groups
// of K, mask; the first two blocks of nqp modes phi_1, phi_2, the third a receiver row's
struct SepMoment { long long blocks, mask; };
inline __host__ __device__ SepMoment sep_moment(const SubDesc &d, const SepGeo &g, int e, int to) {
  const int n = g.nqp / 32, i = to < 2 * n ? e * 2 * n + to : e * n + to - 2 * n;
  return {(to < 2 * n ? d.sep_mb : d.sep_rb) + (long long)i * g.nk1 * SEP_BBLK,
          (to < 2 * n ? d.sep_zm : d.sep_rz) + 4LL * SEP_MASK * i};
}
// the same into the gradient tables: the k-derivatives of the residual's moments
inline __host__ __device__ SepMoment adj_dmoment(const SubDesc &d, const SepGeo &g, int e, int to) {
  const int n = g.nqp / 32, i = to < 2 * n ? e * 2 * n + to : e * n + to - 2 * n;
  return {(to < 2 * n ? d.adj_dmb : d.adj_rb) + (long long)i * g.nk1 * SEP_BBLK,
          (to < 2 * n ? d.adj_zd : d.adj_rz) + 4LL * SEP_MASK * i};
}
// grid column of output s (gamma) and of source c (ring); x-centred: the left ones, the right ones mirrored
inline __host__ __device__ int sep_out_col(const SubDesc &d, int s) {
  return s == 0 ? d.mlo - 1 : s == 1 ? d.mlo : s == 2 ? d.mhi : d.mhi + 1;
}
inline __host__ __device__ int sep_src_col(const SubDesc &d, int c) {
  return c == 0 ? d.mlo : c == 1 ? d.mlo + 1 : c == 2 ? d.mhi - 1 : d.mhi;
}
inline __host__ __device__ int sep_pad128(int n) { return (n + 127) / 128 * 128; }
// The rows of A take an item's basis columns side by side (Dirichlet, then Neumann columns of side 1,
// of side 2, ...), so that a tile's columns share their zeros; user densities stay in order.
// Columns c0 .. c0 + ncols - 1 that are of side s (0..3) and kind k:
inline __host__ __device__ int sep_seg(const SubDesc &d, int c0, int ncols, int s, int k) {
  const int M = d.n_modes, lo = (4 * k + s) * M, hi = lo + M;
  const int a = c0 > lo ? c0 : lo, b = c0 + ncols < hi ? c0 + ncols : hi;
  return b > a ? b - a : 0;
}
// row of the item's column b, and its column
inline __host__ __device__ int sep_row_of(const SubDesc &d, int c0, int ncols, int b) {
  const int M = d.n_modes, c = c0 + b, k = c / (4 * M), s = (c % (4 * M)) / M, lo = (4 * k + s) * M;
  int row = c - (c0 > lo ? c0 : lo);
  for (int t = 0; t < s; ++t) row += sep_seg(d, c0, ncols, t, 0) + sep_seg(d, c0, ncols, t, 1);
  return k ? row + sep_seg(d, c0, ncols, s, 0) : row;
}
inline __host__ __device__ int sep_col_of(const SubDesc &d, int c0, int ncols, int row) {
  for (int s = 0; s < 4; ++s)
    for (int k = 0; k < 2; ++k) {
      const int n = sep_seg(d, c0, ncols, s, k), lo = (4 * k + s) * d.n_modes;
      if (row < n) return (c0 > lo ? c0 : lo) + row - c0;
      row -= n;
    }
  return 0;
}
// Only the basis columns of sides 3 and 4 have residuals on the middle ring rows (the gamma nodes next
// to them belong to these sides): MID has their rows only, the item's last ones; columns of sides 1, 2:
inline __host__ __device__ int sep_first34(const SubDesc &d, int c0, int ncols) {
  return sep_seg(d, c0, ncols, 0, 0) + sep_seg(d, c0, ncols, 0, 1) + sep_seg(d, c0, ncols, 1, 0) + sep_seg(d, c0, ncols, 1, 1);
}
// Rows of A, a multiple of the MMA's 128: the item's columns padded to 128, times real and imaginary
// parts where the data (MID, FWD: user densities) or the results (SYN, INV) are complex, times the
// 4 dense rows (FWD) or the rows transformed back (INV), in the order (row, part, column).
inline __host__ __device__ int sep_rows(const SubDesc &d, int job, int ncols, int col0, bool user) {
  const int cp = sep_pad128(ncols);
  switch (job) {
    case J_MID: return user ? 2 * cp : sep_pad128(ncols - sep_first34(d, col0, ncols));
    case J_FWD: return (user ? 8 : 4) * cp;
    case J_SYN: return (user || d.cplx ? 2 : 1) * cp;
    default: return (d.nrec >= 0 ? 5 : 4) * (user || d.cplx ? 2 : 1) * cp;
  }
}
inline __host__ __device__ int sep_classes(const SepGeo &g, int job) { return job == J_MID || job == J_SYN ? g.ncls : 2; }
inline __host__ __device__ int sep_nk(const SepGeo &g, int job) {
  return job == J_MID ? g.nk1 : job == J_FWD ? g.nkf : job == J_SYN ? g.nk3 : g.nqh / 16;
}
inline __host__ __device__ int sep_nt(const SepGeo &g, int job) {
  return job == J_MID ? g.nt1 : job == J_FWD ? g.nqh / 32 : job == J_SYN ? g.nt3 : g.ntg;
}
// blocks of 8 rows (operand cutting) and tiles of 128 rows x 32 outputs of a job
inline __host__ __device__ int sep_cut_blocks(const SubDesc &d, const SepGeo &g, int job, int ncols, int col0, bool user) {
  return sep_classes(g, job) * (sep_rows(d, job, ncols, col0, user) / 8);
}
inline __host__ __device__ int sep_tiles(const SubDesc &d, const SepGeo &g, int job, int ncols, int col0, bool user) {
  return sep_classes(g, job) * (sep_rows(d, job, ncols, col0, user) / 128) * sep_nt(g, job);
}
// Workspace of an item's separable solve, in doubles from its a_off (sized for complex data and a
// receiver row). Per job: digit blocks of A, exponents of A's rows (ints) [class][rows], masks of
// the nonzero groups of K (words) [class][rows / 128][SEP_MASK]; then the sums.
struct SepWs {
  long long a[4], ex[4], mask;   // mask: of all jobs, job after job
  long long u1, u3;    // sums at the gamma columns [class][output][Pi][rows] of MID and SYN
  long long mom;       // moments [class][3][nqp][rows]
  long long aeff;      // A_b [class][2][nqp][rows]
  long long ui;        // sums on the gamma rows and the receiver row [parity][Ng][rows]
  long long total;
};
inline __host__ __device__ SepWs sep_ws(const SubDesc &d, int ncols) {
  const SepGeo g = sep_geo(d);
  const long long cp = sep_pad128(ncols), R = 2 * cp, u = g.ncls * (long long)g.nS * g.Pi * R;
  const long long rows[4] = {R, 4 * R, R, 5 * R};
  SepWs w;
  long long off = 0;
  auto take = [&](long long n) { const long long o = off; off += (n + 31) & ~31LL; return o; };
  for (int j = 0; j < 4; ++j) {
    w.a[j] = take(sep_classes(g, j) * (rows[j] / 128) * sep_nk(g, j) * (SEP_ABLK / 8));
    w.ex[j] = take(sep_classes(g, j) * rows[j] / 2);
  }
  w.mask = take(2 * 11 * (R / 128) * SEP_MASK / 2);
  w.u1 = take(u);
  w.u3 = take(u);
  w.mom = take(g.ncls * 3LL * g.nqp * R);
  w.aeff = take(g.ncls * 2LL * g.nqp * R);
  w.ui = take(2LL * g.Ng * 5 * R);
  w.total = off;
  return w;
}
// Workspace of a full-grid solve of nr right-hand sides, in doubles (kernels_full.cu).
struct FullWs {
  int rows, R;            // rows of A: (right-hand side, unknown row, part), padded to 128
  int ldf, ldu;           // row lengths of f and u
  long long a, ex, mask;  // digit blocks, exponents (ints) [parity][R], masks (words) [parity][R / 128][SEP_MASK]
  long long f;            // mode space [rows][parity][nqh]
  long long u;            // sums over one parity [parity][R][folded columns]
  long long total;
};
inline __host__ __device__ FullWs full_ws(const SubDesc &d, int nr) {
  const SepGeo g = sep_geo(d);
  FullWs w;
  w.rows = 2 * nr * d.Nt;
  w.R = sep_pad128(w.rows);
  w.ldf = 2 * g.nqh;
  w.ldu = 32 * g.ntx;
  const long long nk = g.nkx > g.nqh / 16 ? g.nkx : g.nqh / 16;
  long long off = 0;
  auto take = [&](long long n) { const long long o = off; off += (n + 31) & ~31LL; return o; };
  w.a = take(2LL * (w.R / 128) * nk * (SEP_ABLK / 8));
  w.ex = take(w.R);
  w.mask = take(2LL * (w.R / 128) * SEP_MASK);   // two masks: of the forward and of the inverse transform
  w.f = take((long long)w.R * w.ldf);
  w.u = take(2LL * w.R * w.ldu);
  w.total = off;
  return w;
}
// ---- separable gradient pass (kernels_sepadj.cu): the same contractions with gamma and the ring exchanged
constexpr int ADJ_MDW = 68;               // doubles per mode of the k-derivative table
constexpr int ADJ_MOM = 4;                // moments of the cotangent per mode: phi_1, phi_2, their k-derivatives
constexpr int ADJ_DMOM = 3;               // k-derivative moments of the residual: phi_1, phi_2, receiver (tables of its own)
enum AdjJob { A_MID = 0, A_FWD, A_SYN, A_INV };
struct AdjGeo {
  int ncls, nS, nqp, nqh;
  int nti, nkj, ND;        // output groups (ring rows nlo+2 .. nhi-2), source groups (gamma rows nlo+1 .. nhi-1)
  int nt3, nt1;            // tiles of 32: ring columns; with the moments
  int nk1, nk3;            // K of MID, SYN ((b, mode), b < 2 or with a receiver row 3)
  int nb;                  // K blocks of SYN
  int nkf, ntr;            // FWD: folded columns mg .. of the gamma rows by 16, INV: mf .. of the ring rows by 32
};
inline __host__ __device__ AdjGeo adj_geo(const SubDesc &d, const SepGeo &g) {
  AdjGeo a;
  a.ncls = g.ncls; a.nS = g.nS; a.nqp = g.nqp; a.nqh = g.nqh;
  a.nti = (g.Pj + 31) / 32;
  a.nkj = (g.Pi + 15) / 16;
  a.ND = 2 * a.nti + a.nkj;
  a.nt3 = g.nS * a.nti;
  a.nt1 = a.nt3 + ADJ_MOM * g.nqp / 32;
  a.nk1 = g.nS * a.nkj;
  a.nb = d.nrec >= 0 ? 3 : 2;
  a.nk3 = a.nb * g.nqp / 16;
  a.nkf = (g.Ng + 15) / 16;
  a.ntr = (g.Kf + 31) / 32;
  return a;
}
// the gradient tables, as sep_tables
template <class D, class F>
inline __host__ __device__ void adj_tables(D &d, F f) {
  if (!d.tc_cols) return;
  const SepGeo g = sep_geo(d);
  const AdjGeo a = adj_geo(d, g);
  const long long n = g.nqp / 32, zw = 4LL * SEP_MASK * g.ncls, pairs = (long long)g.ncls * g.nS * g.nS;
  f(d.adj_rz, zw * n, TAB_MASK | TAB_OWN);
  f(d.adj_r3z, zw * a.nt3, TAB_MASK | TAB_OWN);
  f(d.adj_zm, zw * ADJ_MOM * n, TAB_MASK);
  f(d.adj_z3, zw * a.nt3, TAB_MASK);
  f(d.adj_zd, zw * 2 * n, TAB_MASK);
  f(d.adj_rp, 16LL * d.Nq, TAB_OWN);
  f(d.adj_rb, g.ncls * n * g.nk1 * SEP_BBLK, TAB_OWN);
  f(d.adj_r3, g.ncls * a.nt3 * 2 * n * SEP_BBLK, TAB_OWN);
  f(d.adj_md, 8LL * ADJ_MDW * d.Nq, 0);
  f(d.adj_phid, 16LL * (d.Py + 2) * d.Nq, 0);
  f(d.adj_kdd, 8 * pairs * d.Py, 0);
  f(d.adj_kde, 8LL * g.ncls * g.nS, 0);
  f(d.adj_tb, pairs * a.ND * SEP_BBLK, 0);
  f(d.adj_mb, g.ncls * ADJ_MOM * n * a.nk1 * SEP_BBLK, 0);
  f(d.adj_b3, g.ncls * a.nt3 * 4 * n * SEP_BBLK, 0);
  f(d.adj_bf, 2LL * (g.nqh / 32) * a.nkf * SEP_BBLK, 0);
  f(d.adj_bi, 2LL * a.ntr * (g.nqh / 16) * SEP_BBLK, 0);
  f(d.adj_dtb, pairs * g.ND * SEP_BBLK, 0);
  f(d.adj_dmb, g.ncls * 2 * n * g.nk1 * SEP_BBLK, 0);
}
// rows of A: the columns padded to 128, real and imaginary parts, times the rows transformed
inline __host__ __device__ int adj_rows(const SubDesc &d, int job, int ncols) {
  const int r = 2 * sep_pad128(ncols);
  return job == A_FWD ? (d.nrec >= 0 ? 5 : 4) * r : job == A_INV ? 4 * r : r;
}
inline __host__ __device__ int adj_classes(const AdjGeo &a, int job) { return job == A_MID || job == A_SYN ? a.ncls : 2; }
inline __host__ __device__ int adj_nk(const AdjGeo &a, int job) {
  return job == A_MID ? a.nk1 : job == A_FWD ? a.nkf : job == A_SYN ? a.nk3 : a.nqh / 16;
}
inline __host__ __device__ int adj_nt(const AdjGeo &a, int job) {
  return job == A_MID ? a.nt1 : job == A_FWD ? a.nqh / 32 : job == A_SYN ? a.nt3 : a.ntr;
}
inline __host__ __device__ int adj_cut_blocks(const SubDesc &d, const AdjGeo &a, int job, int ncols) {
  return adj_classes(a, job) * (adj_rows(d, job, ncols) / 8);
}
inline __host__ __device__ int adj_tiles(const SubDesc &d, const AdjGeo &a, int job, int ncols) {
  return adj_classes(a, job) * (adj_rows(d, job, ncols) / 128) * adj_nt(a, job);
}
// tiles of the forward pass's stage 1 for the gradient: dK/dk, the moments and their derivatives, the dense rows
inline __host__ __device__ int grad_mid_tiles(const SubDesc &d, const SepGeo &g) {
  return g.nt3 + (2 + (d.nrec >= 0 ? 3 : 2)) * g.nqp / 32;
}
// Workspace of an item's gradient pass after the projection's (SepWs, whose stage 1 it shares), in doubles.
struct AdjWs {
  long long a[4], ex[4], mask;
  long long dmom;        // k-derivative moments of the residual [class][ADJ_DMOM][nqp][rows] (its moments: SepWs::mom)
  long long mom;         // moments of the cotangent [class][ADJ_MOM][nqp][rows]
  long long ga;          // transforms of its gamma rows and receiver row [5][Nq][ncols] (complex)
  long long u1, u3;      // sums at the ring columns [class][column][Pj][rows]
  long long aeff;        // coefficients [class][3][nqp][rows]
  long long ui;          // sums on the dense ring rows [parity][Kf][rows]
  long long total;
};
inline __host__ __device__ int adj_mask_of(int job, int ncols) {   // jobs of at most R, 5 R, R, 4 R rows
  const int t = 2 * (2 * sep_pad128(ncols) / 128) * SEP_MASK;
  return job == A_MID ? 0 : job == A_FWD ? t : job == A_SYN ? 6 * t : 7 * t;
}
inline __host__ __device__ int adj_mask_words(int ncols) { return 11 * 2 * (2 * sep_pad128(ncols) / 128) * SEP_MASK; }
inline __host__ __device__ AdjWs adj_ws(const SubDesc &d, int ncols) {
  const SepGeo g = sep_geo(d);
  const AdjGeo a = adj_geo(d, g);
  const long long cp = sep_pad128(ncols), R = 2 * cp;
  const long long rows[4] = {R, 5 * R, R, 4 * R}, nk3 = 3LL * g.nqp / 16;   // with room for a receiver row
  AdjWs w;
  long long off = sep_ws(d, ncols).total;
  auto take = [&](long long n) { const long long o = off; off += (n + 31) & ~31LL; return o; };
  for (int j = 0; j < 4; ++j) {
    w.a[j] = take(adj_classes(a, j) * (rows[j] / 128) * (j == A_SYN ? nk3 : adj_nk(a, j)) * (SEP_ABLK / 8));
    w.ex[j] = take(adj_classes(a, j) * rows[j] / 2);
  }
  w.mask = take(adj_mask_words(ncols) / 2);
  w.dmom = take(g.ncls * (long long)ADJ_DMOM * g.nqp * R);
  w.mom = take(g.ncls * (long long)ADJ_MOM * g.nqp * R);
  w.ga = take(10LL * d.Nq * ncols);
  w.u1 = take(g.ncls * (long long)g.nS * g.Pj * R);
  w.u3 = take(g.ncls * (long long)g.nS * g.Pj * R);
  w.aeff = take(g.ncls * 3LL * g.nqp * R);
  w.ui = take(2LL * g.Kf * 4 * R);
  w.total = off;
  return w;
}
// first mask word of a job, in words from SepWs::mask (jobs of at most R, 4 R, R, 5 R rows)
inline __host__ __device__ int sep_mask_of(int job, int ncols) {
  const int t = 2 * (2 * sep_pad128(ncols) / 128) * SEP_MASK;
  return job == J_MID ? 0 : job == J_FWD ? t : job == J_SYN ? 5 * t : 6 * t;
}
inline __host__ __device__ int sep_mask_words(int ncols) { return 11 * 2 * (2 * sep_pad128(ncols) / 128) * SEP_MASK; }
constexpr int TRI_WARPS = 1;  // warps (modes) per block of the per-mode sweep kernel k_tri
constexpr int FFT_POINTS = 4096;        // longest transform (2 Nx) of the dense-row FFT kernels (64 KiB)
constexpr int FFT_BLOCK_POINTS = 1024;  // complex values per block when 2 Nx is shorter: fpb = 1024 / (2 Nx)

// Host buffer of the plan's tables: page-locked (cudaMallocHost) for plans with a device, so
// that uploads (plan creation, mdp_plan_update_k) run at full link speed; plain heap memory for
// host-only plans, which make no CUDA call. Zero-filled on allocation.
template <class T>
struct HostBuf {
  T *p = nullptr;
  size_t n = 0;
  bool pinned = false;
  HostBuf() = default;
  HostBuf(const HostBuf &) = delete;
  HostBuf &operator=(const HostBuf &) = delete;
  ~HostBuf() { release(); }
  void release() {
    if (p) { if (pinned) cudaFreeHost(p); else std::free(p); }
    p = nullptr; n = 0; pinned = false;
  }
  bool alloc(size_t count, bool want_pinned) {
    release();
    const size_t bytes = std::max<size_t>(count, 1) * sizeof(T);
    if (want_pinned && cudaMallocHost((void **)&p, bytes) == cudaSuccess) pinned = true;
    else { p = (T *)std::malloc(bytes); pinned = false; }
    if (!p) return false;
    std::memset((void *)p, 0, bytes);
    n = count;
    return true;
  }
  T *data() { return p; }
  const T *data() const { return p; }
  size_t size() const { return n; }
  T &operator[](size_t i) { return p[i]; }
  const T &operator[](size_t i) const { return p[i]; }
};

struct HostSub {
  SubDesc d;
  std::vector<int> gamma_nm;     // 2*G: (n, m) pairs, row-major order
  std::vector<int> owner;        // G
  std::vector<double> rho, s, L; // G
  // this subdomain's slices of the plan's host tables (written in place by the factorisation)
  double *fact = nullptr;        // [Nq][Nt][FW]
  uint8_t *piv = nullptr;        // [Nq][Nt]
  double *dT = nullptr;          // [Nq][Nt][6]
  double *fs = nullptr;          // [Nq][NYf][FSW]: projection forward-sweep table
  std::vector<int> seg;          // [Nq][5]: see SubDesc::seg_off
};

struct Wave {
  std::vector<Item> items;
  long long ws_doubles;
};

}  // namespace mdp

struct mdp_plan {
  unsigned flags = 0;
  int n_subs = 0;
  int device = -1;
  std::vector<mdp::HostSub> subs;
  mdp::HostBuf<double> host_tables;      // factor / dT / sweep / sine / geometry tables: the first n_light doubles
  long long n_tables = 0, n_light = 0;   // of n_tables, or all of them (bind_tables)
  mdp::HostBuf<uint8_t> host_piv;
  long long out_size = 0;
  long long rec_size = 0;
  int tile_cols = 256;                   // columns per work item of subdomains that take the sweeps
  int sep_cols = 512;                    // of those that take the separable solve, in its gradient pass too
  int fft_block_points = mdp::FFT_BLOCK_POINTS;  // complex values per block of the dense-row FFT kernels
  int tri_stages = 2;                    // table rows the projection sweep stages ahead (2 or 4)
  long long ws_budget = 0;               // bytes of workspace
  // batch schedules: [S_PROJ] mdp_project_batch over every subdomain, [S_GRAD] mdp_ap_adjoint
  // (larger workspace), [S_BASIS] basis columns of the distinct subdomains only (MDP_PLAN_DEDUPE
  // with duplicates; else empty)
  std::vector<mdp::Wave> sched[3];
  std::vector<int> leader;               // per subdomain: the subdomain whose tables and basis columns it shares
  // device side
  mdp::SubDesc *d_subs = nullptr;        // the subdomains, then the same without receiver rows (subs_of)
  double *d_tables = nullptr;
  uint8_t *d_piv = nullptr;
  unsigned char *d_sep = nullptr;        // separable tables (kernels_sep.cu), rebuilt with the factor tables
  unsigned char *d_adj = nullptr;        // gradient tables (kernels_sepadj.cu), one set: rebuilt by the gradient
  long long adj_bytes = 0, adj_masks = 0;   // pass when the wavenumbers have changed since (adj_stale)
  bool adj_stale = true, adj_sines = false, adj_captured = false;
  cudaStream_t side = nullptr;           // an update's factorisation beside its separable tables, with the events
  cudaEvent_t fork_ev = nullptr, join_ev = nullptr;   // that fork it from and join it to the caller's stream
  long long sep_bytes = 0, sep_masks = 0;   // size; its first bytes: the masks, cleared before a rebuild
  double *d_ws = nullptr;
  long long ws_doubles = 0;
  int *d_status = nullptr;
  int *d_fstatus = nullptr;               // status word of the device factorisation
  int fft_smem = 16;                     // dynamic shared memory of the FFT kernels: max fpb * 2 Nx * 16 B
  int n_sm = 0;                          // multiprocessors of the plan's device (persistent grids)
  mdp::HostBuf<mdp::SubDesc> sub_stage;  // pinned copy of the subdomain descriptors (async upload)
  mdp::HostBuf<int> h_fstatus;           // pinned read-back of d_fstatus
  bool host_stale = false;               // device tables refactored since the host tables were built
  bool fs_stale = false;                 // device sweep tables older than the wavenumbers (not read by the
                                         // separable solve; rebuilt when mdp_plan_read_tables asks)
  // second table set of mdp_plan_update_k_async (allocated by its first call). d_subs, d_tables
  // and d_piv name physical set `set`; the alt_* pointers the other. ready_ev[s]: after the last
  // refactorisation into set s; used_ev[s]: after the last compute call that read it.
  mdp::SubDesc *alt_subs = nullptr;
  double *alt_tables = nullptr;
  uint8_t *alt_piv = nullptr;
  unsigned char *alt_sep = nullptr;
  mdp::HostBuf<mdp::SubDesc> alt_stage;  // pinned descriptor stage of set 1 (sub_stage: set 0)
  int set = 0;
  cudaEvent_t ready_ev[2] = {nullptr, nullptr};
  cudaEvent_t used_ev[2] = {nullptr, nullptr};
  bool used_rec[2] = {false, false};
  // per schedule and wave: device items and prefix arrays (one prefix array per kernel family)
  std::vector<mdp::Item *> d_items[3];
  std::vector<int *> d_order[3];         // [wave] -> device int [k_tri + k_adj_tri blocks]: launch orders
  std::vector<int *> d_prefix[3];        // [wave] -> device int [2][NFAM][n_items + 1]: without, with receiver rows
  std::vector<std::vector<int>> h_prefix[3];
  // CUDA graphs of mdp_project_batch, keyed by (xi, out, kind, stream, table set)
  struct GraphEntry {
    const void *xi; void *out; void *out_rec; int kind; cudaStream_t st; const double *tab; cudaGraphExec_t exec;
  };
  std::vector<GraphEntry> graphs;
  // per-kernel event timing (mdp_plan_profile)
  bool prof_on = false;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> prof_ev[48];
  int prof_used[48] = {0};
};

namespace mdp {

enum Sched { S_PROJ = 0, S_GRAD = 1, S_BASIS = 2 };

// the ranges a launch's Batch carries for the bounds-checked build (out_n: complex elements of the
// call's output, density and cotangent arrays)
inline void set_bounds(const mdp_plan *p, Batch &b, long long out_n, bool grad) {
  b.n_subs = p->n_subs;
  b.grad = grad ? 1 : 0;
  b.ws_n = p->ws_doubles;
  b.tab_n = p->n_tables;
  b.piv_n = (long long)p->host_piv.size();
  b.out_n = out_n;
  b.rec_n = p->rec_size;
  b.sep_n = p->sep_bytes;
  b.adj_n = p->adj_bytes;
  b.status = p->d_status;
}

// Device descriptors of a call: with the receiver rows where it reads or writes their values, else without, so that
// such a call does no work for them and one captured before a change of the rows stays what it was.
inline const SubDesc *subs_of(const mdp_plan *p, bool rec) { return p->d_subs + (rec ? 0 : p->n_subs); }
inline SubDesc without_rec(SubDesc d) {
  d.nrec = -1;
  d.rec_off = 0;
  return d;
}
// the descriptors of d_subs, 2 n_subs of them
inline void fill_subs(const mdp_plan *p, SubDesc *s) {
  for (int i = 0; i < p->n_subs; ++i) { s[i] = p->subs[i].d; s[p->n_subs + i] = without_rec(s[i]); }
}

// kernel families (each has its own block decomposition of an item). F_A* are the adjoint's. F_RING (basis
// columns of the separable solve), F_PRES and F_RES make the ring residuals. F_C* cut operands, F_G* contract
// (stage 1 and 3, B: basis columns, U: user densities; F_TCOLS is stage 3 for basis columns), F_SMODE and
// F_SOUT are the separable solve's other kernels; F_ACLR to F_AOUT and F_ATCOLS its gradient pass.
enum Fam { F_EXT = 0, F_RES, F_FROWS, F_TRI, F_IROWS, F_ICOLS, F_AFWD, F_ATRI, F_ARING, F_ARINGC, F_AGAM, F_IREC,
           F_ACOLS, F_TCOLS, F_ATCOLS, F_C1B, F_C1U, F_G1B, F_G1U, F_SMODE, F_C3B, F_C3U, F_G3U, F_SOUT, F_RING, F_PRES,
           F_ACLR, F_GG1B, F_GG1U, F_AC1, F_AG1, F_AMODE, F_AC3, F_AOUT, NFAM };
static_assert(NFAM <= 48, "per-family event lists of mdp_plan");

// Blocks of kernel family f for an item of ncols columns: 32 columns (x) times BY tasks (y).
// The same function numbers the blocks on the host (prefix sums) and in the kernels.
inline __host__ __device__ int blocks_for(int f, const SubDesc &d, int ncols, int col0) {
  const int cb = (ncols + 31) / 32;
  switch (f) {
    case F_EXT: return (d.G + 31) / 32;
    case F_RES: return cb * (((d.xsym ? 4 * d.Ph + 2 * (d.Py - 4) : d.R) + 7) / 8);
    case F_PRES: return d.tc_cols ? 0 : blocks_for(F_RES, d, ncols, col0);
    case F_RING: {
      if (!d.tc_cols) return 0;
      const int dense = d.xsym ? d.Ph : d.Px, side = d.Py + 4;
      return cb * (((dense > side ? dense : side) + 7) / 8);
    }
    case F_FROWS:
      if (d.tc_cols) return 0;
      if (d.rows_fft) return 4 * ((ncols + d.fpb - 1) / d.fpb);
      return cb * ((d.Nx / 2 + 7) / 8);
    case F_TRI: return d.tc_cols ? 0 : cb * ((d.Nq + TRI_WARPS - 1) / TRI_WARPS);
    case F_IROWS:
      if (d.tc_cols) return 0;
      if (d.rows_fft) return 4 * ((ncols + d.fpb - 1) / d.fpb);
      return cb * (((d.xsym ? 4 * (d.Ph + 1) : 4 * (d.Px + 2)) + 7) / 8);
    case F_ICOLS: return d.tc_cols ? 0 : cb * ((d.Py - 2 + 7) / 8);
    case F_C1B: case F_C1U: case F_G1B: case F_G1U: case F_C3B: case F_C3U: case F_TCOLS: case F_G3U: {
      if (!d.tc_cols) return 0;
      const SepGeo g = sep_geo(d);
      const bool user = f == F_C1U || f == F_G1U || f == F_C3U || f == F_G3U;
      const int j = f == F_C1B || f == F_C1U || f == F_G1B || f == F_G1U ? J_MID : J_SYN;   // and the next job
      if (f == F_C1B || f == F_C1U || f == F_C3B || f == F_C3U)
        return sep_cut_blocks(d, g, j, ncols, col0, user) + sep_cut_blocks(d, g, j + 1, ncols, col0, user);
      return sep_tiles(d, g, j, ncols, col0, user) + sep_tiles(d, g, j + 1, ncols, col0, user);
    }
    case F_ACLR: return d.tc_cols ? 1 : 0;
    case F_GG1B: case F_GG1U: {
      if (!d.tc_cols) return 0;
      const SepGeo g = sep_geo(d);
      return g.ncls * (sep_rows(d, J_MID, ncols, col0, f == F_GG1U) / 128) * grad_mid_tiles(d, g) +
             sep_tiles(d, g, J_FWD, ncols, col0, f == F_GG1U);
    }
    case F_AC1: case F_AC3: case F_AG1: case F_ATCOLS: {
      if (!d.tc_cols) return 0;
      const AdjGeo a = adj_geo(d, sep_geo(d));
      const int j = f == F_AC1 || f == F_AG1 ? A_MID : A_SYN;   // and the next job
      if (f == F_AC1 || f == F_AC3) return adj_cut_blocks(d, a, j, ncols) + adj_cut_blocks(d, a, j + 1, ncols);
      return adj_tiles(d, a, j, ncols) + adj_tiles(d, a, j + 1, ncols);
    }
    case F_SMODE: case F_AMODE: {
      if (!d.tc_cols) return 0;
      const int per = sep_modes_per_block(d, ncols);
      return cb * ((d.Nq + per - 1) / per);
    }
    case F_AOUT: {   // ring columns of the middle rows; dense ring rows; dK/dk against the cotangent
      if (!d.tc_cols) return 0;
      const SepGeo g = sep_geo(d);
      return cb * ((g.Pj + 7) / 8 + (4 * g.Kf + 7) / 8 + (g.Pi + 7) / 8);
    }
    case F_SOUT: {   // middle rows, 8 per block, then 32 folded columns of each row transformed back
      if (!d.tc_cols) return 0;
      const SepGeo g = sep_geo(d);
      return cb * ((d.Py - 2 + 7) / 8) + cb * g.slots * g.ntg;
    }
    case F_AFWD:
      if (d.tc_cols) return 0;
      if (d.rows_fft) return 5 * ((ncols + d.fpb - 1) / d.fpb);
      return cb * ((d.Nx / 2 + 7) / 8);
    case F_ATRI: return d.tc_cols ? 0 : cb * ((d.Nq + 3) / 4);
    case F_ARING:
      if (d.tc_cols) return 0;
      if (d.rows_fft) return 4 * ((ncols + d.fpb - 1) / d.fpb);
      return cb * ((4 * d.Px + 7) / 8);
    case F_ARINGC: return d.tc_cols ? 0 : cb * ((d.Py - 4 + 7) / 8);
    case F_AGAM: return cb * ((d.G + 7) / 8);
    case F_IREC: return d.nrec < 0 || d.tc_cols ? 0 : cb * (((d.xsym ? d.Ph - 1 : d.Px - 2) + 7) / 8);
    case F_ACOLS: return cb * ((d.Py - 2 + 7) / 8);
    default: return 0;
  }
}

// slot bases of the per-block gradient partials of an item: [ATRI or AMODE | ARING or AOUT | ARINGC | AGAM],
// total
inline __host__ __device__ void red_slots(const SubDesc &d, int ncols, int base[5]) {
  base[0] = 0;
  base[1] = base[0] + blocks_for(F_ATRI, d, ncols, 0) + blocks_for(F_AMODE, d, ncols, 0);
  base[2] = base[1] + blocks_for(F_ARING, d, ncols, 0) + blocks_for(F_AOUT, d, ncols, 0);
  base[3] = base[2] + blocks_for(F_ARINGC, d, ncols, 0);
  base[4] = base[3] + blocks_for(F_AGAM, d, ncols, 0);
}
// Workspace slices of an item of ncols columns, in doubles from the item's base (each 256-byte
// aligned): basis densities, ring residual, dense-row transforms, mode-space field, and for the
// gradient pass the adjoint field, k-source and per-block partials. With the separable solve the projection
// keeps only the 4 gamma rows and the receiver row of the mode-space field ([Nq][5][ncols]), and its
// operands and sums (SepWs); the gradient pass the adjoint field of the 4 dense ring rows, SepWs and AdjWs.
inline __host__ __device__ void item_workspace(const SubDesc &d, int ncols, bool grad, long long &xi, long long &r,
                                               long long &gr, long long &y, long long &a, long long &s,
                                               long long &red, long long &total) {
  auto al = [](long long v) { return (v + 31) & ~31LL; };
  long long off = 0;
  xi = off; off += al((long long)d.G * ncols * (grad ? 2 : 1));
  r = off;  off += al((long long)(d.R > d.R2 ? d.R : d.R2) * ncols * 2);
  gr = off; off += al(5LL * d.Nq * ncols * 2);  // 4 dense rows (+ the receiver row in the adjoint)
  y = off;  off += al((long long)d.Nq * (d.tc_cols ? 5 : grad ? d.Nt : d.NYf) * ncols * 2);
  a = off;  off += d.tc_cols ? (grad ? adj_ws(d, ncols).total : sep_ws(d, ncols).total)
                             : grad ? al((long long)d.Nq * d.Nt * ncols * 2) : 0;
  s = off;  off += grad ? al((long long)d.R * ncols * 2) : 0;
  int rs[5];
  red_slots(d, ncols, rs);
  red = off; off += grad ? al(rs[4] + 1) : 0;
  total = off;
}
const char *fam_name(int f);
// event pair around a launch when profiling is on
void prof_begin(mdp_plan *p, int fam, cudaStream_t st);
void prof_end(mdp_plan *p, int fam, cudaStream_t st);
// plan construction (host)
bool bind_tables(mdp_plan *p, long long n, bool pinned);
mdp_status build_host_plan(mdp_plan *p, const mdp_subdomain *subs, int n);
mdp_status refactor_host(mdp_plan *p, const double *k);
void mode_entries(const SubDesc &d, int q, double &off, double &diag);   // interior entries of T_q
mdp_status set_k_fields(mdp_plan *p, const double *k);   // validate k, update the k-dependent SubDesc fields
// factor.cu: the factor tables into a table set (descriptors ds, tables tab, pivot flags piv); the
// sweep tables of subdomains that project through the separable solve only with `all`
cudaError_t launch_factor_to(const mdp_plan *p, const SubDesc *ds, double *tab, uint8_t *piv, int *status, bool all,
                             cudaStream_t st);
void host_mode_solve(const HostSub &hs, int q, int adjoint, const double *b, double *x);
// kernel launchers (kernels.cu)
enum { PASS_FWD = 0, PASS_GRAD = 1 };
#ifdef __CUDACC__
// Launch whose set-up overlaps the kernel before it on the stream (programmatic dependent launch): its blocks come
// as that kernel's last ones leave, and every kernel launched so first waits in pdl_wait(), which returns when
// the kernels before it are complete and their writes visible. Eight kernels of a pass of 129^2: 84.6 -> 66.2 us;
// 4 x 257^2: 231 -> 214 us. No earlier trigger: blocks that wait take the registers and shared memory of the
// kernel before (279 us with one at each kernel's start).
template <class... P, class... A>
inline void pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid; c.blockDim = block; c.dynamicSmemBytes = smem; c.stream = st; c.attrs = &at; c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
}
__device__ __forceinline__ void pdl_wait() {
  cudaGridDependencySynchronize();
}
#endif
cudaError_t set_kernel_attributes();      // kernels.cu: opt-in shared memory of the FFT kernels
cudaError_t set_adj_kernel_attributes();  // kernels_adj.cu
cudaError_t set_sep_kernel_attributes();  // kernels_sep.cu
// the separable tables of every subdomain that takes them, for the wavenumbers of the descriptors ds;
// entries: from matrix entries computed here, else from the stored ones (sep_ab)
cudaError_t launch_sep_tables(const mdp_plan *p, const SubDesc *ds, const double *tab, unsigned char *sep, bool entries,
                              cudaStream_t st);
// the sine tables among them, which no wavenumber enters
cudaError_t launch_sep_sines(const mdp_plan *p, const SubDesc *ds, const double *tab, unsigned char *sep, cudaStream_t st);
// the separable solve of the projection, from the ring residuals to the output columns
cudaError_t launch_sep_project(mdp_plan *p, const Batch *fb, int out_kind, const double2 *xi_user, double2 *out,
                               double2 *out_rec, cudaStream_t st);
// kernels_sepadj.cu: the gradient tables for the wavenumbers of the plan's current set, and the k-independent
// ones; the separable gradient pass of a wave (forward: with the k-gradient)
cudaError_t launch_adj_tables(const mdp_plan *p, cudaStream_t st);
cudaError_t launch_adj_sines(const mdp_plan *p, cudaStream_t st);
// (rec: with the receivers' cotangent, see subs_of)
cudaError_t launch_adj_clear(mdp_plan *p, const Batch *fb, bool rec, cudaStream_t st);
cudaError_t launch_sep_adj_residual(mdp_plan *p, const Batch *fb, bool user, bool rec, cudaStream_t st);
cudaError_t launch_sep_adjoint(mdp_plan *p, const Batch *fb, bool user, bool dk, const double2 *cot, const double2 *cot_rec,
                               cudaStream_t st);
cudaError_t launch_sep_cut1(const Batch &b, const SubDesc *subs, double *ws, bool user, int fam, cudaStream_t st);
cudaError_t set_sepadj_kernel_attributes();
cudaError_t launch_project(mdp_plan *p, const Batch *fam_batches, int out_kind, const double2 *xi_user,
                           double2 *out, double2 *out_rec, cudaStream_t st);
cudaError_t launch_adjoint(mdp_plan *p, const Batch *fam_batches, int out_kind, const double2 *xi_user,
                           const double2 *cot, const double2 *cot_rec, double2 *grad_xi, double *grad_k,
                           cudaStream_t st);
// the adjoint's own kernels (kernels_adj.cu), after the forward recompute of the gradient pass
cudaError_t launch_adjoint_tail(mdp_plan *p, const Batch *fb, int out_kind, const double2 *xi_user, const double2 *cot,
                                const double2 *cot_rec, double2 *grad_xi, double *grad_k, cudaStream_t st);

cudaError_t launch_potential(const mdp_plan *p, int sub, int ncols, const double2 *xi, double2 *u, cudaStream_t st);
cudaError_t launch_source_terms(mdp_plan *p, int sub, const double2 *f, const double2 *src4, double2 *F, double2 *u,
                                cudaStream_t st);
cudaError_t launch_basis_densities(const mdp_plan *p, int sub, int col0, int ncols, double2 *out, cudaStream_t st);
// the full-grid solve through the separable Green's function (subdomains with tc_cols; kernels_full.cu)
bool full_solve_fits(const SubDesc &d);   // the grid has no more rows than the separable full-grid solve takes
cudaError_t launch_full_solve(const mdp_plan *p, int sub, int nrhs, const double2 *g, double2 *u, cudaStream_t st);
cudaError_t set_full_kernel_attributes();
__global__ void k_full_modes(const SubDesc *subs, int s0, unsigned char *sep);
cudaError_t launch_solve(const mdp_plan *p, int sub, int nrhs, const double2 *g, double2 *u, int adjoint,
                         cudaStream_t st);
cudaError_t launch_solve_raw(const SubDesc *d_sub, const SubDesc &hd, const double *tab, const uint8_t *piv,
                             double *buf, long long buf_doubles, int nrhs, const double2 *g, double2 *u, int adjoint,
                             cudaStream_t st);
}  // namespace mdp
