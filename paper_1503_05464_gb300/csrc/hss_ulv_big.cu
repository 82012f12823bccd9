// ULV factorization (Algorithm 3) of nodes by blocked operations, spread over
// the whole GPU.
//
// The per-node kernel of hss_ulv.cu runs one CTA per node, which suits nodes
// of a few dozen rows.  Larger ones are factored here, batched over all such
// nodes of a level (and of every handle of the call).  FP64 instructions are
// the scarce unit (two multiply-adds a clock and SM), so every step is either
// a matrix product that keeps all SMs busy or a panel whose serial part is
// kept short:
//   D_tau   diagonal blocks copied, off-diagonal blocks B Vtb^T by batched GEMM;
//   Vhat^T  V^T diag(Vtb_1, Vtb_2)^T by batched GEMM (V = Pi [I; E]);
//   W       Omega D_tau: top rows D(perm(k+i)) - E D(perm(0..k)) by GEMM;
//   LQ      in panels of NB rows: the panel and its compact WY factor T
//           (I - V^T T V = H_i0 ... H_i1) by a cluster of CTAs that split its
//           columns (lq_panel_kernel), then the trailing rows of W and all of
//           Vhat^T -- whose rows the reflectors turn into Vtilde^T =
//           (Q Vhat)^T -- in one launch: R <- R - ((R V^T) T) V, a CTA per 8
//           to 32 rows (lq_update_kernel);
//   root    right-looking blocked LU with partial pivoting: the panel by a
//           cluster that splits its rows (lu_panel_kernel), the block row by
//           substitution, 16 columns a CTA, GEMM update of the rest.
// The factors have the per-node kernel's layout.
// Every launch shape that a node's sums depend on follows from the node's own
// order, so factors do not depend on what shares the launch.
#include "hss_fp.cuh"
#include "hss_internal.cuh"
#include "hss_tree.h"

#include <cooperative_groups.h>

#include <cfloat>

#include <algorithm>
#include <climits>
#include <functional>

namespace cg = cooperative_groups;

namespace hss {

namespace {

constexpr int NB = 32;           // panel width
constexpr int B_THREADS = 256;
constexpr int B_WARPS = B_THREADS / 32;

// dst[i][j] (rows x cols, ld_dst) = src[i][j] (input dtype or FP64), with an
// optional destination row map and an optional lower-triangle mask
struct CopyItem {
  const void* src;
  int64_t lds;
  int src_f64;
  double* dst;
  int64_t ldd;
  int rows, cols;
  const int32_t* dst_row;   // null: row i
  int lower;                // 1: entries j > i become 0
  int trans;                // 1: the source is transposed (src[j][i])
};

__global__ void copy_items_kernel(const CopyItem* items, const int64_t* start, int nitems,
                                  int64_t total) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= total) return;
  int lo = 0, hi = nitems - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  const CopyItem it = items[lo];
  const int64_t e = t - start[lo];
  int i = static_cast<int>(e / it.cols), j = static_cast<int>(e % it.cols);
  if (it.trans) {   // source entries in order: its reads are the contiguous side
    j = static_cast<int>(e / it.rows);
    i = static_cast<int>(e % it.rows);
  }
  const int64_t o = it.trans ? j * it.lds + i : i * it.lds + j;
  double v = it.src_f64 ? reinterpret_cast<const double*>(it.src)[o]
                        : static_cast<double>(reinterpret_cast<const float*>(it.src)[o]);
  if (it.lower && j > i) v = 0.0;
  const int di = it.dst_row ? it.dst_row[i] : i;
  it.dst[di * it.ldd + j] = v;
}

// V = Pi [I; E] of a node (mc x kc): row perm[q] is unit vector q for q < kc,
// else row q - kc of E.  trans: V^T (kc rows, ld ldv) instead.
struct VItem {
  double* V;
  int64_t ldv;
  const int32_t* perm;
  const double* E;
  int mc, kc, trans;
};

__global__ void v_fill_kernel(const VItem* items, const int64_t* start, int nitems, int64_t total) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= total) return;
  int lo = 0, hi = nitems - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  const VItem it = items[lo];
  const int64_t e = t - start[lo];
  const int q = static_cast<int>(e / it.kc), l = static_cast<int>(e % it.kc);
  const double v = q < it.kc ? (q == l ? 1.0 : 0.0) : it.E[static_cast<int64_t>(q - it.kc) * it.kc + l];
  const int row = it.perm[q];
  it.V[it.trans ? l * it.ldv + row : row * it.ldv + l] = v;
}

// Columns of a panel per CTA of its cluster (all pivot columns belong to rank 0)
__host__ __device__ inline int lq_cols(int wid, int C) {
  const int cw = (wid + C - 1) / C;
  return cw < NB ? NB : cw;
}
// CTAs per panel: a function of the node's order alone
inline int panel_ctas(int m) { return m <= 160 ? 1 : m <= 320 ? 2 : m <= 640 ? 4 : 8; }
constexpr size_t PANEL_SMEM_CAP = 160 * 1024;   // larger panels stay in global memory (L2)

struct LqPanel {
  double* W;       // m x m, row-major
  double* hv;      // r x m reflectors
  double* tau;     // r
  double* T;       // NB x NB: the panel's compact WY factor
  int m, i0, nbb;
};

// sums p[0..3] over the 32 lanes; lanes 8 g .. 8 g + 7 return the sum of p[g]
// (six FP64 additions: an addition costs the same for one lane as for 32)
__device__ __forceinline__ double reduce_scatter4(double (&p)[4]) {
  const int lane = threadIdx.x & 31;
  const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
  double a = h16 ? p[2] : p[0], b = h16 ? p[3] : p[1];
  const double oa = h16 ? p[0] : p[2], ob = h16 ? p[1] : p[3];
  a += __shfl_xor_sync(0xffffffffu, oa, 16);
  b += __shfl_xor_sync(0xffffffffu, ob, 16);
  double v = h8 ? b : a;
  v += __shfl_xor_sync(0xffffffffu, h8 ? a : b, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Householder LQ of rows [i0, i0 + nbb) of W over the columns from i0, and
// the compact WY factor of its reflectors, by a cluster of C CTAs that each
// keep a block of columns (all rows) in shared memory.
//
// A step needs one exchange: with a_j = row j right of the pivot, every CTA
// sends the partial sums a_i . a_j of all rows j >= i (and rank 0 the pivot
// column) to its peers, and after one cluster barrier each has sigma, tau,
// the scale of v and, as v is a multiple of a_i, every row's product with it.
// Warp w owns rows w, w + 8, w + 16, w + 24.  The square root and the quotients
// run in one warp, on the integer pipes (hss_fp.cuh: the same bits; a lane's
// FP64 root and divisions, one after the other, took 2100 of a step's 11,600
// cycles; 56 panels 10.5 -> 9.9 ms).
// T = D (I + U D)^{-1} with U the strict upper triangle of V V^T and D =
// diag(tau) (the inverse of a unit triangle: no division, tau may be 0).
//
// Bound: FP64 latency (about 3 us a step).  One CTA per panel, which took the
// sums from global memory and was bound by its SM's two FMAs a clock, needed
// 530 us a panel at m = 1200 against 180.
template <int C>
__global__ void __launch_bounds__(B_THREADS) lq_panel_kernel(const LqPanel* items, int in_smem) {
  extern __shared__ double lsm[];
  double(*gp)[NB * (NB - 1) / 2] = reinterpret_cast<double(*)[NB * (NB - 1) / 2]>(lsm);   // [C]
  double* Asm = lsm + C * (NB * (NB - 1) / 2);
  __shared__ double part[2][C][NB];
  __shared__ double alph[2][NB];
  __shared__ double sc[NB], tq[NB], sh[2];   // scale and tau of each step; this step's
  __shared__ double xl[NB][NB + 1];
  __shared__ double Mu[NB][NB + 1];
  const LqPanel it = items[blockIdx.x / C];
  const int m = it.m, tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nbb = it.nbb;
  int rank = 0;
  if constexpr (C > 1) rank = static_cast<int>(cg::this_cluster().block_rank());
  const int wid = m - it.i0, cw = lq_cols(wid, C);
  const int nloc = max(0, min(cw, wid - rank * cw));
  double* Wg = it.W + static_cast<int64_t>(it.i0) * m + it.i0 + rank * cw;
  double* A = in_smem ? Asm : Wg;
  const int64_t ld = in_smem ? (cw | 1) : m;
  if (in_smem)
    for (int j = w; j < nbb; j += B_WARPS)
      for (int c = lane; c < nloc; c += 32) A[j * ld + c] = Wg[static_cast<int64_t>(j) * m + c];
  auto sync_all = [&]() {
    if constexpr (C > 1) cg::this_cluster().sync();
    else __syncthreads();
  };
  sync_all();   // the columns are in place and every CTA has started
  const int g = lane >> 3, p = lane & 7;   // this lane's row of the warp's four, and its peer
  const int jg = w + 8 * g;
  for (int i = 0; i < nbb; ++i) {
    const int slot = i & 1, c0 = rank == 0 ? i + 1 : 0;
    const double* ai = A + i * ld;
    // a_i . a_j over this CTA's columns right of the pivot, rows j >= i
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    int tlo = 0;   // the warp's first row >= i
    while (tlo < 4 && w + 8 * tlo < i) ++tlo;
    for (int c = c0 + lane; c < nloc; c += 32) {
      const double x = ai[c];
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t >= tlo && w + 8 * t < nbb) acc[t] = fma(A[(w + 8 * t) * ld + c], x, acc[t]);
    }
    const double sum = reduce_scatter4(acc);
    if (jg >= i && jg < nbb && p < C) {
      double* dp = &part[slot][rank][jg];
      double* da = &alph[slot][jg];
      if constexpr (C > 1) {
        dp = cg::this_cluster().map_shared_rank(dp, p);
        da = cg::this_cluster().map_shared_rank(da, p);
      }
      *dp = sum;
      if (rank == 0) *da = A[jg * ld + i];
    }
    sync_all();
    // totals of this lane's row (fixed order over the ranks' eight slots)
    double s = 0.0, al = 0.0;
    if (jg >= i && jg < nbb) {
      if (p < C) s = part[slot][p][jg];
      al = alph[slot][jg];
    }
    if constexpr (C > 1) {
#pragma unroll
      for (int o = C / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    s = __shfl_sync(0xffffffffu, s, lane & 24);
    if (w == (i & 7)) {   // the warp of row i: lanes 0 and 1 the two quotients
      const double si = __shfl_sync(0xffffffffu, s, 8 * (i >> 3));
      const double ali = __shfl_sync(0xffffffffu, al, 8 * (i >> 3));
      double q = 0.0, beta = ali;
      if (si != 0.0) {
        beta = -copysign(fp_sqrt(fma(ali, ali, si)), ali);
        q = fp_div(lane == 0 ? beta - ali : 1.0, lane == 0 ? beta : ali - beta);
      }
      if (lane < 2) {
        sh[lane] = q;
        if (lane == 0) tq[i] = q;
        else sc[i] = q;
      }
      if (rank == 0 && lane == 0) A[i * ld + i] = beta;
    }
    __syncthreads();
    const double tau = sh[0], scal = sh[1];
    const double upd = tau * fma(scal, s, al);   // tau (v . row)
    const double coef = -(upd * scal);
    if (rank == 0 && jg > i && jg < nbb && p == 0) A[jg * ld + i] = al - upd;
    double cf[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) cf[t] = __shfl_sync(0xffffffffu, coef, 8 * t);
    int ulo = 0;   // the warp's first row > i
    while (ulo < 4 && w + 8 * ulo <= i) ++ulo;
    for (int c = c0 + lane; c < nloc; c += 32) {
      const double x = ai[c];
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t >= ulo && w + 8 * t < nbb) {
          double* a = A + (w + 8 * t) * ld + c;
          *a = fma(cf[t], x, *a);
        }
    }
    __syncthreads();
  }
  // L's entries of these rows go to W, the reflectors (0, 1, v) to hv and A
  if (rank == 0 && tid < nbb) it.tau[it.i0 + tid] = tq[tid];
  for (int j = w; j < nbb; j += B_WARPS) {
    double* hv = it.hv + static_cast<int64_t>(it.i0 + j) * m + it.i0 + rank * cw;
    const double scal = sc[j];
    for (int c = lane; c < nloc; c += 32) {
      const int gc = rank * cw + c;
      double v = A[j * ld + c];
      if (gc <= j) {
        Wg[static_cast<int64_t>(j) * m + c] = v;
        v = gc == j ? 1.0 : 0.0;
      } else {
        v *= scal;
      }
      hv[c] = v;
      if (in_smem) A[j * ld + c] = v;
    }
  }
  __syncthreads();
  // strict upper triangle of V V^T: a thread per pair (a < b), this CTA's
  // columns; to rank 0
  const double* Vl = in_smem ? A : it.hv + static_cast<int64_t>(it.i0) * m + it.i0 + rank * cw;
  const int npair = nbb * (nbb - 1) / 2;
  for (int e = tid; e < npair; e += B_THREADS) {
    int b = static_cast<int>((1.0f + sqrtf(1.0f + 8.0f * e)) * 0.5f);
    while (b * (b - 1) / 2 > e) --b;
    while (b * (b + 1) / 2 <= e) ++b;
    const int a = e - b * (b - 1) / 2;
    const double* va = Vl + a * ld;
    const double* vb = Vl + b * ld;
    double s0 = 0.0, s1 = 0.0;
    int c = 0;
    for (; c + 1 < nloc; c += 2) {
      s0 = fma(va[c], vb[c], s0);
      s1 = fma(va[c + 1], vb[c + 1], s1);
    }
    if (c < nloc) s0 = fma(va[c], vb[c], s0);
    double* d = &gp[rank][e];
    if constexpr (C > 1) d = cg::this_cluster().map_shared_rank(d, 0);
    *d = s0 + s1;
  }
  sync_all();
  if (rank != 0) return;   // (rank 0 reads its own shared memory only)
  for (int e = tid; e < npair; e += B_THREADS) {
    int b = static_cast<int>((1.0f + sqrtf(1.0f + 8.0f * e)) * 0.5f);
    while (b * (b - 1) / 2 > e) --b;
    while (b * (b + 1) / 2 <= e) ++b;
    const int a = e - b * (b - 1) / 2;
    double s = gp[0][e];
#pragma unroll
    for (int r = 1; r < C; ++r) s += gp[r][e];
    Mu[a][b] = s * tq[b];
  }
  __syncthreads();
  // X = (I + U D)^{-1}: lane = column, warp w keeps rows w + 8 t
  double x[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) x[t] = (w + 8 * t == lane) ? 1.0 : 0.0;
  for (int l = nbb - 1; l >= 0; --l) {
    if (w == (l & 7)) {
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t == (l >> 3)) xl[l][lane] = x[t];
    }
    __syncthreads();
    const double xv = xl[l][lane];
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (w + 8 * t < l) x[t] = fma(-Mu[w + 8 * t][l], xv, x[t]);
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int a = w + 8 * t;
    it.T[a * NB + lane] = (a < nbb && lane < nbb) ? tq[a] * x[t] : 0.0;
  }
}

// Rows [0, rows) of R (ld ldr, wid columns) <- R - ((R V^T) T) V with V nbb x
// wid (ld ldv), T NB x NB upper triangular: one CTA per 8 NR rows.
struct UpdItem {
  double* R;
  const double* V;
  const double* T;
  int64_t ldr, ldv;
  int rows, wid, nbb;
};

constexpr int UK = 64, UP = UK + 1;   // columns per stage, pitch in shared memory

template <int BYTES>
__device__ __forceinline__ void u_cp(void* dst, const void* src) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES));
}

// Both products of a row block in one pass, so that the panel's update of W
// and Vhat^T is one launch (it was six GEMM launches a panel, three of them
// with a few CTAs: g = V Vhat has 32 rows).  Warp w keeps rows w, w + 8, ...;
// a lane is a row of V in the first product, two columns of a stage in the
// second, so that no lane of an FP64 instruction is idle whatever NR is.
// The next stage of R and V is on its way while the current one is multiplied.
// Bound: FP64 FMAs, and how evenly the row blocks fall on the SMs: 31 GFLOP of
// updates in the factorization of a Schur complement of n = 10,000 took 95 ms
// as GEMMs, 39 ms by blocks of 32 rows (200 blocks on 152 SMs take as long as
// 304), and take 30 ms by blocks of 8 to 32 (see launch_updates).  A row's
// sums run in the order of its columns, whatever its block.
template <int NR>
__global__ void __launch_bounds__(B_THREADS)
lq_update_kernel(const UpdItem* __restrict__ items, const int2* __restrict__ map) {
  constexpr int BR = 8 * NR;
  extern __shared__ double usm[];
  double* Rs = usm;                    // [2][BR][UP]
  double* Vs = Rs + 2 * BR * UP;       // [2][32][UP]
  __shared__ double Ys[BR][NB + 1];
  __shared__ double Y2[BR][NB + 1];
  __shared__ double Ts[NB][NB + 1];
  const int2 tm = map[blockIdx.x];
  const UpdItem it = items[tm.x];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int r0 = tm.y * BR, rows = min(BR, it.rows - r0), wid = it.wid, nbb = it.nbb;
  double* R = it.R + static_cast<int64_t>(r0) * it.ldr;
  const int nst = (wid + UK - 1) / UK;
  const int na = (rows + 7) / 8;   // rows w + 8 a, a >= na, have no work in any warp
  auto load_rows = [&](double* dst, const double* src, int64_t ld, int nr, int nall, int c0) {
    for (int e = tid; e < nall * UK; e += B_THREADS) {
      const int r = e / UK, c = e - r * UK;
      if (r < nr && c0 + c < wid) u_cp<8>(dst + r * UP + c, src + r * ld + c0 + c);
      else dst[r * UP + c] = 0.0;
    }
  };
  for (int e = tid; e < NB * NB; e += B_THREADS) Ts[e / NB][e % NB] = it.T[e];
  load_rows(Rs, R, it.ldr, rows, BR, 0);
  load_rows(Vs, it.V, it.ldv, nbb, NB, 0);
  asm volatile("cp.async.commit_group;");
  double y[NR];
#pragma unroll
  for (int a = 0; a < NR; ++a) y[a] = 0.0;
  for (int k = 0; k < nst; ++k) {
    const int b = k & 1;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (k + 1 < nst) {
      load_rows(Rs + (b ^ 1) * BR * UP, R, it.ldr, rows, BR, (k + 1) * UK);
      load_rows(Vs + (b ^ 1) * NB * UP, it.V, it.ldv, nbb, NB, (k + 1) * UK);
      asm volatile("cp.async.commit_group;");
    }
    const double* rs = Rs + b * BR * UP + w * UP;
    const double* vs = Vs + b * NB * UP + lane * UP;
    const int lim = min(UK, wid - k * UK);
    if (na == NR) {
#pragma unroll 4
      for (int c = 0; c < lim; ++c) {
        const double v = vs[c];
#pragma unroll
        for (int a = 0; a < NR; ++a) y[a] = fma(rs[8 * a * UP + c], v, y[a]);
      }
    } else {
#pragma unroll 4
      for (int c = 0; c < lim; ++c) {
        const double v = vs[c];
#pragma unroll
        for (int a = 0; a + 1 < NR; ++a)
          if (a < na) y[a] = fma(rs[8 * a * UP + c], v, y[a]);
      }
    }
  }
  __syncthreads();
  // V's first stage again, for the second product
  load_rows(Vs, it.V, it.ldv, nbb, NB, 0);
  asm volatile("cp.async.commit_group;");
#pragma unroll
  for (int a = 0; a < NR; ++a) Ys[w + 8 * a][lane] = y[a];
  __syncthreads();
  {   // Y T: warp w has columns 4 w .. 4 w + 3, whose T ends at row 4 w + 3; the
      // lanes are the block's rows, times two or four groups of columns when
      // there are few
    constexpr int G = NR == 1 ? 4 : NR == 2 ? 2 : 1, CG = 4 / G;
    const int row = G == 1 ? min(lane, BR - 1) : lane & (BR - 1);
    const int c0 = 4 * w + (G == 1 ? 0 : lane / BR * CG);
    double z[CG];
#pragma unroll
    for (int q = 0; q < CG; ++q) z[q] = 0.0;
    for (int l = 0; l < 4 * w + 4; ++l) {
      const double v = Ys[row][l];
#pragma unroll
      for (int q = 0; q < CG; ++q) z[q] = fma(v, Ts[l][c0 + q], z[q]);
    }
    if (G > 1 || lane < BR)
#pragma unroll
      for (int q = 0; q < CG; ++q) Y2[row][c0 + q] = z[q];
  }
  for (int k = 0; k < nst; ++k) {
    const int b = k & 1;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (k + 1 < nst) {
      load_rows(Vs + (b ^ 1) * NB * UP, it.V, it.ldv, nbb, NB, (k + 1) * UK);
      asm volatile("cp.async.commit_group;");
    }
    const double* vs = Vs + b * NB * UP + lane;
    double o[NR][2];
#pragma unroll
    for (int a = 0; a < NR; ++a)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int r = w + 8 * a, c = k * UK + lane + 32 * q;
        o[a][q] = (r < rows && c < wid) ? R[r * it.ldr + c] : 0.0;
      }
    // (columns past wid add zeros; a block of 32 columns past it is skipped)
    const bool two = wid - k * UK > 32;
    if (two && na == NR) {
#pragma unroll 4
      for (int l = 0; l < nbb; ++l) {
        const double v0 = vs[l * UP], v1 = vs[l * UP + 32];
#pragma unroll
        for (int a = 0; a < NR; ++a) {
          const double f = -Y2[w + 8 * a][l];
          o[a][0] = fma(f, v0, o[a][0]);
          o[a][1] = fma(f, v1, o[a][1]);
        }
      }
    } else
#pragma unroll 4
    for (int l = 0; l < nbb; ++l) {
      const double v0 = vs[l * UP], v1 = vs[l * UP + 32];
#pragma unroll
      for (int a = 0; a < NR; ++a)
        if (a < na) {
          const double f = -Y2[w + 8 * a][l];
          o[a][0] = fma(f, v0, o[a][0]);
          if (two) o[a][1] = fma(f, v1, o[a][1]);
        }
    }
#pragma unroll
    for (int a = 0; a < NR; ++a)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int r = w + 8 * a, c = k * UK + lane + 32 * q;
        if (r < rows && c < wid) R[r * it.ldr + c] = o[a][q];
      }
  }
}

struct LuPanel {
  double* A;        // m x m
  int32_t* piv;
  int32_t* status;
  int m, j0, nbb;
};

constexpr int LU_PITCH = NB + 1;

// columns [j0, j0 + nbb): partial pivoting (largest |a|, lowest row on ties),
// column scaling and rank-1 updates inside the panel, then whole-row swaps of
// the other columns, by a cluster of C CTAs that split the rows.  A thread
// owns a row (of every 256).  Before a step's one cluster barrier each CTA
// sends its best candidate -- value, row, reciprocal and the row itself -- to
// its peers, and rank 0 the row to be swapped out; after it every thread knows
// the pivot row and updates its own row, and takes the next column's absolute
// value on the way.  (The multipliers scale by the pivot's reciprocal, as
// LAPACK's xGETF2 does for a pivot above the underflow threshold.)
// Bound: the step's latency, about 2 us; one CTA on global memory took 0.8 ms
// a panel at m = 1383 against 0.15 ms.
template <int C>
__global__ void __launch_bounds__(B_THREADS) lu_panel_kernel(const LuPanel* items, int in_smem) {
  extern __shared__ double Asm[];
  __shared__ long long cv[2][C];          // candidate |value| bits, -1: none
  __shared__ int ci[2][C];
  __shared__ double cr[2][C];             // 1 / candidate
  __shared__ double crow[2][C][NB];       // the candidate's row
  __shared__ double drow[2][NB];          // row j
  __shared__ long long wv[B_WARPS];
  __shared__ int wi[B_WARPS];
  __shared__ int pivs[NB];
  __shared__ int src[2 * NB], dst[2 * NB], nmove;
  const LuPanel it = items[blockIdx.x / C];
  const int m = it.m, j0 = it.j0, nbb = it.nbb;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  int rank = 0;
  if constexpr (C > 1) rank = static_cast<int>(cg::this_cluster().block_rank());
  const int hgt = m - j0, rw = lq_cols(hgt, C);   // rows per CTA (at least NB)
  const int nloc = max(0, min(rw, hgt - rank * rw));
  const int row0 = rank * rw;                     // local row 0 is panel row row0
  double* Ag = it.A + static_cast<int64_t>(j0 + row0) * m + j0;
  double* A = in_smem ? Asm : Ag;
  const int64_t ld = in_smem ? LU_PITCH : m;
  if (in_smem)
    for (int r = w; r < nloc; r += B_WARPS)
      if (lane < nbb) A[r * ld + lane] = Ag[static_cast<int64_t>(r) * m + lane];
  auto sync_all = [&]() {
    if constexpr (C > 1) cg::this_cluster().sync();
    else __syncthreads();
  };
  sync_all();
  long long bv = -1;
  int bi = INT_MAX;
  auto consider = [&](int r, int j) {   // row r (local) as the candidate of column j
    const long long v = __double_as_longlong(fabs(A[r * ld + j]));
    if (v > bv) {   // a thread's rows come in increasing order: lowest index on ties
      bv = v;
      bi = row0 + r;
    }
  };
  for (int r = tid; r < nloc; r += B_THREADS) consider(r, 0);
  for (int j = 0; j < nbb; ++j) {
    const int slot = j & 1;
    // this CTA's candidate
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > bv || (ov == bv && oi < bi)) {
        bv = ov;
        bi = oi;
      }
    }
    if (lane == 0) {
      wv[w] = bv;
      wi[w] = bi;
    }
    __syncthreads();
    if (w == 0) {
      bv = lane < B_WARPS ? wv[lane] : -1;
      bi = lane < B_WARPS ? wi[lane] : INT_MAX;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) {
          bv = ov;
          bi = oi;
        }
      }
      bv = __shfl_sync(0xffffffffu, bv, 0);
      bi = __shfl_sync(0xffffffffu, bi, 0);
      const bool have = bv >= 0;
      const double* cand = A + static_cast<int64_t>(have ? bi - row0 : 0) * ld;
      const double rc = have && lane == 0 ? 1.0 / cand[j] : 0.0;
      const double x = have && lane < nbb ? cand[lane] : 0.0;
      const double dj = rank == 0 && lane < nbb ? A[j * ld + lane] : 0.0;
#pragma unroll
      for (int p = 0; p < C; ++p) {
        long long* pv = &cv[slot][rank];
        int* pi = &ci[slot][rank];
        double* pr = &cr[slot][rank];
        double* px = &crow[slot][rank][0];
        double* pd = &drow[slot][0];
        if constexpr (C > 1) {
          pv = cg::this_cluster().map_shared_rank(pv, p);
          pi = cg::this_cluster().map_shared_rank(pi, p);
          pr = cg::this_cluster().map_shared_rank(pr, p);
          px = cg::this_cluster().map_shared_rank(px, p);
          pd = cg::this_cluster().map_shared_rank(pd, p);
        }
        if (lane == 0) {
          *pv = bv;
          *pi = bi;
          *pr = rc;
        }
        px[lane] = x;
        if (rank == 0) pd[lane] = dj;
      }
    }
    sync_all();
    int win = 0;
#pragma unroll
    for (int r = 1; r < C; ++r)
      if (cv[slot][r] > cv[slot][win] ||
          (cv[slot][r] == cv[slot][win] && ci[slot][r] < ci[slot][win]))
        win = r;
    // a zero column, or a NaN in it, whose bits are above every number's (the same
    // decision on every CTA)
    if (cv[slot][win] <= 0 || cv[slot][win] > __double_as_longlong(INFINITY)) {
      if (rank == 0 && tid == 0) *it.status = HSS_ERR_SINGULAR;
      sync_all();   // no CTA leaves while a peer may still write to it
      return;
    }
    const int prow_i = ci[slot][win];
    const double* prow = crow[slot][win];
    const double pv = prow[j], rpv = cr[slot][win];
    const bool scale = fabs(pv) >= DBL_MIN;
    if (tid == 0) pivs[j] = prow_i;
    bv = -1;
    bi = INT_MAX;
    for (int r = tid; r < nloc; r += B_THREADS) {
      const int gr = row0 + r;
      if (gr < j) continue;
      double* a = A + r * ld;
      if (gr == j) {   // row j becomes the pivot row
        for (int c = 0; c < nbb; ++c) a[c] = prow[c];
        continue;
      }
      if (gr == prow_i)   // the pivot's old row takes row j
        for (int c = 0; c < nbb; ++c) a[c] = drow[slot][c];
      const double l = scale ? a[j] * rpv : a[j] / pv;
      a[j] = l;
      for (int c = j + 1; c < nbb; ++c) a[c] = fma(-l, prow[c], a[c]);
      if (j + 1 < nbb) consider(r, j + 1);
    }
    // (a row is read by warp 0 of the next step only after its block barrier)
  }
  __syncthreads();
  if (in_smem)
    for (int r = w; r < nloc; r += B_WARPS)
      if (lane < nbb) Ag[static_cast<int64_t>(r) * m + lane] = A[r * ld + lane];
  // the swaps of this panel as one permutation of at most 2 nbb rows: entry
  // q < nbb is row q, the others are the pivots' rows below (lane q holds
  // entries q and nbb + q)
  if (w == 0) {
    int s0 = lane, d1 = -1, s1 = -1, n1 = 0;
    for (int j = 0; j < nbb; ++j) {
      const int p = pivs[j];
      if (p == j) continue;
      const int a = __shfl_sync(0xffffffffu, s0, j);
      if (p < nbb) {
        const int b = __shfl_sync(0xffffffffu, s0, p);
        if (lane == j) s0 = b;
        if (lane == p) s0 = a;
      } else {
        const unsigned hit = __ballot_sync(0xffffffffu, d1 == p);
        const int q = hit ? __ffs(hit) - 1 : n1++;
        if (!hit && lane == q) d1 = s1 = p;
        const int b = __shfl_sync(0xffffffffu, s1, q);
        if (lane == q) s1 = a;
        if (lane == j) s0 = b;
      }
    }
    if (lane < nbb) {
      dst[lane] = lane;
      src[lane] = s0;
    }
    if (lane < n1) {
      dst[nbb + lane] = d1;
      src[nbb + lane] = s1;
    }
    if (lane == 0) nmove = nbb + n1;
  }
  if (rank == 0 && tid < nbb) it.piv[j0 + tid] = j0 + pivs[tid];
  __syncthreads();
  const int n = nmove;
  for (int c = rank * B_THREADS + tid; c < m - nbb; c += C * B_THREADS) {
    double* col = it.A + static_cast<int64_t>(j0) * m + (c < j0 ? c : c + nbb);
    double v[2 * NB];
#pragma unroll
    for (int q = 0; q < 2 * NB; ++q)
      if (q < n) v[q] = col[static_cast<int64_t>(src[q]) * m];
#pragma unroll
    for (int q = 0; q < 2 * NB; ++q)
      if (q < n) col[static_cast<int64_t>(dst[q]) * m] = v[q];
  }
}

// U12 = L11^{-1} A12 of a batch of panels (one per blockIdx.y) by substitution:
// 16 columns a CTA, thread = (column, rows t and t + 16); row b goes through
// shared memory to the rows below it.  (A thread per column has a chain of 496
// FMAs; with the inverse of L11 the rows are independent, but the error grows
// with L11's condition.)
__global__ void __launch_bounds__(B_THREADS) lu_u12_kernel(const LuPanel* items) {
  __shared__ double L[NB][NB + 1];
  __shared__ double x[NB][17];
  const LuPanel it = items[blockIdx.y];
  const int c0 = it.j0 + it.nbb + blockIdx.x * 16;
  if (c0 >= it.m) return;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, c = c0 + tx;
  double* A = it.A + static_cast<int64_t>(it.j0) * it.m;
  for (int e = tid; e < it.nbb * NB; e += B_THREADS)
    if (e % NB < it.nbb) L[e / NB][e % NB] = A[static_cast<int64_t>(e / NB) * it.m + it.j0 + e % NB];
  double v[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int r = ty + 16 * a;
    v[a] = (r < it.nbb && c < it.m) ? A[static_cast<int64_t>(r) * it.m + c] : 0.0;
  }
  for (int b = 0; b < it.nbb; ++b) {
    if (ty == (b & 15)) x[b][tx] = b < 16 ? v[0] : v[1];
    __syncthreads();
    const double xb = x[b][tx];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const int r = ty + 16 * a;
      if (r > b && r < it.nbb) v[a] = fma(-L[r][b], xb, v[a]);
    }
  }
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int r = ty + 16 * a;
    if (r < it.nbb && c < it.m) A[static_cast<int64_t>(r) * it.m + c] = v[a];
  }
}

template <typename TI>
Err upload(const std::vector<TI>& v, cudaStream_t s, Arena& ar, TI** out) {
  HSS_TRY(ar.alloc_t(out, std::max<size_t>(v.size(), 1), s));
  return ar.upload(*out, v.data(), v.size() * sizeof(TI), s);
}

Err launch_copies(const std::vector<CopyItem>& items, cudaStream_t s, Arena& ar) {
  std::vector<CopyItem> live;
  std::vector<int64_t> start;
  int64_t total = 0;
  for (const CopyItem& c : items) {
    if (c.rows <= 0 || c.cols <= 0) continue;
    live.push_back(c);
    start.push_back(total);
    total += static_cast<int64_t>(c.rows) * c.cols;
  }
  if (live.empty()) return ok();
  CopyItem* di = nullptr;
  int64_t* ds = nullptr;
  HSS_TRY(upload(live, s, ar, &di));
  HSS_TRY(upload(start, s, ar, &ds));
  copy_items_kernel<<<static_cast<unsigned>((total + 255) / 256), 256, 0, s>>>(
      di, ds, static_cast<int>(live.size()), total);
  return check_launch("copy_items_kernel");
}

GemmItem<double> gemm(double* out, int64_t ldo, int rows, int cols, int inner, const double* M,
                      int64_t ldm, int m_trans, const double* Z, int64_t ldz, int z_trans,
                      const double* X, int64_t ldx, double sign) {
  GemmItem<double> g{};
  g.out = out;
  g.ldo = ldo;
  g.rows = rows;
  g.inner = inner;
  g.c0 = 0;
  g.c1 = cols;
  g.M = M;
  g.ldm = ldm;
  g.m_trans = m_trans;
  g.m_is_f64 = 1;
  g.Z.p0 = Z;
  g.Z.ld0 = ldz;
  g.z_trans = z_trans;
  if (X) {
    g.X.p0 = X;
    g.X.ld0 = ldx;
  }
  g.sign = sign;
  return g;
}

Err run_gemms(const std::vector<GemmItem<double>>& v, cudaStream_t s, Arena& ar) {
  std::vector<GemmItem<double>> live;
  for (const auto& g : v)
    if (g.rows > 0 && g.c1 > g.c0) live.push_back(g);
  if (live.empty()) return ok();
  return launch_gemm_batched<double>(live, s, nullptr, 0, &ar, true);
}

}  // namespace

// Nodes of this order or more are factored here: one CTA per node spends its
// time on dependent FP64 operations and on one SM's two multiply-adds a clock.
// Factor times in ms with the line at 32 / 64 / 96 / 160 rows: Toeplitz
// n = 2000 2.11 / 1.70 / 1.71 / 3.28, n = 80,000 12.2 / 12.2 / 13.4 / 14.9,
// Gaussian kernel n = 20,000 13.9 / 14.0 / 14.9 / 20.3 (3.3, 29.3 and 48.0
// with one CTA per node below 320 and the panels on one CTA).
size_t ulv_factor_big_min_m() { return 64; }

namespace {

// Launches a panel kernel on the items of each cluster size (a function of
// the node's order alone).  doubles(item, C): the panel part of one CTA;
// extra(C): doubles it needs besides.
template <typename Item, typename F, typename G>
Err launch_panels(const std::vector<Item>& all, void (*const kern[4])(const Item*, int), F doubles,
                  G extra, cudaStream_t s, Arena& ar, const char* what) {
  if (all.empty()) return ok();
  std::vector<Item> sorted;
  struct Group {
    int first, count, lg, in_smem;
    size_t smem;
  };
  std::vector<Group> groups;
  for (int lg = 0; lg < 4; ++lg)
    for (int big = 0; big < 2; ++big) {
      const int C = 1 << lg;
      Group g{(int)sorted.size(), 0, lg, big ? 0 : 1, sizeof(double) * extra(C)};
      for (const Item& x : all) {
        if (panel_ctas(x.m) != C) continue;
        const size_t need = sizeof(double) * (doubles(x, C) + extra(C));
        if ((need > PANEL_SMEM_CAP) != (big != 0)) continue;
        if (!big) g.smem = std::max(g.smem, need);
        sorted.push_back(x);
        ++g.count;
      }
      if (g.count) groups.push_back(g);
    }
  Item* dev = nullptr;
  HSS_TRY(upload(sorted, s, ar, &dev));
  for (const Group& g : groups) {
    HSS_CUDA_TRY(cudaFuncSetAttribute(kern[g.lg], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)PANEL_SMEM_CAP));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(g.count << g.lg), 1, 1);
    cfg.blockDim = dim3(B_THREADS, 1, 1);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << g.lg;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g.lg ? 1 : 0;
    const cudaError_t le = cudaLaunchKernelEx(&cfg, kern[g.lg], (const Item*)(dev + g.first), g.in_smem);
    if (le != cudaSuccess) {
      cudaGetLastError();
      return fail(HSS_ERR_CUDA, std::string(what) + " launch: " + cudaGetErrorString(le));
    }
    HSS_TRY(check_launch(what));
  }
  return ok();
}

// Rows per block: 8, 16, 24 or 32, whichever lets the launch end first with its
// blocks handed to the SMs as they become free (longest first).  A block costs
// its width times its rows, in eights, and 0.06 of its width for what does not
// shrink with the rows (V's stages, barriers); if some SM gets a second block,
// half of the longest on top (blocks resident together end together, so the
// rounds are coarser than that).  With eight blocks of 32 rows or more per SM
// the last round no longer matters.
Err launch_updates(const std::vector<UpdItem>& items, cudaStream_t s, Arena& ar) {
  std::vector<UpdItem> live;
  for (const UpdItem& u : items)
    if (u.rows > 0) live.push_back(u);
  if (live.empty()) return ok();
  std::stable_sort(live.begin(), live.end(),
                   [](const UpdItem& a, const UpdItem& b) { return a.wid > b.wid; });
  int dev = 0, sms = 0;
  HSS_CUDA_TRY(cudaGetDevice(&dev));
  HSS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  int64_t rows32 = 0;
  for (const UpdItem& u : live) rows32 += (u.rows + 31) / 32;
  int best = 4;
  if (rows32 < 8 * sms) {
    double best_t = 0.0;
    std::vector<double> end;
    for (int nr = 4; nr >= 1; --nr) {
      end.assign(static_cast<size_t>(sms), 0.0);   // a heap: the SM free first on top
      double t = 0.0;
      int blocks = 0;
      for (const UpdItem& u : live)
        for (int r0 = 0; r0 < u.rows; r0 += 8 * nr, ++blocks) {
          std::pop_heap(end.begin(), end.end(), std::greater<double>());
          end.back() += u.wid * ((std::min(8 * nr, u.rows - r0) + 7) / 8 + 0.06);
          t = std::max(t, end.back());
          std::push_heap(end.begin(), end.end(), std::greater<double>());
        }
      if (blocks > sms) t += 0.5 * nr * live.front().wid;
      if (nr == 4 || t < best_t) {
        best = nr;
        best_t = t;
      }
    }
  }
  std::vector<int2> map;
  for (size_t q = 0; q < live.size(); ++q)
    for (int t = 0; t * 8 * best < live[q].rows; ++t) map.push_back(make_int2((int)q, t));
  UpdItem* di = nullptr;
  int2* dm = nullptr;
  HSS_TRY(upload(live, s, ar, &di));
  HSS_TRY(upload(map, s, ar, &dm));
  static void (*const kern[4])(const UpdItem*, const int2*) = {lq_update_kernel<1>, lq_update_kernel<2>,
                                                               lq_update_kernel<3>, lq_update_kernel<4>};
  const size_t smem = sizeof(double) * 2 * (NB + 8 * best) * UP;
  HSS_CUDA_TRY(cudaFuncSetAttribute(kern[best - 1], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem));
  kern[best - 1]<<<(unsigned)map.size(), B_THREADS, smem, s>>>(di, dm);
  return check_launch("lq_update_kernel");
}

Err launch_v_fill(const std::vector<VItem>& items, cudaStream_t s, Arena& ar) {
  std::vector<int64_t> start;
  int64_t total = 0;
  for (const VItem& v : items) {
    start.push_back(total);
    total += static_cast<int64_t>(v.mc) * v.kc;
  }
  if (total == 0) return ok();
  VItem* di = nullptr;
  int64_t* ds = nullptr;
  HSS_TRY(upload(items, s, ar, &di));
  HSS_TRY(upload(start, s, ar, &ds));
  v_fill_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(di, ds, (int)items.size(), total);
  return check_launch("v_fill_kernel");
}

}  // namespace

// Factor the nodes `items` ((handle, node) pairs of one level round of any
// number of handles; status[q] is item q's root-LU status slot): the nodes
// share every launch.
Err ulv_factor_big_multi(const std::vector<std::pair<hss_s*, int>>& items,
                         const std::vector<int32_t*>& status, cudaStream_t s) {
  if (items.empty()) return ok();
  Arena ar{(size_t)8 << 20};
  struct Node {
    hss_s* h;
    int id, m, k, r, kc, mc, leaf, root, f64in;
    int32_t* status;
    double *Dw, *W, *VhT, *Vd, *Tall;
  };
  std::vector<Node> N;
  for (size_t q = 0; q < items.size(); ++q) {
    hss_s* h = items[q].first;
    const int id = items[q].second;
    const TNode& nd = h->tree.nodes[id];
    UlvFactors& F = h->ulv;
    const UlvNode& u = F.nodes[id];
    const NodeGen& g = h->gen[id];
    Node x{};
    x.h = h;
    x.status = status[q];
    x.f64in = h->dtype == HSS_F64;
    x.id = id;
    x.m = u.m;
    x.root = id == 0;
    x.leaf = nd.c1 < 0;
    x.k = x.root ? 0 : u.k;
    x.r = x.m - x.k;
    x.kc = x.root ? 0 : u.kc;
    x.mc = x.root ? 0 : g.mc;
    const size_t mm = static_cast<size_t>(x.m) * x.m;
    if (x.root) {
      x.Dw = F.root_lu;
    } else {
      HSS_TRY(ar.alloc_t(&x.Dw, mm, s));
      HSS_TRY(ar.alloc_t(&x.W, mm, s));
      HSS_TRY(ar.alloc_t(&x.VhT, static_cast<size_t>(x.m) * std::max(x.kc, 1), s));
      if (!x.leaf)
        HSS_TRY(ar.alloc_t(&x.Vd, static_cast<size_t>(std::max(x.mc, 1)) * std::max(x.kc, 1), s));
      x.Tall = F.nodes[id].T;
    }
    N.push_back(x);
  }

  // ---- D_tau
  {
    std::vector<CopyItem> cp;
    std::vector<GemmItem<double>> gm;
    for (Node& x : N) {
      const TNode& nd = x.h->tree.nodes[x.id];
      const NodeGen& g = x.h->gen[x.id];
      if (x.leaf) {
        cp.push_back({g.D, x.m, x.f64in, x.Dw, x.m, x.m, x.m, nullptr, 0, 0});
        continue;
      }
      const UlvNode& a = x.h->ulv.nodes[nd.c1];
      const UlvNode& b = x.h->ulv.nodes[nd.c2];
      const int k1 = a.k, k2 = b.k;
      cp.push_back({a.Dtil, k1, 1, x.Dw, x.m, k1, k1, nullptr, 0, 0});
      cp.push_back({b.Dtil, k2, 1, x.Dw + static_cast<size_t>(k1) * x.m + k1, x.m, k2, k2, nullptr, 0, 0});
      // B12 Vtb_2^T and B21 Vtb_1^T (B in the handle's dtype)
      GemmItem<double> b12 =
          gemm(x.Dw + k1, x.m, k1, k2, b.kc, nullptr, b.kc, 0, b.Vtb, b.kc, 1, nullptr, 0, 1.0);
      GemmItem<double> b21 = gemm(x.Dw + static_cast<size_t>(k1) * x.m, x.m, k2, k1, a.kc, nullptr,
                                  a.kc, 0, a.Vtb, a.kc, 1, nullptr, 0, 1.0);
      b12.M = g.B12;
      b21.M = g.B21;
      b12.m_is_f64 = b21.m_is_f64 = x.f64in ? 1 : 2;
      gm.push_back(b12);
      gm.push_back(b21);
    }
    HSS_TRY(launch_copies(cp, s, ar));
    HSS_TRY(run_gemms(gm, s, ar));
  }

  // ---- roots: blocked LU with partial pivoting, the roots of all handles
  // side by side (panel j0 of every root in one launch, its row block in
  // one, the trailing updates in one; each root's operations and their
  // order are those it has alone)
  {
    int maxm = 0;
    for (const Node& x : N)
      if (x.root) maxm = std::max(maxm, x.m);
    for (int j0 = 0; j0 < maxm; j0 += NB) {
      std::vector<LuPanel> lp, lt;
      std::vector<GemmItem<double>> gm;
      int maxrest = 0;
      for (Node& x : N) {
        if (!x.root || j0 >= x.m) continue;
        const int m = x.m, nbb = std::min(NB, m - j0), rest = m - j0 - nbb;
        lp.push_back({x.Dw, x.h->ulv.root_piv, x.status, m, j0, nbb});
        if (rest <= 0) continue;
        lt.push_back(lp.back());
        maxrest = std::max(maxrest, rest);
        double* a22 = x.Dw + static_cast<size_t>(j0 + nbb) * m + j0 + nbb;
        gm.push_back(gemm(a22, m, rest, rest, nbb, x.Dw + static_cast<size_t>(j0 + nbb) * m + j0,
                          m, 0, x.Dw + static_cast<size_t>(j0) * m + j0 + nbb, m, 0, a22, m, -1.0));
      }
      if (lp.empty()) break;
      static void (*const kern[4])(const LuPanel*, int) = {lu_panel_kernel<1>, lu_panel_kernel<2>,
                                                           lu_panel_kernel<4>, lu_panel_kernel<8>};
      HSS_TRY(launch_panels(
          lp, kern,
          [](const LuPanel& p, int C) { return static_cast<size_t>(lq_cols(p.m - p.j0, C)) * LU_PITCH; },
          [](int) { return static_cast<size_t>(0); }, s, ar, "lu_panel_kernel"));
      if (lt.empty()) continue;
      LuPanel* dlt = nullptr;
      HSS_TRY(upload(lt, s, ar, &dlt));
      lu_u12_kernel<<<dim3(static_cast<unsigned>((maxrest + 15) / 16), static_cast<unsigned>(lt.size())),
                      B_THREADS, 0, s>>>(dlt);
      HSS_TRY(check_launch("lu_u12_kernel"));
      HSS_TRY(run_gemms(gm, s, ar));
    }
  }
  N.erase(std::remove_if(N.begin(), N.end(), [](const Node& x) { return x.root != 0; }), N.end());
  if (N.empty()) {
    ar.release(s);
    return ok();
  }

  // ---- Vhat^T = V^T (leaf) or V^T diag(Vtb_1, Vtb_2)^T, with V = Pi [I; E^c]
  {
    std::vector<VItem> vi;
    std::vector<GemmItem<double>> gm;
    for (Node& x : N) {
      if (x.kc == 0) continue;
      const TNode& nd = x.h->tree.nodes[x.id];
      const NodeGen& g = x.h->gen[x.id];
      if (x.leaf) {
        vi.push_back({x.VhT, x.m, g.permc, g.Ec, x.mc, x.kc, 1});
        continue;
      }
      vi.push_back({x.Vd, x.kc, g.permc, g.Ec, x.mc, x.kc, 0});
      const UlvNode& a = x.h->ulv.nodes[nd.c1];
      const UlvNode& b = x.h->ulv.nodes[nd.c2];
      gm.push_back(gemm(x.VhT, x.m, x.kc, a.k, a.kc, x.Vd, x.kc, 1, a.Vtb, a.kc, 1, nullptr, 0, 1.0));
      gm.push_back(gemm(x.VhT + a.k, x.m, x.kc, b.k, b.kc, x.Vd + static_cast<size_t>(a.kc) * x.kc,
                        x.kc, 1, b.Vtb, b.kc, 1, nullptr, 0, 1.0));
    }
    HSS_TRY(launch_v_fill(vi, s, ar));
    HSS_TRY(run_gemms(gm, s, ar));
  }

  // ---- W = Omega D_tau
  {
    std::vector<GemmItem<double>> gm;
    for (Node& x : N) {
      const NodeGen& g = x.h->gen[x.id];
      GemmItem<double> top = gemm(x.W, x.m, x.r, x.m, x.k, g.Er, x.k, 0, x.Dw, x.m, 0, x.Dw, x.m, -1.0);
      top.Z.map = g.permr;
      top.X.map = g.permr + x.k;
      gm.push_back(top);
      GemmItem<double> bot =
          gemm(x.W + static_cast<size_t>(x.r) * x.m, x.m, x.k, x.m, 0, nullptr, 1, 0, nullptr, 1, 0,
               x.Dw, x.m, 1.0);
      bot.X.map = g.permr;
      gm.push_back(bot);
    }
    HSS_TRY(run_gemms(gm, s, ar));
  }

  // ---- LQ of the top r rows in panels; W's trailing rows and Vhat^T follow
  int maxr = 0;
  for (Node& x : N) maxr = std::max(maxr, x.r);
  for (int i0 = 0; i0 < maxr; i0 += NB) {
    std::vector<LqPanel> lp;
    std::vector<UpdItem> up;
    for (Node& x : N) {
      if (i0 >= x.r) continue;
      const UlvNode& u = x.h->ulv.nodes[x.id];
      const int nbb = std::min(NB, x.r - i0), wid = x.m - i0;
      double* T = x.Tall + static_cast<size_t>(i0 / NB) * NB * NB;
      lp.push_back({x.W, u.hv, u.tau, T, x.m, i0, nbb});
      const double* vp = u.hv + static_cast<size_t>(i0) * x.m + i0;
      up.push_back({x.W + static_cast<size_t>(i0 + nbb) * x.m + i0, vp, T, x.m, x.m, wid - nbb, wid, nbb});
      if (x.kc) up.push_back({x.VhT + i0, vp, T, x.m, x.m, x.kc, wid, nbb});
    }
    static void (*const kern[4])(const LqPanel*, int) = {lq_panel_kernel<1>, lq_panel_kernel<2>,
                                                         lq_panel_kernel<4>, lq_panel_kernel<8>};
    HSS_TRY(launch_panels(
        lp, kern,
        [](const LqPanel& p, int C) { return static_cast<size_t>(NB) * (lq_cols(p.m - p.i0, C) | 1); },
        [](int C) { return static_cast<size_t>(C) * (NB * (NB - 1) / 2); }, s, ar, "lq_panel_kernel"));
    HSS_TRY(launch_updates(up, s, ar));
  }

  // ---- L, W_b Q_t^T, Dtil, Vtilde
  {
    std::vector<CopyItem> cp;
    for (Node& x : N) {
      const UlvNode& u = x.h->ulv.nodes[x.id];
      cp.push_back({x.W, x.m, 1, u.L, x.r, x.r, x.r, nullptr, 1, 0});
      cp.push_back({x.W + static_cast<size_t>(x.r) * x.m, x.m, 1, u.WbQt, x.r, x.k, x.r, nullptr, 0, 0});
      cp.push_back({x.W + static_cast<size_t>(x.r) * x.m + x.r, x.m, 1, u.Dtil, x.k, x.k, x.k,
                    nullptr, 0, 0});
      if (x.kc == 0) continue;
      cp.push_back({x.VhT, x.m, 1, u.Vtt, x.kc, x.r, x.kc, nullptr, 0, 1});
      cp.push_back({x.VhT + x.r, x.m, 1, u.Vtb, x.kc, x.k, x.kc, nullptr, 0, 1});
    }
    HSS_TRY(launch_copies(cp, s, ar));
  }
  ar.release(s);
  return ok();
}

}  // namespace hss
