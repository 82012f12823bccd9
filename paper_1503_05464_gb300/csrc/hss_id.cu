// Batched interpolative decomposition [X, J] = ID(Y, eps) by truncated
// column-pivoted Householder QR in FP64 (Section 2.2; Section 3.1: the QR
// with column pivoting stops as soon as |R_ii| <= eps |R_11|).
//
// One thread-block cluster of C CTAs (C = 1..16, one SM each) factors one Y.
// Y is d x m and is stored transposed: its column j is the contiguous row j
// of the input.  Column j belongs to CTA j % C, which keeps it in its shared
// memory (or, for matrices too large for the cluster's shared memory, in a
// global work copy) together with its residual norm.  One cluster barrier per
// elimination step:
//   1. before the barrier every CTA pushes its candidate (largest residual
//      norm among its active columns, lowest index on ties) into every CTA's
//      shared memory, with the Householder reflector that the candidate
//      column would give: sigma, tau and the scale of v, from the column's
//      exact residual (the entry at the next pivot row and the sum of squares
//      below it in a fixed order);
//   2. after the barrier every CTA picks the same pivot from the C local
//      candidates, reads |R_ii| = sigma, takes the stopping decision against
//      max(rtol |R_11|, atol), and copies and scales the pivot column from the
//      owner -- so no CTA waits for the owner, and all agree bitwise;
//   3. every CTA applies the reflector to its active columns (a team of
//      threads per column: dot product, fixed-order reduction, update), then
//      downdates their norms with one lane per column -- recomputing a norm
//      when cancellation makes the downdate inaccurate (LAPACK xGEQP3's
//      safeguard, threshold sqrt(eps)) -- and pushes its next candidate into
//      the other of two slots (a CTA can be at most one step ahead of
//      another, so the slot being read is never the one being written).
// Columns never move and a pivot column is never written after it is chosen
// (its R_ii is kept aside), so peers can read it while its owner goes on.
// perm[0..k) records the pivot order, the remaining columns follow in
// increasing index order.  The pivot columns' R entries go to a global k x k
// buffer, and each CTA solves T = R1^{-1} R2 for the remaining columns it owns
// (column-oriented back substitution by blocks of 16 rows), writing E = T^T
// so that the generator is Pi [I; E].
//
// Group mode: when a launch holds a few large items (a CTA's share of one
// step is long), each item instead gets floor(SMs / items) CTAs of one
// cooperative launch, so that every SM works.  They keep their columns in the
// global work copy, exchange candidates through global memory and meet at a
// bounded barrier in global memory (a counter per item); each column's
// arithmetic is that of the cluster mode, so the bits do not depend on the
// number of CTAs.
//
// What bounds it: the chain of one step.  At 16 columns or so per CTA a step
// takes 12600 cycles (n = 20000, m 150-340): the barrier 800, the pick and the
// pivot column 1000-1500, the columns' pass 4000-5000, the downdates 1700 and
// the candidate with its reflector 3800 -- forming the reflector before the
// barrier (once, not in every CTA after it), integer arg-max reductions and
// the integer root and quotient took that compression (all of it) from 17.2 to
// 16.0 ms; large items (n = 60000, m to 4700) are bound by the FP64 pipe in
// the pass: the registers kept under 128, so that two CTAs fit an SM, took
// that compression from 1451 to 1299 ms.
#include "hss_internal.cuh"
#include "hss_fp.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <array>
#include <cfloat>
#include <climits>
#include <cstdlib>
#include <map>
#include <mutex>
#include <cstddef>
#include <tuple>

namespace cg = cooperative_groups;

namespace hss {

namespace {

constexpr int ID_THREADS = 256;
constexpr int ID_WARPS = ID_THREADS / 32;
constexpr size_t ID_SMEM_CAP = 200 * 1024;   // shared-memory budget per CTA

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Doubles of a block of the back substitution (16 x 17 entries of R1 and 4 x 32
// of T), which takes the place of the candidate's column, or where that is
// shorter of the columns' limits and downdates (3 mloc doubles), and gets
// doubles of its own only where both are short: with few samples the number of
// columns a CTA can hold must not fall for it
constexpr int ID_BS = 16, ID_BLK = ID_BS * (ID_BS + 1) + 128;
__host__ __device__ inline int id_cbuf(int d, int mloc) {
  return d < ID_BLK && 3 * mloc < ID_BLK ? ID_BLK : d;
}

// Residual norms are >= 0 and inactive columns carry -1: as 64-bit integers
// their bit patterns order the same way (the sign bit makes -1 negative), so
// the arg-max runs on the integer pipes instead of the narrow FP64 one.
// Three integer reductions (high word, low word, index) take a third of the
// time of five shuffle rounds.
__device__ __forceinline__ void warp_argmax_bits(long long& v, int& j) {
  const int hi = static_cast<int>(v >> 32);
  const unsigned lo = static_cast<unsigned>(v);
  const int mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  j = __reduce_min_sync(0xffffffffu, (hi == mh && lo == ml) ? j : INT_MAX);
  v = (static_cast<long long>(mh) << 32) | ml;
}

// a / b, correctly rounded, from y = 1 / b (itself correctly rounded): two
// residual corrections of a y (P. Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34,
// 1990: the second gives the rounded quotient when the first is within an
// ulp).  Five dependent FP64 operations instead of a division's ten or so;
// operands whose quotient or residuals could leave the normal range, and a b
// whose significand is all ones, take the division.
__device__ __forceinline__ double div_by(double a, double b, double y) {
  const int ea = (__double2hiint(a) >> 20) & 0x7ff, eb = (__double2hiint(b) >> 20) & 0x7ff;
  const bool ones = (__double_as_longlong(b) & 0xfffffffffffffll) == 0xfffffffffffffll;
  const bool zero = (__double_as_longlong(a) & LLONG_MAX) == 0;   // a y is the quotient
  if (!zero && (ea < 600 || ea > 1400 || eb < 700 || eb > 1300 || ones)) return a / b;
  double q = a * y;
  if (zero) return q;
  q = fma(fma(-q, b, a), y, q);
  return fma(fma(-q, b, a), y, q);
}

// Sum over the column entries c >= i of f(c) with a summation order that does
// not depend on the team size TS: entry c accumulates (in increasing c) into
// partial c mod 32, and the 32 partials are combined by a fixed butterfly
// (pairs p, p + o for o = 16, 8, ..., 1).  Levels o >= TS pair partials held
// by the same thread, the others go through shuffles within the team.  So a
// node's ID is bitwise the same whatever cluster size or batch it runs in.
template <int TS, typename F>
__device__ __forceinline__ double team_sum(int i, int d, int member, F f) {
  constexpr int NP = 32 / TS;
  double acc[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) acc[q] = 0.0;
  for (int base = (i / 32) * 32; base < d; base += 32) {
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const int c = base + member + q * TS;
      if (c >= i && c < d) acc[q] = f(c, acc[q]);
    }
  }
#pragma unroll
  for (int o = 16; o >= TS; o >>= 1) {
#pragma unroll
    for (int q = 0; q < o / TS; ++q) acc[q] = acc[q] + acc[q + o / TS];
  }
  double v = acc[0];
#pragma unroll
  for (int o = TS >> 1; o > 0; o >>= 1) v = v + __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One pass over a column for two elimination steps: the pending update of
// step i-1, w[c] += a * up[c - (i-1)] for c >= i-1 (when `pending`), and the
// dot product of the updated column with u_i over c >= i, summed in
// team_sum's order.  Each entry gets the same operations, in the same order,
// as an update pass followed by a dot-product pass, so the bits are those of
// the two passes; the column is read and written once instead of read twice
// and written once.  Chunks of 32 rows; the inner ones carry no bounds, and a
// column in global memory (WS false) has its next chunk on the way.
template <int TS, bool WS>
__device__ __forceinline__ double team_update_dot(int i, int d, int member, bool pending, double a,
                                                  const double* __restrict__ up,
                                                  const double* __restrict__ u, double* w) {
  constexpr int NP = 32 / TS;              // partial sums per thread
  constexpr int NG = NP < 8 ? NP : 8;      // rows of a chunk in flight per thread
  constexpr bool PF = !WS && TS >= 4;      // next chunk loaded ahead
  double acc[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) acc[q] = 0.0;
  const int lo = pending ? i - 1 : i;
  int base = (lo / 32) * 32;
  double x[PF ? NP : 1];
  auto load = [&](int b, int q) -> double {
    const int c = b + member + q * TS;
    return (c >= lo && c < d) ? w[c] : 0.0;
  };
  if constexpr (PF) {
#pragma unroll
    for (int q = 0; q < NP; ++q) x[q] = load(base, q);
  }
  for (; base < d; base += 32) {
    double nx[PF ? NP : 1];
    if constexpr (PF) {
      if (base + 64 <= d) {
#pragma unroll
        for (int q = 0; q < NP; ++q) nx[q] = w[base + 32 + member + q * TS];
      } else {
#pragma unroll
        for (int q = 0; q < NP; ++q) nx[q] = load(base + 32, q);
      }
    }
    if (base >= i && base + 32 <= d) {
#pragma unroll
      for (int g = 0; g < NP; g += NG) {
        double pp[NG], uu[NG], xx[NG];
#pragma unroll
        for (int q = 0; q < NG; ++q) {
          const int c = base + member + (g + q) * TS;
          pp[q] = up[c - lo];
          uu[q] = u[c - i];
          if constexpr (PF) xx[q] = x[g + q];
          else xx[q] = w[c];
        }
#pragma unroll
        for (int q = 0; q < NG; ++q) {
          const int c = base + member + (g + q) * TS;
          const double t = fma(a, pp[q], xx[q]);
          if (pending) {
            xx[q] = t;
            w[c] = t;
          }
          acc[g + q] = fma(uu[q], xx[q], acc[g + q]);
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < NP; ++q) {
        const int c = base + member + q * TS;
        if (c >= lo && c < d) {
          double xq;
          if constexpr (PF) xq = x[q];
          else xq = w[c];
          if (pending) {
            xq = fma(a, up[c - lo], xq);
            w[c] = xq;
          }
          if (c >= i) acc[q] = fma(u[c - i], xq, acc[q]);
        }
      }
    }
    if constexpr (PF) {
#pragma unroll
      for (int q = 0; q < NP; ++q) x[q] = nx[q];
    }
  }
#pragma unroll
  for (int o = 16; o >= TS; o >>= 1) {
#pragma unroll
    for (int q = 0; q < o / TS; ++q) acc[q] = acc[q] + acc[q + o / TS];
  }
  double r = acc[0];
#pragma unroll
  for (int o = TS >> 1; o > 0; o >>= 1) r = r + __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

// A CTA's pivot candidate as its peers receive it, with the reflector it
// would give.
struct alignas(16) Cand {
  long long v;    // bit pattern of its largest active residual norm (LLONG_MIN: none)
  int j;          // its global column index
  int pad;
  double sigma;   // |R_ii| if it is the pivot
  double tau;
  double scal;    // v = x scal below the pivot row
  double pad2;
};
// (v, j), (sigma, tau) and scal are read as 16-byte loads
static_assert(offsetof(Cand, j) == 8 && offsetof(Cand, sigma) == 16 && offsetof(Cand, scal) == 32 &&
                  sizeof(Cand) == 48,
              "Cand layout");

// A node side spread over more CTAs than a cluster holds (a "group"): the
// group's CTAs meet at a barrier in global memory (a counter per item) and
// exchange their candidates there; their columns stay in the global work
// copy.  Used when one step's update is long enough (large m and d) that the
// barrier's few microseconds are small beside it.
struct GroupArgs {
  int gsz;          // CTAs per item (0: the launch uses clusters)
  Cand* cand;       // [items][2][gsz]
  unsigned* ctr;    // [items] barrier counters, zero at launch
  int* abort;       // set when a barrier wait gives up
  int* err;         // first error code
  long long limit;  // clock cycles a barrier wait may take
};
constexpr long long GROUP_WAIT_LIMIT = 1ll << 33;   // clock cycles (about 4 s)
// smallest per-CTA update of one step in cluster mode (columns x sample
// count) for which the group mode is used
constexpr long GROUP_MIN_STEP_WORK = 1l << 15;

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// WS: the columns are in shared memory, else in the global work copy
template <int TS, bool GRP, int MINB = 1, bool WS = false>
__global__ void __launch_bounds__(ID_THREADS, MINB)
id_cpqr_cluster_kernel(const IdItem* __restrict__ items, int f64in,
                       double* __restrict__ r1buf_base,
                       const int64_t* __restrict__ r1off, GroupArgs ga) {
  extern __shared__ __align__(16) double smem[];
  __shared__ Cand cands[2][16];
  __shared__ long long redb[ID_WARPS];
  __shared__ int redi[ID_WARPS];
  __shared__ double cbeta;   // R_ii of this CTA's last candidate
  __shared__ int nrest;
  __shared__ int nact;
  __shared__ int gstop;

  int C, crank;
  if constexpr (GRP) {
    C = ga.gsz;
    crank = static_cast<int>(blockIdx.x) % C;
  } else {
    cg::cluster_group cl = cg::this_cluster();
    C = (int)cl.num_blocks();
    crank = (int)cl.block_rank();
  }
  const int item = blockIdx.x / C;
  const IdItem it = items[item];
  const int m = it.m, d = it.d;
  const double rtol = it.rtol, atol = it.atol;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // every CTA of the cluster / group: a cluster barrier, or a barrier in
  // global memory (bounded: on a timeout the launch is abandoned and every
  // CTA returns at its next barrier)
  unsigned nsync = 0;
  auto sync_all = [&]() -> bool {
    if constexpr (GRP) {
      __syncthreads();
      if (tid == 0) {
        // arrive after a device-wide fence (the CTA's writes, ordered before
        // by the block barrier, become visible first), then poll with
        // acquire loads; the abort flag and the clock are looked at every
        // 16th poll
        __threadfence();
        atomicAdd(ga.ctr + item, 1u);
        const unsigned target = (++nsync) * static_cast<unsigned>(C);
        const long long t0 = clock64();
        int st = 0;
        unsigned polls = 0;
        while (ld_acquire_gpu(ga.ctr + item) < target) {
          if ((++polls & 15u) != 0u) continue;
          if (*reinterpret_cast<volatile int*>(ga.abort)) {
            st = 1;
            break;
          }
          if (clock64() - t0 > ga.limit) {
            atomicExch(ga.abort, 1);
            atomicCAS(ga.err, 0, 1);
            st = 1;
            break;
          }
        }
        __threadfence();
        gstop = st;
      }
      __syncthreads();
      return gstop == 0;
    } else {
      cg::this_cluster().sync();
      return true;
    }
  };
  if (m <= 0) {
    if (crank == 0 && tid == 0) *it.k = 0;
    return;   // uniform across the cluster
  }
  const int mloc = (m - crank + C - 1) / C;       // columns crank, crank+C, ...
  const int mloc_max = (m + C - 1) / C;
  // reflectors of steps i (vbuf + (i & 1) d) and i - 1: the update of a step
  // is applied in the same pass as the next step's dot product; then the
  // candidate's column (cbuf).  The buffer of u_{i-1} also takes the (at most
  // 128) partial sums of a candidate's residual, at the end of step i.  After the
  // elimination: R1's diagonal, its reciprocals, and a block of the back
  // substitution
  double* vbuf = smem;                            // 2 d
  double* cbuf = vbuf + 2 * d;                    // id_cbuf(d, mloc_max)
  double* nrm = cbuf + id_cbuf(d, mloc_max);      // mloc_max
  double* lim = nrm + mloc_max;                   // mloc_max: tol3z * (norm at last recompute)^2
  double* rdiag = lim + mloc_max;                 // mloc_max: R_ii of the pivot columns
  double* dprev = rdiag + mloc_max;               // mloc_max: tau (u_i . w), update pending
  int* pstep = reinterpret_cast<int*>(dprev + mloc_max);   // mloc_max: pivot step or -1
  // the active (not yet pivoted) local columns, compacted: alist[0..nact)
  // holds their local indices, apos[jl] is jl's position in alist.  Teams and
  // norm-downdate lanes are dealt over this list, so no FP64 instruction is
  // issued for a pivoted column (an FP64 instruction costs the same however
  // few lanes are active).  Removal swaps in the last entry: which thread
  // takes which column changes, the arithmetic of every column does not.
  int* alist = pstep + ((mloc_max + 1) & ~1);
  int* apos = alist + ((mloc_max + 1) & ~1);
  int* pend = apos + ((mloc_max + 1) & ~1);       // 1: the column's update by dprev is pending
  double* Wsm = reinterpret_cast<double*>(pend + ((mloc_max + 1) & ~1));
  // odd column stride in shared memory: a thread per column reads without
  // bank conflicts
  const int ldw = d | 1;
  // (telling the compiler the address space: generic loads and stores could
  // alias the reflectors in shared memory and wait for each other)
  auto col = [&](int jl) -> double* {
    if constexpr (WS) {
      return Wsm + (size_t)jl * ldw;
    } else {
      double* q = it.work + (size_t)(jl * C + crank) * d;
      __builtin_assume(__isGlobal(q));
      return q;
    }
  };
  // team of TS threads per column (power of two, chosen by the launcher):
  // all 256 threads stay busy whether a CTA owns 8 columns or 500
  const int member = lane & (TS - 1);
  const int cols_per_warp = 32 / TS;
  const double tol3z = sqrt(DBL_EPSILON * 0.5);
  int32_t* perm = it.perm;

  // load the owned columns (FP64 copy) and their norms
  for (int jl = warp; jl < mloc; jl += ID_WARPS) {
    const int j = jl * C + crank;
    double* w = col(jl);
    double ss = 0.0;
    if (f64in) {
      const double* y = reinterpret_cast<const double*>(it.Yt) + (size_t)j * it.ldy;
      for (int c = lane; c < d; c += 32) {
        double x = y[c];
        w[c] = x;
        ss = fma(x, x, ss);
      }
    } else {
      const float* y = reinterpret_cast<const float*>(it.Yt) + (size_t)j * it.ldy;
      for (int c = lane; c < d; c += 32) {
        double x = (double)y[c];
        w[c] = x;
        ss = fma(x, x, ss);
      }
    }
    ss = warp_sum(ss);
    if (lane == 0) {
      nrm[jl] = sqrt(ss);
      lim[jl] = tol3z * (nrm[jl] * nrm[jl]);
      pstep[jl] = -1;
      alist[jl] = jl;
      apos[jl] = jl;
      pend[jl] = 0;
    }
  }
  if (tid == 0) nact = mloc;
  // every CTA of the cluster has started (its shared memory may now be
  // written by peers) and the columns and norms are loaded
  if (!sync_all()) return;
  // each CTA's candidate (largest residual norm of its active columns, as the
  // norm's bit pattern; lowest index on ties) goes into slot s of every CTA's
  // cands[s][crank], so the reads after the next cluster barrier are local.
  // The whole CTA brings the candidate's column up to date (its update by
  // u = u_{r-1} may be pending) and leaves it in cbuf as well; four warps on
  // four schedulers sum its squares below the pivot row r, and warp 0 forms
  // the reflector (lanes 0 and 1 the two quotients in one division) and
  // pushes.  The sum: entry c goes to partial (c / 32) mod 4 of lane c mod 32,
  // in increasing c, then ((p0 + p1) + (p2 + p3)) and a butterfly over the
  // lanes: a fixed order, computed by the owner alone.
  auto push_candidate = [&](int s, long long v, int j, int r, const double* u, double* psum) {
    const bool have = v != LLONG_MIN;
    const int jl = have ? (j - crank) / C : 0;
    if (have) {
      double* w = col(jl);
      const bool pd = pend[jl] != 0;
      const double a = -dprev[jl];
      constexpr int U = 4;
      for (int c0 = (pd ? r - 1 : r) + tid; c0 < d; c0 += U * ID_THREADS) {
        double x[U];
#pragma unroll
        for (int q = 0; q < U; ++q) x[q] = c0 + q * ID_THREADS < d ? w[c0 + q * ID_THREADS] : 0.0;
#pragma unroll
        for (int q = 0; q < U; ++q) {
          const int c = c0 + q * ID_THREADS;
          if (c >= d) continue;
          if (pd) {
            x[q] = fma(a, u[c - (r - 1)], x[q]);
            w[c] = x[q];
          }
          cbuf[c] = x[q];
        }
      }
    }
    __syncthreads();
    if (warp >= 4) return;
    if (have && tid == 0) pend[jl] = 0;
    double pa = 0.0;
    if (have)
      for (int base = ((r + 1) / 128) * 128; base < d; base += 128) {
        const int c = base + 32 * warp + lane;
        const double x = (c >= r + 1 && c < d) ? cbuf[c] : 0.0;
        pa = fma(x, x, pa);
      }
    if (32 * warp + lane < d) psum[32 * warp + lane] = pa;   // (the others are zero)
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (warp != 0) return;
    double ps[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) ps[q] = 32 * q + lane < d ? psum[32 * q + lane] : 0.0;
    double st = (ps[0] + ps[1]) + (ps[2] + ps[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) st = st + __shfl_xor_sync(0xffffffffu, st, o);
    const double alpha = have && r < d ? cbuf[r] : 0.0;
    const double sigma = fp_sqrt(fma(alpha, alpha, st));
    const bool refl = st != 0.0;
    const double beta = refl ? -copysign(sigma, alpha) : alpha;
    double q = 0.0;
    if (refl && lane < 2) {
      const double num = lane == 0 ? beta - alpha : 1.0;
      const double den = lane == 0 ? beta : alpha - beta;
      q = fp_div(num, den);
    }
    const double tau = __shfl_sync(0xffffffffu, q, 0), scal = __shfl_sync(0xffffffffu, q, 1);
    if (lane == 0) cbeta = beta;
    Cand* dst = nullptr;
    if constexpr (GRP) {
      if (lane == 0) dst = ga.cand + (static_cast<size_t>(item) * 2 + s) * C + crank;
    } else if (lane < C) {
      dst = cg::this_cluster().map_shared_rank(&cands[s][crank], lane);
    }
    if (dst != nullptr) {
      dst->v = v;
      dst->j = j;
      dst->sigma = sigma;
      dst->tau = tau;
      dst->scal = scal;
    }
  };
  {
    long long bv = LLONG_MIN;
    int bj = INT_MAX;
    if (warp == 0) {
      for (int jl = lane; jl < mloc; jl += 32) {
        const long long x = __double_as_longlong(nrm[jl]);
        const int j = jl * C + crank;
        if (x > bv || (x == bv && j < bj)) {
          bv = x;
          bj = j;
        }
      }
      warp_argmax_bits(bv, bj);
      if (lane == 0) {
        redb[0] = bv;
        redi[0] = bj;
      }
    }
    __syncthreads();
    push_candidate(0, redb[0], redi[0], 0, vbuf, vbuf + d);
  }

  const int kmax = min(m, d);
  // warps that downdate the norms (one lane per column: an FP64 instruction
  // costs the same however few lanes are active)
  const int nwd = min(ID_WARPS, (mloc_max + 31) / 32);
  int k = kmax;
  long long thr = 0;   // bit pattern of max(rtol |R_11|, atol)
  for (int i = 0; i < kmax; ++i) {
    if (!sync_all()) return;   // candidates of step i pushed, dot products of step i-1 done
    const int slot = i & 1;
    double* vloc = vbuf + (i & 1) * d;         // reflector u_i
    const double* vprev = vbuf + ((i + 1) & 1) * d;  // u_{i-1}
    // every warp reduces the C candidates (lane r <- CTA r): all threads agree
    // on the pivot without a block barrier
    long long bv = LLONG_MIN;
    int p = INT_MAX;
    const Cand* gc = nullptr;
    if constexpr (GRP) {
      gc = ga.cand + (static_cast<size_t>(item) * 2 + slot) * C;
      // every candidate (v, j) is loaded before any is compared: one round
      // trip to L2 for up to 320 CTAs instead of one per 32
      constexpr int U = 10;
      for (int r0 = lane; r0 < C; r0 += 32 * U) {
        longlong2 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int r = r0 + 32 * u;
          x[u] = r < C ? __ldcg(reinterpret_cast<const longlong2*>(&gc[r]))
                       : make_longlong2(LLONG_MIN, INT_MAX);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int j = static_cast<int>(x[u].y & 0xffffffffll);
          if (x[u].x > bv || (x[u].x == bv && j < p)) {
            bv = x[u].x;
            p = j;
          }
        }
      }
    } else if (lane < C) {
      bv = cands[slot][lane].v;
      p = cands[slot][lane].j;
    }
    warp_argmax_bits(bv, p);
    const int owner = p % C;
    // the winner's reflector and its column, entries i..d-1, from the owner
    double sigma, tau, scal;
    if constexpr (GRP) {
      const double2 y = __ldcg(reinterpret_cast<const double2*>(&gc[owner]) + 1);
      scal = __ldcg(&gc[owner].scal);
      sigma = y.x;
      tau = y.y;
    } else {
      sigma = cands[slot][owner].sigma;
      tau = cands[slot][owner].tau;
      scal = cands[slot][owner].scal;
    }
    // the stopping test on bit patterns (all values are >= 0): |R_11| = 0 or
    // |R_ii| <= max(rtol |R_11|, atol)
    const long long sb = __double_as_longlong(sigma) & LLONG_MAX;   // (a NaN is above all)
    if (i == 0) thr = sb == 0 ? LLONG_MAX : __double_as_longlong(fmax(rtol * sigma, atol) + 0.0);
    if (sb <= thr) {
      k = i;
      break;   // every CTA of the cluster takes the same decision
    }
    if (tid == 0) {
      if (owner == crank) {
        const int jp = p / C;
        rdiag[jp] = cbeta;
        nrm[jp] = -1.0;
        pstep[jp] = i;
        const int pos = apos[jp], last = alist[nact - 1];
        alist[pos] = last;
        apos[last] = pos;
        --nact;
      }
      if (crank == 0) perm[i] = p;
    }
    if constexpr (WS) {
      const double* src = cg::this_cluster().map_shared_rank(Wsm + (size_t)(p / C) * ldw, owner);
      for (int c = i + tid; c < d; c += ID_THREADS) vloc[c - i] = c == i ? 1.0 : src[c] * scal;
    } else {
      // written by another CTA: read from L2, eight loads in flight per
      // thread before the stores
      const double* src = it.work + (size_t)p * d;
      constexpr int U = 8;
      for (int c0 = i + tid; c0 < d; c0 += ID_THREADS * U) {
        double x[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          x[u] = c0 + ID_THREADS * u < d ? __ldcg(src + c0 + ID_THREADS * u) : 0.0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int c = c0 + ID_THREADS * u;
          if (c < d) vloc[c - i] = c == i ? 1.0 : x[u] * scal;
        }
      }
    }
    __syncthreads();
    // one pass per active column (a team of TS threads, the teams dealt over
    // the compacted list): the pending update of step i-1 and the dot
    // product with u_i; the update of step i is left pending (dprev)
    const int na = nact;
    for (int jb = warp * cols_per_warp; jb < na; jb += ID_WARPS * cols_per_warp) {
      const int q = jb + lane / TS;
      const bool act = q < na;
      const int jl = act ? alist[q] : 0;
      double* wj = col(jl);
      const bool pd = act && pend[jl] != 0;
      const double dot = team_update_dot<TS, WS>(i, act ? d : 0, member, pd, pd ? -dprev[jl] : 0.0,
                                             vprev, vloc, wj);
      if (act && member == 0) {
        dprev[jl] = dot * tau;
        pend[jl] = 1;
      }
    }
    __syncthreads();
    // norm downdates (LAPACK xGEQP3's formula and safeguard), one lane per
    // column, and this CTA's next candidate
    if (warp < nwd) {
      long long cv = LLONG_MIN;
      int cj = INT_MAX;
      for (int q0 = warp * 32; q0 < na; q0 += nwd * 32) {
        const int jl = q0 + lane < na ? alist[q0 + lane] : 0;
        const double nj = q0 + lane < na ? nrm[jl] : -1.0;
        const bool act = nj >= 0.0;
        bool recompute = false;
        double newn = nj;
        if (act && nj != 0.0) {
          // xGEQP3's downdate nj sqrt(max(0, (1 - t)(1 + t))), t = |r| / nj,
          // and its test t (nj / nrm0)^2 <= tol3z, both multiplied out by nj^2;
          // r = the column's entry i after the (pending) update of step i
          const double r = fabs(fma(-dprev[jl], 1.0, col(jl)[i]));
          const double q = fmax(0.0, (nj - r) * (nj + r));
          if (q <= lim[jl]) recompute = true;
          else newn = fp_sqrt(q);
        }
        // cancellation: recompute those norms, one column at a time with the
        // whole warp (the fixed summation tree gives the same bits as a team)
        unsigned rm = __ballot_sync(0xffffffffu, recompute);
        while (rm) {
          const int src = __ffs(rm) - 1;
          rm &= rm - 1;
          const int jr = __shfl_sync(0xffffffffu, jl, src);
          double* wr = col(jr);
          if (pend[jr]) {   // the exact norm needs the updated column
            const double a = -dprev[jr];
#pragma unroll 8
            for (int c = i + lane; c < d; c += 32) wr[c] = fma(a, vloc[c - i], wr[c]);
            __syncwarp();
            if (lane == 0) pend[jr] = 0;
            __syncwarp();
          }
          const double ss = team_sum<32>(i + 1, d, lane, [&](int c, double a) {
            return fma(wr[c], wr[c], a);
          });
          if (lane == src) {
            newn = sqrt(ss);
            lim[jl] = tol3z * (newn * newn);
          }
        }
        if (act) {
          nrm[jl] = newn;
          const long long nb = __double_as_longlong(newn);
          const int j = jl * C + crank;
          if (nb > cv || (nb == cv && j < cj)) {
            cv = nb;
            cj = j;
          }
        }
      }
      warp_argmax_bits(cv, cj);
      if (lane == 0) {
        redb[warp] = cv;
        redi[warp] = cj;
      }
    }
    __syncthreads();
    {
      // the CTA's candidate (the same total order as the warps' arg-max),
      // known to every thread
      long long cv = LLONG_MIN;
      int cj = INT_MAX;
      for (int w = 0; w < nwd; ++w)
        if (redb[w] > cv || (redb[w] == cv && redi[w] < cj)) {
          cv = redb[w];
          cj = redi[w];
        }
      push_candidate(slot ^ 1, cv, cj, i + 1, vloc, vbuf + ((i + 1) & 1) * d);
    }
  }

  if (k > it.fail_above) {
    // the caller discards this side (its node fails the adaptive test): no
    // generator; the barrier keeps every CTA's shared memory alive until the
    // cluster's last reads and pushes of the loop are done
    if (crank == 0 && tid == 0) *it.k = k;
    sync_all();
    return;
  }
  // the update of step k - 1 is still pending on the remaining columns
  if (k > 0) {
    const double* ul = vbuf + ((k - 1) & 1) * d;
    const int na = nact;
    for (int q = warp; q < na; q += ID_WARPS) {
      const int jl = alist[q];
      if (!pend[jl]) continue;
      double* w = col(jl);
      const double a = -dprev[jl];
      for (int c = k - 1 + lane; c < d; c += 32) w[c] = fma(a, ul[c - (k - 1)], w[c]);
      __syncwarp();
      if (lane == 0) pend[jl] = 0;
    }
    __syncthreads();
  }
  // R1 (k x k, column b = pivot b's first b+1 entries) to global, remaining
  // columns flagged for the ordering of perm[k..m)
  double* R1 = r1buf_base + r1off[item];
  int* flag = reinterpret_cast<int*>(it.norms);   // m ints of the norms scratch
  for (int jl = warp; jl < mloc; jl += ID_WARPS) {
    const int j = jl * C + crank;
    const int b = pstep[jl];
    if (b >= 0 && b < k) {
      const double* w = col(jl);
      for (int a = lane; a <= b; a += 32) R1[(size_t)b * k + a] = (a == b) ? rdiag[jl] : w[a];
    }
    if (lane == 0) flag[j] = (b < 0 || b >= k) ? 1 : 0;
  }
  if (!sync_all()) return;   // R1 and flags visible to the whole cluster
  if (crank == 0 && tid == 0) *it.k = k;
  // position of each remaining column in perm[k..m): the count of remaining
  // columns of lower index.  Warp 0 walks the flags 32 at a time with the
  // count so far; the columns this CTA owns are among them, and go to rlist
  // in order
  int* restpos = pstep;   // reuse: local rest position
  int* rlist = reinterpret_cast<int*>(nrm);   // local indices of the remaining columns
  __syncthreads();        // pstep and nrm have been read
  if (warp == 0) {
    constexpr int U = 8;
    int before = 0, mine = 0;
    for (int j0 = 0; j0 < m; j0 += 32 * U) {
      int f[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + 32 * u + lane;
        f[u] = j < m ? __ldcg(flag + j) : 0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + 32 * u + lane;
        const unsigned rest = __ballot_sync(0xffffffffu, f[u] != 0);
        const bool own = j < m && j % C == crank;
        const unsigned keep = __ballot_sync(0xffffffffu, own && f[u] != 0);
        const unsigned below = (1u << lane) - 1u;
        if (own) {
          const int jl = (j - crank) / C;
          restpos[jl] = f[u] ? before + __popc(rest & below) : -1;
          if (f[u]) rlist[mine + __popc(keep & below)] = jl;
        }
        before += __popc(rest);
        mine += __popc(keep);
      }
    }
    if (lane == 0) nrest = mine;
  }
  // T = R1^{-1} R2 for the remaining columns this CTA owns, by column-oriented
  // back substitution: T_a = rhs_a / R_aa, then rhs_c -= R_ca T_a for c < a, a
  // from k-1 down to 0, solved in place in the columns' first k entries.  By
  // blocks of 16 rows: the block itself by groups of four warps (lane =
  // column, warp q rows q mod 4 of the block: a row's quotient goes through
  // shared memory to the group), then all its terms for the rows above in one
  // pass (a thread per row, R's 16 entries in registers).  Each entry gets
  // its terms one by one in the order of decreasing a, so neither the blocks
  // nor the CTA or cluster size change its bits.  (Two block barriers and a
  // division's 680 cycles of latency per row: 0.38 ms at m = 342, k = 241;
  // by blocks 0.24 ms.)
  double* diag = vbuf;        // k <= d entries
  double* rinv = vbuf + d;    // their reciprocals
  double* blk = d < ID_BLK && 3 * mloc_max >= ID_BLK ? lim : cbuf;
  double(*Rb)[ID_BS + 1] = reinterpret_cast<double(*)[ID_BS + 1]>(blk);
  double(*xs)[2][32] = reinterpret_cast<double(*)[2][32]>(blk + ID_BS * (ID_BS + 1));
  for (int a = tid; a < k; a += ID_THREADS) {
    const double x = __ldcg(R1 + (size_t)a * k + a);
    diag[a] = x;
    rinv[a] = 1.0 / x;
  }
  __syncthreads();
  const int nr = nrest;
  for (int u = tid; u < nr; u += ID_THREADS) perm[k + restpos[rlist[u]]] = rlist[u] * C + crank;
  constexpr int BS = ID_BS;
  for (int a1 = k; a1 > 0 && nr > 0; a1 -= BS) {
    const int a0 = max(0, a1 - BS), nb = a1 - a0;
    for (int e = tid; e < nb * nb; e += ID_THREADS) {
      const int q = e / nb, t = e - q * nb;
      if (t < q) Rb[t][q] = __ldcg(R1 + (size_t)(a0 + q) * k + a0 + t);
    }
    __syncthreads();
    const int grp = warp >> 2, w4 = warp & 3;
    for (int u0 = 0; u0 < nr; u0 += 64) {
      const int u = u0 + 32 * grp + lane;
      const bool act = u < nr;
      const int jl = act ? rlist[u] : 0;
      double* r2 = col(jl);
      double v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) v[t] = act && w4 + 4 * t < nb ? r2[a0 + w4 + 4 * t] : 0.0;
      if (u0 + 32 * grp < nr) {   // uniform in the group
        for (int q = nb - 1; q >= 0; --q) {
          if ((q & 3) == w4) {
#pragma unroll
            for (int t = 0; t < 4; ++t)
              if (t == (q >> 2)) {
                v[t] = div_by(v[t], diag[a0 + q], rinv[a0 + q]);
                xs[grp][q & 1][lane] = v[t];
              }
          }
          asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory");
          const double xq = xs[grp][q & 1][lane];   // (two slots: a barrier lies between uses)
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (w4 + 4 * t < q) v[t] = fma(-Rb[w4 + 4 * t][q], xq, v[t]);
        }
      }
      if (act) {
        double* E = it.E + (size_t)restpos[jl] * k;
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (w4 + 4 * t < nb) {
            r2[a0 + w4 + 4 * t] = v[t];
            E[a0 + w4 + 4 * t] = v[t];
          }
      }
    }
    __syncthreads();
    if (a0 > 0) {
      // rows c < a0: threads over (row, every ng-th column)
      const int cw = min(ID_THREADS, (a0 + 31) & ~31), ng = ID_THREADS / cw, ug = tid / cw;
      for (int c = tid - ug * cw; c < a0 && ug < ng; c += cw) {
        double rq[BS];
#pragma unroll
        for (int q = 0; q < BS; ++q) rq[q] = q < nb ? __ldcg(R1 + (size_t)(a0 + q) * k + c) : 0.0;
        // four columns at a time: an entry's 16 terms are a chain of 67
        // cycles each
        for (int u = ug; u < nr; u += 4 * ng) {
          double* r2[4];
          double v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            r2[e] = col(rlist[min(u + e * ng, nr - 1)]);
            v[e] = r2[e][c];
          }
#pragma unroll
          for (int q = BS - 1; q >= 0; --q)
            if (q < nb) {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (u + e * ng < nr) v[e] = fma(-rq[q], r2[e][a0 + q], v[e]);
            }
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (u + e * ng < nr) r2[e][c] = v[e];
        }
      }
    }
    __syncthreads();
  }
}

using IdKernel = void (*)(const IdItem*, int, double*, const int64_t*, GroupArgs);
std::array<IdKernel, 6> kernels() {
  return {id_cpqr_cluster_kernel<1, false>, id_cpqr_cluster_kernel<2, false>,
          id_cpqr_cluster_kernel<4, false>, id_cpqr_cluster_kernel<8, false>,
          id_cpqr_cluster_kernel<16, false>, id_cpqr_cluster_kernel<32, false>};
}
// Columns in shared memory.  At most 128 registers a thread where that does
// not spill: with one CTA per SM only 15 clusters of 8 (7 of 16) fit on the
// GPU at once, so a launch of 128 CTAs would run a second wave for its last
// cluster (897 -> 1343 us and 1304 -> 2122 us on two levels of a Gaussian
// kernel's compression).
std::array<IdKernel, 6> smem_kernels() {
  return {id_cpqr_cluster_kernel<1, false, 1, true>,  id_cpqr_cluster_kernel<2, false, 1, true>,
          id_cpqr_cluster_kernel<4, false, 2, true>,  id_cpqr_cluster_kernel<8, false, 2, true>,
          id_cpqr_cluster_kernel<16, false, 2, true>, id_cpqr_cluster_kernel<32, false, 2, true>};
}
std::array<IdKernel, 6> group_kernels() {
  return {id_cpqr_cluster_kernel<1, true>, id_cpqr_cluster_kernel<2, true>,
          id_cpqr_cluster_kernel<4, true>, id_cpqr_cluster_kernel<8, true>,
          id_cpqr_cluster_kernel<16, true>, id_cpqr_cluster_kernel<32, true>};
}
// the group mode with two CTAs per SM (at most 128 registers a thread): while
// one CTA waits at a barrier or runs the serial part of a step (pivot choice,
// reflector, norm downdates), the other keeps the SM's FP64 pipes busy
std::array<IdKernel, 6> group_kernels2() {
  return {id_cpqr_cluster_kernel<4, true, 2>, id_cpqr_cluster_kernel<4, true, 2>,
          id_cpqr_cluster_kernel<4, true, 2>, id_cpqr_cluster_kernel<8, true, 2>,
          id_cpqr_cluster_kernel<16, true, 2>, id_cpqr_cluster_kernel<32, true, 2>};
}

// cluster mode with two CTAs per SM, for launches of more CTAs than SMs
// (the leaf levels): one wave instead of two, and the same overlap of one
// CTA's serial part with the other's FP64 work
std::array<IdKernel, 6> kernels2() {
  return {id_cpqr_cluster_kernel<4, false, 2>, id_cpqr_cluster_kernel<4, false, 2>,
          id_cpqr_cluster_kernel<4, false, 2>, id_cpqr_cluster_kernel<8, false, 2>,
          id_cpqr_cluster_kernel<16, false, 2>, id_cpqr_cluster_kernel<32, false, 2>};
}

// Measuring tuner of the team size (threads per column) of the ID launches.
// The results do not depend on the team size (fixed summation tree), so the
// tuner may try several on real launches: launches are grouped into classes
// (spread-out or cluster mode, columns in shared or global memory, the powers
// of two of the largest side, the sample count and the item count, and whether
// the launch may change its group or cluster size: a class's choice is made for
// every launch of the class, so it has to be one that each of them can run);
// the first launches of a class try the instruction-count model's choice and
// its two neighbours, twice each, timed with CUDA events and normalised by
// the launch's sum of m d min(m, d); later launches of the class take the
// fastest.  Events are read without waiting, when the next ID launch comes.
// HSS_AUTOTUNE=0 in the environment keeps the model's choice everywhere.
class TeamTuner {
 public:
  struct Key {
    int dev, group, smem, lg_m, lg_d, lg_n;
    bool alt;   // the launch may also halve its group or double its clusters
    bool operator<(const Key& o) const {
      return std::tie(dev, group, smem, lg_m, lg_d, lg_n, alt) <
             std::tie(o.dev, o.group, o.smem, o.lg_m, o.lg_d, o.lg_n, o.alt);
    }
  };
  struct Trial {
    Key key;
    int ti;
    double units;
    cudaEvent_t e0, e1;
  };

  static TeamTuner& get() {
    static TeamTuner t;
    return t;
  }
  // team index for this launch; *trial receives events to record around it
  // (nullptr when the class has settled).  half_group: the launch may also
  // run with half as many CTAs per item (a spread-out launch whose CTAs own
  // few columns each): that candidate is the model's team index + 8.
  // double_cluster: a cluster launch may also run with clusters twice as
  // large: the model's team index + 16.
  int choose(const Key& k, int model_ti, int min_ti, double units, Trial** trial,
             bool half_group = false, bool double_cluster = false) {
    std::lock_guard<std::mutex> lock(mu_);
    harvest();
    *trial = nullptr;
    if (!enabled_) return model_ti;
    Cls& c = cls_[k];
    if (c.cand.empty()) {
      for (int t : {model_ti, model_ti - 1, model_ti + 1})
        if (t >= min_ti && t <= 5) c.cand.push_back(t);
      if (half_group) c.cand.push_back(model_ti + 8);
      if (double_cluster) c.cand.push_back(model_ti + 16);
      c.sum.assign(c.cand.size(), 0.0);
      c.cnt.assign(c.cand.size(), 0);
      c.issued.assign(c.cand.size(), 0);
    }
    if (c.best >= 0) return c.best;
    for (size_t q = 0; q < c.cand.size(); ++q) {
      if (c.issued[q] < kTrials) {
        Trial* t = new Trial{k, c.cand[q], units, nullptr, nullptr};
        if (cudaEventCreate(&t->e0) != cudaSuccess || cudaEventCreate(&t->e1) != cudaSuccess) {
          cudaGetLastError();
          if (t->e0) cudaEventDestroy(t->e0);
          delete t;
          return model_ti;
        }
        ++c.issued[q];
        ++trials_;
        *trial = t;
        return t->ti;
      }
    }
    return model_ti;   // every trial issued, some not yet measured
  }
  void launched(Trial* t, bool ok) {
    std::lock_guard<std::mutex> lock(mu_);
    if (!ok) {
      cudaEventDestroy(t->e0);
      cudaEventDestroy(t->e1);
      delete t;
      return;
    }
    pending_.push_back(t);
  }
  void stats(int32_t* classes, int32_t* settled, int32_t* trials) {
    std::lock_guard<std::mutex> lock(mu_);
    harvest();
    int s = 0;
    for (auto& kv : cls_) s += kv.second.best >= 0;
    if (classes) *classes = (int32_t)cls_.size();
    if (settled) *settled = s;
    if (trials) *trials = (int32_t)trials_;
  }

 private:
  static constexpr int kTrials = 2;
  struct Cls {
    std::vector<int> cand, cnt, issued;
    std::vector<double> sum;
    int best = -1;
  };
  TeamTuner() {
    const char* e = std::getenv("HSS_AUTOTUNE");
    enabled_ = !(e && e[0] == '0');
  }
  void harvest() {
    for (size_t q = 0; q < pending_.size();) {
      Trial* t = pending_[q];
      const cudaError_t st = cudaEventQuery(t->e1);
      if (st == cudaErrorNotReady) {
        ++q;
        continue;
      }
      float ms = 0.f;
      if (st == cudaSuccess && cudaEventElapsedTime(&ms, t->e0, t->e1) == cudaSuccess) {
        Cls& c = cls_[t->key];
        for (size_t i = 0; i < c.cand.size(); ++i)
          if (c.cand[i] == t->ti) {
            c.sum[i] += ms / std::max(t->units, 1.0);
            ++c.cnt[i];
          }
        bool all = true;
        for (int n : c.cnt) all = all && n >= kTrials;
        if (all && c.best < 0) {
          size_t b = 0;
          for (size_t i = 1; i < c.cand.size(); ++i)
            if (c.sum[i] < c.sum[b]) b = i;
          c.best = c.cand[b];
        }
      } else {
        cudaGetLastError();
      }
      cudaEventDestroy(t->e0);
      cudaEventDestroy(t->e1);
      delete t;
      pending_[q] = pending_.back();
      pending_.pop_back();
    }
  }
  std::mutex mu_;
  std::map<Key, Cls> cls_;
  std::vector<Trial*> pending_;
  int64_t trials_ = 0;
  bool enabled_ = true;
};

int ilog2(long x) {
  int l = 0;
  while (x > 1) {
    x >>= 1;
    ++l;
  }
  return l;
}

}  // namespace

void id_tuner_stats(int32_t* classes, int32_t* settled, int32_t* trials) {
  TeamTuner::get().stats(classes, settled, trials);
}

Err launch_id_batched(const IdItem* items_dev, const std::vector<IdItem>& h, bool f64,
                      cudaStream_t s, Arena* scratch) {
  const int count = (int)h.size();
  if (count <= 0) return ok();
  int max_m = 1, max_d = 1;
  for (const IdItem& x : h) {
    max_m = std::max(max_m, x.m);
    max_d = std::max(max_d, x.d);
  }
  int sms = 152;
  {
    int dev = 0;
    HSS_CUDA_TRY(cudaGetDevice(&dev));
    HSS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  }
  // cluster size: spread each item over more SMs when the batch is small,
  // keeping at least ~16 columns per CTA
  int C = 1;
  while (C < 16 && (long)count * C * 2 <= sms && max_m / (C * 2) >= 16) C *= 2;
  const int d = std::max(max_d, 1);
  auto need = [&](int c) {
    auto bytes = [](int d, int mloc) {
      return sizeof(double) * (2 * (size_t)d + (size_t)id_cbuf(d, mloc) + 4 * (size_t)mloc) +
             4 * sizeof(int) * (size_t)((mloc + 1) & ~1);
    };
    // (an item smaller than the largest may need the block's own doubles)
    const int mloc = (max_m + c - 1) / c;
    return std::max(bytes(d, mloc), bytes(std::min(d, ID_BLK - 1), std::min(mloc, (ID_BLK - 1) / 3)));
  };
  // a large side among many items: more CTAs per item until its share of the
  // per-column arrays fits in shared memory
  while (C < 16 && need(C) > 227 * 1024 - 2048) C *= 2;
  size_t base = need(C);
  size_t wbytes = sizeof(double) * (size_t)((max_m + C - 1) / C) * (d | 1);
  int w_in_smem = base + wbytes <= ID_SMEM_CAP ? 1 : 0;
  size_t smem = base + (w_in_smem ? wbytes : 0);
  if (smem > 227 * 1024 - 2048)   // room for the static shared memory
    return fail(HSS_ERR_INVALID, "ID: sample count d too large for the reflector buffers");
  // R1 buffers: k <= min(m, d) per item
  std::vector<int64_t> off(count);
  int64_t tot = 0;
  for (int q = 0; q < count; ++q) {
    off[q] = tot;
    int64_t kk = std::min(h[q].m, h[q].d);
    tot += std::max<int64_t>(kk * kk, 1);
  }
  double* r1 = nullptr;
  int64_t* offd = nullptr;
  if (scratch) {
    HSS_TRY(scratch->alloc_t(&r1, (size_t)tot, s));
    HSS_TRY(scratch->alloc_t(&offd, (size_t)count, s));
  } else {
    HSS_TRY(dalloc_t(&r1, (size_t)tot, s));
    HSS_TRY(dalloc_t(&offd, (size_t)count, s));
  }
  if (scratch) HSS_TRY(scratch->upload(offd, off.data(), count * sizeof(int64_t), s));
  else HSS_CUDA_TRY(cudaMemcpyAsync(offd, off.data(), count * sizeof(int64_t), cudaMemcpyHostToDevice, s));
  {
    // kernel attributes: once per device (the shared-memory cap is the
    // hardware maximum; each launch asks for what it needs)
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    HSS_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if (dev >= 0 && dev < 64 && !done[dev]) {
      int optin = 0;
      HSS_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
      std::vector<IdKernel> ck;
      for (auto fn : kernels()) ck.push_back(fn);
      for (auto fn : smem_kernels()) ck.push_back(fn);
      for (auto fn : kernels2()) ck.push_back(fn);
      for (auto fn : ck) {
        cudaFuncAttributes fa;
        HSS_CUDA_TRY(cudaFuncGetAttributes(&fa, fn));
        HSS_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          optin - (int)fa.sharedSizeBytes));
        HSS_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
      }
      std::vector<IdKernel> gk;
      for (auto fn : group_kernels()) gk.push_back(fn);
      for (auto fn : group_kernels2()) gk.push_back(fn);
      for (auto fn : gk) {
        cudaFuncAttributes fa;
        HSS_CUDA_TRY(cudaFuncGetAttributes(&fa, fn));
        HSS_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          optin - (int)fa.sharedSizeBytes));
      }
      done[dev] = true;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(count * C), 1, 1);
  cfg.blockDim = dim3(ID_THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // the cluster must fit in one GPC with this shared memory: shrink C if not
  // (answers cached per cluster size and shared-memory size)
  static std::mutex occ_mu;
  static std::map<std::pair<int, size_t>, int> occ_cache;
  while (C > 1) {
    int nclusters = 0;
    {
      std::lock_guard<std::mutex> lock(occ_mu);
      auto key = std::make_pair(C, smem);
      auto itc = occ_cache.find(key);
      if (itc != occ_cache.end()) {
        nclusters = itc->second;
      } else {
        cudaError_t oe = cudaOccupancyMaxActiveClusters(&nclusters, id_cpqr_cluster_kernel<1, false>, &cfg);
        if (oe != cudaSuccess) {
          cudaGetLastError();
          nclusters = 0;
        }
        occ_cache[key] = nclusters;
      }
    }
    if (nclusters > 0) break;
    C /= 2;
    attr[0].val.clusterDim.x = C;
    cfg.gridDim = dim3((unsigned)(count * C), 1, 1);
    base = need(C);
    wbytes = sizeof(double) * (size_t)((max_m + C - 1) / C) * (d | 1);
    w_in_smem = base + wbytes <= ID_SMEM_CAP ? 1 : 0;
    smem = base + (w_in_smem ? wbytes : 0);
    cfg.dynamicSmemBytes = smem;
  }
  // group mode: a few large items, whose clusters would leave most SMs idle
  // and whose steps are long (the update of a CTA's share of the columns
  // dominates a barrier in global memory): each item gets gsz CTAs, all
  // resident at once (cooperative launch), at least 8 columns per CTA
  int gsz = 0;
  bool two_per_sm = false;
  {
    const int per_item = sms / count;
    const long step_work = (long)((max_m + C - 1) / C) * d;   // per CTA, cluster mode
    const int g = std::min(per_item, max_m / 8);
    // twice the CTAs, two on each SM, when both fit (registers, shared
    // memory) and each still has at least 8 columns
    const int g2 = std::min(2 * per_item, max_m / 8);
    if (step_work >= GROUP_MIN_STEP_WORK && g2 > 2 * C && g2 >= 2 * g - 1) {
      int nb = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, group_kernels2()[5], ID_THREADS,
                                                        need(g2)) == cudaSuccess &&
          nb >= 2) {
        gsz = g2;
        two_per_sm = true;
      }
      cudaGetLastError();
    }
    if (!two_per_sm && g > 2 * C && step_work >= GROUP_MIN_STEP_WORK) gsz = g;
  }
  // threads per column: results do not depend on it (fixed summation tree),
  // so pick the team size with the fewest FP64 instructions on the busiest of
  // the 4 schedulers.  An FP64 instruction costs the same however few lanes
  // are active; per team and step: 2 d / TS fused multiply-adds (dot product
  // and update), 32 / TS - 1 in-thread and log2 TS shuffle additions, and the
  // multiplication by tau.  Team groups go to warps round-robin, warp w runs
  // on scheduler w % 4.
  auto team_index = [&](int ctas, bool global_cols) {
    const int mloc = (max_m + ctas - 1) / ctas;
    long best = -1;
    int ti = 0;
    // columns in global memory: at least 4 threads per column (a thread per
    // column streams its entries one at a time and measured slower)
    for (int ts = global_cols ? 4 : 1, lg = global_cols ? 2 : 0; ts <= 32; ts *= 2, ++lg) {
      const long groups = ((long)mloc * ts + 31) / 32;
      const long per = 2 * ((d + ts - 1) / ts) + (32 / ts - 1) + lg + 1;
      const long cost = (groups + 3) / 4 * per;
      if (best < 0 || cost < best) {
        best = cost;
        ti = lg;
      }
    }
    return ti;
  };
  // the tuner's work measure of this launch and the device it runs on
  double units = 0.0;
  for (const IdItem& x : h) units += (double)x.m * x.d * std::min(x.m, x.d);
  int dev_ordinal = 0;
  HSS_CUDA_TRY(cudaGetDevice(&dev_ordinal));
  GroupArgs ga = {};
  Err res;
  bool done = false;
  if (gsz > 0) {
    // the tuner may also try half as many CTAs per item when each owns few
    // columns (the per-step serial part -- barrier, candidates, reflector --
    // then weighs less against the columns' work); results do not depend on
    // the choice
    TeamTuner::Trial* trial = nullptr;
    const bool half_ok = (max_m + gsz - 1) / gsz < 32 && gsz >= 4 &&
                         need(gsz / 2) <= 227 * 1024 - 2048;
    const int choice = TeamTuner::get().choose(
        TeamTuner::Key{dev_ordinal, two_per_sm ? 2 : 1, 0, ilog2(max_m), ilog2(d), ilog2(count), half_ok},
        team_index(gsz, true), 2, units, &trial, half_ok);
    const int ti = choice & 7;
    if (choice >> 3) gsz /= 2;
    const size_t gsmem = need(gsz);
    // candidates [count][2][gsz], then the counters, the abort flag and the
    // error code (zeroed together)
    const size_t cand_bytes = sizeof(Cand) * 2 * (size_t)gsz * count;
    const size_t ctl_bytes = sizeof(unsigned) * ((size_t)count + 2);
    char* gbuf = nullptr;
    if (scratch) HSS_TRY(scratch->alloc(reinterpret_cast<void**>(&gbuf), cand_bytes + ctl_bytes, s));
    else HSS_TRY(dalloc(reinterpret_cast<void**>(&gbuf), cand_bytes + ctl_bytes, s));
    ga.gsz = gsz;
    ga.limit = fault_wait_limit() > 0 ? fault_wait_limit() : GROUP_WAIT_LIMIT;
    ga.cand = reinterpret_cast<Cand*>(gbuf);
    ga.ctr = reinterpret_cast<unsigned*>(gbuf + cand_bytes);
    ga.abort = reinterpret_cast<int*>(ga.ctr + count);
    ga.err = ga.abort + 1;
    HSS_CUDA_TRY(cudaMemsetAsync(ga.ctr, 0, ctl_bytes, s));
    // one spread-out launch at a time in the process: its CTAs wait for one
    // another, so two of them sharing the GPU (two threads, two streams)
    // could each hold SMs the other's waiting CTAs need; the lock is held
    // until this launch has completed (the stream is synchronized below)
    static std::mutex coop_mu;
    std::lock_guard<std::mutex> coop_lock(coop_mu);
    cudaLaunchConfig_t gcfg = {};
    gcfg.gridDim = dim3((unsigned)(count * gsz), 1, 1);
    gcfg.blockDim = dim3(ID_THREADS, 1, 1);
    gcfg.dynamicSmemBytes = gsmem;
    gcfg.stream = s;
    cudaLaunchAttribute gattr[1];
    gattr[0].id = cudaLaunchAttributeCooperative;
    gattr[0].val.cooperative = 1;
    gcfg.attrs = gattr;
    gcfg.numAttrs = 1;
    if (trial) cudaEventRecord(trial->e0, s);
    cudaError_t e = cudaLaunchKernelEx(&gcfg, (two_per_sm ? group_kernels2() : group_kernels())[ti],
                                       items_dev,
                                       f64 ? 1 : 0, r1, (const int64_t*)offd, ga);
    if (trial) {
      if (e == cudaSuccess) cudaEventRecord(trial->e1, s);
      TeamTuner::get().launched(trial, e == cudaSuccess);
    }
    if (e == cudaErrorCooperativeLaunchTooLarge) {
      // fewer SMs than expected are free for this context: clusters instead
      cudaGetLastError();
    } else {
      done = true;
      if (e != cudaSuccess) {
        cudaGetLastError();
        res = fail(HSS_ERR_CUDA, std::string("id_cpqr group launch: ") + cudaGetErrorString(e));
      } else {
        res = check_launch("id_cpqr_cluster_kernel");
      }
      if (res.st == HSS_OK) {
        int herr = 0;
        HSS_CUDA_TRY(cudaMemcpyAsync(&herr, ga.err, sizeof(int), cudaMemcpyDeviceToHost, s));
        HSS_CUDA_TRY(cudaStreamSynchronize(s));
        if (herr) res = fail(HSS_ERR_TIMEOUT, "id_cpqr: a group barrier wait timed out");
      }
    }
    if (!scratch) dfree(gbuf, s);
    ga = GroupArgs{};
  }
  if (!done) {
    // more CTAs than SMs, columns in global memory: two CTAs per SM when
    // they fit (registers, shared memory)
    auto two_fit = [&](int c, size_t sm_bytes, int in_smem) {
      if ((long)count * c <= sms || in_smem) return false;
      int nb = 0;
      const bool ok = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                          &nb, kernels2()[5], ID_THREADS, sm_bytes) == cudaSuccess && nb >= 2;
      cudaGetLastError();
      return ok;
    };
    bool two = two_fit(C, smem, w_in_smem);
    // the tuner may also try clusters twice as large when the launch leaves
    // SMs with fewer than two CTAs and the columns are in global memory
    // (more warps per SM to hide the columns' memory latency, a cluster
    // barrier per step in exchange); results do not depend on the choice
    const int C2 = 2 * C;
    const size_t smem2 = need(C2);
    bool dbl_ok = !w_in_smem && C2 <= 16 && (long)count * C < 2L * sms && max_m / C2 >= 16 &&
                  smem2 <= 227 * 1024 - 2048;
    if (dbl_ok) {
      cudaLaunchConfig_t c2 = cfg;
      cudaLaunchAttribute a2[1];
      a2[0] = attr[0];
      a2[0].val.clusterDim.x = C2;
      c2.attrs = a2;
      c2.gridDim = dim3((unsigned)(count * C2), 1, 1);
      c2.dynamicSmemBytes = smem2;
      int ncl = 0;
      if (cudaOccupancyMaxActiveClusters(&ncl, id_cpqr_cluster_kernel<1, false>, &c2) != cudaSuccess)
        ncl = 0;
      cudaGetLastError();
      dbl_ok = ncl > 0;
    }
    TeamTuner::Trial* trial = nullptr;
    const int choice = TeamTuner::get().choose(
        TeamTuner::Key{dev_ordinal, two ? 3 : 0, w_in_smem, ilog2(max_m), ilog2(d), ilog2(count), dbl_ok},
        team_index(C, w_in_smem == 0), w_in_smem ? 0 : 2, units, &trial, false, dbl_ok);
    const int ti = choice & 7;
    if (choice & 16) {   // clusters of C2: the columns stay in global memory
      C = C2;
      smem = smem2;
      attr[0].val.clusterDim.x = C;
      cfg.gridDim = dim3((unsigned)(count * C), 1, 1);
      cfg.dynamicSmemBytes = smem;
      two = two_fit(C, smem, 0);
    }
    if (trial) cudaEventRecord(trial->e0, s);
    // (clusters of 4 and more: two CTAs per SM also where there are SMs enough,
    // as for the columns in shared memory)
    const IdKernel fn = (w_in_smem ? smem_kernels() : two || C >= 4 ? kernels2() : kernels())[ti];
    cudaError_t e = cudaLaunchKernelEx(&cfg, fn, items_dev, f64 ? 1 : 0, r1, (const int64_t*)offd, ga);
    if (trial) {
      if (e == cudaSuccess) cudaEventRecord(trial->e1, s);
      TeamTuner::get().launched(trial, e == cudaSuccess);
    }
    if (e != cudaSuccess) cudaGetLastError();   // (reported here, not to the caller's next call)
    res = e == cudaSuccess ? check_launch("id_cpqr_cluster_kernel")
                           : fail(HSS_ERR_CUDA, std::string("id_cpqr_cluster_kernel launch: ") +
                                                    cudaGetErrorString(e));
  }
  if (!scratch) {
    dfree(r1, s);
    dfree(offd, s);
  }
  return res;
}

}  // namespace hss
