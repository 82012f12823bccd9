// Solution with the ULV factors (Algorithm 4, Appendix A) of one or many
// handles in one launch, in FP64 whatever the handles' dtype.
//
//   up    b = B(I) at a leaf, [g_1 - B12 z_2; g_2 - B21 z_1] above;
//         y = L^{-1} (b(perm(k..)) - E b(perm(0..k)))   (Omega b = [.; .])
//         g = b(perm(0..k)) - W_b Q_t^T y,
//         z = Vtilde_t^T y (+ V^T [z_1; z_2]);
//   root  x = U^{-1} L^{-1} P b;
//   down  x = Q^T [y; the parent's part], the reflectors by panels of 32 in
//         compact WY form: t_p = T_p V_p v, v <- v - V_p^T t_p, last panel first.
//
// Every line is a product with a stored matrix, so the whole solve is a table
// of tasks as in the HSS product (hss_matvec.cu): at most 32 rows of one
// result for NC right-hand sides, claimed in dependence order from a ticket
// counter, each polling the values it needs (the work buffer starts as
// all-ones NaNs; a poll is bounded, and on a timeout the NaN reaches the
// solution and the handle's next call reports it).  Triangular systems go by blocks of 32 rows: a task subtracts
// the rows of L it needs and multiplies by the inverse of its diagonal block
// (hss_factor leaves these, hss_ulv.cu; an ill-conditioned block is left as it
// is, and the task substitutes), so the chain is one task per 32 rows.
// One launch per tree level and operation (23 to 112 a solve), a warp per
// right-hand side on its triangular chain, spent 5 FP64 instructions for
// every useful one on narrow reductions: an FP64 instruction holds its pipe
// for 64 cycles whatever it computes.  Here a thread sums one row for all NC
// columns, and the partial sums of a task meet once.
//
// A column's sums depend neither on nrhs nor on what shares the launch.  A
// handle's table depends on its tree and ranks; it is built at the first solve
// after a factorization and kept with the factors.
//
// What bounds it: at one column the chain of dependent tasks (about 4 us per
// 32-row block of a triangular system, 10 us per panel of Q at m = 600), at
// many columns FP64 work at about half its rate.  Measured (GB300, whole call,
// against one launch per tree level and operation): Toeplitz n = 80,000, FP64, 1
// / 16 columns 1.80 -> 0.45, 4.6 -> 1.34 ms; Schur complement n = 5041, FP32, 1 /
// 32 columns 4.8 -> 0.90, 9.9 -> 2.26 ms; n = 10,000, 64 columns 82 -> 8.9 ms.
#include "hss_internal.cuh"
#include "hss_tree.h"

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <climits>

using namespace hss;

namespace hss {

namespace {

constexpr int SV_ROWS = 32, SV_THREADS = 128;
// A stage holds 1024 matrix entries: 32 inner indices of 32 rows, 64 of 16 or
// 128 of 8.  (A chain's task waits for its last stage only, so stages of 32
// rows are short; 8-row tasks have long sums and want few stages.)
constexpr int SV_ENT = 1024;
constexpr int SV_LMAX = SV_ENT / 8;
constexpr int SV_FINE_M = 160;
constexpr int SV_COLS = 64;   // right-hand sides per launch, fewer where memory is short
constexpr long long SV_WAIT_LIMIT = 1ll << 33;   // clock cycles (about 4 s)

enum {   // SvTerm::flags
  ST_TRANS = 1,    // M(row, l) = M[l * ld + row], else M[row * ld + l]
  ST_NATIVE = 2,   // M has the handle's dtype, else FP64
  ST_INPUT = 4,    // the vector is the caller's B, else the work buffer
  ST_LOWER = 8,    // l < r0 only (r0 = the task's first row)
  ST_UPPER = 16    // l >= r0 + SV_ROWS only
};
enum {   // SvDesc::flags
  SD_POST_LOWER = 32,   // post is lower triangular
  SD_POST_UPPER = 64,   // ... upper
  SD_X = 1,          // an entry of a vector besides the sums
  SD_XINPUT = 2,     // ... of the caller's B
  SD_NEG = 4,        // the sums are subtracted
  SD_BUF = 8,        // the result goes to the work buffer
  SD_OUT = 16        // ... to the caller's X
};

// sum_l M(row, l) v[l] over vector rows zmap[l] (or l): rows below split start
// at z0, the others at z1
struct SvTerm {
  const void* M;
  const int32_t* zmap;
  int64_t z0, z1;
  int32_t ld, inner, split, flags;
};

// rows r of one result: entry xmap[r] (or r) of the X vector (rows below
// xsplit start at x0, the others at x1) plus or minus the terms, then times
// the task's 32 x 32 block of `post`
struct alignas(16) SvDesc {
  SvTerm t[2];
  const int32_t* xmap;
  const double* post;
  int64_t x0, x1, out, outx;
  int32_t xsplit, rows, flags, nterm, trows;   // trows: rows per task (8, 16 or 32)
  int32_t pad[3];
};
static_assert(sizeof(SvDesc) == 176, "copied as 16-byte pieces");

// one handle's system
struct SvJob {
  const SvDesc* descs;
  double* buf;
  const void* B;
  void* X;
  unsigned* timeout;   // the handle's word for a poll that has run out
  int64_t ldb, ldx;
  int32_t nrhs, pad;
};

struct SvArgs {
  SvJob job;           // the only job (list null)
  const int2* tasks;   // ... its tasks: (description, r0)
  const SvJob* jobs;   // several jobs
  const int4* list;    // ... (job, description, r0, column chunk)
  unsigned* ctl;       // [0] ticket, [1] a poll has timed out
  long long limit;     // of a poll, in clock cycles
  unsigned total;
  int nch;
};

__device__ __forceinline__ double sv_ld(const double* p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ bool sv_unset(double v) { return __double_as_longlong(v) == -1ll; }

// *p once it has been written (bounded; the flag ends the other polls early)
__device__ __forceinline__ double sv_poll(const double* p, const SvArgs& g, const SvJob& jb) {
  double v = sv_ld(p);
  if (!sv_unset(v)) return v;
  const long long t0 = clock64();
  unsigned polls = 0;
  while (sv_unset(v = sv_ld(p))) {
    if ((++polls & 31u) != 0u) continue;
    bool out = *reinterpret_cast<volatile unsigned*>(g.ctl + 1) != 0;
    if (!out && clock64() - t0 > g.limit) {
      atomicExch(g.ctl + 1, 1u);
      out = true;
    }
    if (out) {   // (the other jobs' polls end early as well: each marks its own)
      *reinterpret_cast<volatile unsigned*>(jb.timeout) = 1u;
      break;
    }
  }
  return v;
}

template <int BYTES>
__device__ __forceinline__ void sv_cp(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES));
}

// one stage of a matrix: rows r0 .. and inner indices l0 .., [row][l] (odd
// pitch), or (trans) [l][trows]
template <typename S>
__device__ __forceinline__ void sv_load(S* dst, const S* M, int64_t ld, bool trans, int r0,
                                        int rows, int trows, int l0, int lc) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (trans) {
    const int r = threadIdx.x & (trows - 1);
    if (r < rows)
      for (int l = threadIdx.x / trows; l < lc; l += SV_THREADS / trows)
        sv_cp<sizeof(S)>(dst + l * trows + r, M + (int64_t)(l0 + l) * ld + r0 + r);
    return;
  }
  const int pitch = SV_ENT / trows + 1;
  for (int r = w; r < rows; r += SV_THREADS / 32) {
    const S* row = M + (int64_t)(r0 + r) * ld + l0;
    for (int l = lane; l < lc; l += 32) sv_cp<sizeof(S)>(dst + r * pitch + l, row + l);
  }
}

// a += the terms l = part, part + parts, ... of this thread's row, in turn
// into two chains (an FP64 operation takes 67 cycles)
template <typename S, int NC>
__device__ __forceinline__ void sv_fma(double (&a)[2][NC], const S* ms, const double* zs, int row,
                                       int part, int parts, int srow, int sl, int lc) {
  const S* m = ms + row * srow;
  int l = part;
#pragma unroll 2
  for (; l + parts < lc; l += 2 * parts) {
    const double m0 = (double)m[l * sl], m1 = (double)m[(l + parts) * sl];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      a[0][c] = fma(m0, zs[l * NC + c], a[0][c]);
      a[1][c] = fma(m1, zs[(l + parts) * NC + c], a[1][c]);
    }
  }
  if (l < lc) {
    const double m0 = (double)m[l * sl];
#pragma unroll
    for (int c = 0; c < NC; ++c) a[0][c] = fma(m0, zs[l * NC + c], a[0][c]);
  }
}

// v <- B^-1 v for the columns of v ([row][NC]) by substitution, a warp per
// column, lane = row.  divided: B's rows are divided by its diagonal, where the
// reciprocals stand; else B itself.
template <int NC>
__device__ __forceinline__ void sv_substitute(double* v, const double* B, int rows, bool upper,
                                              bool divided) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (w >= NC) return;
  const double* row = B + lane * (SV_ROWS + 1);
  double x = lane < rows ? v[lane * NC + w] : 0.0;
  if (divided) {
    x *= row[lane];
    if (upper) {
#pragma unroll 8
      for (int t = SV_ROWS - 1; t > 0; --t) {
        const double xt = __shfl_sync(0xffffffffu, x, t);
        if (lane < t && t < rows) x = fma(-row[t], xt, x);
      }
    } else {
#pragma unroll 8
      for (int t = 0; t < SV_ROWS - 1; ++t) {
        const double xt = __shfl_sync(0xffffffffu, x, t);
        if (lane > t) x = fma(-row[t], xt, x);
      }
    }
  } else {
    for (int q = 0; q < rows; ++q) {
      const int t = upper ? rows - 1 - q : q;
      if (lane == t) x /= row[t];
      const double xt = __shfl_sync(0xffffffffu, x, t);
      if (upper ? lane < t : lane > t) x = fma(-row[t], xt, x);
    }
  }
  if (lane < rows) v[lane * NC + w] = x;
}

constexpr int SV_MS = SV_ENT + SV_ROWS;   // a stage's matrix with its odd pitch
template <int NC>
constexpr size_t sv_smem() {   // two stages, their vectors, the post block
  return sizeof(double) * (2 * SV_MS + 2 * SV_LMAX * NC + SV_ROWS * (SV_ROWS + 1));
}

template <typename T, int NC, bool BATCH>
__global__ void __launch_bounds__(SV_THREADS, NC == 4 ? 5 : 6) ulv_solve_kernel(const SvArgs g) {
  extern __shared__ __align__(16) double sv_raw[];
  double* ms = sv_raw;                              // [2][SV_MS]
  double* zs = ms + 2 * SV_MS;                      // [2][SV_LMAX * NC]
  double* ps = zs + 2 * SV_LMAX * NC;               // [SV_ROWS][SV_ROWS + 1]
  static_assert(SV_LMAX >= SV_THREADS / 2, "the partial sums take the place of the vectors");
  static_assert(SV_ENT / SV_ROWS % (2 * SV_THREADS / 8) == 0, "whole turns of the chains in a stage");
  double* red = zs;                                 // [part][row][NC], after the last stage
  __shared__ int idx[2][SV_LMAX];
  __shared__ SvDesc tk;
  __shared__ SvJob jb;
  __shared__ unsigned snext;
  constexpr int EO = SV_ROWS * NC > SV_THREADS ? SV_ROWS * NC / SV_THREADS : 1;   // outputs per thread
  const int tid = threadIdx.x, lane = tid & 31;
  unsigned claim = 0;
  if (tid == 0) snext = atomicAdd(g.ctl, 1u);
  if (!BATCH && tid == 0) jb = g.job;
  __syncthreads();
  while (true) {
    const unsigned tick = snext;
    if (tick >= g.total) return;
    int4 task;
    if (BATCH) {
      task = g.list[tick];
      if (tid < (int)(sizeof(SvJob) / 4))
        reinterpret_cast<uint32_t*>(&jb)[tid] = reinterpret_cast<const uint32_t*>(g.jobs + task.x)[tid];
      const SvDesc* d = g.jobs[task.x].descs + task.y;
      if (tid < (int)(sizeof(SvDesc) / 16))
        reinterpret_cast<uint4*>(&tk)[tid] = reinterpret_cast<const uint4*>(d)[tid];
    } else {
      const int2 t2 = g.tasks[tick / (unsigned)g.nch];
      task = make_int4(0, t2.x, t2.y, (int)(tick % (unsigned)g.nch));
      if (tid < (int)(sizeof(SvDesc) / 16))
        reinterpret_cast<uint4*>(&tk)[tid] = reinterpret_cast<const uint4*>(g.job.descs + t2.x)[tid];
    }
    __syncthreads();
    if (tid == 0) claim = atomicAdd(g.ctl, 1u);   // the next ticket, needed at the end only
    const int r0 = task.z, cb = task.w * NC, nr = jb.nrhs, nc = min(NC, nr - cb);
    const int rows = min(tk.trows, tk.rows - r0);
    const int trows = tk.trows;
    const int rows8 = rows <= 8 ? 8 : rows <= 16 ? 16 : 32, parts = SV_THREADS / rows8;
    const int SL = SV_ENT / trows;   // inner indices per stage
    const int row = tid & (rows8 - 1), part = tid / rows8;
    double* buf = jb.buf;
    // inner range of a term
    auto lbeg = [&](const SvTerm& t) { return t.flags & ST_UPPER ? min(t.inner, r0 + SV_ROWS) : 0; };
    auto lend = [&](const SvTerm& t) { return t.flags & ST_LOWER ? min(t.inner, r0) : t.inner; };
    auto stages = [&](const SvTerm& t) { return (lend(t) - lbeg(t) + SL - 1) / SL; };
    // first inner index of a term's q-th stage: in the order in which a chain
    // makes the entries, so that only the last stage waits for its neighbour
    auto lfirst = [&](const SvTerm& t, int q) {
      return lbeg(t) + (t.flags & ST_UPPER ? stages(t) - 1 - q : q) * SL;
    };
    const int n0 = tk.nterm > 0 ? stages(tk.t[0]) : 0;
    const int nst = n0 + (tk.nterm > 1 ? stages(tk.t[1]) : 0);
    auto issue = [&](int k) {   // stage k's matrix entries and row indices
      if (k < nst) {
        const SvTerm& t = tk.t[k < n0 ? 0 : 1];
        const int l0 = lfirst(t, k < n0 ? k : k - n0), lc = min(SL, lend(t) - l0);
        if (t.zmap && tid < lc) sv_cp<4>(&idx[k & 1][tid], t.zmap + l0 + tid);
        double* d = ms + (k & 1) * SV_MS;
        const bool tr = (t.flags & ST_TRANS) != 0;
        if (t.flags & ST_NATIVE)
          sv_load(reinterpret_cast<T*>(d), reinterpret_cast<const T*>(t.M), t.ld, tr, r0, rows, trows, l0, lc);
        else
          sv_load(d, reinterpret_cast<const double*>(t.M), t.ld, tr, r0, rows, trows, l0, lc);
      }
      asm volatile("cp.async.commit_group;");
    };
    if (tk.post) {   // the block's inverse (or T): 32 x 32
      const double* P = tk.post + (size_t)(r0 / SV_ROWS) * SV_ROWS * SV_ROWS;
      for (int e = tid; e < SV_ROWS * SV_ROWS; e += SV_THREADS)
        sv_cp<8>(ps + (e / SV_ROWS) * (SV_ROWS + 1) + e % SV_ROWS, P + e);
    }
    issue(0);
    const int nrow_b = nr;   // pitch of the work buffer
    const T* Bin = reinterpret_cast<const T*>(jb.B) + cb;
    // indices of this thread's outputs' X entries
    int xr[EO];
#pragma unroll
    for (int o = 0; o < EO; ++o) {
      const int e = tid + o * SV_THREADS, r = e / NC, c = e - r * NC;
      xr[o] = -1;
      if ((tk.flags & SD_X) && r < rows && c < nc) xr[o] = tk.xmap ? tk.xmap[r0 + r] : r0 + r;
    }
    double acc[2][NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[0][c] = acc[1][c] = 0.0;
    constexpr int U = SV_LMAX * NC / SV_THREADS;
    // addresses of this thread's vector entries of stage k in the work buffer
    // (null: no entry, or the caller's B)
    auto entries = [&](int k, const double* (&p)[U]) {
      const SvTerm& t = tk.t[k < n0 ? 0 : 1];
      const int l0 = lfirst(t, k < n0 ? k : k - n0), lc = min(SL, lend(t) - l0);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = tid + u * SV_THREADS, l = e / NC, c = e - l * NC;
        p[u] = nullptr;
        if (l < lc && c < nc) {
          const int q = t.zmap ? idx[k & 1][l] : l0 + l;
          p[u] = buf + (q < t.split ? t.z0 + q : t.z1 + (q - t.split)) * nrow_b + cb + c;
        }
      }
    };
    double v[U];
    bool ahead = false;   // v holds stage k's entries, read while stage k - 1 was multiplied
    for (int k = 0; k < nst; ++k) {
      const SvTerm& t = tk.t[k < n0 ? 0 : 1];
      const int l0 = lfirst(t, k < n0 ? k : k - n0), lc = min(SL, lend(t) - l0);
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      const bool mapped = t.zmap != nullptr;
      if (mapped) __syncthreads();   // idx was copied by other threads
      if (t.flags & ST_INPUT) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = tid + u * SV_THREADS, l = e / NC, c = e - l * NC;
          v[u] = 0.0;
          if (l < lc && c < nc)
            v[u] = (double)Bin[(t.z0 + (mapped ? idx[k & 1][l] : l0 + l)) * jb.ldb + c];
        }
      } else {
        const double* p[U];
        entries(k, p);
        if (!ahead) {
          // one lane of each warp polls until its value is there, then every
          // value is read
          if (lane == 0 && p[0]) sv_poll(p[0], g, jb);
          __syncwarp();
#pragma unroll
          for (int u = 0; u < U; ++u) v[u] = p[u] ? sv_ld(p[u]) : 0.0;
        }
        if (__any_sync(0xffffffffu, p[0] && sv_unset(v[0]))) {
          if (lane == 0 && p[0]) sv_poll(p[0], g, jb);
          __syncwarp();
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (p[u] && sv_unset(v[u])) v[u] = sv_poll(p[u], g, jb);
      }
      double* z = zs + (k & 1) * SV_LMAX * NC;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = tid + u * SV_THREADS;
        if (e < lc * NC) z[e] = v[u];
      }
      __syncthreads();
      issue(k + 1);
      ahead = false;
      if (k + 1 < nst) {
        const SvTerm& tn = tk.t[k + 1 < n0 ? 0 : 1];
        if (!(tn.flags & ST_INPUT) && !tn.zmap) {
          const double* p[U];
          entries(k + 1, p);
#pragma unroll
          for (int u = 0; u < U; ++u) v[u] = p[u] ? sv_ld(p[u]) : 0.0;
          ahead = true;
        }
      }
      {
        const double* m = ms + (k & 1) * SV_MS;
        const bool tr = (t.flags & ST_TRANS) != 0;
        const int srow = tr ? 1 : SL + 1, sl = tr ? trows : 1;
        if (t.flags & ST_NATIVE)
          sv_fma<T, NC>(acc, reinterpret_cast<const T*>(m), z, row, part, parts, srow, sl, lc);
        else
          sv_fma<double, NC>(acc, m, z, row, part, parts, srow, sl, lc);
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    double xv[EO];
#pragma unroll
    for (int o = 0; o < EO; ++o) {
      const int c = (tid + o * SV_THREADS) % NC;
      xv[o] = 0.0;
      if (xr[o] < 0) continue;
      if (tk.flags & SD_XINPUT) xv[o] = (double)Bin[(tk.x0 + xr[o]) * jb.ldb + c];
      else
        xv[o] = sv_poll(buf + (xr[o] < tk.xsplit ? tk.x0 + xr[o] : tk.x1 + (xr[o] - tk.xsplit)) * nrow_b +
                            cb + c, g, jb);
    }
    __syncthreads();   // every warp is done with zs
    {
#pragma unroll
      for (int c = 0; c < NC; ++c) red[(part * rows8 + row) * NC + c] = acc[0][c] + acc[1][c];
    }
    if (tid == 0) snext = claim;
    __syncthreads();
    double val[EO];
#pragma unroll
    for (int o = 0; o < EO; ++o) {
      const int e = tid + o * SV_THREADS;
      val[o] = 0.0;
      if (e >= rows * NC) continue;
      double v = red[e];
      for (int q = 1; q < parts; ++q) v += red[q * rows8 * NC + e];
      val[o] = tk.flags & SD_NEG ? xv[o] - v : xv[o] + v;
    }
    if (tk.post) {   // the block's rows meet in ms, then the 32 x 32 product
#pragma unroll
      for (int o = 0; o < EO; ++o) {
        const int e = tid + o * SV_THREADS;
        if (e < rows * NC) ms[e] = val[o];
      }
      __syncthreads();
      const bool up = (tk.flags & SD_POST_UPPER) != 0;
      const double kind = ps[up ? (SV_ROWS - 1) * (SV_ROWS + 1) : SV_ROWS - 1];
      if (kind == 0.0) {
#pragma unroll
        for (int o = 0; o < EO; ++o) {
          const int e = tid + o * SV_THREADS, r = e / NC, c = e - r * NC;
          if (r >= rows) continue;
          double s[4] = {0.0, 0.0, 0.0, 0.0};
          const double* p = ps + r * (SV_ROWS + 1);
          // (the zeros of a triangular block are left out four at a time)
          int l = up ? r & ~3 : 0;
          const int end = tk.flags & SD_POST_LOWER ? min(rows, (r & ~3) + 4) : rows;
          for (; l + 3 < end; l += 4)
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] = fma(p[l + q], ms[(l + q) * NC + c], s[q]);
#pragma unroll
          for (int q = 0; q < 3; ++q)
            if (l + q < end) s[q] = fma(p[l + q], ms[(l + q) * NC + c], s[q]);
          val[o] = (s[0] + s[1]) + (s[2] + s[3]);
        }
      } else {   // the block, not its inverse
        sv_substitute<NC>(ms, ps, rows, up, kind == 1.0);
        __syncthreads();
#pragma unroll
        for (int o = 0; o < EO; ++o) {
          const int e = tid + o * SV_THREADS;
          if (e < rows * NC) val[o] = ms[e];
        }
      }
    }
#pragma unroll
    for (int o = 0; o < EO; ++o) {
      const int e = tid + o * SV_THREADS, r = e / NC, c = e - r * NC;
      if (r >= rows || c >= nc) continue;
      if (tk.flags & SD_OUT)
        reinterpret_cast<T*>(jb.X)[(tk.outx + r0 + r) * jb.ldx + cb + c] = (T)val[o];
      if (tk.flags & SD_BUF) {   // (a NaN of the caller's may carry the unset pattern through)
        const double w = sv_unset(val[o]) ? (double)NAN : val[o];
        asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(
                         buf + (tk.out + r0 + r) * nrow_b + cb + c), "d"(w) : "memory");
      }
    }
    // (the shared buffers are written again only after every thread has passed here)
    __syncthreads();
  }
}

using SvKernel = void (*)(const SvArgs);
template <typename T, bool BATCH>
SvKernel sv_kernel(int nc, size_t* smem) {
  switch (nc) {
    case 1: *smem = sv_smem<1>(); return ulv_solve_kernel<T, 1, BATCH>;
    case 2: *smem = sv_smem<2>(); return ulv_solve_kernel<T, 2, BATCH>;
    default: *smem = sv_smem<4>(); return ulv_solve_kernel<T, 4, BATCH>;
  }
}

// The task table of a factored handle.  phases: first task of each phase
// (tasks of a phase do not depend on one another), for interleaving handles.
struct SvPlan {
  std::vector<SvDesc> descs;
  std::vector<int2> tasks;
  std::vector<int> phases;
  int64_t rows = 0;   // of the work buffer
  double entries = 0.0;   // matrix entries that the tasks multiply by
};

void sv_build(const hss_s* h, SvPlan& pl) {
  const Tree& tr = h->tree;
  const UlvFactors& F = h->ulv;
  const int nn = (int)tr.nodes.size();
  std::vector<int64_t> ob(nn, 0), oy(nn, 0), og(nn, 0), oz(nn, 0), ox(nn, 0);
  int64_t tot = 0;
  auto take = [&](int64_t rows) {
    const int64_t o = tot;
    tot += rows;
    return o;
  };
  for (int id = 0; id < nn; ++id) {
    const UlvNode& u = F.nodes[id];
    if (tr.nodes[id].c1 >= 0) ob[id] = take(u.m);
    oy[id] = take(id == 0 ? u.m : u.m - u.k);
    if (id == 0) continue;
    og[id] = take(u.k);
    oz[id] = take(u.kc);
  }
  pl.descs.reserve(8 * (size_t)nn);
  // one phase: the tiles [t0, t1) of descriptions (all tiles by default)
  auto phase = [&]() {
    if (pl.phases.empty() || pl.phases.back() != (int)pl.tasks.size())
      pl.phases.push_back((int)pl.tasks.size());
  };
  auto tile = [&](int desc, int r0) { pl.tasks.push_back(make_int2(desc, r0)); };
  auto add = [&](const SvDesc& d) {
    pl.descs.push_back(d);
    return (int)pl.descs.size() - 1;
  };
  auto add_all = [&](const SvDesc& d) {
    if (d.rows <= 0) return;
    const int q = add(d);
    for (int r0 = 0; r0 < d.rows; r0 += d.trows) tile(q, r0);
  };
  auto blank = [](int rows, int64_t out, int flags) {
    SvDesc d{};
    d.rows = rows;
    d.out = out;
    d.flags = flags;
    d.xsplit = INT32_MAX;
    d.trows = SV_ROWS;
    return d;
  };
  // rows per task of a node of order m: nodes of a few hundred rows are few
  // (the top of the tree) and their sums long, so they go by 8 rows
  auto fine = [](int m) { return m > SV_FINE_M; };

  auto term = [](SvDesc& d, const void* M, int64_t ld, int inner, int flags, int64_t z0,
                 const int32_t* zmap = nullptr, int split = INT32_MAX, int64_t z1 = 0) {
    if (inner <= 0) return;
    SvTerm& t = d.t[d.nterm++];
    t.M = M;
    t.ld = (int32_t)ld;
    t.inner = inner;
    t.flags = flags;
    t.z0 = z0;
    t.z1 = z1;
    t.zmap = zmap;
    t.split = split;
  };
  // a triangular system's tasks, one phase per 32-row block across the level's
  // nodes: (description, rows)
  auto chain = [&](const std::vector<std::pair<int, int>>& ds, bool up) {
    int maxb = 0;
    for (auto& q : ds) maxb = std::max(maxb, (q.second + SV_ROWS - 1) / SV_ROWS);
    for (int b = 0; b < maxb; ++b) {
      phase();
      for (auto& q : ds) {
        const int nb = (q.second + SV_ROWS - 1) / SV_ROWS;
        if (b < nb) tile(q.first, SV_ROWS * (up ? nb - 1 - b : b));
      }
    }
  };
  for (int depth = tr.maxdepth; depth >= 0; --depth) {
    phase();
    for (int id : tr.levels[depth]) {   // b of non-leaves
      const TNode& nd = tr.nodes[id];
      if (nd.c1 < 0) continue;
      const NodeGen& g = h->gen[id];
      const UlvNode& a = F.nodes[nd.c1];
      const UlvNode& b = F.nodes[nd.c2];
      SvDesc d = blank(a.k, ob[id], SD_X | SD_NEG | SD_BUF);
      d.x0 = og[nd.c1];
      if (fine(a.k + b.k)) d.trows = 8;
      term(d, g.B12, b.kc, b.kc, ST_NATIVE, oz[nd.c2]);
      add_all(d);
      d = blank(b.k, ob[id] + a.k, SD_X | SD_NEG | SD_BUF);
      d.x0 = og[nd.c2];
      if (fine(a.k + b.k)) d.trows = 8;
      term(d, g.B21, a.kc, a.kc, ST_NATIVE, oz[nd.c1]);
      add_all(d);
    }
    if (depth == 0) break;
    std::vector<std::pair<int, int>> ys;
    for (int id : tr.levels[depth]) {   // y
      const TNode& nd = tr.nodes[id];
      const NodeGen& g = h->gen[id];
      const UlvNode& u = F.nodes[id];
      const int r = u.m - u.k, leaf = nd.c1 < 0;
      if (r <= 0) continue;
      SvDesc d = blank(r, oy[id], SD_X | SD_NEG | SD_BUF | SD_POST_LOWER | (leaf ? SD_XINPUT : 0));
      d.x0 = leaf ? nd.lo : ob[id];
      d.xmap = g.permr + u.k;
      d.post = u.Li;
      term(d, g.Er, u.k, u.k, leaf ? ST_INPUT : 0, d.x0, g.permr);
      term(d, u.L, r, r, ST_LOWER, oy[id]);
      ys.push_back({add(d), r});
    }
    chain(ys, false);
    phase();
    for (int id : tr.levels[depth]) {   // g and z
      const TNode& nd = tr.nodes[id];
      const NodeGen& g = h->gen[id];
      const UlvNode& u = F.nodes[id];
      const int r = u.m - u.k, leaf = nd.c1 < 0;
      SvDesc d = blank(u.k, og[id], SD_X | SD_NEG | SD_BUF | (leaf ? SD_XINPUT : 0));
      d.x0 = leaf ? nd.lo : ob[id];
      d.xmap = g.permr;
      if (fine(u.m)) d.trows = 8;
      term(d, u.WbQt, r, r, 0, oy[id]);
      add_all(d);
      d = blank(u.kc, oz[id], SD_BUF | (leaf ? 0 : SD_X));
      if (fine(u.m)) d.trows = 8;
      term(d, u.Vtt, u.kc, r, ST_TRANS, oy[id]);
      if (!leaf) {
        d.x0 = oz[nd.c1];
        d.x1 = oz[nd.c2];
        d.xsplit = F.nodes[nd.c1].kc;
        d.xmap = g.permc;
        term(d, g.Ec, u.kc, g.mc - u.kc, ST_TRANS, d.x0, g.permc + u.kc, d.xsplit, d.x1);
      }
      add_all(d);
    }
  }
  {   // root: x = U^{-1} L^{-1} P b
    const int m = F.root_m, leaf = nn == 1;
    ox[0] = take(m);
    SvDesc d = blank(m, oy[0], SD_X | SD_NEG | SD_BUF | SD_POST_LOWER | (leaf ? SD_XINPUT : 0));
    d.x0 = leaf ? 0 : ob[0];
    d.xmap = F.root_perm;
    d.post = F.root_li;
    term(d, F.root_lu, m, m, ST_LOWER, oy[0]);
    chain({{add(d), m}}, false);
    d = blank(m, ox[0], SD_X | SD_NEG | SD_BUF | SD_POST_UPPER | (leaf ? SD_OUT : 0));
    d.x0 = oy[0];
    d.post = F.root_ui;
    term(d, F.root_lu, m, m, ST_UPPER, ox[0]);
    chain({{add(d), m}}, true);
  }
  for (int depth = 0; depth < tr.maxdepth; ++depth) {
    // the children of this depth's nodes, panels of each from its last; rows
    // [i0, m) of the running v: below `split` the entries of y not touched
    // yet, then the last panel's result (or the parent's part)
    struct Kid {
      int id, np;
      int64_t tail, xp;   // where the part behind y starts, the parent's part
      int split;          // first row of that part
    };
    std::vector<Kid> kids;
    int maxp = 0;
    for (int id : tr.levels[depth]) {
      const TNode& nd = tr.nodes[id];
      if (nd.c1 < 0) continue;
      for (int side = 0; side < 2; ++side) {
        const int c = side ? nd.c2 : nd.c1;
        const UlvNode& u = F.nodes[c];
        const int r = u.m - u.k, np = (r + SV_ROWS - 1) / SV_ROWS;
        const int64_t xp = ox[id] + (side ? F.nodes[nd.c1].k : 0);
        ox[c] = xp;   // (np = 0: x is the parent's part)
        kids.push_back({c, np, xp, xp, r});
        maxp = std::max(maxp, np);
      }
    }
    phase();
    for (Kid& k : kids) {   // leaves without reflectors
      const TNode& nd = tr.nodes[k.id];
      if (k.np > 0 || nd.c1 >= 0) continue;
      SvDesc d = blank(F.nodes[k.id].m, 0, SD_X | SD_OUT);
      d.x0 = k.xp;
      d.outx = nd.lo;
      add_all(d);
    }
    for (int q = 0; q < maxp; ++q) {
      std::vector<int64_t> ot(kids.size(), 0);
      phase();
      for (size_t e = 0; e < kids.size(); ++e) {   // t = T V v
        Kid& k = kids[e];
        if (q >= k.np) continue;
        const UlvNode& u = F.nodes[k.id];
        const int p = k.np - 1 - q, i0 = p * SV_ROWS, nbb = std::min(SV_ROWS, u.m - u.k - i0);
        ot[e] = take(nbb);
        SvDesc d = blank(nbb, ot[e], SD_BUF | SD_POST_UPPER);
        if (fine(u.m)) d.trows = 8;   // (T in a task of its own, below)
        else d.post = u.T + (size_t)p * SV_ROWS * SV_ROWS;
        term(d, u.hv + (size_t)i0 * u.m + i0, u.m, u.m - i0, 0, oy[k.id] + i0, nullptr,
             k.split - i0, k.tail);
        add_all(d);
      }
      phase();
      for (size_t e = 0; e < kids.size(); ++e) {
        Kid& k = kids[e];
        const UlvNode& u = F.nodes[k.id];
        if (q >= k.np || !fine(u.m)) continue;
        const int p = k.np - 1 - q, nbb = std::min(SV_ROWS, u.m - u.k - p * SV_ROWS);
        const int64_t os = take(nbb);
        SvDesc d = blank(nbb, os, SD_BUF);
        d.trows = 8;
        term(d, u.T + (size_t)p * SV_ROWS * SV_ROWS, SV_ROWS, nbb, 0, ot[e]);
        add_all(d);
        ot[e] = os;
      }
      phase();
      for (size_t e = 0; e < kids.size(); ++e) {   // v <- v - V^T t
        Kid& k = kids[e];
        if (q >= k.np) continue;
        const TNode& nd = tr.nodes[k.id];
        const UlvNode& u = F.nodes[k.id];
        const int p = k.np - 1 - q, i0 = p * SV_ROWS, nbb = std::min(SV_ROWS, u.m - u.k - i0);
        const bool fin = p == 0 && nd.c1 < 0;   // the leaf's rows of the solution
        const int64_t ov = fin ? 0 : take(u.m - i0);
        SvDesc d = blank(u.m - i0, ov, SD_X | SD_NEG | (fin ? SD_OUT : SD_BUF));
        d.outx = nd.lo;
        if (fine(u.m)) d.trows = 16;
        d.x0 = oy[k.id] + i0;
        d.xsplit = k.split - i0;
        d.x1 = k.tail;
        term(d, u.hv + (size_t)i0 * u.m + i0, u.m, nbb, ST_TRANS, ot[e]);
        add_all(d);
        k.tail = ov;
        k.split = i0;
        if (p == 0) ox[k.id] = ov;
      }
    }
  }
  for (const SvDesc& d : pl.descs)
    for (int t = 0; t < d.nterm; ++t) {
      const double part = d.t[t].flags & (ST_LOWER | ST_UPPER) ? 0.5 : 1.0;
      pl.entries += part * d.rows * d.t[t].inner;
    }
  phase();   // (the end)
  if (pl.phases.empty() || pl.phases.back() != (int)pl.tasks.size())
    pl.phases.push_back((int)pl.tasks.size());
  pl.rows = tot;
}

// One solve of a batch.
struct SolveJob {
  hss_s* h;
  const void* B;
  int64_t ldb;
  int nr;
  void* X;
  int64_t ldx;
  hss_status* st;
};

// the handle's task table, built at the first solve after a factorization
Err sv_plan(hss_s* h) {
  std::lock_guard<std::mutex> lock(h->plan_mu);
  UlvFactors& F = h->ulv;
  HSS_TRY(h->take_timeout_word());
  if (F.plan) return ok();
  SvPlan pl;
  sv_build(h, pl);
  F.plan_off = pl.descs.size() * sizeof(SvDesc);
  HSS_TRY(upload_kept(&F.plan, {{pl.descs.data(), F.plan_off},
                                {pl.tasks.data(), pl.tasks.size() * sizeof(int2)}}));
  F.plan_rows = pl.rows;
  F.plan_entries = pl.entries;
  F.plan_tasks = std::move(pl.tasks);
  F.plan_phases = std::move(pl.phases);
  return ok();
}

// columns [c0, c0 + width) of every job (those that have them)
template <typename T>
Err solve_slab(const std::vector<SolveJob*>& jobs, int c0, int width, cudaStream_t s) {
  std::vector<SvJob> js;
  std::vector<const UlvFactors*> fs;
  size_t rows = 0;
  int maxnr = 1;
  std::vector<size_t> off;
  for (SolveJob* j : jobs) {
    const int nr = std::min(width, j->nr - c0);
    if (nr <= 0) continue;
    const UlvFactors& F = j->h->ulv;
    SvJob q{};
    q.descs = static_cast<const SvDesc*>(F.plan);
    q.B = static_cast<const T*>(j->B) + c0;
    q.X = static_cast<T*>(j->X) + c0;
    q.ldb = j->ldb;
    q.ldx = j->ldx;
    q.nrhs = nr;
    q.timeout = j->h->timeout;
    js.push_back(q);
    fs.push_back(&F);
    off.push_back(rows);
    rows += (size_t)F.plan_rows * nr;
    maxnr = std::max(maxnr, nr);
  }
  if (js.empty()) return ok();
  // Columns per task.  More make better use of a matrix entry; fewer make the
  // tasks shorter and the chains of dependent tasks with them.  So it follows
  // from the tasks that stand side by side: one column until a phase has 250 to
  // 550 one-column tasks on average (the SMs hold 900; the longer the tasks, the
  // more), two until 700 to 1900, then four.  Deep trees and single nodes, with
  // few tasks a phase, go by the columns alone.  Measured on 113 handles
  // (Toeplitz n = 315 to 160,000, QChem, Schur, Gaussian, BEM and random ones,
  // combs, dense nodes, leaves of 16 to 1000, both dtypes) at 2 to 64 right-hand
  // sides: 1.6% above the best of the three on average (a line at a size of the
  // work buffer, 4.4%).  In us with 1 / 2 / 4 columns: Toeplitz n = 8000, 8
  // right-hand sides 208 / 217 / 240, 32 480 / 364 / 358; n = 80,000, 2: 559 / 524 /
  // 684, 8: 1273 / 952 / 898; Schur complement n = 10,000, 4: 2169 / 2406 / 3110, 16:
  // 4475 / 3817 / 4021, 64: 14539 / 10383 / 8859; dense n = 3000, 64: 2294 / 2006 /
  // 1822; leaves of 16, n = 1376, 32: 258 / 185 / 164.
  double phases = 1.0, tasks = 0.0, entries = 0.0, side = 0.0;
  for (size_t q = 0; q < js.size(); ++q) {
    phases = std::max(phases, (double)fs[q]->plan_phases.size() - 1.0);
    tasks += (double)fs[q]->plan_tasks.size();
    side += (double)fs[q]->plan_tasks.size() * js[q].nrhs;
    entries += fs[q]->plan_entries;
  }
  side /= phases;
  const double len = std::min(entries / std::max(tasks, 1.0), 2000.0);   // entries per task
  int nc = 4;
  if (maxnr < 2) nc = 1;
  else if (tasks < 6.0 * phases) nc = maxnr <= 4 ? 1 : maxnr <= 16 ? 2 : 4;
  else if (side <= 250.0 + 0.15 * len) nc = 1;
  else if (maxnr < 3 || side <= 700.0 + 0.6 * len) nc = 2;
  // several handles: their phases interleaved, so that one handle's chain of
  // dependent tasks does not hold every CTA
  std::vector<int4> list;
  size_t total = 0;
  if (js.size() > 1) {
    size_t nph = 0;
    for (size_t q = 0; q < js.size(); ++q) {
      total += fs[q]->plan_tasks.size() * ((js[q].nrhs + nc - 1) / nc);
      nph = std::max(nph, fs[q]->plan_phases.size());
    }
    list.reserve(total);
    for (size_t ph = 0; ph + 1 < nph; ++ph)
      for (size_t q = 0; q < js.size(); ++q) {
        const UlvFactors& F = *fs[q];
        if (ph + 1 >= F.plan_phases.size()) continue;
        const int nch = (js[q].nrhs + nc - 1) / nc;
        for (int t = F.plan_phases[ph]; t < F.plan_phases[ph + 1]; ++t)
          for (int c = 0; c < nch; ++c)
            list.push_back(make_int4((int)q, F.plan_tasks[t].x, F.plan_tasks[t].y, c));
      }
  } else {
    total = fs[0]->plan_tasks.size() * ((js[0].nrhs + nc - 1) / nc);
  }
  if (total >= UINT32_MAX / 2) return fail(HSS_ERR_INVALID, "hss_solve: too many tasks");
  // control words, job and task tables, then the work buffer
  const size_t jb = (js.size() * sizeof(SvJob) + 255) & ~size_t(255);
  const size_t lb = (list.size() * sizeof(int4) + 255) & ~size_t(255);
  char* mem = nullptr;
  HSS_TRY(dalloc_t(&mem, 256 + jb + lb + rows * sizeof(double), s));
  double* buf = reinterpret_cast<double*>(mem + 256 + jb + lb);
  for (size_t q = 0; q < js.size(); ++q) js[q].buf = buf + off[q];
  Err e;
  SvArgs g{};
  g.ctl = reinterpret_cast<unsigned*>(mem);
  g.total = (unsigned)total;
  g.limit = fault_wait_limit() > 0 ? fault_wait_limit() : SV_WAIT_LIMIT;
  if (cudaMemsetAsync(mem, 0, 256, s) != cudaSuccess ||
      cudaMemsetAsync(buf, 0xff, rows * sizeof(double), s) != cudaSuccess) {
    cudaGetLastError();
    e = fail(HSS_ERR_CUDA, "hss_solve: memset");
  }
  size_t smem = 0;
  SvKernel fn;
  if (js.size() > 1) {
    fn = sv_kernel<T, true>(nc, &smem);
    g.jobs = reinterpret_cast<const SvJob*>(mem + 256);
    g.list = reinterpret_cast<const int4*>(mem + 256 + jb);
    if (e.st == HSS_OK) e = upload_async(mem + 256, js.data(), js.size() * sizeof(SvJob), s);
    if (e.st == HSS_OK) e = upload_async(mem + 256 + jb, list.data(), list.size() * sizeof(int4), s);
  } else {
    fn = sv_kernel<T, false>(nc, &smem);
    g.job = js[0];
    g.tasks = reinterpret_cast<const int2*>(static_cast<const char*>(fs[0]->plan) + fs[0]->plan_off);
    g.nch = (js[0].nrhs + nc - 1) / nc;
  }
  int per_sm = 0, sms = 0, dev = 0;
  if (e.st == HSS_OK &&
      (cudaGetDevice(&dev) != cudaSuccess ||
       cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
       cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
       cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, SV_THREADS, smem) != cudaSuccess)) {
    cudaGetLastError();
    e = fail(HSS_ERR_CUDA, "hss_solve: device query");
  }
  if (e.st == HSS_OK) {
    const size_t grid = std::min<size_t>(total, (size_t)sms * std::max(per_sm, 1));
    fn<<<(unsigned)grid, SV_THREADS, smem, s>>>(g);
    e = check_launch("ulv_solve_kernel");
  }
  dfree(mem, s);
  return e;
}

// Solves every job (all of one dtype).
void solve_many(std::vector<SolveJob>& jobs, cudaStream_t s) {
  std::vector<SolveJob*> live;
  int maxnr = 0;
  for (SolveJob& j : jobs) {
    Err e = sv_plan(j.h);
    if (e.st) {
      j.h->err = e.msg;
      *j.st = e.st;
      continue;
    }
    live.push_back(&j);
    maxnr = std::max(maxnr, j.nr);
  }
  // The work buffer holds a value only once (its values are their own flags), so
  // each panel of Q has rows of its own: about r (m - r / 2) / 32 rows for r
  // reflectors of a node of order m.  Where that does not fit, half as many
  // columns at a time (a column's bits do not depend on it).
  int width = SV_COLS;
  for (int c0 = 0; c0 < maxnr;) {
    width = std::min(width, maxnr - c0);
    const Err e = live[0]->h->dtype == HSS_F64 ? solve_slab<double>(live, c0, width, s)
                                               : solve_slab<float>(live, c0, width, s);
    if (e.st == HSS_OK) {
      c0 += width;
      continue;
    }
    if (e.st == HSS_ERR_OOM && width > 1) {
      width /= 2;
      continue;
    }
    for (SolveJob* j : live) {
      j->h->err = e.msg;
      *j->st = e.st;
    }
    return;
  }
}

// argument checks of one solve; INVALID / STATE with the handle's message
hss_status check_solve(hss_s* h, const void* B, int64_t ldb, int64_t nrhs, const void* X,
                       int64_t ldx) {
  if (!h) return HSS_ERR_INVALID;
  if (!h->ulv.done) {
    h->err = "hss_solve: hss_factor has not run on this handle";
    return HSS_ERR_STATE;
  }
  if (!B || !X || nrhs < 0 || ldb < nrhs || ldx < nrhs || nrhs > INT32_MAX) {
    h->err = "hss_solve: bad B, X, nrhs or leading dimension";
    return HSS_ERR_INVALID;
  }
  if (h->timed_out("hss_solve")) return HSS_ERR_TIMEOUT;
  return HSS_OK;
}

}  // namespace
}  // namespace hss

extern "C" hss_status hss_solve(hss_t h, const void* B, int64_t ldb, int64_t nrhs, void* X,
                                int64_t ldx, void* stream) {
  hss_status st = check_solve(h, B, ldb, nrhs, X, ldx);
  if (st != HSS_OK || nrhs == 0) return st;
  std::vector<SolveJob> jobs(1);
  jobs[0].h = h;
  jobs[0].B = B;
  jobs[0].ldb = ldb;
  jobs[0].nr = (int)nrhs;
  jobs[0].X = X;
  jobs[0].ldx = ldx;
  jobs[0].st = &st;
  solve_many(jobs, (cudaStream_t)stream);
  return st;
}

extern "C" hss_status hss_solve_batched(int32_t count, hss_t* hs, const void* const* B,
                                        const int64_t* ldb, const int64_t* nrhs,
                                        void* const* X, const int64_t* ldx, void* stream,
                                        hss_status* status) {
  if (count < 0 || (count > 0 && (!hs || !B || !ldb || !nrhs || !X || !ldx)))
    return HSS_ERR_INVALID;
  std::vector<hss_status> st(std::max(count, 1), HSS_OK);
  std::vector<SolveJob> jobs;
  const hss_s* one = nullptr;   // the first handle there is: one launch, one dtype
  for (int32_t q = 0; q < count; ++q) {
    st[q] = check_solve(hs[q], B[q], ldb[q], nrhs[q], X[q], ldx[q]);
    if (!one) one = hs[q];
    if (st[q] == HSS_OK && hs[q]->dtype != one->dtype) {
      hs[q]->err = "hss_solve_batched: handles of different dtypes";
      st[q] = HSS_ERR_INVALID;
    }
    if (st[q] != HSS_OK || nrhs[q] == 0) continue;
    SolveJob j;
    j.h = hs[q];
    j.B = B[q];
    j.ldb = ldb[q];
    j.nr = (int)nrhs[q];
    j.X = X[q];
    j.ldx = ldx[q];
    j.st = &st[q];
    jobs.push_back(std::move(j));
  }
  solve_many(jobs, (cudaStream_t)stream);
  hss_status first = HSS_OK;
  for (int32_t q = 0; q < count; ++q) {
    if (status) status[q] = st[q];
    if (st[q] != HSS_OK && first == HSS_OK) {
      first = st[q];
      if (hs[q]) set_thread_error(hs[q]->err);
    }
  }
  return first;
}
