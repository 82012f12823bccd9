// HSS matrix-vector product (Algorithm 2) in one launch, for few right-hand
// sides.
//
// The product is an upward sweep (y_tau = V_tau^T x), a downward sweep (z of
// the children from B, y and the parent's U z) and the leaves (b = U z + D x).
// One launch per tree level and phase left the device waiting between short
// launches (31 of them at n = 80,000: 0.46 ms for 78 MB of generators), so the
// whole product is one launch of small tasks.  A task computes at most 16 rows
// of one y_tau, z_tau or leaf of b for NC right-hand sides.
//
// The data carry their own flags: the work buffer starts as all-ones words (a
// NaN that no arithmetic instruction returns: their NaN has a zero sign bit),
// a task's reader polls the very values it needs until they are there.  That
// leaves one store and one load between a producer and its consumer; counters
// with release / acquire took two more round trips to L2 for each tree level
// (4.4 us a tree level against 2.3).  CTAs claim tasks in table order from a ticket
// counter, and whatever a task reads is written by tasks of lower tickets, so
// its CTA is running or has finished: the polls end whatever number of CTAs is
// resident and whatever else is on the device.  Each poll is bounded all the
// same: on a timeout the value stays NaN and reaches the product, and the next
// call with the handle reports it (hss_s::timeout).
//
// A task's matrix rows never depend on a wait: they are on their way to shared
// memory (cp.async, 16 rows by 64 inner indices a stage) while the task
// waits for its vectors, and the part of its sum that does not need the parent's z
// (B y) is taken first; D x is tasks of its own.  The 128 threads are (row,
// part) pairs, rows rounded up to 8 (an FP64 instruction costs the same
// however few lanes it has work for, so 35 rows are 40, not 64); the parts
// split the inner indices and their sums meet in shared memory once, in
// order.  A column's sums do not depend on NC or on the number of CTAs.
//
// The task table depends on the tree and the ranks alone; it is built at the
// handle's first product and kept with the handle.
//
// What bounds it is the chain of 2 x depth + 1 dependent tasks (2.3 us each:
// a poll's round trip to L2, the gather, the FP64 chains, the store) and, at
// the bottom, the tasks' own latency over eight CTAs an SM.  Measured (GB300,
// FP64, one right-hand side, whole call): n = 2000 (5 levels) 93 -> 26 us;
// n = 80,000 (11 levels, rank 178, 78 MB) 498 -> 104 us.
#include "hss_internal.cuh"
#include "hss_tree.h"

#include <algorithm>
#include <cmath>

namespace hss {

namespace {

constexpr int MV_ROWS = 16, MV_THREADS = 128, MV_WARPS = MV_THREADS / 32;
constexpr int MV_L = 64;   // inner indices per stage (128 and six CTAs per SM: 112 us, below)
constexpr long long MV_WAIT_LIMIT = 1ll << 33;   // clock cycles (about 4 s)

enum { MV_UP = 0, MV_DOWN = 1, MV_DX = 2, MV_LEAF = 3 };

// The tasks of one y_tau (MV_UP), one child's z (MV_DOWN), one leaf's D x
// (MV_DX) or one leaf of b (MV_LEAF: b += U z): rows r0 .. r0 + 15 of
//   first term  M(row, l) = M[row * ld + l], or (MV_UP) M[l * ld + row], times
//     the vector rows zmap[l] (or l): rows below split start at off0, the
//     others at off1 (rows of the work buffer, or of X when from_x);
//   MV_UP: + vector row xmap[row] (the identity part of V);
//   second term (U z of node p = Pi [z; E z], when iperm is not null): with
//     q = iperm[row], z row q if q < k2, else row q - k2 of E times z;
//   MV_LEAF: + D x, from its MV_DX task (rows `dx` of the work buffer).
struct alignas(16) MvDesc {
  const void* M;
  const int32_t* zmap;
  const int32_t* xmap;
  const double* E;
  const int32_t* iperm;
  int64_t off0, off1, out, off2, dx;
  int32_t ld, inner, split, k2;
  int32_t rows, kind, from_x, pad;
};
static_assert(sizeof(MvDesc) == 112, "copied as 16-byte pieces");

struct MvArgs {
  const int2* tasks;   // (description, r0)
  const MvDesc* descs;
  unsigned* ctl;       // [0] ticket, [1] a poll has timed out
  unsigned* timeout;   // the handle's word for that
  long long limit;     // of a poll, in clock cycles
  void* buf;
  const void* X;
  void* B;
  int64_t ldx, ldb;
  int ntasks, nch, nrhs;
};

__device__ __forceinline__ double mv_ld(const double* p) {
  double v;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float mv_ld(const float* p) {
  float v;
  asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void mv_st(double* p, double v) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ void mv_st(float* p, float v) {
  asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
// not yet written (all ones)
__device__ __forceinline__ bool mv_unset(double v) { return __double_as_longlong(v) == -1ll; }
__device__ __forceinline__ bool mv_unset(float v) { return __float_as_int(v) == -1; }

// *p once it has been written (bounded; the flag ends the other polls early)
template <typename T>
__device__ __forceinline__ T mv_poll(const T* p, const MvArgs& g) {
  T v = mv_ld(p);
  if (!mv_unset(v)) return v;
  const long long t0 = clock64();
  unsigned polls = 0;
  while (mv_unset(v = mv_ld(p))) {
    if ((++polls & 31u) != 0u) continue;
    if (*reinterpret_cast<volatile unsigned*>(g.ctl + 1)) break;
    if (clock64() - t0 > g.limit) {
      atomicExch(g.ctl + 1, 1u);
      *reinterpret_cast<volatile unsigned*>(g.timeout) = 1u;
      break;
    }
  }
  return v;
}

template <int BYTES>
__device__ __forceinline__ void mv_cp(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES));
}

// entries of M of one stage: rows r0 .. of a row-major M, [row][l] (odd
// pitch: rows on different banks); rmap: row r is rmap[r] - rsub, dead (zeros) when negative
template <int L, typename S>
__device__ __forceinline__ void mv_load_rows(S* dst, const S* M, int64_t ld,
                                             const int32_t* rmap, int rsub, int r0, int rows,
                                             int l0, int lc) {
  const int lane = threadIdx.x & 31;
  for (int r = threadIdx.x >> 5; r < rows; r += MV_WARPS) {
    const int ri = rmap ? rmap[r0 + r] - rsub : r0 + r;
    S* d = dst + r * (L + 1);
    if (ri < 0) {
      for (int l = lane; l < lc; l += 32) d[l] = S(0);
      continue;
    }
    const S* row = M + (int64_t)ri * ld + l0;
    for (int l = lane; l < lc; l += 32) mv_cp<sizeof(S)>(d + l, row + l);
  }
}

// the transposed form: [l][MV_ROWS] from columns r0 .. of M
__device__ __forceinline__ void mv_load_cols(double* dst, const double* M, int64_t ld, int r0,
                                             int rows, int l0, int lc) {
  const int r = threadIdx.x % MV_ROWS;
  if (r < rows)
    for (int l = threadIdx.x / MV_ROWS; l < lc; l += MV_THREADS / MV_ROWS)
      mv_cp<8>(dst + l * MV_ROWS + r, M + (int64_t)(l0 + l) * ld + r0 + r);
}

// a += the terms l = part, part + parts, ... of this thread's row, the
// terms in turn into two chains (an FP64 operation takes 67 cycles)
template <typename T, typename S, int NC>
__device__ __forceinline__ void mv_fma(T (&a)[2][NC], const S* ms, const T* zs, int row, int part,
                                       int parts, int srow, int sl, int lc) {
  const S* m = ms + row * srow;
  int l = part;
#pragma unroll 2
  for (; l + parts < lc; l += 2 * parts) {
    const T m0 = (T)m[l * sl], m1 = (T)m[(l + parts) * sl];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      a[0][c] = fma(m0, zs[l * NC + c], a[0][c]);
      a[1][c] = fma(m1, zs[(l + parts) * NC + c], a[1][c]);
    }
  }
  if (l < lc) {
    const T m0 = (T)m[l * sl];
#pragma unroll
    for (int c = 0; c < NC; ++c) a[0][c] = fma(m0, zs[l * NC + c], a[0][c]);
  }
}

template <typename T, int NC>
__global__ void __launch_bounds__(MV_THREADS, NC == 8 ? 6 : 8) matvec_kernel(const MvArgs g) {
  constexpr int L = MV_L;
  __shared__ __align__(16) double ms[2][MV_ROWS * (L + 1)];
  __shared__ T zs[2][L * NC];
  __shared__ int idx[2][L];
  static_assert(2 * L >= MV_THREADS, "the partial sums take the place of the vectors");
  static_assert(L <= MV_THREADS && L % (2 * MV_THREADS / 8) == 0, "one index a thread; whole turns");
  static_assert(MV_ROWS * NC <= MV_THREADS, "one output a thread");
  T* red = &zs[0][0];   // [part][row][NC]
  __shared__ MvDesc tk;
  __shared__ unsigned snext;
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned total = (unsigned)g.ntasks * (unsigned)g.nch;
  T* buf = reinterpret_cast<T*>(g.buf);
  const int64_t nr = g.nrhs;
  unsigned claim = 0;
  if (tid == 0) snext = atomicAdd(g.ctl, 1u);
  __syncthreads();
  while (true) {
    const unsigned tick = snext;
    if (tick >= total) return;
    const int chunk = (int)(tick % (unsigned)g.nch);
    const int2 task = g.tasks[tick / (unsigned)g.nch];
    const int r0 = task.y;
    if (tid < (int)(sizeof(MvDesc) / 16))
      reinterpret_cast<uint4*>(&tk)[tid] = reinterpret_cast<const uint4*>(g.descs + task.x)[tid];
    __syncthreads();
    if (tid == 0) claim = atomicAdd(g.ctl, 1u);   // the next ticket, needed at the end only
    const int cb = chunk * NC, nc = min(NC, g.nrhs - cb);
    const int rows = min(MV_ROWS, tk.rows - r0);
    const bool up = tk.kind == MV_UP, second = tk.iperm != nullptr;
    const int rows8 = (rows + 7) & ~7, parts = MV_THREADS / rows8;
    const int row = tid % rows8, part = tid / rows8;   // part >= parts: idle
    const int n0 = (tk.inner + L - 1) / L;
    const int nst = n0 + (second ? (tk.k2 + L - 1) / L : 0);
    auto issue = [&](int k) {   // stage k's matrix entries and row indices
      if (k < n0) {
        const int l0 = k * L, lc = min(L, tk.inner - l0);
        if (tk.zmap && tid < lc) mv_cp<4>(&idx[k & 1][tid], tk.zmap + l0 + tid);
        if (up)
          mv_load_cols(&ms[k & 1][0], reinterpret_cast<const double*>(tk.M), tk.ld, r0, rows, l0, lc);
        else
          mv_load_rows<L>(reinterpret_cast<T*>(&ms[k & 1][0]), reinterpret_cast<const T*>(tk.M), tk.ld,
                       nullptr, 0, r0, rows, l0, lc);
      } else if (k < nst) {
        const int l0 = (k - n0) * L, lc = min(L, tk.k2 - l0);
        mv_load_rows<L>(&ms[k & 1][0], tk.E, tk.k2, tk.iperm, tk.k2, r0, rows, l0, lc);
      }
      asm volatile("cp.async.commit_group;");
    };
    // row r of a term's vector in the work buffer, column cb
    auto zrow = [&](bool first, int r) -> const T* {
      const int64_t q = !first ? tk.off2 + r : r < tk.split ? tk.off0 + r : tk.off1 + (r - tk.split);
      return buf + q * nr + cb;
    };
    const T* Xb = reinterpret_cast<const T*>(g.X) + tk.off0 * g.ldx + cb;   // from_x only
    issue(0);
    // this thread's output (row orow, column oc) and what it takes besides its
    // sum: entry xi of the first (MV_UP) or second term's vector, and D x
    const int orow = tid / NC, oc = tid - orow * NC;
    const bool has_out = orow < rows && oc < nc;
    int xi = -1;
    if (has_out) {
      if (up) xi = tk.xmap[r0 + orow];
      else if (second) xi = tk.iperm[r0 + orow];
      if (!up && xi >= tk.k2) xi = -1;
    }
    T acc[2][NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[0][c] = acc[1][c] = T(0);
    for (int k = 0; k < nst; ++k) {
      const bool first = k < n0;
      const int l0 = (first ? k : k - n0) * L;
      const int lc = min(L, (first ? tk.inner : tk.k2) - l0);
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      const bool mapped = first && tk.zmap;
      if (mapped) __syncthreads();   // idx was copied by other threads
      constexpr int U = (L * NC + MV_THREADS - 1) / MV_THREADS;
      T v[U];
      if (first && tk.from_x) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = tid + u * MV_THREADS, l = e / NC, c = e - l * NC;
          v[u] = T(0);
          if (l < lc && c < nc) v[u] = Xb[(int64_t)(mapped ? idx[k & 1][l] : l0 + l) * g.ldx + c];
        }
      } else {
        const T* p[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = tid + u * MV_THREADS, l = e / NC, c = e - l * NC;
          p[u] = nullptr;
          if (l < lc && c < nc) p[u] = zrow(first, mapped ? idx[k & 1][l] : l0 + l) + c;
        }
        // one lane of each warp polls until its value is there, so that a
        // wait costs one load a warp; then every value is read
        if (lane == 0 && p[0]) mv_poll(p[0], g);
        __syncwarp();
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = p[u] ? mv_ld(p[u]) : T(0);
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (p[u] && mv_unset(v[u])) v[u] = mv_poll(p[u], g);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = tid + u * MV_THREADS;
        if (e < lc * NC) zs[k & 1][e] = v[u];
      }
      __syncthreads();
      issue(k + 1);
      if (part < parts) {
        if (up) mv_fma<T, double, NC>(acc, ms[k & 1], zs[k & 1], row, part, parts, 1, MV_ROWS, lc);
        else if (!first)
          mv_fma<T, double, NC>(acc, ms[k & 1], zs[k & 1], row, part, parts, L + 1, 1, lc);
        else
          mv_fma<T, T, NC>(acc, reinterpret_cast<const T*>(ms[k & 1]), zs[k & 1], row, part, parts,
                           L + 1, 1, lc);
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    T xv = T(0), xb = T(0);
    if (xi >= 0) {
      if (up && tk.from_x) xv = Xb[(int64_t)xi * g.ldx + oc];
      else xv = mv_poll(zrow(up, xi) + oc, g);
    }
    if (has_out && tk.kind == MV_LEAF) xb = mv_poll(buf + (tk.dx + r0 + orow) * nr + cb + oc, g);
    __syncthreads();   // every warp is done with zs
    if (part < parts) {
#pragma unroll
      for (int c = 0; c < NC; ++c) red[(part * rows8 + row) * NC + c] = acc[0][c] + acc[1][c];
    }
    if (tid == 0) snext = claim;
    __syncthreads();
    if (has_out) {
      T v = red[tid];
      for (int q = 1; q < parts; ++q) v += red[q * rows8 * NC + tid];
      v += xv;
      const int64_t o = tk.out + r0 + orow;
      if (tk.kind == MV_LEAF) reinterpret_cast<T*>(g.B)[o * g.ldb + cb + oc] = v + xb;
      // (a NaN of the caller's may carry the unset pattern through)
      else mv_st(buf + o * nr + cb + oc, mv_unset(v) ? T(NAN) : v);
    }
    // (tk, zs and snext are written again only after every thread has passed here)
    __syncthreads();
  }
}

template <typename T>
using MvKernel = void (*)(const MvArgs);
template <typename T>
MvKernel<T> mv_kernel(int nc) {
  switch (nc) {
    case 1: return matvec_kernel<T, 1>;
    case 2: return matvec_kernel<T, 2>;
    case 4: return matvec_kernel<T, 4>;
    default: return matvec_kernel<T, 8>;
  }
}

// The task table of a handle: upward tasks from the deepest level, downward
// tasks from the root, then the leaves (D x between the sweeps).  rows_out:
// rows of the work buffer (y_tau and z_tau of every non-root node, D x).
void mv_build(const hss_s* h, std::vector<MvDesc>& descs, std::vector<int2>& tasks,
              int64_t* rows_out) {
  const Tree& tr = h->tree;
  const int nn = (int)tr.nodes.size();
  std::vector<int64_t> oy(nn, 0), oz(nn, 0);
  int64_t tot = 0;
  auto tiles = [](int rows) { return (rows + MV_ROWS - 1) / MV_ROWS; };
  size_t nt = 0;
  for (int i = 0; i < nn; ++i) {
    const TNode& nd = tr.nodes[i];
    if (i) {
      oy[i] = tot;
      tot += h->gen[i].kc;
      oz[i] = tot;
      tot += h->gen[i].kr;
      nt += tiles(h->gen[i].kc) + tiles(h->gen[i].kr);
    }
    if (nd.c1 < 0) nt += 2 * tiles(nd.hi - nd.lo);
  }
  *rows_out = tot + h->n;
  descs.reserve(4 * (size_t)nn);
  tasks.reserve(nt);
  auto add = [&](const MvDesc& d) {
    if (d.rows <= 0) return;
    for (int r0 = 0; r0 < d.rows; r0 += MV_ROWS)
      tasks.push_back(make_int2((int)descs.size(), r0));
    descs.push_back(d);
  };
  auto blank = [&](int kind, int rows, int64_t out) {
    MvDesc d{};
    d.kind = kind;
    d.rows = rows;
    d.out = out;
    d.split = INT32_MAX;
    return d;
  };
  // U z of node p through iperm_r
  auto u_term = [&](MvDesc& d, int p, const int32_t* iperm) {
    const NodeGen& g = h->gen[p];
    d.E = g.Er;
    d.k2 = g.kr;
    d.iperm = iperm;
    d.off2 = oz[p];
  };
  for (int depth = tr.maxdepth; depth >= 1; --depth)
    for (int id : tr.levels[depth]) {
      const TNode& nd = tr.nodes[id];
      const NodeGen& g = h->gen[id];
      MvDesc d = blank(MV_UP, g.kc, oy[id]);
      d.xmap = g.permc;
      d.M = g.Ec;
      d.ld = g.kc;
      d.inner = g.mc - g.kc;
      d.zmap = g.permc + g.kc;
      if (nd.c1 < 0) {
        d.from_x = 1;
        d.off0 = nd.lo;
      } else {
        d.off0 = oy[nd.c1];
        d.off1 = oy[nd.c2];
        d.split = h->gen[nd.c1].kc;
      }
      add(d);
    }
  // D x: nothing to wait for, and most of the bytes; the CTAs that have run
  // out of upward tasks take these while the top of the tree is worked on
  for (int id = 0; id < nn; ++id) {
    const TNode& nd = tr.nodes[id];
    if (nd.c1 >= 0) continue;
    MvDesc d = blank(MV_DX, nd.hi - nd.lo, tot + nd.lo);
    d.M = h->gen[id].D;
    d.ld = d.inner = nd.hi - nd.lo;
    d.from_x = 1;
    d.off0 = nd.lo;
    add(d);
  }
  for (int depth = 0; depth < tr.maxdepth; ++depth)
    for (int id : tr.levels[depth]) {
      const TNode& nd = tr.nodes[id];
      if (nd.c1 < 0) continue;
      const NodeGen& g = h->gen[id];
      for (int side = 0; side < 2; ++side) {
        const int c = side ? nd.c2 : nd.c1, o = side ? nd.c1 : nd.c2;
        MvDesc d = blank(MV_DOWN, h->gen[c].kr, oz[c]);
        d.M = side ? g.B21 : g.B12;
        d.ld = d.inner = h->gen[o].kc;
        d.off0 = oy[o];
        if (id != 0) u_term(d, id, g.iperm_r + (side ? h->gen[nd.c1].kr : 0));
        add(d);
      }
    }
  for (int id = 0; id < nn; ++id) {
    const TNode& nd = tr.nodes[id];
    if (nd.c1 >= 0) continue;
    MvDesc d = blank(MV_LEAF, nd.hi - nd.lo, nd.lo);
    d.dx = tot + nd.lo;
    if (id != 0) u_term(d, id, h->gen[id].iperm_r);
    add(d);
  }
}

}  // namespace

template <typename T>
Err matvec_tasks(hss_s* h, const T* X, int64_t ldx, int nrhs, T* B, int64_t ldb, cudaStream_t s) {
  {
    std::lock_guard<std::mutex> lock(h->plan_mu);
    HSS_TRY(h->take_timeout_word());
    if (!h->mv_tasks) {
      std::vector<MvDesc> descs;
      std::vector<int2> tasks;
      mv_build(h, descs, tasks, &h->mv_rows);
      h->mv_ntasks = (int)tasks.size();
      h->mv_off = descs.size() * sizeof(MvDesc);
      const size_t tb = tasks.size() * sizeof(int2);
      HSS_TRY(upload_kept(&h->mv_tasks, {{descs.data(), h->mv_off}, {tasks.data(), tb}}));
    }
  }
  const int nc = nrhs <= 1 ? 1 : nrhs == 2 ? 2 : nrhs <= 4 ? 4 : 8;
  MvArgs g{};
  g.descs = static_cast<const MvDesc*>(h->mv_tasks);
  g.tasks = reinterpret_cast<const int2*>(static_cast<const char*>(h->mv_tasks) + h->mv_off);
  g.ntasks = h->mv_ntasks;
  g.nch = (nrhs + nc - 1) / nc;
  g.nrhs = nrhs;
  g.timeout = h->timeout;
  g.limit = fault_wait_limit() > 0 ? fault_wait_limit() : MV_WAIT_LIMIT;
  g.X = X;
  g.B = B;
  g.ldx = ldx;
  g.ldb = ldb;
  // the control words (zero), then y, z and D x (all ones: not yet written)
  const size_t vec = (size_t)h->mv_rows * nrhs * sizeof(T);
  char* buf = nullptr;
  HSS_TRY(dalloc_t(&buf, 256 + vec, s));
  g.ctl = reinterpret_cast<unsigned*>(buf);
  g.buf = buf + 256;
  Err e;
  if (cudaMemsetAsync(g.ctl, 0, 256, s) != cudaSuccess ||
      cudaMemsetAsync(g.buf, 0xff, vec, s) != cudaSuccess) {
    cudaGetLastError();
    e = fail(HSS_ERR_CUDA, "hss_matvec: memset");
  } else {
    const MvKernel<T> fn = mv_kernel<T>(nc);
    int per_sm = 0, sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, MV_THREADS, 0) != cudaSuccess) {
      cudaGetLastError();
      e = fail(HSS_ERR_CUDA, "hss_matvec: device query");
    } else {
      const int64_t total = (int64_t)g.ntasks * g.nch;
      if (h->tree.nodes.size() == 1) {
        // H = D: half of the tasks are D x and all of the work, and none waits
        // for long.  A CTA claims a task ahead, so the CTAs per SM are those
        // whose rounds over the D x tasks are the fewest tasks per SM in all
        // (three or more if there are several rounds).  FP64, n = 1000, 3000,
        // 8000: 1 column 35, 103, 313 -> 34, 90, 286 us, 8 columns 66, 348, 1619 ->
        // 66, 258, 1111, 16 columns 95, 523, 2910 -> 68, 348, 2280 with eight
        // (six) CTAs per SM before.
        const int64_t dx = total / 2;
        int best = per_sm;
        int64_t least = INT64_MAX;
        for (int p = per_sm; p >= 1; --p) {
          const int64_t rounds = (dx + (int64_t)sms * p - 1) / ((int64_t)sms * p);
          if (rounds * p < least && (p >= 3 || rounds == 1)) {
            least = rounds * p;
            best = p;
          }
        }
        per_sm = best;
      }
      const int grid = (int)std::min<int64_t>(total, (int64_t)sms * std::max(per_sm, 1));
      fn<<<grid, MV_THREADS, 0, s>>>(g);
      e = check_launch("matvec_kernel");
    }
  }
  dfree(buf, s);
  return e;
}

template Err matvec_tasks<float>(hss_s*, const float*, int64_t, int, float*, int64_t, cudaStream_t);
template Err matvec_tasks<double>(hss_s*, const double*, int64_t, int, double*, int64_t,
                                  cudaStream_t);

}  // namespace hss
