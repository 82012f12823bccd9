// Fused sampling S^r = (A - D) R, S^c = (A - D)^T R (Section 2.2, step 2 of
// the compression; Algorithm 1's leaf samples S^r(I,:) - D R(I,:)).
//
// One pass over A serves both products: the (128-row panel, column tile) pairs
// of a chunk of DC sample columns are dealt evenly over the CTAs, and a CTA walks
// its range.  Its part of a panel's row sample (accumulated on chip) and the
// column sample of each tile, a partial sum over the panel's rows, go to two
// slabs, which a second kernel reduces in a fixed order (deterministic: no
// floating-point atomics).  Entries with leaf(i) == leaf(j) are masked to zero
// while A is staged, which subtracts the leaf diagonal blocks D exactly (no
// cancellation).  In FP32 the row sample is summed per 32 columns and these sums
// are added with Kahan compensation, whose remainder goes to the slab as well;
// the partials of both samples are summed with compensation: the sample error
// stays near one rounding instead of growing like sqrt(n).
#include "hss_internal.cuh"

#include <algorithm>
#include <cstdlib>
#include <cstring>

namespace hss {

namespace {

constexpr int S_BM = 128;   // panel rows
constexpr int S_DC = 64;    // sample columns per chunk (the mma.sync kernel's slabs)
constexpr int S_THREADS = 256;

// SIMT (FP32 or FP64 FMA) fused sampling.
//
// Bound: the FMA pipe (4 n^2 c flops; FP32 128, FP64 2 multiply-adds a clock
// and SM), so the split has to give every SM the same share and the FMAs few
// shared-memory reads.  The (panel, column tile) pairs of a chunk are
// numbered panel-major and dealt evenly over G CTAs (one per SM): a CTA's
// range may start or end inside a panel, and its part of the panel's row
// sample goes to slot q + panel of a row slab (q the CTA), which the second
// kernel sums; a grid of one CTA per panel leaves SMs idle below 152 panels
// and a ragged last wave above.  The next tile of A and of R is on its way
// (cp.async) while the current one is multiplied.  A's tile stays row-major
// in shared memory for both products: a thread takes rows ty, ty + NTY, ...
// of the row product, four inner indices per 16-byte load (the odd multiple
// of 16 bytes in the pitch keeps the rows of a warp on different banks), and
// CJ adjacent columns of the column product.  Chunks are 64 or 32 columns wide
// (simt_plan).
// What is left above the FMA floor is shared-memory bandwidth: a read of 16
// bytes a lane takes about three of the SM's shared-memory cycles even where
// lanes share addresses, and the 8 x 4 and 4 x 4 register blocks need 12 and
// 8 words for 32 and 16 FMAs.
// Measured (GB300, hss_sample, 64 columns, both products; one CTA per panel
// with 8 x 4 / 2 x 4 blocks and scalar reads before): FP32 n = 10000 4.64 ->
// 0.78 ms (floor 0.37 ms; this kernel 0.72, the reduction 0.04), FP64
// n = 2000 8.5 -> 0.96 ms (floor 0.82 ms).
template <typename T, int DC>
struct Simt {
  static constexpr int BK = sizeof(T) == 4 ? 64 : 32;   // column tile of A
  static constexpr int VEC = 16 / sizeof(T);            // elements of 16 bytes
  static constexpr int PA = BK + VEC;                   // pitch of A's tile
  static constexpr int NTX = DC / 4;                    // threads along the sample columns
  static constexpr int NTY = S_THREADS / NTX;
  static constexpr int RR = S_BM / NTY;                 // rows per thread (row product)
  static constexpr int CJ = BK / NTY;                   // columns of A per thread (column product)
  static constexpr size_t a_elems = (size_t)S_BM * PA, r_elems = (size_t)BK * DC;
  static constexpr size_t smem = sizeof(T) * (2 * (a_elems + r_elems) + (size_t)S_BM * DC);
};

struct SimtPlan {
  int npanel, ntile, nchunk, dc;
  long long T;   // (panel, tile) pairs of a chunk
  int G;         // CTAs per chunk
};

template <typename T>
SimtPlan simt_plan(int64_t n, int64_t ncols, int sms) {
  SimtPlan pl;
  // FP64: 32-column chunks where they pad less, as the pipe's time is the padded
  // columns' (n = 8000, in chunks of 64 / 32: 32 columns 13.8 / 7.0 ms, 64 13.8 /
  // 14.0, 96 27.5 / 21.1, 128 27.5 / 27.8).  FP32 is bound by shared memory, where
  // the smaller register blocks of 32 columns cost more than the padding unless
  // one chunk holds all (n = 10000: 32 columns 0.75 / 0.54 ms, 48 0.75 / 1.05, 65
  // 1.55 / 1.64, 96 1.47 / 1.59, 160 2.23 / 2.62).
  const bool narrow = sizeof(T) == 4 ? ncols <= 32
                                     : (ncols + 63) / 64 * 64 != (ncols + 31) / 32 * 32;
  pl.dc = narrow ? 32 : 64;
  const int bk = sizeof(T) == 4 ? 64 : 32;
  pl.npanel = (int)((n + S_BM - 1) / S_BM);
  pl.ntile = (int)((n + bk - 1) / bk);
  pl.nchunk = (int)((ncols + pl.dc - 1) / pl.dc);
  pl.T = (long long)pl.npanel * pl.ntile;
  // one CTA per SM in all; with many chunks about four per SM, so that the
  // last wave is a small part
  const long long want = std::max<long long>((pl.nchunk <= 8 ? 1LL : 4LL) * sms / pl.nchunk, 1);
  pl.G = (int)std::min<long long>(want, pl.T);
  return pl;
}
// column partials [npanel][nchunk][n][dc], then row partials [nchunk][G + npanel][128][dc];
// FP32: then the row partials' remainders, laid out the same
size_t simt_col_elems(const SimtPlan& pl, int64_t n) {
  return (size_t)pl.npanel * pl.nchunk * n * pl.dc;
}
__host__ __device__ inline size_t simt_row_elems(const SimtPlan& pl) {
  return (size_t)pl.nchunk * (pl.G + pl.npanel) * S_BM * pl.dc;
}

__host__ __device__ __forceinline__ long long simt_begin(long long q, long long T, long long G) {
  return q * T / G;
}
// the CTA whose range holds pair t
__host__ __device__ __forceinline__ int simt_owner(long long t, long long T, long long G) {
  return (int)(((t + 1) * G - 1) / T);
}

// copies 16 bytes (or one element) to shared memory; 0 source bytes: zeros
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool live) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int sz = live ? BYTES : 0;
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(sz));
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES),
                 "r"(sz));
}

template <typename T>
__device__ __forceinline__ void ld_vec4(T (&v)[4], const T* p) {
  if constexpr (sizeof(T) == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
  } else {
    const double2 x = reinterpret_cast<const double2*>(p)[0];
    const double2 y = reinterpret_cast<const double2*>(p)[1];
    v[0] = x.x;
    v[1] = x.y;
    v[2] = y.x;
    v[3] = y.y;
  }
}

template <typename T>
__device__ __forceinline__ void st_vec4(T* p, const T (&v)[4]) {
  if constexpr (sizeof(T) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
  }
}

// rows x cols of src (row r0 + r, column q0 + q; live rows / columns below
// rmax, cmax) to dst (pitch): 16-byte copies when VECOK, else one element each
template <typename T, int ROWS, int COLS>
__device__ __forceinline__ void stage(T* dst, int pitch, const T* src, int64_t ld, int64_t r0,
                                      int64_t rmax, int64_t q0, int64_t cmax, bool vecok) {
  constexpr int V = 16 / sizeof(T);
  if (vecok) {
    for (int e = threadIdx.x; e < ROWS * (COLS / V); e += S_THREADS) {
      const int r = e / (COLS / V), q = (e - r * (COLS / V)) * V;
      const int64_t i = r0 + r, j = q0 + q;
      T* d = dst + r * pitch + q;
      if (j + V <= cmax || i >= rmax || j >= cmax) {
        const bool live = i < rmax && j < cmax;
        cp_async<16>(d, live ? src + i * ld + j : src, live);
      } else {   // the ragged edge: element by element
#pragma unroll
        for (int x = 0; x < V; ++x) {
          const bool live = j + x < cmax;
          cp_async<sizeof(T)>(d + x, live ? src + i * ld + j + x : src, live);
        }
      }
    }
  } else {
    for (int e = threadIdx.x; e < ROWS * COLS; e += S_THREADS) {
      const int r = e / COLS, q = e - r * COLS;
      const int64_t i = r0 + r, j = q0 + q;
      const bool live = i < rmax && j < cmax;
      cp_async<sizeof(T)>(dst + r * pitch + q, live ? src + i * ld + j : src, live);
    }
  }
}

template <typename T, int DC>
__global__ void __launch_bounds__(S_THREADS, 1)
sample_simt_kernel(const T* __restrict__ A, int64_t n, int64_t lda, const T* __restrict__ R,
                   int64_t ldr, int64_t c0, int64_t ncols, SimtPlan pl, int a_vec, int r_vec,
                   int want_cols, const int32_t* __restrict__ leaf_of, T* __restrict__ P,
                   T* __restrict__ PR) {
  using S = Simt<T, DC>;
  constexpr int BK = S::BK, PA = S::PA, RR = S::RR, CJ = S::CJ, NTY = S::NTY;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* As = reinterpret_cast<T*>(smem_raw);           // [2][S_BM][PA]
  T* Rs = As + 2 * S::a_elems;                       // [2][BK][DC]
  T* Rp = Rs + 2 * S::r_elems;                       // [S_BM][DC]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // a warp covers 8 threads along the sample columns and 4 along the rows
  const int tx = (lane & 7) + 8 * (warp % (S::NTX / 8));
  const int ty = (lane >> 3) + 4 * (warp / (S::NTX / 8));
  const int chunk = blockIdx.x % pl.nchunk;
  const int cta = blockIdx.x / pl.nchunk;
  const int64_t cq = (int64_t)chunk * DC;            // offset inside [c0, c0 + ncols)
  const int cw = (int)(ncols - cq < (int64_t)DC ? ncols - cq : (int64_t)DC);
  const T* Rc = R + c0 + cq;
  const long long tb = simt_begin(cta, pl.T, pl.G), te = simt_begin(cta + 1, pl.T, pl.G);

  // Row sample: partial sums per 32 columns of A, in FP32 added with Kahan
  // compensation (cmp) so that the error does not grow with n.
  constexpr bool kCompensate = sizeof(T) == 4;
  T acc[RR][4], cmp[RR][4];

  auto load_tile = [&](long long t, int buf) {
    const int64_t i0 = (t / pl.ntile) * S_BM, j0 = (t % pl.ntile) * BK;
    stage<T, S_BM, BK>(As + buf * S::a_elems, PA, A, lda, i0, n, j0, n, a_vec != 0);
    stage<T, BK, DC>(Rs + buf * S::r_elems, DC, Rc, ldr, j0, n, 0, cw, r_vec != 0);
  };
  if (tb < te) load_tile(tb, 0);
  asm volatile("cp.async.commit_group;");
  for (long long t = tb; t < te; ++t) {
    const int buf = (int)((t - tb) & 1);
    const int64_t panel = t / pl.ntile, tile = t % pl.ntile;
    const int64_t i0 = panel * S_BM, j0 = tile * BK;
    const bool first = t == tb || tile == 0, last = t == te - 1 || tile == pl.ntile - 1;
    if (first) {   // this panel's rows of R (feed the column sample)
      stage<T, S_BM, DC>(Rp, DC, Rc, ldr, i0, n, 0, cw, r_vec != 0);
      asm volatile("cp.async.commit_group;");
#pragma unroll
      for (int r = 0; r < RR; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = cmp[r][c] = T(0);
    }
    if (t + 1 < te) load_tile(t + 1, buf ^ 1);
    asm volatile("cp.async.commit_group;");
    asm volatile("cp.async.wait_group 1;");
    __syncthreads();
    T* at = As + buf * S::a_elems;
    const T* rt = Rs + buf * S::r_elems;
    // leaf blocks are zeroed here.  Leaves are contiguous index ranges, so a
    // tile whose rows all precede its columns holds masked entries only if
    // the last row's leaf is the first column's (and the other way round)
    if (leaf_of != nullptr) {
      const int64_t il = min(i0 + S_BM, n) - 1, jl = min(j0 + BK, n) - 1;
      bool hit = true;
      if (il < j0) hit = leaf_of[il] == leaf_of[j0];
      else if (jl < i0) hit = leaf_of[jl] == leaf_of[i0];
      if (hit) {
        for (int e = tid; e < S_BM * BK; e += S_THREADS) {
          const int r = e / BK, c = e - r * BK;
          if (i0 + r < n && j0 + c < n && leaf_of[i0 + r] == leaf_of[j0 + c]) at[r * PA + c] = T(0);
        }
        __syncthreads();
      }
    }
    // row sample: acc += A_tile * R_tile
    // (operands of the next four inner indices are read while the current
    // ones are multiplied: two warps a scheduler do not hide the reads)
    T av[RR][4], bv[2][4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) ld_vec4(bv[0][u], rt + u * DC + tx * 4);
#pragma unroll
    for (int r = 0; r < RR; ++r) ld_vec4(av[r], at + (ty + NTY * r) * PA);
#pragma unroll 1
    for (int kb = 0; kb < BK; kb += 32) {
      T tp[RR][4];
#pragma unroll
      for (int r = 0; r < RR; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) tp[r][c] = T(0);
#pragma unroll
      for (int k4 = 0; k4 < 8; ++k4) {
        // (past the tile's end: its first indices again, read but not used)
        const int kn = kb + 4 * k4 + 4 < BK ? kb + 4 * k4 + 4 : 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          ld_vec4(bv[(k4 + 1) & 1][u], rt + (kn + u) * DC + tx * 4);
#pragma unroll
        for (int r = 0; r < RR; ++r) {
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < 4; ++c) tp[r][c] = fma(av[r][u], bv[k4 & 1][u][c], tp[r][c]);
          ld_vec4(av[r], at + (ty + NTY * r) * PA + kn);
        }
      }
#pragma unroll
      for (int r = 0; r < RR; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (kCompensate) {
            const T y = tp[r][c] - cmp[r][c];
            const T s = acc[r][c] + y;
            cmp[r][c] = (s - acc[r][c]) - y;
            acc[r][c] = s;
          } else {
            acc[r][c] += tp[r][c];
          }
        }
    }
    if (want_cols) {
      // column sample of this tile: pc = A_tile^T * R_panel
      T pc[CJ][4];
#pragma unroll
      for (int r = 0; r < CJ; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) pc[r][c] = T(0);
      // a ring of four rows' operands, read two rows ahead
      T ar[4][CJ], br[4][4];
      auto ld_row = [&](int slot, int i) {
        ld_vec4(br[slot], Rp + i * DC + tx * 4);
        if constexpr (CJ == 4) {
          ld_vec4(ar[slot], at + i * PA + ty * 4);
        } else {
#pragma unroll
          for (int r = 0; r < CJ; ++r) ar[slot][r] = at[i * PA + ty * CJ + r];
        }
      };
      ld_row(0, 0);
      ld_row(1, 1);
#pragma unroll 2
      for (int i0b = 0; i0b < S_BM; i0b += 4) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          ld_row((x + 2) & 3, min(i0b + x + 2, S_BM - 1));
#pragma unroll
          for (int r = 0; r < CJ; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) pc[r][c] = fma(ar[x][r], br[x][c], pc[r][c]);
        }
      }
      T* Pp = P + ((size_t)panel * pl.nchunk + chunk) * n * DC;
#pragma unroll
      for (int r = 0; r < CJ; ++r) {
        const int64_t j = j0 + ty * CJ + r;
        if (j >= n) continue;
        st_vec4(Pp + j * DC + tx * 4, pc[r]);
      }
    }
    if (last) {   // this CTA's part of the panel's row sample
      T* o = PR + ((size_t)chunk * (pl.G + pl.npanel) + cta + panel) * S_BM * DC;
#pragma unroll
      for (int r = 0; r < RR; ++r) {
        st_vec4(o + (ty + NTY * r) * DC + tx * 4, acc[r]);
        if (kCompensate) st_vec4(o + simt_row_elems(pl) + (ty + NTY * r) * DC + tx * 4, cmp[r]);
      }
    }
    __syncthreads();   // before the next copies into these buffers
  }
}

// Sr[i][c0 + q*DC + cc] = the sum of its panel's row partials, in CTA order:
// one thread per entry.  FP32: compensated, and with the remainders of the
// partials' own compensation (without them a cut cost a rounding: the error
// 1.10e-7 to 1.17e-7 instead of 1.06e-7 to 1.14e-7).
template <typename T>
__device__ __forceinline__ void reduce_row_entry(const T* __restrict__ PR, int64_t n, SimtPlan pl,
                                                 int64_t c0, int64_t ncols, T* __restrict__ Sr,
                                                 int64_t lds, int64_t t) {
  const int dc = pl.dc;
  const int q = (int)(t / (n * dc));
  const int64_t rem = t - (int64_t)q * n * dc;
  const int64_t i = rem / dc;
  const int cc = (int)(rem - i * dc);
  const int64_t col = (int64_t)q * dc + cc;
  if (col >= ncols) return;
  const int p = (int)(i / S_BM), r = (int)(i % S_BM);
  const int q0 = simt_owner((long long)p * pl.ntile, pl.T, pl.G);
  const int q1 = simt_owner((long long)(p + 1) * pl.ntile - 1, pl.T, pl.G);
  const T* src = PR + (((size_t)q * (pl.G + pl.npanel) + p) * S_BM + r) * dc + cc;
  T s = T(0), k = T(0);
  for (int g = q0; g <= q1; ++g) {
    const T x = src[(size_t)g * S_BM * dc];
    if (sizeof(T) == 4) {
      const T u = s + x;
      k += (fabs(s) >= fabs(x)) ? ((s - u) + x) : ((x - u) + s);
      k -= src[(size_t)g * S_BM * dc + simt_row_elems(pl)];
      s = u;
    } else {
      s += x;
    }
  }
  Sr[i * lds + c0 + col] = isfinite(s) ? s + k : s;
}

// Sc[j][c0 + q*DC + cc] = sum over panels p (in order) of P[p][q][j][cc];
// one thread sums four adjacent columns, eight panels in flight per step
template <typename T>
__device__ __forceinline__ void reduce_col_entries(const T* __restrict__ P, int64_t n, int npanel,
                                                   int nchunk, int dc, int64_t c0, int64_t ncols,
                                                   T* __restrict__ Sc, int64_t lds, int64_t t) {
  const int g4 = dc / 4;
  int q = (int)(t / (n * g4));
  int64_t rem = t - (int64_t)q * n * g4;
  int64_t j = rem / g4;
  int cc = (int)(rem - j * g4) * 4;
  const int64_t pstride = (int64_t)nchunk * n * dc;
  const T* src = P + (int64_t)q * n * dc + j * dc + cc;
  // FP32: compensated (Neumaier) FP32 sums: s + k carries 48 bits, so the error
  // is that of the partials and one rounding, as with FP64 sums (n = 1000 to
  // 20000, 16 to 128 columns: the same error to four digits, 1.7e-7 to
  // 2.2e-7); FP64 additions and conversions would cost more than reading the
  // slab
  T s[4] = {T(0), T(0), T(0), T(0)}, k[4] = {T(0), T(0), T(0), T(0)};
  auto add = [&](int e, T x) {
    if (sizeof(T) == 4) {
      const T u = s[e] + x;
      k[e] += (fabs(s[e]) >= fabs(x)) ? ((s[e] - u) + x) : ((x - u) + s[e]);
      s[e] = u;
    } else {
      s[e] += x;
    }
  };
  int p = 0;
  for (; p + 8 <= npanel; p += 8) {
    T v[8][4];
#pragma unroll
    for (int u = 0; u < 8; ++u) ld_vec4(v[u], src + (int64_t)(p + u) * pstride);
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int e = 0; e < 4; ++e) add(e, v[u][e]);
  }
  for (; p < npanel; ++p) {
    T v[4];
    ld_vec4(v, src + (int64_t)p * pstride);
#pragma unroll
    for (int e = 0; e < 4; ++e) add(e, v[e]);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    int64_t col = (int64_t)q * dc + cc + e;
    if (col >= ncols) continue;
    T v = s[e] + k[e];
    if (sizeof(T) == 4 && !isfinite(s[e])) {
      // a partial is infinite or NaN, or the running sum has left FP32's range
      // (the total may still lie in it): in FP64
      double w = 0.0;
#pragma unroll 1
      for (p = 0; p < npanel; ++p) w += (double)src[(int64_t)p * pstride + e];
      v = (T)w;
    }
    Sc[j * lds + c0 + col] = v;
  }
}

template <typename T>
__global__ void reduce_partials_kernel(const T* __restrict__ P, int64_t n, int npanel, int nchunk,
                                       int64_t c0, int64_t ncols, T* __restrict__ Sc, int64_t lds) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < (int64_t)nchunk * n * (S_DC / 4))
    reduce_col_entries(P, n, npanel, nchunk, S_DC, c0, ncols, Sc, lds, t);
}

// both slabs of the SIMT kernel (Sc == nullptr: the row samples only)
template <typename T>
__global__ void reduce_simt_kernel(const T* __restrict__ P, const T* __restrict__ PR, int64_t n,
                                   SimtPlan pl, int64_t c0, int64_t ncols, T* __restrict__ Sr,
                                   T* __restrict__ Sc, int64_t lds) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t nc = Sc != nullptr ? (int64_t)pl.nchunk * n * (pl.dc / 4) : 0;
  if (t < nc)
    reduce_col_entries(P, n, pl.npanel, pl.nchunk, pl.dc, c0, ncols, Sc, lds, t);
  else if (t - nc < (int64_t)pl.nchunk * n * pl.dc)
    reduce_row_entry(PR, n, pl, c0, ncols, Sr, lds, t - nc);
}

// The SIMT path: scratch of sample_scratch_bytes
template <typename T, int DC>
Err launch_simt(const T* A, int64_t n, int64_t lda, const T* R, int64_t ldr, int64_t c0,
                int64_t ncols, T* Sr, T* Sc, int64_t lds, const int32_t* leaf_of,
                const SimtPlan& pl, T* scratch, cudaStream_t s) {
  using S = Simt<T, DC>;
  HSS_CUDA_TRY(cudaFuncSetAttribute(sample_simt_kernel<T, DC>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem));
  T* P = scratch;
  T* PR = P + simt_col_elems(pl, n);
  // 16-byte copies need 16-byte aligned rows
  auto aligned = [](const T* p, int64_t ld) {
    return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld * sizeof(T)) % 16 == 0;
  };
  sample_simt_kernel<T, DC><<<(unsigned)(pl.nchunk * pl.G), S_THREADS, S::smem, s>>>(
      A, n, lda, R, ldr, c0, ncols, pl, aligned(A, lda) ? 1 : 0, aligned(R + c0, ldr) ? 1 : 0,
      Sc != nullptr ? 1 : 0, leaf_of, P, PR);
  HSS_TRY(check_launch("sample_simt_kernel"));
  const int64_t total = (int64_t)pl.nchunk * n * ((Sc != nullptr ? pl.dc / 4 : 0) + pl.dc);
  reduce_simt_kernel<T><<<(unsigned)((total + 255) / 256), 256, 0, s>>>(P, PR, n, pl, c0, ncols,
                                                                        Sr, Sc, lds);
  return check_launch("reduce_simt_kernel");
}

Err sm_count(int* sms) {
  int dev = 0;
  HSS_CUDA_TRY(cudaGetDevice(&dev));
  HSS_CUDA_TRY(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
  return ok();
}

}  // namespace

Err launch_reduce_partials(const float* P, int64_t n, int npanel, int nchunk, int64_t c0,
                           int64_t ncols, float* Sc, int64_t lds, cudaStream_t s) {
  int64_t total = (int64_t)nchunk * n * (S_DC / 4);
  reduce_partials_kernel<float><<<(unsigned)((total + 255) / 256), 256, 0, s>>>(
      P, n, npanel, nchunk, c0, ncols, Sc, lds);
  return check_launch("reduce_partials_kernel");
}

Err launch_sample_mma(const float* A, int64_t n, int64_t lda, const float* R, int64_t ldr,
                      int64_t c0, int64_t ncols, float* Sr, float* Sc, int64_t lds,
                      const int32_t* leaf_of, int mode, float* P, cudaStream_t s);

bool sample_tc_supported(const float* A, int64_t n, int64_t lda, int mode);
Err sample_tc_need(int64_t n, int64_t ncols, int mode, size_t* need);
Err launch_sample_tc(const float* A, int64_t n, int64_t lda, const float* R, int64_t ldr,
                     int64_t c0, int64_t ncols, float* Sr, float* Sc, int64_t lds,
                     const int32_t* leaf_of, int mode, SampleScratch* scratch, cudaStream_t s);

static bool legacy_mma_requested() {
  static const bool v = [] {
    const char* e = std::getenv("HSS_SAMPLE_KERNEL");
    return e != nullptr && std::strcmp(e, "mma") == 0;
  }();
  return v;
}

// the SIMT kernel's slabs (NATIVE), or the mma.sync kernel's column slab
static Err sample_scratch_bytes(int64_t n, int64_t ncols, int mode, bool f64, size_t* need) {
  if (mode == HSS_SAMPLE_NATIVE) {
    int sms = 0;
    HSS_TRY(sm_count(&sms));
    const SimtPlan pl = f64 ? simt_plan<double>(n, ncols, sms) : simt_plan<float>(n, ncols, sms);
    *need = (simt_col_elems(pl, n) + simt_row_elems(pl) * (f64 ? 1 : 2)) * (f64 ? 8 : 4);
    return ok();
  }
  int64_t npanel = (n + S_BM - 1) / S_BM;
  int64_t nchunk = (ncols + S_DC - 1) / S_DC;
  *need = (size_t)npanel * nchunk * n * S_DC * sizeof(float);
  return ok();
}

Err sample_scratch_need(const void* A, int64_t n, int64_t lda, int64_t ncols, int mode, bool f64,
                        size_t* need) {
  *need = 0;
  if (n <= 0 || ncols <= 0) return ok();
  if (!f64 && !legacy_mma_requested() &&
      sample_tc_supported(reinterpret_cast<const float*>(A), n, lda, mode))
    return sample_tc_need(n, ncols, mode, need);
  return sample_scratch_bytes(n, ncols, mode, f64, need);
}

template <typename T>
Err launch_sample(const T* A, int64_t n, int64_t lda, const T* R, int64_t ldr, int64_t c0,
                  int64_t c1, T* Sr, T* Sc, int64_t lds, const int32_t* leaf_of, int mode,
                  SampleScratch* scratch, cudaStream_t s, float* ms_out) {
  int64_t ncols = c1 - c0;
  if (n <= 0 || ncols <= 0) return ok();
  const bool f64 = sizeof(T) == 8;
  // the TF32 and split-bfloat16 modes run on tcgen05 when A's layout suits
  // TMA (16-byte aligned rows); HSS_SAMPLE_KERNEL=mma selects the warp-level
  // mma.sync kernel
  const bool tc = !f64 && !legacy_mma_requested() &&
                  sample_tc_supported(reinterpret_cast<const float*>(A), n, lda, mode);
  size_t need = 0;
  if (!tc) HSS_TRY(sample_scratch_bytes(n, ncols, mode, f64, &need));
  if (scratch->bytes < need && scratch->fixed)
    return fail(HSS_ERR_INVALID, "sampling: the fixed scratch is smaller than this call needs");
  if (scratch->bytes < need) {
    dfree(scratch->part, s);
    scratch->part = nullptr;
    scratch->bytes = 0;
    HSS_TRY(dalloc(&scratch->part, need, s));
    scratch->bytes = need;
  }
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (ms_out) {
    HSS_CUDA_TRY(cudaEventCreate(&e0));
    HSS_CUDA_TRY(cudaEventCreate(&e1));
    HSS_CUDA_TRY(cudaEventRecord(e0, s));
  }
  T* P = reinterpret_cast<T*>(scratch->part);
  if (tc) {
    HSS_TRY(launch_sample_tc(reinterpret_cast<const float*>(A), n, lda,
                             reinterpret_cast<const float*>(R), ldr, c0, ncols,
                             reinterpret_cast<float*>(Sr), reinterpret_cast<float*>(Sc), lds,
                             leaf_of, mode, scratch, s));
  } else if (sizeof(T) == 4 && mode != HSS_SAMPLE_NATIVE) {
    HSS_TRY(launch_sample_mma(reinterpret_cast<const float*>(A), n, lda,
                              reinterpret_cast<const float*>(R), ldr, c0, ncols,
                              reinterpret_cast<float*>(Sr), reinterpret_cast<float*>(Sc), lds,
                              leaf_of, mode, reinterpret_cast<float*>(P), s));
  } else {
    int sms = 0;
    HSS_TRY(sm_count(&sms));
    const SimtPlan pl = simt_plan<T>(n, ncols, sms);
    HSS_TRY((pl.dc == 64 ? launch_simt<T, 64> : launch_simt<T, 32>)(
        A, n, lda, R, ldr, c0, ncols, Sr, Sc, lds, leaf_of, pl, P, s));
  }
  if (ms_out) {
    HSS_CUDA_TRY(cudaEventRecord(e1, s));
    HSS_CUDA_TRY(cudaEventSynchronize(e1));
    HSS_CUDA_TRY(cudaEventElapsedTime(ms_out, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
  }
  return ok();
}

template Err launch_sample<float>(const float*, int64_t, int64_t, const float*, int64_t, int64_t,
                                  int64_t, float*, float*, int64_t, const int32_t*, int,
                                  SampleScratch*, cudaStream_t, float*);
template Err launch_sample<double>(const double*, int64_t, int64_t, const double*, int64_t,
                                   int64_t, int64_t, double*, double*, int64_t, const int32_t*,
                                   int, SampleScratch*, cudaStream_t, float*);

}  // namespace hss
