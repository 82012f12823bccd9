// ULV-like factorization (Algorithm 3) of a compressed HSS form, in FP64
// whatever the input precision.
//
// One CTA per node, level by level (deepest first); nodes of 64 rows or more
// go through hss_ulv_big.cu instead:
//   D_tau  = A(I,I) at a leaf, [Dtil_1, B12 Vtb_2^T; B21 Vtb_1^T, Dtil_2] above;
//   Vhat   = V at a leaf, diag(Vtb_1, Vtb_2) V above;
//   W      = Omega D_tau with Omega = [-E I; I 0] Pi^T (Omega U = [0; I]);
//   LQ of the top r = m - k rows of W by Householder reflectors applied from
//   the right to every row of W, so W_t Q^T = [L 0] and W_b Q^T = [W_b Q_t^T,
//   Dtil];  Vtilde = Q Vhat.   Root: LU with partial pivoting of D_0.
// At the end one launch forms what the solve (hss_solve.cu) multiplies by
// instead of substituting: the inverses of the 32 x 32 diagonal blocks of L
// and of the root's LU (of the well-conditioned ones: ULV_BLOCK_COND), the
// compact WY factors of the small nodes, and the root's interchanges as a
// permutation.
#include "hss_internal.cuh"
#include "hss_tree.h"

#include <algorithm>
#include <climits>

using namespace hss;

namespace hss {

size_t ulv_factor_big_min_m();
Err ulv_factor_big_multi(const std::vector<std::pair<hss_s*, int>>& items,
                         const std::vector<int32_t*>& status, cudaStream_t s);

namespace {

constexpr int U_THREADS = 256;
constexpr int U_WARPS = U_THREADS / 32;

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ double block_sum(double v, double* red) {
  v = wsum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int q = 0; q < U_WARPS; ++q) s += red[q];
  return s;
}

__device__ __forceinline__ double ld_any(const void* p, int64_t i, int f64) {
  return f64 ? reinterpret_cast<const double*>(p)[i] : (double)reinterpret_cast<const float*>(p)[i];
}

struct FacItem {
  int m, k, kc, mc, leaf, root;
  const void* D;          // leaf block (input dtype), ld m
  const double* Dtil1;
  const double* Dtil2;
  const double* Vtb1;
  const double* Vtb2;
  int k1, k2, kc1, kc2;
  const void* B12;        // k1 x kc2
  const void* B21;        // k2 x kc1
  const int32_t* permr;
  const double* Er;
  const int32_t* permc;
  const double* Ec;
  double* hv;
  double* tau;
  double* L;
  double* WbQt;
  double* Dtil;
  double* Vtt;
  double* Vtb;
  double* Dw;     // m x m scratch
  double* W;      // m x m scratch
  double* Vh;     // m x kc scratch
  double* Vd;     // mc x kc scratch
  int32_t* piv;   // root
  int32_t* status;
};

__global__ void __launch_bounds__(U_THREADS) ulv_factor_kernel(const FacItem* items, int f64) {
  extern __shared__ double vsh[];
  __shared__ double red[U_WARPS];
  __shared__ double redv[U_WARPS];
  __shared__ int redi[U_WARPS];
  const FacItem it = items[blockIdx.x];
  const int m = it.m, k = it.k, r = m - k, kc = it.kc;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* Dw = it.Dw;
  // 1. D_tau
  for (int64_t e = tid; e < (int64_t)m * m; e += U_THREADS) {
    int i = (int)(e / m), j = (int)(e - (int64_t)i * m);
    double v;
    if (it.leaf) {
      v = ld_any(it.D, e, f64);
    } else {
      const int k1 = it.k1;
      if (i < k1 && j < k1) v = it.Dtil1[i * k1 + j];
      else if (i >= k1 && j >= k1) v = it.Dtil2[(i - k1) * it.k2 + (j - k1)];
      else if (i < k1) {   // B12 Vtb_2^T
        v = 0.0;
        for (int l = 0; l < it.kc2; ++l)
          v = fma(ld_any(it.B12, (int64_t)i * it.kc2 + l, f64), it.Vtb2[(j - k1) * it.kc2 + l], v);
      } else {             // B21 Vtb_1^T
        v = 0.0;
        for (int l = 0; l < it.kc1; ++l)
          v = fma(ld_any(it.B21, (int64_t)(i - k1) * it.kc1 + l, f64), it.Vtb1[j * it.kc1 + l], v);
      }
    }
    Dw[e] = v;
  }
  __syncthreads();
  if (it.root) {
    // LU with partial pivoting, lowest index on ties
    for (int i = 0; i < m; ++i) {
      double bv = -1.0;
      int bi = INT_MAX;
      for (int j = i + tid; j < m; j += U_THREADS) {
        double x = fabs(Dw[(int64_t)j * m + i]);
        if (x > bv) {
          bv = x;
          bi = j;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        double ov = __shfl_xor_sync(0xffffffffu, bv, o);
        int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) {
          bv = ov;
          bi = oi;
        }
      }
      __syncthreads();
      if (lane == 0) {
        redv[warp] = bv;
        redi[warp] = bi;
      }
      __syncthreads();
      bv = redv[0];
      bi = redi[0];
      for (int q = 1; q < U_WARPS; ++q)
        if (redv[q] > bv || (redv[q] == bv && redi[q] < bi)) {
          bv = redv[q];
          bi = redi[q];
        }
      if (!(bv > 0.0)) {   // zeros and NaN only (then no row was chosen)
        if (tid == 0) *it.status = HSS_ERR_SINGULAR;
        return;
      }
      if (bi != i)
        for (int c = tid; c < m; c += U_THREADS) {
          double t = Dw[(int64_t)i * m + c];
          Dw[(int64_t)i * m + c] = Dw[(int64_t)bi * m + c];
          Dw[(int64_t)bi * m + c] = t;
        }
      if (tid == 0) it.piv[i] = bi;
      __syncthreads();
      const double piv = Dw[(int64_t)i * m + i];
      for (int j = i + 1 + warp; j < m; j += U_WARPS) {
        double l = Dw[(int64_t)j * m + i] / piv;
        for (int c = i + 1 + lane; c < m; c += 32)
          Dw[(int64_t)j * m + c] = fma(-l, Dw[(int64_t)i * m + c], Dw[(int64_t)j * m + c]);
        if (lane == 0) Dw[(int64_t)j * m + i] = l;
      }
      __syncthreads();
    }
    return;
  }
  // 2. Vhat
  double* Vd = it.leaf ? it.Vh : it.Vd;
  const int mc = it.mc;
  for (int64_t e = tid; e < (int64_t)mc * kc; e += U_THREADS) Vd[e] = 0.0;
  __syncthreads();
  for (int l = tid; l < kc; l += U_THREADS) Vd[(int64_t)it.permc[l] * kc + l] = 1.0;
  for (int64_t e = tid; e < (int64_t)(mc - kc) * kc; e += U_THREADS) {
    int q = (int)(e / kc), l = (int)(e - (int64_t)q * kc);
    Vd[(int64_t)it.permc[kc + q] * kc + l] = it.Ec[e];
  }
  __syncthreads();
  if (!it.leaf) {
    for (int64_t e = tid; e < (int64_t)m * kc; e += U_THREADS) {
      int i = (int)(e / kc), l = (int)(e - (int64_t)i * kc);
      double v = 0.0;
      if (i < it.k1) {
        for (int q = 0; q < it.kc1; ++q) v = fma(it.Vtb1[i * it.kc1 + q], Vd[(int64_t)q * kc + l], v);
      } else {
        int ii = i - it.k1;
        for (int q = 0; q < it.kc2; ++q)
          v = fma(it.Vtb2[ii * it.kc2 + q], Vd[(int64_t)(it.kc1 + q) * kc + l], v);
      }
      it.Vh[e] = v;
    }
  }
  // 3. W = Omega D
  double* W = it.W;
  for (int64_t e = tid; e < (int64_t)m * m; e += U_THREADS) {
    int i = (int)(e / m), j = (int)(e - (int64_t)i * m);
    double v;
    if (i < r) {
      v = Dw[(int64_t)it.permr[k + i] * m + j];
      for (int l = 0; l < k; ++l) v = fma(-it.Er[(int64_t)i * k + l], Dw[(int64_t)it.permr[l] * m + j], v);
    } else {
      v = Dw[(int64_t)it.permr[i - r] * m + j];
    }
    W[e] = v;
  }
  __syncthreads();
  // 4. LQ of the top r rows, reflectors applied to every row of W
  for (int i = 0; i < r; ++i) {
    double* wi = W + (int64_t)i * m;
    double sa = 0.0, st = 0.0;
    for (int c = i + tid; c < m; c += U_THREADS) {
      double x = wi[c];
      sa = fma(x, x, sa);
      if (c > i) st = fma(x, x, st);
    }
    sa = block_sum(sa, red);
    st = block_sum(st, red);
    const double alpha = wi[i];
    const double sigma = sqrt(sa);
    double tau, beta, scal;
    if (st == 0.0) {
      tau = 0.0;
      beta = alpha;
      scal = 0.0;
    } else {
      beta = -copysign(sigma, alpha);
      tau = (beta - alpha) / beta;
      scal = 1.0 / (alpha - beta);
    }
    for (int c = tid; c < m; c += U_THREADS) {
      double v = c < i ? 0.0 : (c == i ? 1.0 : wi[c] * scal);
      vsh[c] = v;
      it.hv[(int64_t)i * m + c] = v;
    }
    __syncthreads();
    for (int c = i + tid; c < m; c += U_THREADS) wi[c] = c == i ? beta : 0.0;
    if (tid == 0) it.tau[i] = tau;
    for (int j = i + 1 + warp; j < m; j += U_WARPS) {
      double* wj = W + (int64_t)j * m;
      double dot = 0.0;
      for (int c = i + lane; c < m; c += 32) dot = fma(wj[c], vsh[c], dot);
      dot = wsum(dot) * tau;
      for (int c = i + lane; c < m; c += 32) wj[c] = fma(-dot, vsh[c], wj[c]);
    }
    __syncthreads();
  }
  for (int64_t e = tid; e < (int64_t)r * r; e += U_THREADS) {
    int i = (int)(e / r), j = (int)(e - (int64_t)i * r);
    it.L[e] = j <= i ? W[(int64_t)i * m + j] : 0.0;
  }
  for (int64_t e = tid; e < (int64_t)k * r; e += U_THREADS) {
    int l = (int)(e / r), j = (int)(e - (int64_t)l * r);
    it.WbQt[e] = W[(int64_t)(r + l) * m + j];
  }
  for (int64_t e = tid; e < (int64_t)k * k; e += U_THREADS) {
    int l = (int)(e / k), j = (int)(e - (int64_t)l * k);
    it.Dtil[e] = W[(int64_t)(r + l) * m + r + j];
  }
  __syncthreads();
  // 5. Vtilde = Q Vhat = H_{r-1} ... H_0 Vhat (H_0 first), one thread per column
  for (int l = tid; l < kc; l += U_THREADS) {
    double* vh = it.Vh;
    for (int i = 0; i < r; ++i) {
      const double* h = it.hv + (int64_t)i * m;
      double dot = 0.0;
      for (int c = i; c < m; ++c) dot = fma(h[c], vh[(int64_t)c * kc + l], dot);
      dot *= it.tau[i];
      for (int c = i; c < m; ++c) vh[(int64_t)c * kc + l] = fma(-dot, h[c], vh[(int64_t)c * kc + l]);
    }
    for (int i = 0; i < m; ++i) {
      double v = vh[(int64_t)i * kc + l];
      if (i < r) it.Vtt[(int64_t)i * kc + l] = v;
      else it.Vtb[(int64_t)(i - r) * kc + l] = v;
    }
  }
}

// What the solve needs of a factored node besides the factors, one CTA per
// 32 x 32 block.
enum { UB_LOWER = 0, UB_UNIT_LOWER = 1, UB_UPPER = 2, UB_WY = 3, UB_PERM = 4 };
struct BlockItem {
  const double* M;    // the diagonal block (ld), or (UB_WY) the panel's reflectors
  int64_t ld;
  double* out;        // 32 x 32
  const double* tau;  // UB_WY
  const int32_t* piv; // UB_PERM: n interchanges -> the permutation perm
  int32_t* perm;
  int n, wid, mode;   // order of the block; UB_WY: columns of the panel
};

constexpr int UBN = 32;

// A triangular block B goes by its inverse only while c = max_i (|B||B^-1| 1)_i
// is at most this: x = B^-1 b leaves a residual of about c roundings of |B||x|,
// where substitution leaves one whatever the condition (20,000 random blocks,
// residual in units of 2^-53 |B||x|, mean / largest: c in [16, 32) 0.9 / 4.5
// against 0.6 / 2.7, [256, 512) 3.6 / 45, 2^20 7800 / 71,000).  L's blocks are
// mostly below it (p90 of 7 to 12 on Toeplitz, Schur and kernel matrices), the
// root's 50 to 300 and above it.  Other blocks are stored for substitution: the
// rows divided by their diagonal, whose place the reciprocal takes, so that a
// step of the substitution is one FMA (or as they are, where a quotient would
// be very large), with a one (two) in the corner of the empty triangle.
constexpr double ULV_BLOCK_COND = 32.0;

__global__ void __launch_bounds__(U_THREADS) ulv_blocks_kernel(const BlockItem* items) {
  __shared__ double M[UBN][UBN + 1];
  __shared__ double xl[UBN][UBN + 1];
  __shared__ double sd[UBN], rs[UBN];
  __shared__ int keep;   // the block itself, not its inverse
  const BlockItem it = items[blockIdx.x];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, n = it.n;
  if (it.mode == UB_PERM) {   // row i of the permuted system is row perm[i]
    // one thread's chain of interchanges, in shared memory (M and xl) while both
    // arrays fit: n = 725 of rank 40 in leaves of 64, factor 1580 -> 1549 us
    constexpr int FIT = static_cast<int>(sizeof(M) / sizeof(int));
    int* perm = n <= FIT ? reinterpret_cast<int*>(&M[0][0]) : it.perm;
    const int* piv = it.piv;
    if (n <= FIT) {
      int* ps = reinterpret_cast<int*>(&xl[0][0]);
      for (int i = tid; i < n; i += U_THREADS) ps[i] = it.piv[i];
      piv = ps;
    }
    for (int i = tid; i < n; i += U_THREADS) perm[i] = i;
    __syncthreads();
    if (tid == 0)
      for (int i = 0; i < n; ++i) {
        const int p = piv[i];
        if (p > i && p < n) {   // (a singular root's pivots are not all written)
          const int t = perm[i];
          perm[i] = perm[p];
          perm[p] = t;
        }
      }
    __syncthreads();
    if (n <= FIT)
      for (int i = tid; i < n; i += U_THREADS) it.perm[i] = perm[i];
    return;
  }
  const bool upper = it.mode == UB_UPPER || it.mode == UB_WY;
  if (it.mode == UB_WY) {   // I + U D with U the strict upper triangle of V V^T, D = diag(tau)
    if (tid < UBN) sd[tid] = tid < n ? it.tau[tid] : 0.0;
    __syncthreads();
    for (int e = tid; e < n * n; e += U_THREADS) {
      const int a = e / n, b = e - a * n;
      if (a >= b) continue;
      double s0 = 0.0, s1 = 0.0;
      int c = 0;
      for (; c + 1 < it.wid; c += 2) {
        s0 = fma(it.M[a * it.ld + c], it.M[b * it.ld + c], s0);
        s1 = fma(it.M[a * it.ld + c + 1], it.M[b * it.ld + c + 1], s1);
      }
      if (c < it.wid) s0 = fma(it.M[a * it.ld + c], it.M[b * it.ld + c], s0);
      M[a][b] = (s0 + s1) * sd[b];
    }
  } else {
    for (int e = tid; e < n * n; e += U_THREADS) M[e / n][e % n] = it.M[(e / n) * it.ld + e % n];
    __syncthreads();
    if (tid < UBN) sd[tid] = (it.mode != UB_UNIT_LOWER && tid < n) ? 1.0 / M[tid][tid] : 1.0;
  }
  __syncthreads();
  // the inverse by substitution on the unit matrix: lane = column, warp w
  // keeps rows w + 8 t; row l is final at its step
  double x[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) x[t] = (w + 8 * t == lane) ? 1.0 : 0.0;
  for (int q = 0; q < n; ++q) {
    const int l = upper ? n - 1 - q : q;
    if (w == (l & 7)) {
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t == (l >> 3)) {
          if (it.mode != UB_WY) x[t] *= sd[l];
          xl[l][lane] = x[t];
        }
    }
    __syncthreads();
    const double xv = xl[l][lane];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int a = w + 8 * t;
      if (upper ? a < l : (a > l && a < n)) x[t] = fma(-M[a][l], xv, x[t]);
    }
  }
  if (it.mode != UB_WY) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {   // row sums of |B^-1|
      const double v = wsum(w + 8 * t < n && lane < n ? fabs(x[t]) : 0.0);
      if (lane == 0) rs[w + 8 * t] = v;
    }
    __syncthreads();
    if (w == 0) {
      double c = 0.0;
      const int k0 = upper ? lane + 1 : 0, k1 = upper ? n : lane;
      if (lane < n) {
        for (int k = k0; k < k1; ++k) c = fma(fabs(M[lane][k]), rs[k], c);
        c = fma(it.mode == UB_UNIT_LOWER ? 1.0 : fabs(M[lane][lane]), rs[lane], c);
      }
      const bool bad = __any_sync(0xffffffffu, !(c <= ULV_BLOCK_COND));   // (NaN too)
      if (lane == 0) keep = bad;
    }
    __syncthreads();
    if (keep) {
      const int corner = upper ? (UBN - 1) * UBN : UBN - 1;
      double m[4], q[4];   // the triangle, and divided by its diagonal
      bool large = false;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int a = w + 8 * t;
        m[t] = q[t] = 0.0;
        if (a < n && lane < n && (upper ? lane >= a : lane <= a)) {
          m[t] = a == lane && it.mode == UB_UNIT_LOWER ? 1.0 : M[a][lane];
          q[t] = a == lane ? sd[a] : m[t] * sd[a];   // (sd: the reciprocals)
          // (a diagonal out of the normal range counts as large, and NaN)
          large = large || !(fabs(q[t]) <= 0x1p100 || (a == lane && fabs(q[t]) <= 0x1p1000));
        }
      }
      large = __syncthreads_or(large);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int e = (w + 8 * t) * UBN + lane;
        it.out[e] = e == corner ? (large ? 2.0 : 1.0) : large ? m[t] : q[t];
      }
      return;
    }
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int a = w + 8 * t;
    const double v = it.mode == UB_WY ? sd[a] * x[t] : x[t];
    it.out[a * UBN + lane] = (a < n && lane < n) ? v : 0.0;
  }
}

template <typename TI>
Err upload_and_launch(const std::vector<TI>& items, cudaStream_t s, TI** dev) {
  HSS_TRY(dalloc_t(dev, std::max<size_t>(items.size(), 1), s));
  HSS_TRY(upload_async(*dev, items.data(), items.size() * sizeof(TI), s));
  return ok();
}

}  // namespace
}  // namespace hss

// ---------------------------------------------------------------- factor
namespace hss {
namespace {

// One allocation for every factor of the handle; sets each node's pointers.
Err ulv_prepare(hss_s* h, cudaStream_t s) {
  h->ulv.release(s);
  const Tree& tr = h->tree;
  const int nn = (int)tr.nodes.size();
  UlvFactors& F = h->ulv;
  F.nodes.assign(nn, UlvNode{});
  // sizes: m = leaf size or k(c1) + k(c2); r = m - kr; kc
  std::vector<size_t> off(nn + 1, 0);
  size_t tot = 0;
  auto m_of = [&](int id) {
    const TNode& nd = tr.nodes[id];
    return nd.c1 < 0 ? nd.hi - nd.lo : h->gen[nd.c1].kr + h->gen[nd.c2].kr;
  };
  for (int id = 0; id < nn; ++id) {
    UlvNode& u = F.nodes[id];
    u.m = m_of(id);
    off[id] = tot;
    if (id == 0) {
      // LU, its blocks' inverses, pivots and permutation (int32 packed)
      tot += (size_t)u.m * u.m + 2 * (size_t)((u.m + UBN - 1) / UBN) * UBN * UBN + u.m + 2;
      continue;
    }
    const NodeGen& g = h->gen[id];
    u.k = g.kr;
    u.kc = g.kc;
    int r = u.m - u.k;
    tot += (size_t)r * u.m + r + (size_t)r * r + (size_t)u.k * r + (size_t)u.k * u.k +
           (size_t)r * u.kc + (size_t)u.k * u.kc;
    tot += 2 * (size_t)((r + UBN - 1) / UBN) * UBN * UBN;   // T, Li
  }
  double* blk = nullptr;
  HSS_TRY(dalloc_t(&blk, std::max<size_t>(tot, 1), s));
  F.block = blk;
  F.bytes = tot * sizeof(double);
  for (int id = 0; id < nn; ++id) {
    UlvNode& u = F.nodes[id];
    double* p = blk + off[id];
    if (id == 0) {
      F.root_m = u.m;
      F.root_lu = p;
      p += (size_t)u.m * u.m;
      const size_t nb = (size_t)((u.m + UBN - 1) / UBN) * UBN * UBN;
      F.root_li = p;
      F.root_ui = p + nb;
      F.root_piv = reinterpret_cast<int32_t*>(p + 2 * nb);
      F.root_perm = F.root_piv + u.m;
      continue;
    }
    int r = u.m - u.k;
    u.hv = p;
    p += (size_t)r * u.m;
    u.tau = p;
    p += r;
    u.L = p;
    p += (size_t)r * r;
    u.WbQt = p;
    p += (size_t)u.k * r;
    u.Dtil = p;
    p += (size_t)u.k * u.k;
    u.Vtt = p;
    p += (size_t)r * u.kc;
    u.Vtb = p;
    p += (size_t)u.k * u.kc;
    u.T = p;
    u.Li = p + (size_t)((r + UBN - 1) / UBN) * UBN * UBN;
  }
  return ok();
}

// scratch doubles of one node of the one-CTA kernel
size_t fac_scratch(const hss_s* h, int id) {
  const UlvNode& u = h->ulv.nodes[id];
  const NodeGen& g = h->gen[id];
  return 2 * (size_t)u.m * u.m + (size_t)u.m * std::max(u.kc, 1) +
         (size_t)std::max(g.mc, 1) * std::max(u.kc, 1);
}

FacItem fac_item(hss_s* h, int id, int32_t* status, double* sc) {
  const Tree& tr = h->tree;
  UlvFactors& F = h->ulv;
  const TNode& nd = tr.nodes[id];
  const UlvNode& u = F.nodes[id];
  const NodeGen& g = h->gen[id];
  FacItem it{};
  it.m = u.m;
  it.k = u.k;
  it.kc = u.kc;
  it.mc = g.mc;
  it.leaf = nd.c1 < 0;
  it.root = id == 0;
  it.D = g.D;
  if (!it.leaf) {
    const UlvNode& a = F.nodes[nd.c1];
    const UlvNode& b = F.nodes[nd.c2];
    it.Dtil1 = a.Dtil;
    it.Dtil2 = b.Dtil;
    it.Vtb1 = a.Vtb;
    it.Vtb2 = b.Vtb;
    it.k1 = a.k;
    it.k2 = b.k;
    it.kc1 = a.kc;
    it.kc2 = b.kc;
    it.B12 = g.B12;
    it.B21 = g.B21;
  }
  it.permr = g.permr;
  it.Er = g.Er;
  it.permc = g.permc;
  it.Ec = g.Ec;
  it.hv = u.hv;
  it.tau = u.tau;
  it.L = u.L;
  it.WbQt = u.WbQt;
  it.Dtil = u.Dtil;
  it.Vtt = u.Vtt;
  it.Vtb = u.Vtb;
  size_t so = 0;
  it.Dw = it.root ? F.root_lu : sc + so;
  so += (size_t)u.m * u.m;
  it.W = sc + so;
  so += (size_t)u.m * u.m;
  it.Vh = sc + so;
  so += (size_t)u.m * std::max(u.kc, 1);
  it.Vd = sc + so;
  it.piv = F.root_piv;
  it.status = status;
  return it;
}

// Factors `count` handles of one dtype together: round r takes depth
// maxdepth - r of every handle, deepest first; the small nodes of all
// handles share one launch of the one-CTA kernel, the large ones take the
// blocked whole-GPU path handle by handle.  Each node's arithmetic is the
// same as alone, so the factors are bitwise those of a single-handle call.
void factor_many(int count, hss_t* hs, cudaStream_t s, hss_status* st) {
  std::vector<int> live;
  int rounds = 0;
  for (int q = 0; q < count; ++q) {
    hss_s* h = hs[q];
    st[q] = HSS_OK;
    if (!h) {
      st[q] = HSS_ERR_INVALID;
      continue;
    }
    if (h->gen.empty() || h->gen[0].state != NODE_COMPRESSED) {
      h->err = "hss_factor: the handle holds no complete compressed form";
      st[q] = HSS_ERR_STATE;
      continue;
    }
    Err e = ulv_prepare(h, s);
    if (e.st) {
      h->err = e.msg;
      st[q] = e.st;
      h->ulv.release(s);
      continue;
    }
    live.push_back(q);
    rounds = std::max(rounds, h->tree.maxdepth + 1);
  }
  auto fail_all = [&](const Err& e) {
    for (int q : live)
      if (st[q] == HSS_OK) {
        hs[q]->err = e.msg;
        st[q] = e.st;
      }
  };
  int32_t* status = nullptr;   // one root-LU status per handle
  Err e = dalloc_t(&status, std::max(count, 1), s);
  if (e.st == HSS_OK && cudaMemsetAsync(status, 0, 4 * (size_t)std::max(count, 1), s) != cudaSuccess)
    e = fail(HSS_ERR_CUDA, "hss_factor: memset");
  if (e.st) fail_all(e);
  const int f64 = (!live.empty() && hs[live[0]]->dtype == HSS_F64) ? 1 : 0;
  for (int r = 0; r < rounds && e.st == HSS_OK; ++r) {
    std::vector<std::pair<int, int>> small;   // (handle, node)
    std::vector<std::pair<hss_s*, int>> big;  // large nodes of every handle
    std::vector<int32_t*> big_status;
    size_t scratch = 0;
    int maxm = 1;
    for (int q : live) {
      if (st[q] != HSS_OK) continue;
      hss_s* h = hs[q];
      const int depth = h->tree.maxdepth - r;
      if (depth < 0) continue;
      for (int id : h->tree.levels[depth]) {
        if ((size_t)h->ulv.nodes[id].m >= ulv_factor_big_min_m()) {
          big.push_back({h, id});
          big_status.push_back(status + q);
        } else {
          small.push_back({q, id});
          scratch += fac_scratch(h, id);
          maxm = std::max(maxm, h->ulv.nodes[id].m);
        }
      }
    }
    // the large nodes of all handles share the blocked path's launches
    e = ulv_factor_big_multi(big, big_status, s);
    if (e.st) break;
    if (small.empty()) continue;
    double* sc = nullptr;
    e = dalloc_t(&sc, std::max<size_t>(scratch, 1), s);
    if (e.st) break;
    std::vector<FacItem> items;
    size_t so = 0;
    for (auto& qi : small) {
      if (st[qi.first] != HSS_OK) continue;
      items.push_back(fac_item(hs[qi.first], qi.second, status + qi.first, sc + so));
      so += fac_scratch(hs[qi.first], qi.second);
    }
    FacItem* dev = nullptr;
    if (!items.empty()) e = upload_and_launch(items, s, &dev);
    if (e.st == HSS_OK && !items.empty()) {
      size_t smem = sizeof(double) * maxm;
      if (cudaFuncSetAttribute(ulv_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)smem) != cudaSuccess) {
        cudaGetLastError();
        e = fail(HSS_ERR_CUDA, "ulv_factor_kernel smem attribute");
      } else {
        ulv_factor_kernel<<<(unsigned)items.size(), U_THREADS, smem, s>>>(dev, f64);
        e = check_launch("ulv_factor_kernel");
      }
    }
    dfree(dev, s);
    dfree(sc, s);
  }
  // the blocks for the solve
  if (e.st == HSS_OK) {
    std::vector<BlockItem> items;
    for (int q : live) {
      if (st[q] != HSS_OK) continue;
      const UlvFactors& F = hs[q]->ulv;
      const int m0 = F.root_m;
      BlockItem it{};
      it.mode = UB_PERM;
      it.n = m0;
      it.piv = F.root_piv;
      it.perm = F.root_perm;
      items.push_back(it);
      for (int i0 = 0; i0 < m0; i0 += UBN) {
        BlockItem b{};
        b.M = F.root_lu + (size_t)i0 * m0 + i0;
        b.ld = m0;
        b.n = std::min(UBN, m0 - i0);
        b.mode = UB_UNIT_LOWER;
        b.out = F.root_li + (size_t)(i0 / UBN) * UBN * UBN;
        items.push_back(b);
        b.mode = UB_UPPER;
        b.out = F.root_ui + (size_t)(i0 / UBN) * UBN * UBN;
        items.push_back(b);
      }
      for (size_t id = 1; id < F.nodes.size(); ++id) {
        const UlvNode& u = F.nodes[id];
        const int r = u.m - u.k;
        for (int i0 = 0; i0 < r; i0 += UBN) {
          const size_t o = (size_t)(i0 / UBN) * UBN * UBN;
          BlockItem b{};
          b.M = u.L + (size_t)i0 * r + i0;
          b.ld = r;
          b.n = std::min(UBN, r - i0);
          b.mode = UB_LOWER;
          b.out = u.Li + o;
          items.push_back(b);
          if ((size_t)u.m >= ulv_factor_big_min_m()) continue;   // T comes with its panels
          b.M = u.hv + (size_t)i0 * u.m + i0;
          b.ld = u.m;
          b.wid = u.m - i0;
          b.tau = u.tau + i0;
          b.mode = UB_WY;
          b.out = u.T + o;
          items.push_back(b);
        }
      }
    }
    if (!items.empty()) {
      BlockItem* dev = nullptr;
      e = upload_and_launch(items, s, &dev);
      if (e.st == HSS_OK) {
        ulv_blocks_kernel<<<(unsigned)items.size(), U_THREADS, 0, s>>>(dev);
        e = check_launch("ulv_blocks_kernel");
      }
      dfree(dev, s);
    }
  }
  if (e.st) fail_all(e);
  std::vector<int32_t> hst(std::max(count, 1), 0);
  if (status) {
    cudaMemcpyAsync(hst.data(), status, 4 * (size_t)count, cudaMemcpyDeviceToHost, s);
    if (cudaStreamSynchronize(s) != cudaSuccess) {
      cudaGetLastError();
      fail_all(fail(HSS_ERR_CUDA, "hss_factor: sync"));
    }
  }
  dfree(status, s);
  for (int q : live) {
    hss_s* h = hs[q];
    if (st[q] == HSS_OK && hst[q] != 0) {
      h->err = "hss_factor: no pivot (zeros or NaN) in a column of the root LU";
      st[q] = HSS_ERR_SINGULAR;
    }
    if (st[q] != HSS_OK) {
      h->ulv.release(s);
      continue;
    }
    h->ulv.done = true;
    h->info.factored = 1;
    h->info.bytes_ulv = (int64_t)h->ulv.bytes;
  }
}

}  // namespace
}  // namespace hss

extern "C" hss_status hss_factor(hss_t h, void* stream) {
  if (!h) return HSS_ERR_INVALID;
  hss_status st = HSS_OK;
  factor_many(1, &h, (cudaStream_t)stream, &st);
  return st;
}

extern "C" hss_status hss_factor_batched(int32_t count, hss_t* hs, void* stream,
                                         hss_status* status) {
  if (count < 0 || (count > 0 && !hs)) return HSS_ERR_INVALID;
  const hss_s* one = nullptr;   // the first handle there is: one launch, one dtype
  for (int32_t q = 0; q < count; ++q) {
    if (!one) one = hs[q];
    if (hs[q] && hs[q]->dtype != one->dtype) {
      set_thread_error("hss_factor_batched: handles of different dtypes");
      return HSS_ERR_INVALID;
    }
  }
  std::vector<hss_status> st(std::max(count, 1), HSS_OK);
  factor_many(count, hs, (cudaStream_t)stream, st.data());
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
