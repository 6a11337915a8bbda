// Orthogonalisation kernels of the subspace iteration (eig_si.cu).
//
// One CholeskyQR pass of an n x m block is two launches:
//
//   k_gram_chol32  one 8-CTA cluster per problem: FP32 Gram matrix of the CTAs'
//                  rows (runs of 16 rows in FP32, added up in two floats), the
//                  partials summed in FP64 through distributed shared memory,
//                  then W by one CTA;
//   k_si_rotate    Out = A W in FP64 (the span of the block is kept to FP64
//                  whatever the accuracy of W).
//
// What bounds them: the factorisation is a chain of m dependent pivots
// (broadcast of a row through shared memory, one barrier, a reciprocal, the
// updates), kept free of FP64 (conversions included: FP32 -> FP64 by an
// instruction on that chain cost 10 us of 31); the rotation is FP64 arithmetic
// (two FMAs per clock and SM), so its tiles are sized to spread n m^2 / 2 FMAs
// over all SMs.  Measured at n = 1024, m = 48, two problems: Gram partials, their
// sum and the factor as three launches took 14.7 + 9.6 + 28 us and take 21.1 us
// as one; the rotation 19.1 us and 9.2 us; an FP64 Gram matrix with its sum
// 50 us and 16 us; the FP64 factor (one rank-1 update and three barriers per
// column before) 115 us and 34 us.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>

#include "eig_orth.cuh"
#include "kernel_attr.cuh"
#include "launch.cuh"
#include "eig_si.cuh"

namespace cg = cooperative_groups;

namespace hotrg {
namespace {

constexpr int kOrthCluster = 8;
constexpr int kSlab = 32;                    // rows staged at a time
constexpr float kChol32Retry = 0x1.0p-12f;   // diagonal shift of a retried FP32 factorisation

__device__ __forceinline__ float reciprocal(float p) { return __frcp_rn(p); }
__device__ __forceinline__ double reciprocal(double p) {     // p within the FP32 range
  double r = (double)__frcp_rn((float)p);
  r = fma(r, fma(-p, r, 1.0), r);
  return fma(r, fma(-p, r, 1.0), r);
}
__device__ __forceinline__ float inv_sqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double inv_sqrt(double x) { return rsqrt_fp64(x); }

// Factor and inverse in one elimination, 256 threads as 16 x 16, thread (ty, tx)
// holding the entries (ty + 16 u, tx + 16 v) in registers: element (i, k) is the
// scaled matrix for k >= i and the growing L^-1 (L = R^T) for k < i, which
// starts at zero.  A step takes two pivots j, j + 1 (m is even): rows j and j + 1
// go through shared memory (two buffers, one barrier per step); every thread
// eliminates row j from its part of row j + 1, and both update every row below.
// A row's part right of the diagonal also holds (the matrix being symmetric) the
// multipliers of the rows below, its L^-1 part is k < j, and 1 at k = j.  At the
// end the L^-1 rows over the square roots of the pivots are the columns of
// W = diag(d) R^-1 = diag(d) L^-T.  Which row values an entry takes depends on
// its tile alone off the diagonal tiles (right of them the matrix part, left of
// them the L^-1 part), so the updates carry no tests.  One pivot per barrier took
// 14 us at m = 48 and 41 at m = 88, two take 10 and 28 us.
//
// Nearly dependent columns break the unshifted factorisation; attempt a adds
// shift(a) to the unit diagonal.  cmat(i, k), i <= k: the unscaled matrix.
template <class T, int U, class Cmat, class Shift>
__device__ void chol_inverse(Cmat cmat, Shift shift, int attempts, int m, double *W, int *flag, T *rowbuf, T *d,
                             T *piv) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  constexpr int LD = 16 * U;
  for (int j = tid; j < LD; j += 256) {
    const T cjj = j < m ? cmat(j, j) : T(0);
    d[j] = (cjj > T(0) && isfinite(cjj)) ? inv_sqrt(cjj) : T(1);
    piv[j] = T(1);
  }
  __syncthreads();
  T e[U][U];
  bool bad = true;
  for (int attempt = 0; attempt < attempts && bad; ++attempt) {
    const T sh = shift(attempt);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int v = 0; v < U; ++v) {
        const int i = ty + 16 * u, k = tx + 16 * v;
        e[u][v] = (i <= k && k < m) ? cmat(i, k) * (d[i] * d[k]) + (i == k ? sh : T(0)) : T(0);
      }
    bad = false;
    for (int j = 0; j < m; j += 2) {
      T *b0 = rowbuf + (j & 2) * LD, *b1 = b0 + LD;
      if (ty == (j & 15) || ty == (j & 15) + 1) {          // j is even: both rows lie in one tile
        const int ju = j >> 4;
        T *buf = ty == (j & 15) ? b0 : b1;
#pragma unroll
        for (int v = 0; v < U; ++v) {
          T x = e[0][v];             // selected, not indexed: e stays in registers
#pragma unroll
          for (int u = 1; u < U; ++u) x = ju == u ? e[u][v] : x;
          buf[tx + 16 * v] = x;
        }
      }
      __syncthreads();
      const T p0 = b0[j], c01 = b0[j + 1];
      const T r0 = reciprocal(p0), l = c01 * r0;           // row j + 1 loses l times row j
      const T p1 = fma(-l, c01, b1[j + 1]);
      if (!(p0 > T(0)) || !isfinite(p0) || !(p1 > T(0)) || !isfinite(p1)) {   // the same for every thread
        bad = true;
        break;
      }
      if (tid == 0) {
        piv[j] = p0;
        piv[j + 1] = p1;
      }
      const T r1 = reciprocal(p1);
      T right0[U], left0[U], diag0[U], right1[U], left1[U], diag1[U];
#pragma unroll
      for (int v = 0; v < U; ++v) {
        const int k = tx + 16 * v;
        const T x0 = b0[k], x1 = b1[k];
        right0[v] = x0;
        left0[v] = k < j ? x0 : k == j ? T(1) : T(0);
        diag0[v] = tx >= ty ? right0[v] : left0[v];
        right1[v] = fma(-l, x0, x1);
        left1[v] = fma(-l, left0[v], k < j ? x1 : k == j + 1 ? T(1) : T(0));
        diag1[v] = tx >= ty ? right1[v] : left1[v];
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (j >= 16 * u + 15) continue;        // every row of the tile is done
        const int i = ty + 16 * u;
        const T x0 = b0[i];
        const T m0 = i > j ? -(x0 * r0) : T(0), m1 = i > j + 1 ? -(fma(-l, x0, b1[i]) * r1) : T(0);
#pragma unroll
        for (int v = 0; v < U; ++v) {
          const T a0 = v > u ? right0[v] : v < u ? left0[v] : diag0[v];
          const T a1 = v > u ? right1[v] : v < u ? left1[v] : diag1[v];
          e[u][v] = fma(m1, a1, fma(m0, a0, e[u][v]));
        }
      }
    }
    __syncthreads();
  }
  if (bad) {
    if (tid == 0) atomicExch(flag, 1);
    return;
  }
  for (int j = tid; j < m; j += 256) piv[j] = inv_sqrt(piv[j]);
  __syncthreads();
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int i = ty + 16 * u, k = tx + 16 * v;
      if (i < m && k < m) {
        const T z = (k < i ? e[u][v] : k == i ? T(1) : T(0)) * piv[i] * d[k];
        if constexpr (sizeof(T) == 4) W[k + (size_t)i * m] = to_f64(z);
        else W[k + (size_t)i * m] = z;
      }
    }
}

// FP32 attempts: as given, then with kChol32Retry, which always succeeds and
// leaves a basis with condition number below about kChol32Retry^-1/2 for the
// next pass to finish
struct Shift32 {
  float s;
  __device__ float operator()(int a) const { return a == 0 ? s : fmaxf(s, kChol32Retry); }
};
// FP64 attempts: as given, then 2^-26 and 2^-12 of the unit diagonal
struct Shift64 {
  double s;
  __device__ double operator()(int a) const { return a == 0 ? s : fmax(s, a == 1 ? 0x1.0p-26 : 0x1.0p-12); }
};

template <int U>
constexpr size_t gram_chol_smem(int m) {
  return ((size_t)m * m) * (sizeof(float2) + sizeof(float)) +
         (size_t)(kSlab * (16 * U + 1) + 6 * 16 * U) * sizeof(float);
}

template <int U>
__global__ void __launch_bounds__(256) __cluster_dims__(kOrthCluster, 1, 1)
    k_gram_chol32(PSet Yin, int n, int m, float shift, PSet Wout, int *flag) {
  pdl_enter();
  extern __shared__ float2 gsh[];
  constexpr int LD = 16 * U;
  float2 *part = gsh;                                              // m x m, upper triangle
  float *tot = reinterpret_cast<float *>(part + (size_t)m * m);    // m x m, upper triangle (rank 0)
  float *slab = tot + (size_t)m * m;                               // kSlab x (LD + 1)
  float *rowbuf = slab + kSlab * (LD + 1);                         // 2 x 2 x LD
  float *d = rowbuf + 4 * LD, *piv = d + LD;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), z = blockIdx.z;
  const double *y = Yin.at(z);
  const int rp = (n + kOrthCluster - 1) / kOrthCluster;
  const int r0 = rank * rp, r1 = min(n, r0 + rp);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  // a run of 16 rows is summed in FP32, the runs in two floats (TwoSum, Knuth)
  float hi[U][U], lo[U][U];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) hi[u][v] = lo[u][v] = 0.0f;
  auto two_sum = [](float &h, float &l, float x) {
    const float s = h + x, bb = s - h;
    l += (h - (s - bb)) + (x - bb);
    h = s;
  };
  constexpr int PER = kSlab * LD / 256;                        // staged elements per thread
  double nxt[PER];
  auto fetch = [&](int rr) {
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int e = tid + 256 * k, ii = e & (kSlab - 1), col = e / kSlab, row = rr + ii;
      nxt[k] = (row < r1 && col < m) ? y[(size_t)col * n + row] : 0.0;
    }
  };
  fetch(r0);
  for (int rr = r0; rr < r1; rr += kSlab) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int e = tid + 256 * k, ii = e & (kSlab - 1), col = e / kSlab;
      slab[ii * (LD + 1) + col] = to_f32(nxt[k]);
    }
    __syncthreads();
    fetch(rr + kSlab);
#pragma unroll 1
    for (int half = 0; half < kSlab; half += 16) {
      float acc[U][U];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = 0; v < U; ++v) acc[u][v] = 0.0f;
#pragma unroll 4
      for (int ii = half; ii < half + 16; ++ii) {
        float av[U], bv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          av[u] = slab[ii * (LD + 1) + ty + 16 * u];
          bv[u] = slab[ii * (LD + 1) + tx + 16 * u];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int v = u; v < U; ++v) acc[u][v] = fmaf(av[u], bv[v], acc[u][v]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int v = u; v < U; ++v) two_sum(hi[u][v], lo[u][v], acc[u][v]);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = u; v < U; ++v) {
      const int a = ty + 16 * u, b = tx + 16 * v;
      if (a <= b && b < m) part[a * m + b] = make_float2(hi[u][v], lo[u][v]);
    }
  cluster.sync();
  // every CTA sums its share of the entries over the cluster, into rank 0
  float *dst = cluster.map_shared_rank(tot, 0);
  for (int e = rank * 256 + tid; e < m * m; e += kOrthCluster * 256) {
    if (e / m > e % m) continue;
    float2 v[kOrthCluster];
#pragma unroll
    for (int q = 0; q < kOrthCluster; ++q) v[q] = *cluster.map_shared_rank(part + e, q);
    float h = v[0].x, l = v[0].y;
#pragma unroll
    for (int q = 1; q < kOrthCluster; ++q) {
      two_sum(h, l, v[q].x);
      l += v[q].y;
    }
    dst[e] = h + l;
  }
  cluster.sync();                    // the partials have been read, the totals written
  if (rank != 0) return;
  chol_inverse<float, U>([&](int i, int k) { return tot[i * m + k]; }, Shift32{shift}, 2, m, Wout.at(z), flag,
                         rowbuf, d, piv);
}

template <int U>
__global__ void __launch_bounds__(256) k_chol32(PSet Cin, int m, float shift, PSet Wout, int *flag) {
  pdl_enter();
  __shared__ float rowbuf[4 * 16 * U], d[16 * U], piv[16 * U];
  const double *C = Cin.at(blockIdx.z);
  chol_inverse<float, U>([&](int i, int k) { return to_f32(C[(size_t)i * m + k]); }, Shift32{shift}, 2, m,
                         Wout.at(blockIdx.z), flag, rowbuf, d, piv);
}

// the same in FP64; only_if (optional): run for problem z only if only_if.at(z)[2]
// != 0, and without a first shift if it is 1
template <int U>
__global__ void __launch_bounds__(256) k_chol64(PSet Cin, int m, double shift, PSet Wout, int *flag, PSet only_if) {
  pdl_enter();
  const double cond = only_if.b0 ? only_if.at(blockIdx.z)[2] : 2.0;
  if (cond == 0.0) return;
  __shared__ double rowbuf[4 * 16 * U], d[16 * U], piv[16 * U];
  const double *C = Cin.at(blockIdx.z);
  chol_inverse<double, U>([&](int i, int k) { return C[(size_t)i * m + k]; }, Shift64{cond == 1.0 ? 0.0 : shift}, 3, m,
                          Wout.at(blockIdx.z), flag, rowbuf, d, piv);
}

// Sums of two FP32 numbers, ~2^-44 of the value: twelve FP32 instructions for a
// multiply-add (Dekker's product by fused multiply-add, Knuth's sum), where the
// FP64 unit takes the time of 64 for one.
struct F2 { float h, l; };
__device__ __forceinline__ F2 f2_norm(float h, float l) {
  const float s = __fadd_rn(h, l);
  return F2{s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  const float p = __fmul_rn(a.h, b.h);
  return F2{p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)))};
}
// c + a b, the low part not yet normalised
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
  const F2 p = f2_mul(a, b);
  const float s = __fadd_rn(c.h, p.h), t = __fsub_rn(s, c.h);
  const float r = __fadd_rn(__fsub_rn(c.h, __fsub_rn(s, t)), __fsub_rn(p.h, t));
  return F2{s, __fadd_rn(c.l, __fadd_rn(p.l, r))};
}
__device__ __forceinline__ F2 f2_neg(F2 a) { return F2{-a.h, -a.l}; }
__device__ __forceinline__ F2 f2_reciprocal(F2 p) {
  const float r = __frcp_rn(p.h);
  return F2{r, __fmul_rn(r, fmaf(-p.l, r, fmaf(-p.h, r, 1.0f)))};
}
__device__ __forceinline__ F2 f2_rsqrt(F2 p) {          // one Newton step y + y (1 - p y^2) / 2
  const float y = rsqrtf(p.h);
  const float q = __fmul_rn(p.h, y), ql = fmaf(p.h, y, -q);
  return F2{y, 0.5f * y * (fmaf(-q, y, 1.0f) - y * fmaf(p.l, y, ql))};
}

// Cholesky factor (see lr_factor), laid out and stepped like chol_inverse without
// the inverse: the rows of R = L^T go to shared memory once each, as they become
// pivots, so a step (two pivots) has one barrier and no buffer is reused.  The
// square roots of the pivots are taken at the end, off the chain of steps.  L only
// has to be one matrix whose columns the caller rotates: what it misses of H is
// seen, and removed, by the FP64 passes after it.  In FP64 the kernel was bound by
// that unit (87 us at m = 60; 29 us in pairs of FP32 numbers); FP32 alone takes
// the caller four more sweeps, which cost as much as FP64.
template <int U>
__global__ void __launch_bounds__(256) k_lr_factor(PSet Hin, int m, PSet Lout, PSet Bout) {
  pdl_enter();
  constexpr int LD = 16 * U;
  extern __shared__ __align__(16) F2 lr_rows[];       // m rows of LD: row j as it was published
  __shared__ F2 rs[LD], ls[LD / 2];                   // pivot, then 1 / sqrt of it; row j + 1's multiple of row j
  __shared__ int s_exp;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const double *H = Hin.at(blockIdx.z);
  double *L = Lout.at(blockIdx.z), *B = Bout.at(blockIdx.z);
  if (tid == 0) s_exp = 0;
  __syncthreads();
  double x[U][U];
  int ex = 0;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = u; v < U; ++v) {
      const int i = ty + 16 * u, k = tx + 16 * v;
      x[u][v] = i <= k && k < m ? H[(size_t)i * m + k] : 0.0;
      ex = max(ex, (__double2hiint(x[u][v]) >> 20) & 0x7FF);
    }
  for (int o = 16; o > 0; o >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
  if ((tid & 31) == 0) atomicMax(&s_exp, ex);
  __syncthreads();
  ex = s_exp;
  // 2^-(exponent); a matrix of zeros, or with entries no scale helps, keeps its own
  const double sc = ex > 0 && ex < 2046 ? __longlong_as_double((long long)(2046 - ex) << 52) : 1.0;
  F2 e[U][U];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = u; v < U; ++v) {
      const double y = fma(x[u][v], sc, ty + 16 * u == tx + 16 * v ? kLrShift : 0.0);
      const float h = to_f32(y);
      e[u][v] = F2{h, to_f32(y - to_f64(h))};
    }
  bool bad = false;
  for (int j = 0; j < m; j += 2) {
    F2 *b0 = lr_rows + (size_t)j * LD, *b1 = b0 + LD;
    if (ty == (j & 15) || ty == (j & 15) + 1) {          // j is even: both rows lie in one tile
      const int ju = j >> 4;
      F2 *buf = ty == (j & 15) ? b0 : b1;
#pragma unroll
      for (int v = 0; v < U; ++v) {
        F2 w = e[0][v];              // selected, not indexed: e stays in registers
#pragma unroll
        for (int u = 1; u <= v; ++u) w = ju == u ? e[u][v] : w;
        buf[tx + 16 * v] = f2_norm(w.h, w.l);
      }
    }
    __syncthreads();
    const F2 p0 = b0[j], c01 = b0[j + 1];
    const F2 r0 = f2_reciprocal(p0), l = f2_neg(f2_mul(c01, r0));
    const F2 q1 = f2_fma(l, c01, b1[j + 1]), p1 = f2_norm(q1.h, q1.l);
    if (!(p0.h > kLrPivot) || !isfinite(p0.h) || !(p1.h > kLrPivot) || !isfinite(p1.h)) {   // the same for every thread
      bad = true;
      break;
    }
    if (tid == 0) {
      rs[j] = p0;
      rs[j + 1] = p1;
      ls[j >> 1] = l;
    }
    const F2 r1 = f2_reciprocal(p1);
    F2 x0[U], x1[U];
#pragma unroll
    for (int v = 0; v < U; ++v) {
      x0[v] = b0[tx + 16 * v];
      const F2 w = f2_fma(l, x0[v], b1[tx + 16 * v]);
      x1[v] = f2_norm(w.h, w.l);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j >= 16 * u + 14) continue;        // every row of the tile is done
      const int i = ty + 16 * u;
      if (i <= j + 1) continue;
      const F2 y0 = b0[i], w = f2_fma(l, y0, b1[i]), y1 = f2_norm(w.h, w.l);
      const F2 m0 = f2_neg(f2_mul(y0, r0)), m1 = f2_neg(f2_mul(y1, r1));
#pragma unroll
      for (int v = u; v < U; ++v) e[u][v] = f2_fma(m1, x1[v], f2_fma(m0, x0[v], e[u][v]));
    }
  }
  __syncthreads();
  if (bad) {
    for (int q = tid; q < m * m; q += 256) {
      const int i = q % m, k = q / m;
      L[q] = i == k ? 1.0 : 0.0;
      B[q] = 0.5 * (H[q] + H[(size_t)i * m + k]);
    }
    return;
  }
  if (tid < m) rs[tid] = f2_rsqrt(rs[tid]);
  __syncthreads();
  for (int q = tid; q < m * m; q += 256) {
    const int i = q % m, k = q / m;          // L(i, k) = R(k, i)
    double v = 0.0;
    if (i >= k) {
      F2 w = lr_rows[(size_t)k * LD + i];
      if (k & 1) w = f2_fma(ls[k >> 1], lr_rows[(size_t)(k - 1) * LD + i], w);
      w = f2_mul(f2_norm(w.h, w.l), rs[k]);
      v = to_f64(w.h) + to_f64(w.l);
    }
    L[q] = v;
    B[q] = v;
  }
}

// Cp[c] = A[rows of chunk c]^T B[same rows] in FP64 (m x m, row-major; the second
// product's chunks follow the first's), 256 threads as 16 x 16 with entries
// (ty + 16 u, tx + 16 v): every thread works whatever m is.  Of a symmetric
// product, entries u <= v only (all of the upper triangle).
template <int U>
__global__ void __launch_bounds__(256) k_si_gram(PSet A, PSet B0, PSet B1, PSet Cp, int n, int m, int P, int rows) {
  pdl_enter();
  constexpr int LD = 16 * U;
  __shared__ double As[16][LD + 1];
  __shared__ double Bs[16][LD + 1];
  // problem z's products A^T B0 and, from blockIdx.z = P on, A^T B1; one with
  // B == A is symmetric
  const bool second = (int)blockIdx.z >= P;
  const int z = second ? (int)blockIdx.z - P : (int)blockIdx.z, c = blockIdx.x;
  const double *a = A.at(z);
  const double *b = (second ? B1 : B0).at(z);
  const bool sym = a == b;
  const int r0 = c * rows, r1 = min(n, r0 + rows);
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  double acc[U][U];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) acc[u][v] = 0.0;
  for (int rr = r0; rr < r1; rr += 16) {
    for (int e = threadIdx.x; e < 16 * LD; e += 256) {
      const int j = e >> 4, ii = e & 15;
      const int row = rr + ii;
      const bool in = row < r1 && j < m;
      As[ii][j] = in ? a[(size_t)j * n + row] : 0.0;
      if (!sym) Bs[ii][j] = in ? b[(size_t)j * n + row] : 0.0;
    }
    __syncthreads();
    // a test of sym at every FMA would cost as much as the FMAs it saves
    if (sym) {
#pragma unroll 2
      for (int ii = 0; ii < 16; ++ii) {
        double av[U], bv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          av[u] = As[ii][ty + 16 * u];
          bv[u] = As[ii][tx + 16 * u];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int v = u; v < U; ++v) acc[u][v] = fma(av[u], bv[v], acc[u][v]);
      }
    } else {
#pragma unroll 2
      for (int ii = 0; ii < 16; ++ii) {
        double av[U], bv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          av[u] = As[ii][ty + 16 * u];
          bv[u] = Bs[ii][tx + 16 * u];
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int v = 0; v < U; ++v) acc[u][v] = fma(av[u], bv[v], acc[u][v]);
      }
    }
    __syncthreads();
  }
  double *out = Cp.at(z) + (size_t)(second ? gridDim.x + c : c) * m * m;
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int v = 0; v < U; ++v) {
      const int ia = ty + 16 * u, ib = tx + 16 * v;
      if (ia < m && ib < m && (!sym || ia <= ib)) out[ia * m + ib] = acc[u][v];
    }
}

// C = sum over the chunks (fixed order), symmetrised.  A block takes 64 entries,
// four threads to an entry, each with its own run of chunks: the sum is bound
// by load latency, so many loads are kept in flight.
// blockIdx.z as in k_si_gram; sym0, sym1: whether the products are symmetric.
__global__ void __launch_bounds__(256) k_si_gram_reduce(PSet Cp, PSet C0, PSet C1, int nchunks, int m, int P, int sym0,
                                                        int sym1) {
  pdl_enter();
  __shared__ double sum[4][64];
  const bool second = (int)blockIdx.z >= P;
  const int z = second ? (int)blockIdx.z - P : (int)blockIdx.z, l = threadIdx.x & 63, g = threadIdx.x >> 6;
  const bool sym = second ? sym1 : sym0;
  const PSet &C = second ? C1 : C0;
  const long long mm = (long long)m * m;
  const int e = blockIdx.x * 64 + l, a = e / m, b = e % m;
  const bool in = e < m * m && a <= b;
  const int per = (nchunks + 3) / 4, c0 = g * per, c1 = min(nchunks, c0 + per);
  double s = 0.0;
  if (in) {
    const double *src = Cp.at(z) + (second ? nchunks * mm : 0);
    const long long o = (long long)a * m + b, ot = (long long)b * m + a;
    double v[4] = {0.0, 0.0, 0.0, 0.0}, w[4] = {0.0, 0.0, 0.0, 0.0};
    int c = c0;
    for (; c + 4 <= c1; c += 4) {
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] += src[(c + q) * mm + o];
      if (!sym)
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] += src[(c + q) * mm + ot];
    }
    for (; c < c1; ++c) {
      v[0] += src[c * mm + o];
      if (!sym) w[0] += src[c * mm + ot];
    }
    s = (v[0] + v[1]) + (v[2] + v[3]);
    if (!sym) s = 0.5 * (s + ((w[0] + w[1]) + (w[2] + w[3])));
  }
  sum[g][l] = s;
  __syncthreads();
  if (g == 0 && in) {
    s = (sum[0][l] + sum[1][l]) + (sum[2][l] + sum[3][l]);
    C.at(z)[a * m + b] = s;
    C.at(z)[b * m + a] = s;
  }
}

// Out = A W: a CTA takes RT rows and all columns; a warp takes 32 / RT
// neighbouring columns at a time (lanes run along the rows), so that for a
// triangular W its sum stops at their last nonzero, and the warps take the
// column groups forwards and backwards in turn (equal shares).  FP64-bound:
// RT is chosen so that the CTAs fill the SMs.
template <int RT>
__global__ void __launch_bounds__(256) k_si_rotate(PSet A0, PSet A1, PSet W, PSet Out0, PSet Out1, int n, int m, int P,
                                                   int tri) {
  pdl_enter();
  extern __shared__ double rsh[];
  double *As = rsh;                       // [column][RT]
  double *Ws = rsh + (size_t)m * RT;      // [column][m + 1]
  constexpr int CPW = 32 / RT;
  const bool second = (int)blockIdx.z >= P;      // A0 W, and from blockIdx.z = P on A1 W
  const int z = second ? (int)blockIdx.z - P : (int)blockIdx.z, i0 = blockIdx.x * RT;
  const double *a = (second ? A1 : A0).at(z), *w = W.at(z);
  double *out = (second ? Out1 : Out0).at(z);
  for (int e = threadIdx.x; e < m * RT; e += 256) {
    const int j = e / RT, r = e % RT;
    As[e] = i0 + r < n ? a[(size_t)j * n + i0 + r] : 0.0;
  }
  for (int e = threadIdx.x; e < m * m; e += 256) {
    const int c = e / m, j = e % m;
    if (!tri || j <= c) Ws[c * (m + 1) + j] = w[e];
    else Ws[c * (m + 1) + j] = 0.0;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = lane % RT, cl = lane / RT;
  const int ng = (m + CPW - 1) / CPW;
  for (int k = 0; k * 8 < ng; ++k) {
    const int g = k * 8 + ((k & 1) ? 7 - warp : warp);
    if (g >= ng) continue;
    const int c = min(g * CPW + cl, m - 1);
    const int jend = tri ? min(m, g * CPW + CPW) : m;
    double acc = 0.0;
#pragma unroll 8
    for (int j = 0; j < jend; ++j) acc = fma(As[j * RT + r], Ws[c * (m + 1) + j], acc);
    if (g * CPW + cl < m && i0 + r < n) out[(size_t)c * n + i0 + r] = acc;
  }
}

int tile_of(int m) { return m <= 32 ? 2 : (m + 15) / 16; }   // 16-wide tiles per dimension, 2..6

template <int U>
cudaError_t launch_gram_chol(PSet Y, int n, int m, float shift, PSet W, int *flag, int P, cudaStream_t s) {
  static SmemLimit limit;
  if (cudaError_t e = limit.raise(reinterpret_cast<const void *>(k_gram_chol32<U>), (int)gram_chol_smem<U>(16 * U)))
    return e;
  launch_pdl(k_gram_chol32<U>, dim3(kOrthCluster, 1, P), 256, gram_chol_smem<U>(m), s, Y, n, m, shift, W, flag);
  return cudaGetLastError();
}

template <int RT>
cudaError_t launch_rotate(PSet A0, PSet A1, PSet W, PSet Out0, PSet Out1, int count, int n, int m, bool tri, int P,
                          cudaStream_t s) {
  static SmemLimit limit;
  if (cudaError_t e = limit.raise(reinterpret_cast<const void *>(k_si_rotate<RT>),
                                  (int)(sizeof(double) * kSiMaxBlock * (RT + kSiMaxBlock + 1))))
    return e;
  // a plain launch: started early, its blocks would be dealt out while the factor's
  // cluster still holds SMs, and the others would get two (D = 48 job: 57.6 ms
  // started early, 55.5 ms like this)
  k_si_rotate<RT><<<dim3((n + RT - 1) / RT, 1, count * P), 256, sizeof(double) * m * (RT + m + 1), s>>>(
      A0, A1, W, Out0, Out1, n, m, P, tri ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace

cudaError_t gram_reduce(PSet part, PSet out, int chunks, int m, int P, cudaStream_t s, long long *launches) {
  launch_pdl(k_si_gram_reduce, dim3((m * m + 63) / 64, 1, P), 256, 0, s, part, out, out, chunks, m, P, 0, 0);
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t gram64(PSet A, PSet B0, PSet out0, const PSet *B1, const PSet *out1, int n, int m, PSet part, int P,
                   cudaStream_t s, long long *launches) {
  // chunks of 16 rows until two CTAs per SM have one; longer ones beyond that
  // keep the partials (m x m doubles per chunk) few
  const int count = B1 && 2 * P <= 65535 ? 2 : 1;
  const int want = std::max(1, std::min(kGramChunks / count, (304 + P * count - 1) / (P * count)));
  const int rows = std::max(16, ((n + want - 1) / want + 15) / 16 * 16);
  const int chunks = (n + rows - 1) / rows;
  if (chunks * count > kGramChunks || m > kSiMaxBlock) return cudaErrorInvalidValue;
  const PSet b1 = count == 2 ? *B1 : B0, o1 = count == 2 ? *out1 : out0;
  const dim3 g(chunks, 1, count * P);
  switch (tile_of(m)) {
    case 2: launch_pdl(k_si_gram<2>, g, 256, 0, s, A, B0, b1, part, n, m, P, rows); break;
    case 3: launch_pdl(k_si_gram<3>, g, 256, 0, s, A, B0, b1, part, n, m, P, rows); break;
    case 4: launch_pdl(k_si_gram<4>, g, 256, 0, s, A, B0, b1, part, n, m, P, rows); break;
    case 5: launch_pdl(k_si_gram<5>, g, 256, 0, s, A, B0, b1, part, n, m, P, rows); break;
    default: launch_pdl(k_si_gram<6>, g, 256, 0, s, A, B0, b1, part, n, m, P, rows); break;
  }
  auto same = [](const PSet &x, const PSet &y) { return x.b0 == y.b0 && x.b1 == y.b1 && x.stride == y.stride; };
  launch_pdl(k_si_gram_reduce, dim3((m * m + 63) / 64, 1, count * P), 256, 0, s, part, out0, o1, chunks, m, P,
             same(A, B0) ? 1 : 0, same(A, b1) ? 1 : 0);
  *launches += 2;
  cudaError_t e = cudaGetLastError();
  if (e || !B1 || count == 2) return e;
  return gram64(A, *B1, *out1, nullptr, nullptr, n, m, part, P, s, launches);
}

cudaError_t cholqr32_factor(PSet Y, int n, int m, float shift, PSet W, int *flag, int P, cudaStream_t s,
                            long long *launches) {
  *launches += 1;
  switch (tile_of(m)) {
    case 2: return launch_gram_chol<2>(Y, n, m, shift, W, flag, P, s);
    case 3: return launch_gram_chol<3>(Y, n, m, shift, W, flag, P, s);
    case 4: return launch_gram_chol<4>(Y, n, m, shift, W, flag, P, s);
    case 5: return launch_gram_chol<5>(Y, n, m, shift, W, flag, P, s);
    case 6: return launch_gram_chol<6>(Y, n, m, shift, W, flag, P, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t chol32(PSet C, int m, float shift, PSet W, int *flag, int P, cudaStream_t s, long long *launches) {
  const dim3 g(1, 1, P);
  switch (tile_of(m)) {
    case 2: launch_pdl(k_chol32<2>, g, 256, 0, s, C, m, shift, W, flag); break;
    case 3: launch_pdl(k_chol32<3>, g, 256, 0, s, C, m, shift, W, flag); break;
    case 4: launch_pdl(k_chol32<4>, g, 256, 0, s, C, m, shift, W, flag); break;
    case 5: launch_pdl(k_chol32<5>, g, 256, 0, s, C, m, shift, W, flag); break;
    case 6: launch_pdl(k_chol32<6>, g, 256, 0, s, C, m, shift, W, flag); break;
    default: return cudaErrorInvalidValue;
  }
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t chol64(PSet C, int m, double shift, PSet W, int *flag, PSet only_if, int P, cudaStream_t s,
                   long long *launches) {
  const dim3 g(1, 1, P);
  switch (tile_of(m)) {
    case 2: launch_pdl(k_chol64<2>, g, 256, 0, s, C, m, shift, W, flag, only_if); break;
    case 3: launch_pdl(k_chol64<3>, g, 256, 0, s, C, m, shift, W, flag, only_if); break;
    case 4: launch_pdl(k_chol64<4>, g, 256, 0, s, C, m, shift, W, flag, only_if); break;
    case 5: launch_pdl(k_chol64<5>, g, 256, 0, s, C, m, shift, W, flag, only_if); break;
    case 6: launch_pdl(k_chol64<6>, g, 256, 0, s, C, m, shift, W, flag, only_if); break;
    default: return cudaErrorInvalidValue;
  }
  *launches += 1;
  return cudaGetLastError();
}

template <int U>
static cudaError_t launch_lr(PSet H, int m, PSet L, PSet B, int P, cudaStream_t s) {
  constexpr size_t smem = (size_t)(16 * U) * (16 * U) * sizeof(F2);
  static SmemLimit limit;
  if (cudaError_t e = limit.raise(reinterpret_cast<const void *>(k_lr_factor<U>), (int)smem)) return e;
  launch_pdl(k_lr_factor<U>, dim3(1, 1, P), 256, smem, s, H, m, L, B);
  return cudaGetLastError();
}

cudaError_t lr_factor(PSet H, int m, PSet L, PSet B, int P, cudaStream_t s, long long *launches) {
  *launches += 1;
  switch (tile_of(m)) {
    case 2: return launch_lr<2>(H, m, L, B, P, s);
    case 3: return launch_lr<3>(H, m, L, B, P, s);
    case 4: return launch_lr<4>(H, m, L, B, P, s);
    case 5: return launch_lr<5>(H, m, L, B, P, s);
    case 6: return launch_lr<6>(H, m, L, B, P, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t rotate_basis(PSet A0, PSet Out0, const PSet *A1, const PSet *Out1, PSet W, int n, int m, bool tri, int P,
                         cudaStream_t s, long long *launches) {
  if (m > kSiMaxBlock) return cudaErrorInvalidValue;
  const int count = A1 && 2 * P <= 65535 ? 2 : 1;
  const PSet a1 = count == 2 ? *A1 : A0, o1 = count == 2 ? *Out1 : Out0;
  *launches += 1;
  // the tallest tile that still gives most of the 152 SMs a CTA (each CTA reads
  // all of W)
  const long long rows = (long long)n * P * count;
  const cudaError_t e = rows >= 16 * 120  ? launch_rotate<16>(A0, a1, W, Out0, o1, count, n, m, tri, P, s)
                        : rows >= 8 * 120 ? launch_rotate<8>(A0, a1, W, Out0, o1, count, n, m, tri, P, s)
                                          : launch_rotate<4>(A0, a1, W, Out0, o1, count, n, m, tri, P, s);
  if (e || !A1 || count == 2) return e;
  return rotate_basis(*A1, *Out1, nullptr, nullptr, W, n, m, tri, P, s, launches);
}

}  // namespace hotrg
