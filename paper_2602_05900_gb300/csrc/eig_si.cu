// Batched FP64 subspace-iteration eigensolver for the environments (see
// eig_si.cuh).  GB300's FP64 rate is a few flops per clock per SM, so the
// work is arranged for the whole GPU: the products with G, the Gram matrices
// and the basis rotations are tall-skinny FP64 GEMMs spread over all SMs (the
// two environments of a step run in the same launches), and only the small
// m x m factorisations run on one CTA per problem.
//
// The iteration runs on G + sigma I with sigma = 2^-40 Tr G (same
// eigenvectors; the Ritz values are shifted back at the end).  The shift keeps
// the columns of G X that belong to the numerical null space of G at least
// sigma long and along their own direction when the products are nearly
// exact (HOTRG fixed points far from criticality have numerically rank
// deficient G).  Where columns still become nearly dependent (G from
// reduced-precision contractions is indefinite at their rounding level, and a
// Ritz value can sit at zero), the FP32 CholeskyQR pass restarts with a shift
// instead of breaking down.
//
// One iteration:  Y = G X  ->  X = orth(Y): CholeskyQR with FP32 Cholesky
// factors and FP64 rotations -- two passes while the block may be ill
// conditioned (or shifted CholeskyQR3 in FP64 for large batches), one pass once
// its columns are close to eigenvectors, two FP64 passes where the block holds
// numerically null directions.  A Rayleigh-Ritz step works with C0 = X^T X:
// W = C0^(-1/2) (Newton-Schulz on the m x m side, or a shifted FP64 Cholesky
// where C0 is far from I), H = W^T (X^T Y) W, H diagonalised by the parallel
// two-sided Jacobi method (FP32, then an FP64 finish), and X, Y rotated onto
// the Ritz vectors.  The iteration stops when ||G x_i - theta_i x_i|| <= tol *
// theta_0 for i < k (or at the accuracy floor of G); the next check is
// scheduled from the observed Ritz-value ratio theta_m / theta_k.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <vector>

#include "eig_orth.cuh"
#include "launch.cuh"
#include "eig_si.cuh"
#include "eig_small.cuh"
#include "tc_exact.cuh"

namespace hotrg {
namespace {

constexpr int kSplitMax = 8;     // split-K partials of G X
// FP64 FMAs of one n x m x m product batch from which its rotations and Gram
// matrices run as exact-slice products: few problems are latency bound and stay
// with the single FP64 launches longer (24-instance TF32 sweep: 150.4 ms with 2^25
// for all, 142.4 ms like this; with 2^22 for all the one pair of a D = 32 run, 2^22.2,
// took 65 ms against 50).  The lower line is for environments of reduced precision
// only, whose isometries are rounded to 2^-24 or coarser before they are used: the
// slices leave U^T U within 4e-13 of I, the FP64 launches within 2e-15 (five D = 32
// instances in TF32: 3.3e-13 and 1.4e-15; ln Z of 192 TF32 instances against the FP64
// mode: geometric mean 6.06e-5 and maximum 3.22e-4 either way).
constexpr double kXsSmallWork = 0x1p25, kXsBatchWork = 0x1p23;
constexpr int kSiSmallBatch = 8;      // problems up to which the solve is latency bound
constexpr double kSiFloorTol = 1e-10;  // residuals accepted once they stop decreasing
constexpr int kSiSlowIters = 24;       // iterations after which a residual below the floor is accepted


// splitmix64 finaliser (Steele, Lea, Flood 2014) -> uniform double in [-1, 1)
__device__ inline double hash_uniform(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  x ^= x >> 31;
  return static_cast<double>(x >> 11) * 0x1.0p-52 - 1.0;
}

__global__ void k_si_init(PSet X, PSet warm, int has_warm, int kw, int n, int m) {
  pdl_enter();
  const int z = blockIdx.z;
  const long long total = (long long)n * m;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(e / n);
    double v;
    if (has_warm && j < kw) v = warm.at(z)[e];
    else v = hash_uniform(((unsigned long long)z << 56) ^ ((unsigned long long)j << 32) ^ (unsigned long long)(e % n));
    X.at(z)[e] = v;
  }
}

// Out_s = G[rows i0.., cols in split s] . X[those rows, :]  (X, Out column-major n x m)
__global__ void __launch_bounds__(256) k_si_gemm(PSet G, PSet X, PSet Out, int n, int m, int chunk) {
  pdl_enter();
  __shared__ double Gs[16][65];
  __shared__ double Xs[16][kSiMaxBlock];
  const int z = blockIdx.z;
  const double *g = G.at(z);
  const double *x = X.at(z);
  double *out = Out.at(z) + (size_t)blockIdx.y * n * m;
  const int i0 = blockIdx.x * 64;
  const int k0 = blockIdx.y * chunk;
  const int k1 = min(n, k0 + chunk);
  const int t = threadIdx.x, r = t & 63, cg = t >> 6;
  double acc[kSiMaxBlock / 4];
#pragma unroll
  for (int c = 0; c < kSiMaxBlock / 4; ++c) acc[c] = 0.0;
  for (int kk = k0; kk < k1; kk += 16) {
    for (int e = t; e < 64 * 16; e += 256) {
      const int row = e >> 4, col = e & 15;
      const int gi = i0 + row, gk = kk + col;
      Gs[col][row] = (gi < n && gk < k1) ? g[(size_t)gi * n + gk] : 0.0;
    }
    for (int e = t; e < 16 * m; e += 256) {
      const int j = e >> 4, col = e & 15;
      const int gk = kk + col;
      Xs[col][j] = (gk < k1) ? x[(size_t)j * n + gk] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int l = 0; l < 16; ++l) {
      const double gv = Gs[l][r];
#pragma unroll
      for (int c = 0; c < kSiMaxBlock / 4; ++c) {
        const int j = cg + 4 * c;
        if (j < m) acc[c] = fma(gv, Xs[l][j], acc[c]);
      }
    }
    __syncthreads();
  }
  const int i = i0 + r;
  if (i < n) {
#pragma unroll
    for (int c = 0; c < kSiMaxBlock / 4; ++c) {
      const int j = cg + 4 * c;
      if (j < m) out[(size_t)j * n + i] = acc[c];
    }
  }
}

// Shift of the iteration (see si_solve): sig[0] is the shift of the current
// Y = (G + sig[0] I) X, sig[1] the shift of the next product (equal to it in
// this solver; kept apart so that a shift change can never mix the two).
__global__ void k_si_sigma_init(PSet sig, PSet trace, double factor) {
  pdl_enter();
  const int z = blockIdx.z;
  if (threadIdx.x == 0) {
    const double t = trace.at(z)[0];
    const double v = (t > 0.0 && isfinite(t)) ? factor * t : 0.0;
    sig.at(z)[0] = v;
    sig.at(z)[1] = v;
  }
}

// Y += sig[1] X; block (0, 0, z) records sig[0] = sig[1] (the shift now in Y)
__global__ void k_si_shift_add(PSet Y, PSet X, PSet sig, long long nm) {
  pdl_enter();
  const int z = blockIdx.z;
  const double sg = sig.at(z)[1];
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nm;
       e += (long long)gridDim.x * blockDim.x)
    Y.at(z)[e] = fma(sg, X.at(z)[e], Y.at(z)[e]);
  if (blockIdx.x == 0 && threadIdx.x == 0) sig.at(z)[0] = sg;
}

// theta_z[i] -= sig[0] for i < m (the shift of the last Rayleigh-Ritz step)
__global__ void k_si_unshift(PSet theta, PSet sig, int m) {
  pdl_enter();
  const int z = blockIdx.z;
  const double sg = sig.at(z)[0];
  for (int i = threadIdx.x; i < m; i += blockDim.x) theta.at(z)[i] -= sg;
}

// ks[j] = power of two within a factor 2 of 1 / sqrt(C_jj) (1 if C_jj is not
// positive and finite): the column scales of a CholeskyQR basis change
__global__ void k_si_colscale(PSet C, PSet ks, int m) {
  pdl_enter();
  const int z = blockIdx.z;
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    const double c = C.at(z)[(size_t)j * m + j];
    int e = 0;
    if (c > 0.0 && isfinite(c)) (void)frexp(c, &e);
    ks.at(z)[j] = ldexp(1.0, -(e / 2));
  }
}

// out = sum of the S K-parts; with shift, + sig[1] X as well (the iteration's
// shift, the same fma as k_si_shift_add) and sig[0] = sig[1]
__global__ void k_si_sum_split(PSet part, PSet out, int S, long long nm, PSet X, PSet sig, int shift) {
  pdl_enter();
  const int z = blockIdx.z;
  const double sg = shift ? sig.at(z)[1] : 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nm;
       e += (long long)gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int s = 0; s < S; ++s) v += part.at(z)[s * nm + e];
    if (shift) v = fma(sg, X.at(z)[e], v);
    out.at(z)[e] = v;
  }
  if (shift && blockIdx.x == 0 && threadIdx.x == 0) sig.at(z)[0] = sg;
}

// Start of W = C^-1/2: W1 = (3 I - C) / 2, and how far C is from I (largest entry
// of C - I): flags[2] = 0 up to kNearChol (Newton-Schulz converges to rounding in
// two steps: the norm of C - I is at most 96 times that, 3/8 of its square the error
// of W1, and a step squares it again), 1 up to 1/4, else 2; flags[3] = 1 where
// one step is enough.
constexpr float kNearChol = 1e-4f, kNearOne = 3e-6f;

__global__ void __launch_bounds__(1024) k_rr_start(PSet Cin, int m, PSet W, PSet flags) {
  pdl_enter();
  const int z = blockIdx.z;
  const double *C = Cin.at(z);
  float far = 0.0f;
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
    const double one = (e % m == e / m) ? 1.0 : 0.0, c = C[e];
    W.at(z)[e] = fma(-0.5, c, 1.5 * one);
    const float d = fabsf(to_f32(c - one));
    far = fmaxf(far, d == d ? d : INFINITY);
  }
  for (int o = 16; o > 0; o >>= 1) far = fmaxf(far, __shfl_xor_sync(0xffffffffu, far, o));
  __shared__ float part[32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = far;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) far = fmaxf(far, part[i]);
    flags.at(z)[2] = far > 0.25f ? 2.0 : far > kNearChol ? 1.0 : 0.0;
    flags.at(z)[3] = far <= kNearOne ? 1.0 : 0.0;
  }
}

// Out = op(A) (bs B + bd I) for m x m column-major FP64 matrices of every
// problem z (op(A) = A^T if ta).  One CTA per 8 x 8 output tile; the sum over
// k is split four ways across the CTA's threads and combined in a fixed order.
// unless (optional): nothing is done for problem z where unless.at(z)[3] != 0;
// copy (optional): receives the result too.
__global__ void __launch_bounds__(256) k_rr_mm(PSet A, int ta, PSet B, double bs, double bd,
                                               PSet Out, int m, PSet unless, PSet copy) {
  pdl_enter();
  if (unless.b0 && unless.at(blockIdx.z)[3] != 0.0) return;
  __shared__ double As[8][kSiMaxBlock + 1];   // op(A) rows i0..i0+7, all k
  __shared__ double Bs[8][kSiMaxBlock + 1];   // B columns j0..j0+7, all k
  __shared__ double part[4][8][9];
  const int z = blockIdx.z;
  const int i0 = blockIdx.x * 8, j0 = blockIdx.y * 8;
  const double *a = A.at(z), *b = B.at(z);
  for (int e = threadIdx.x; e < 8 * m; e += blockDim.x) {
    const int r = e / m, k = e % m;
    const int i = i0 + r, j = j0 + r;
    // op(A)(i, k): A[i + k m] or (transposed) A[k + i m]
    As[r][k] = (i < m) ? (ta ? a[(size_t)i * m + k] : a[(size_t)k * m + i]) : 0.0;
    Bs[r][k] = (j < m) ? bs * b[(size_t)j * m + k] + (k == j ? bd : 0.0) : 0.0;
  }
  __syncthreads();
  const int ti = threadIdx.x & 7, tj = (threadIdx.x >> 3) & 7, ks = threadIdx.x >> 6;
  double acc = 0.0;
  for (int k = ks; k < m; k += 4) acc = fma(As[ti][k], Bs[tj][k], acc);
  part[ks][ti][tj] = acc;
  __syncthreads();
  if (threadIdx.x < 64) {
    const int i = i0 + ti, j = j0 + tj;
    if (i < m && j < m) {
      const double v = (part[0][ti][tj] + part[1][ti][tj]) + (part[2][ti][tj] + part[3][ti][tj]);
      Out.at(z)[(size_t)j * m + i] = v;
      if (copy.b0) copy.at(z)[(size_t)j * m + i] = v;
    }
  }
}

// Out = (A^T B + B^T A) / 2, symmetric to the last bit, with the tiles and sums of
// k_rr_mm: the mean of the two triangles of H = W^T (X^T Y W).  Where W is large (a
// block that holds numerically null directions) the triangles differ by far more
// than small_eig resolves; given as they are they took its last stage 200 to 280
// rounds (5 at most now), and one of them for both costs the iteration more steps
// than their mean (Ising beta = 8, D = 13 to 24, BF16X3: 186 and 117 in twelve steps).
__global__ void __launch_bounds__(256) k_rr_sym(PSet A, PSet B, PSet Out, int m) {
  pdl_enter();
  if (blockIdx.x > blockIdx.y) return;
  __shared__ double As[2][8][kSiMaxBlock + 1], Bs[2][8][kSiMaxBlock + 1];   // columns of tile I, of tile J
  __shared__ double part[2][4][8][9];
  const int z = blockIdx.z, i0 = blockIdx.x * 8, j0 = blockIdx.y * 8;
  const double *a = A.at(z), *b = B.at(z);
  for (int e = threadIdx.x; e < 8 * m; e += blockDim.x) {
    const int r = e / m, k = e % m;
    const int i = i0 + r, j = j0 + r;
    As[0][r][k] = i < m ? a[(size_t)i * m + k] : 0.0;
    As[1][r][k] = j < m ? a[(size_t)j * m + k] : 0.0;
    Bs[0][r][k] = i < m ? b[(size_t)i * m + k] : 0.0;
    Bs[1][r][k] = j < m ? b[(size_t)j * m + k] : 0.0;
  }
  __syncthreads();
  const int ti = threadIdx.x & 7, tj = (threadIdx.x >> 3) & 7, ks = threadIdx.x >> 6;
  double ab = 0.0, ba = 0.0;
  for (int k = ks; k < m; k += 4) {
    ab = fma(As[0][ti][k], Bs[1][tj][k], ab);
    ba = fma(Bs[0][ti][k], As[1][tj][k], ba);
  }
  part[0][ks][ti][tj] = ab;
  part[1][ks][ti][tj] = ba;
  __syncthreads();
  if (threadIdx.x < 64) {
    const int i = i0 + ti, j = j0 + tj;
    if (i < m && j < m) {
      double v[2];
      for (int q = 0; q < 2; ++q) v[q] = (part[q][0][ti][tj] + part[q][1][ti][tj]) + (part[q][2][ti][tj] + part[q][3][ti][tj]);
      const double h = 0.5 * (v[0] + v[1]);
      Out.at(z)[(size_t)j * m + i] = h;
      if (i0 != j0) Out.at(z)[(size_t)i * m + j] = h;
    }
  }
}

// res[i] = ||Y_i - theta_i X_i|| / |theta_0|, i < k
// res_i = ||y_i - theta_i x_i|| / theta_0, or 0 for a pair whose unshifted
// value lies below half the shift (2^-41 Tr G: inside the band where G's own
// rounding makes the eigenpairs arbitrary; any orthonormal completion there
// is as good as another)
__global__ void k_si_residual(PSet X, PSet Y, PSet theta, PSet res, PSet sig, int use_sig, int n,
                              int k) {
  pdl_enter();
  const int z = blockIdx.z, i = blockIdx.x;
  const double th = theta.at(z)[i];
  if (use_sig && th - sig.at(z)[0] <= 0.5 * sig.at(z)[1] && i > 0) {
    if (threadIdx.x == 0) res.at(z)[i] = 0.0;
    return;
  }
  const double *x = X.at(z) + (size_t)i * n;
  const double *y = Y.at(z) + (size_t)i * n;
  double v = 0.0;
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    const double d = y[r] - th * x[r];
    v = fma(d, d, v);
  }
  __shared__ double part[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += part[w];
    res.at(z)[i] = sqrt(s) / fabs(theta.at(z)[0]);
  }
}

// G (n x n) into an m x m zero-padded square (m = n or n + 1) for the direct Jacobi path.
__global__ void k_si_copy_square(PSet G, PSet out, int n, int m) {
  pdl_enter();
  const int z = blockIdx.z;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * m; e += gridDim.x * blockDim.x) {
    const int a = e / m, b = e % m;
    out.at(z)[e] = (a < n && b < n) ? G.at(z)[a * n + b] : 0.0;
  }
}

// Copy of problem z's n x m block from src to dst (final placement of Ritz vectors).
__global__ void k_si_copy(PSet src, PSet dst, long long nm) {
  pdl_enter();
  const int z = blockIdx.z;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nm;
       e += (long long)gridDim.x * blockDim.x)
    dst.at(z)[e] = src.at(z)[e];
}

// ---- host helpers ----

struct Layout {
  int S, m;
  long long nm, mm;
  long long per;   // doubles per problem
  // slot offsets (doubles) inside a problem's workspace
  long long oY, oZ, oX, oYp, oCp, oC, oW, oRes, oTh, oSig;
  // exact-slice operands (BF16 slices and row scales): G, and two general
  // slots for the n x m / m x n / m x m operands of the other products
  int xsp;
  long long oGs, oGsc, oSa, oSasc, oSb, oSbsc, oKs;
};

Layout layout(int P, int n, int m) {
  Layout L;
  L.nm = (long long)n * m;
  L.mm = (long long)m * m;
  L.m = m;
  const int tiles = (n + 63) / 64;
  L.S = std::max(1, std::min(kSplitMax, (2 * 152 + tiles * P - 1) / std::max(1, tiles * P)));
  while (L.S > 1 && (n + L.S - 1) / L.S < 64) --L.S;
  auto up = [](long long v) { return (v + 31) / 32 * 32; };   // 256-byte aligned slots
  long long o = 0;
  L.oY = o; o += up(L.nm);
  L.oZ = o; o += up(L.nm);
  L.oX = o; o += up(L.nm);
  L.oYp = o; o += up(kSplitMax * L.nm);
  L.oCp = o; o += up(kGramChunks * L.mm);
  L.oC = o; o += up(L.mm);
  L.oW = o; o += up(L.mm);
  L.oRes = o; o += up(m);
  L.oTh = o; o += up(m);
  L.oSig = o; o += up(2);
  L.xsp = xs_pitch(n);
  const long long sa = std::max(xs_elems(n, m, kSiSlices), xs_elems(m, n, kSiSlices));
  const long long sb = std::max(xs_elems(m, n, kSiSlices), xs_elems(m, m, kSiSlices));
  L.oGs = o; o += up((xs_elems(n, n, kSiSlices) + 3) / 4);
  L.oGsc = o; o += up(n);
  L.oSa = o; o += up((sa + 3) / 4);
  L.oSasc = o; o += up(std::max(n, m));
  L.oSb = o; o += up((sb + 3) / 4);
  L.oSbsc = o; o += up(std::max(n, m));
  L.oKs = o; o += up(m);
  L.per = o;
  return L;
}

struct Bufs {
  PSet Y, Z, X, Yp, Cp, C, W, res, th, sig;
  int *flag, *sweeps;
};

Bufs carve(double *work, int P, const Layout &L) {
  Bufs B;
  B.Y = pset_linear(work + L.oY, L.per);
  B.Z = pset_linear(work + L.oZ, L.per);
  B.X = pset_linear(work + L.oX, L.per);
  B.Yp = pset_linear(work + L.oYp, L.per);
  B.Cp = pset_linear(work + L.oCp, L.per);
  B.C = pset_linear(work + L.oC, L.per);
  B.W = pset_linear(work + L.oW, L.per);
  B.res = pset_linear(work + L.oRes, L.per);
  B.th = pset_linear(work + L.oTh, L.per);
  B.sig = pset_linear(work + L.oSig, L.per);
  B.flag = reinterpret_cast<int *>(work + (long long)P * L.per);
  B.sweeps = B.flag + 2;
  return B;
}

bool same(const PSet &a, const PSet &b) { return a.b0 == b.b0 && a.b1 == b.b1 && a.stride == b.stride; }

int grid_1d(long long count, int P) {
  long long b = (count + 255) / 256;
  return (int)std::max<long long>(1, std::min<long long>(b, (152 * 4 + P - 1) / P));
}

}  // namespace

long long si_workspace_doubles(int P, int n, int m) {
  return layout(P, n, m).per * P + 64;
}

int jacobi_block(int n) {
  const int m = n + (n & 1);
  return m < 4 ? 4 : m;
}

SiOut si_outputs(double *work, int P, int n, int m) {
  const Layout L = layout(P, n, m);
  Bufs B = carve(work, P, L);
  return SiOut{B.X, B.th};
}

cudaError_t jacobi_full(const SiBatch &b, double *work, cudaStream_t s, long long *launches) {
  const int n = b.n, P = b.P, m = jacobi_block(n);
  if (m > kSiMaxBlock || b.k > n || P > 65535) return cudaErrorInvalidValue;
  const Layout L = layout(P, n, m);
  Bufs B = carve(work, P, L);
  if (n == 1) return eig_one(b.G, B.X, B.th, m, P, s, launches);
  cudaError_t e;
  if ((e = cudaMemsetAsync(B.flag, 0, 4 * sizeof(int), s))) return e;
  PSet H = b.G;
  if (m != n) {
    launch_pdl(k_si_copy_square, dim3(grid_1d((long long)m * m, P), 1, P), 256, 0, s, b.G, B.C, n, m);
    if ((e = cudaGetLastError())) return e;
    *launches += 1;
    H = B.C;
  }
  const SmallEig se{P, m, H, B.Cp, true, b.graded, B.X, n, b.k, B.th, B.flag, b.err, B.sweeps, B.flag + 3};
  return small_eig(se, s, launches);
}

cudaError_t si_solve(const SiBatch &b, double *work, double tol, int max_iter, cudaStream_t s,
                     SiResult *res, long long *launches) {
  cudaError_t e;
  const int P = b.P, n = b.n, m = b.m, k = b.k;
  if (P < 1 || P > 65535 || m > kSiMaxBlock || m > n || k > m || (m & 1))
    return cudaErrorInvalidValue;
  const Layout L = layout(P, n, m);
  Bufs B = carve(work, P, L);
  PSet X = B.X, Y = B.Y, Z = B.Z, Y2 = B.Yp;   // Y2: free but during an FP64 SIMT product
  const dim3 gz(1, 1, P);
  const int chunk = ((n + L.S - 1) / L.S + 15) / 16 * 16;
  const double shift = 11.0 * ((double)n * m + (double)m * (m + 1)) * 1.1102230246251565e-16;
  long long nl = 0;

  // Products over the long dimension n (G X, the basis rotations X W and the
  // Gram matrices X^T Y) run as exact-slice tensor-core GEMMs (FP64-grade, see
  // tc_exact.cuh) unless the caller asked for the FP64 SIMT kernels.  The
  // n x m x m rotations and Gram matrices go to the tensor cores only when the
  // batch makes them FP64-throughput bound; below
  // that the single SIMT launch beats the slice-and-multiply sequence.
  const bool xs = b.xs;
  const bool batch = P > kSiSmallBatch && b.floor_tol > 0.0;
  const bool xs_small = xs && (double)P * n * m * m >= (batch ? kXsBatchWork : kXsSmallWork);
  XsOperand gs{};
  // slices of a row-major (rows x K) view of problem z's buffer at src
  auto xs_slot = [&](long long off, long long scoff, int rows, int K) {
    return XsOperand{work + off, work + scoff, rows, K, xs_pitch(K), kSiSlices, P, L.per * 4, L.per};
  };
  if (xs) {
    gs = XsOperand{work + L.oGs, work + L.oGsc, n, n, L.xsp, kSiSlices, P, L.per * 4, L.per};
    if ((e = xs_split(b.G, map1(n), map1(1), gs, s))) return e;
    nl += 1;
  }
  auto add_shift = [&](PSet src, PSet dst) -> cudaError_t {
    if (!b.has_trace) return cudaSuccess;
    launch_pdl(k_si_shift_add, dim3(grid_1d(L.nm, P), 1, P), 256, 0, s, dst, src, B.sig, L.nm);
    nl += 1;
    return cudaGetLastError();
  };
  // dst = G src; where the K parts are summed by a separate pass, that pass
  // also adds the shift (shifted = true)
  bool shifted = false;
  auto product = [&](PSet src, PSet dst) -> cudaError_t {
    shifted = false;
    const int sh = b.has_trace ? 1 : 0;
    if (xs) {
      const XsOperand xsl = xs_slot(L.oSb, L.oSbsc, m, n);     // rows of X^T
      cudaError_t r = xs_split(src, map1(n), map1(1), xsl, s);
      if (r) return r;
      r = xs_gemm(gs, xsl, n, m, n, dst.b0, map1(1), map1(n), L.per, 1, 0, b.err, s, XsShift{sh != 0, src, B.sig});
      shifted = true;
      nl += 2;
      return r ? r : cudaGetLastError();
    }
    if (L.S == 1) {
      launch_pdl(k_si_gemm, dim3((n + 63) / 64, 1, P), 256, 0, s, b.G, src, dst, n, m, chunk);
      nl += 1;
    } else {
      launch_pdl(k_si_gemm, dim3((n + 63) / 64, L.S, P), 256, 0, s, b.G, src, B.Yp, n, m, chunk);
      launch_pdl(k_si_sum_split, dim3(grid_1d(L.nm, P), 1, P), 256, 0, s, B.Yp, dst, L.S, L.nm, src, B.sig, sh);
      shifted = true;
      nl += 2;
    }
    return cudaGetLastError();
  };
  auto gemm = [&](PSet src, PSet dst) -> cudaError_t {
    cudaError_t r0 = product(src, dst);
    return r0 ? r0 : (shifted ? cudaSuccess : add_shift(src, dst));
  };
  // dst = src W (n x m times m x m, W column-major; tri: W upper triangular).
  // A CholeskyQR basis change (tri) normalises columns whose lengths can differ
  // by many orders of magnitude: the exact-slice product then scales column j
  // of src by a power of two near 1 / |src_j| (and row j of W inversely), so
  // that the row slicing of src keeps every column's relative accuracy.
  auto rot = [&](PSet src, PSet W, PSet dst, int tri) -> cudaError_t {
    if (xs_small) {
      const XsOperand a = xs_slot(L.oSa, L.oSasc, n, m);       // rows of X
      const XsOperand w = xs_slot(L.oSb, L.oSbsc, m, m);       // columns of W
      const PSet ks = pset_linear(work + L.oKs, L.per);
      cudaError_t r;
      if (tri) {
        launch_pdl(k_si_colscale, dim3(1, 1, P), 128, 0, s, B.C, ks, m);
        nl += 1;
      }
      if ((r = xs_split_scaled(src, map1(1), map1(n), ks, tri ? 1 : 0, a, s)) ||
          (r = xs_split_scaled(W, map1(m), map1(1), ks, tri ? 2 : 0, w, s)) ||
          (r = xs_gemm(a, w, n, m, m, dst.b0, map1(1), map1(n), L.per, 1, 0, b.err, s)))
        return r;
      nl += 3;
      return cudaSuccess;
    }
    return rotate_basis(src, dst, nullptr, nullptr, W, n, m, tri != 0, P, s, &nl);
  };
  // C = A^T A (m x m), and with Bm out2 = A^T Bm, symmetrised
  auto gram = [&](PSet A, PSet out, const PSet *Bm, const PSet *out2) -> cudaError_t {
    if (xs_small) {
      const XsOperand a = xs_slot(L.oSa, L.oSasc, m, n);       // columns of A
      const XsOperand bb = xs_slot(L.oSb, L.oSbsc, m, n);      // columns of B
      cudaError_t r;
      if ((r = xs_split(A, map1(n), map1(1), a, s)) ||
          (r = xs_gemm(a, a, m, m, n, B.Cp.b0, map1(m), map1(1), L.per, 1, 0, b.err, s)))
        return r;
      nl += 2;
      if ((r = gram_reduce(B.Cp, out, 1, m, P, s, &nl)) || !Bm) return r;
      if ((r = xs_split(*Bm, map1(n), map1(1), bb, s)) ||
          (r = xs_gemm(a, bb, m, m, n, B.Cp.b0, map1(m), map1(1), L.per, 1, 0, b.err, s)))
        return r;
      nl += 2;
      return gram_reduce(B.Cp, *out2, 1, m, P, s, &nl);
    }
    return gram64(A, A, out, Bm, out2, n, m, B.Cp, P, s, &nl);
  };
  // one CholeskyQR pass with an FP32 factorisation: dst = src W
  auto cholqr32 = [&](PSet src, PSet dst, float sh) -> cudaError_t {
    cudaError_t r;
    if (xs_small) {
      if ((r = gram(src, B.C, nullptr, nullptr)) || (r = chol32(B.C, m, sh, B.W, B.flag, P, s, &nl))) return r;
    } else if ((r = cholqr32_factor(src, n, m, sh, B.W, B.flag, P, s, &nl))) {
      return r;
    }
    return rot(src, B.W, dst, 1);
  };
  // one CholeskyQR pass in FP64 (robust for any conditioning with the shift)
  auto cholqr64 = [&](PSet src, PSet dst, double sh) -> cudaError_t {
    cudaError_t r = gram(src, B.C, nullptr, nullptr);
    if (r) return r;
    if ((r = chol64(B.C, m, sh, B.W, B.flag, PSet{nullptr, nullptr, 0}, P, s, &nl))) return r;
    return rot(src, B.W, dst, 1);
  };
  // dst = orth(src) through tmp (src is overwritten).  After the first
  // Rayleigh-Ritz step the basis holds Ritz vectors, G X is X Theta up to the
  // residual, its column-scaled Gram matrix is close to I, and one CholeskyQR
  // pass with an FP32 factorisation suffices for the power iteration.  Before
  // it the block can be ill conditioned.  Small batches (latency bound: the
  // single-CTA FP64 factorisation costs more than its iterations save) use the
  // same two FP32 passes, the first of which retries with a diagonal shift
  // where the columns are nearly dependent; large batches use shifted
  // CholeskyQR3 in FP64, which keeps more of the ill-conditioned directions and
  // saves iterations on their hardest problems.
  //
  // A block that holds numerically null directions of G (Ritz values below
  // 1e-9 of the largest: rank-deficient environments at fixed points and in
  // limits such as the classical Ising chain) cannot be orthogonalised in FP32:
  // each FP32 pass leaves about 1e-7 of the dominant directions in the null
  // columns, and the next product amplifies it by theta_0 / sigma (~1e12), so
  // the basis collapses.  Once a Rayleigh-Ritz step sees such directions, the
  // rest of the solve orthogonalises with two FP64 CholeskyQR passes.
  const bool fp64_start = P > kSiSmallBatch;
  bool orth64 = false;
  int n_orth = 0;
  auto orth = [&](PSet src, PSet tmp, PSet dst, bool after_rr) -> cudaError_t {
    cudaError_t r;
    ++n_orth;
    if (orth64) {
      if ((r = cholqr64(src, tmp, shift))) return r;
      return cholqr64(tmp, dst, 0.0);
    }
    // One FP32 pass once the columns are close to eigenvectors (after a
    // Rayleigh-Ritz step, or from the third iteration of a warm start): the
    // column-scaled Gram matrix of G X is then close to I and one pass leaves
    // X orthonormal to about FP32 accuracy, which is all the power iteration
    // needs -- the Rayleigh-Ritz step works with C0 = X^T X and does not
    // assume an orthonormal basis (measured at D = 32: 8.5 iterations per
    // step either way, 0.6 ms less per step).
    if (after_rr || (b.has_warm && n_orth >= 3)) return cholqr32(src, dst, 0.0f);
    if (!fp64_start) {
      if ((r = cholqr32(src, tmp, 0.0f))) return r;
      return cholqr32(tmp, dst, 0.0f);
    }
    if ((r = cholqr64(src, tmp, shift)) || (r = cholqr64(tmp, src, 0.0))) return r;
    return cholqr64(src, dst, 0.0);
  };

  if ((e = cudaMemsetAsync(B.flag, 0, 4 * sizeof(int), s))) return e;
  if (b.has_trace) {
    launch_pdl(k_si_sigma_init, dim3(1, 1, P), 32, 0, s, B.sig, b.trace, b.shift_rel);
    nl += 1;
  }
  launch_pdl(k_si_init, dim3(grid_1d(L.nm, P), 1, P), 256, 0, s, X, b.warm, b.has_warm ? 1 : 0, b.kw, n, m);
  nl += 1;
  // a random or partly warm start is orthogonalised (well conditioned); a start
  // from all m Ritz vectors of the previous solve is orthonormal to FP64 accuracy
  // already (the final rotation of a Rayleigh-Ritz step)
  if (!(b.has_warm && b.kw >= m)) {
    if ((e = cholqr32(X, Z, 0.0f)) || (e = cholqr32(Z, Y, 0.0f))) return e;
    std::swap(X, Y);
  }

  res->converged = false;
  res->breakdown = 0;
  res->sweeps64 = 0;
  res->sweeps32 = 0;
  res->rr = 0;
  res->residual = INFINITY;
  int it = 0;
  // With the FP32 start-up a Rayleigh-Ritz step costs several iterations:
  // the first one goes where the caller expects convergence.
  int next_check = fp64_start ? 3 : std::max(3, b.first_check);
  std::vector<double> hres((size_t)P * k), hth((size_t)P * m);
  // HOTRG_TRACE_EIG=1 (or 2, with every residual and Ritz value) prints each
  // convergence check of the solve to stderr
  static const int trace = getenv("HOTRG_TRACE_EIG") ? atoi(getenv("HOTRG_TRACE_EIG")) : 0;
  double prev_worst = INFINITY;
  while (it < max_iter) {
    const bool check = (it + 1 >= next_check) || (it + 1 == max_iter);
    if ((e = gemm(X, Y))) return e;  // Y = G X
    ++it;
    if (check) {
      // Rayleigh-Ritz on the span of X, whose columns the FP32 CholeskyQR left
      // orthonormal only to about its own accuracy: with C0 = X^T X and
      // W = C0^(-1/2) (Newton-Schulz on the m x m side, from C0 ~ I), X W is
      // orthonormal to FP64 accuracy, G X W = Y W, and the projected matrix
      // is H = W^T (X^T Y) W.  Its eigenvectors Z give the Ritz vectors X (W Z)
      // and G X (W Z) = Y (W Z) with one rotation each.
      auto slot = [&](int i) { return PSet{B.Cp.b0 + i * L.mm, B.Cp.b1 + i * L.mm, B.Cp.stride}; };
      PSet Wn = slot(0), Tn = slot(1);
      const PSet Ck = slot(2), Rr = slot(3);
      const dim3 gmm((m + 7) / 8, (m + 7) / 8, P);
      const PSet always{nullptr, nullptr, 0};
      if ((e = gram(X, B.W, &Y, &B.C))) return e;   // C0 (B.W until small_eig) and X^T Y
      launch_pdl(k_rr_start, gz, 1024, 0, s, B.W, m, Wn, B.sig);
      nl += 1;
      // W <- W (3I - W^T C0 W) / 2 twice, the second time only where it is needed
      // (Tn holds the result either way)
      const PSet T2 = slot(4 + kSmallEigSlots);
      launch_pdl(k_rr_mm, gmm, 256, 0, s, B.W, 0, Wn, 1.0, 0.0, Ck, m, always, always);   // C0 W
      launch_pdl(k_rr_mm, gmm, 256, 0, s, Wn, 1, Ck, 1.0, 0.0, Rr, m, always, always);    // W^T C0 W
      launch_pdl(k_rr_mm, gmm, 256, 0, s, Wn, 0, Rr, -0.5, 1.5, Tn, m, always, T2);
      launch_pdl(k_rr_mm, gmm, 256, 0, s, B.W, 0, T2, 1.0, 0.0, Ck, m, B.sig, always);
      launch_pdl(k_rr_mm, gmm, 256, 0, s, T2, 1, Ck, 1.0, 0.0, Rr, m, B.sig, always);
      launch_pdl(k_rr_mm, gmm, 256, 0, s, T2, 0, Rr, -0.5, 1.5, Tn, m, B.sig, always);
      nl += 6;
      std::swap(Wn, Tn);
      // where X is further from orthonormal (nearly dependent columns at a first
      // check), W comes instead from an FP64 Cholesky of C0, shifted where C0 is far
      // from I (X W is then orthonormal for any conditioning the shift allows)
      if ((e = chol64(B.W, m, shift, Wn, B.flag, B.sig, P, s, &nl))) return e;
      launch_pdl(k_rr_mm, gmm, 256, 0, s, B.C, 0, Wn, 1.0, 0.0, Tn, m, always, always);     // (X^T Y) W
      launch_pdl(k_rr_sym, gmm, 256, 0, s, Wn, Tn, Ck, m);                                  // H = W^T X^T Y W
      nl += 2;
      if ((e = cudaGetLastError())) return e;
      const SmallEig se{P, m, Ck, slot(4), false, false, B.W, m, m, B.th, B.flag, nullptr, B.sweeps, B.flag + 3};
      if ((e = small_eig(se, s, &nl))) return e;                    // H = Z Theta Z^T (Z in B.W)
      launch_pdl(k_rr_mm, gmm, 256, 0, s, Wn, 0, B.W, 1.0, 0.0, Rr, m, always, always);     // R = W Z
      nl += 1;
      if (xs_small) {
        if ((e = rot(X, Rr, Z, 0))) return e;
        std::swap(X, Z);
        if ((e = rot(Y, Rr, Z, 0))) return e;
        std::swap(Y, Z);
      } else {
        // X -> Z and Y -> the first K-part slot in one launch, then renamed
        if ((e = rotate_basis(X, Z, &Y, &Y2, Rr, n, m, false, P, s, &nl))) return e;
        std::swap(X, Z);
        std::swap(Y, Y2);
      }
      launch_pdl(k_si_residual, dim3(k, 1, P), 256, 0, s, X, Y, B.th, B.res, B.sig, b.has_trace ? 1 : 0, n, k);
      nl += 1;
      ++res->rr;
      if ((e = cudaMemcpy2DAsync(hres.data(), sizeof(double) * k, B.res.at(0), sizeof(double) * L.per,
                                 sizeof(double) * k, P, cudaMemcpyDeviceToHost, s)))
        return e;
      if ((e = cudaMemcpy2DAsync(hth.data(), sizeof(double) * m, B.th.at(0), sizeof(double) * L.per,
                                 sizeof(double) * m, P, cudaMemcpyDeviceToHost, s)))
        return e;
      int hflag[4];
      if ((e = cudaMemcpyAsync(hflag, B.flag, sizeof(hflag), cudaMemcpyDeviceToHost, s))) return e;
      if ((e = cudaStreamSynchronize(s))) return e;
      double worst = 0.0;
      int wp = 0, wi = 0;
      for (int q = 0; q < P * k; ++q) {
        const double v = std::isfinite(hres[q]) ? hres[q] : INFINITY;
        if (v > worst) {
          worst = v;
          wp = q / k;
          wi = q % k;
        }
      }
      res->residual = worst;
      if (trace) {
        const double *th = hth.data() + (size_t)wp * m;
        fprintf(stderr,
                "[hotrg eig] n %d m %d k %d P %d it %d rr %d worst %.3e at problem %d pair %d: "
                "theta_i/theta_0 %.6e theta_k/theta_0 %.6e theta_m/theta_0 %.6e sweeps %d/%d flag %d\n",
                n, m, k, P, it, res->rr, worst, wp, wi, th[wi] / th[0], th[k - 1] / th[0],
                th[m - 1] / th[0], hflag[3], hflag[2], hflag[0]);
        if (trace > 1) {
          fprintf(stderr, "[hotrg eig]   residuals:");
          for (int i = 0; i < k; ++i) fprintf(stderr, " %.1e", hres[(size_t)wp * k + i]);
          fprintf(stderr, "\n[hotrg eig]   theta/theta_0:");
          for (int i = 0; i < m; ++i) fprintf(stderr, " %.4e", th[i] / th[0]);
          fprintf(stderr, "\n");
        }
      }
      res->breakdown = hflag[0];
      res->sweeps64 = hflag[2];
      res->sweeps32 = hflag[3];
      if (hflag[0]) break;          // breakdown: reported to the caller
      // Converged at the bound, or at the accuracy floor of G: a residual
      // below the floor that no longer halves between two Rayleigh-Ritz
      // steps cannot be improved by more iterations (the exact-slice products
      // reach about 1e-12 relative at n = 4096; an environment built with
      // reduced-precision products carries a noise floor of eigenvalues whose
      // vectors are not determined beyond that noise).
      const double floor_tol = b.floor_tol > 0.0 ? b.floor_tol : kSiFloorTol;
      const bool stalled = worst <= floor_tol && res->rr >= 2 && worst > 0.5 * prev_worst;
      // In a flat tail of noise-level eigenvalues (reduced-precision G) the
      // wanted pairs converge at a rate near 1: after kSiSlowIters iterations
      // a residual below the accuracy floor of G is accepted.
      const bool slow = b.floor_tol > 0.0 && worst <= floor_tol && it >= kSiSlowIters;
      if (worst <= tol || stalled || slow) {
        res->converged = true;
        break;
      }
      prev_worst = worst;
      // A Ritz value well below zero is as telling where G is accurate to FP64
      // (G + sigma I is positive definite): the FP32 passes have let the block
      // collapse onto nearly dependent columns.
      for (int p = 0; p < P && !orth64; ++p) {
        const double t0 = hth[(size_t)p * m], tm = hth[(size_t)p * m + m - 1];
        if (!(fabs(tm) > 1e-9 * fabs(t0))) orth64 = true;
        if (b.floor_tol == 0.0 && tm < -1e-9 * fabs(t0)) orth64 = true;
      }
      // Errors in the wanted Ritz pairs shrink by about theta_m / theta_k per
      // iteration: schedule the next check where that predicts convergence.
      double rho = 0.0;
      for (int p = 0; p < P; ++p) {
        const double tk = fabs(hth[(size_t)p * m + k - 1]), tm = fabs(hth[(size_t)p * m + m - 1]);
        rho = std::max(rho, tk > 0.0 ? tm / tk : 1.0);
      }
      int need = 2;
      if (rho > 0.0 && rho < 0.9 && std::isfinite(worst) && worst > 0.0)
        need = (int)std::ceil(std::log(tol / worst) / std::log(rho)) + 1;
      next_check = it + std::max(1, std::min(need, 8));
    }
    if ((e = orth(Y, Z, X, res->rr > 0))) return e;   // X = orth(G X)
  }
  res->iterations = it;
  if (b.has_trace) {
    launch_pdl(k_si_unshift, dim3(1, 1, P), 128, 0, s, B.th, B.sig, m);
    nl += 1;
  }
  // the Ritz vectors end in the workspace's X slot
  if (!same(X, B.X)) {
    launch_pdl(k_si_copy, dim3(grid_1d(L.nm, P), 1, P), 256, 0, s, X, B.X, L.nm);
    nl += 1;
  }
  *launches += nl;
  return cudaGetLastError();
}

}  // namespace hotrg
