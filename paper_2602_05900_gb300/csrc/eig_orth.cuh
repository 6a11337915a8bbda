// Orthogonalisation kernels of the subspace iteration (see eig_orth.cu): Gram
// matrices of n x m blocks, the FP32 CholeskyQR factor, and the basis rotation.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace hotrg {

// 2^-e scaling factor with e the binary exponent of x (exact, x > 0 finite)
__device__ inline double pow2_inv_of(double x) {
  const long long bits = __double_as_longlong(x);
  const int e = (int)((bits >> 52) & 0x7FF) - 1023;
  return __longlong_as_double((long long)(1023 - e) << 52);
}

// GB300 executes FP64 square roots and divisions as long dependent instruction
// sequences; on latency-bound paths they are replaced by an FP32 estimate
// refined with FP64 fused multiply-adds (Newton's method), which is accurate to
// FP64 rounding after two steps.
//
// 1/sqrt(x) for x > 0 to FP64 accuracy: FP32 seed on a power-of-two scaled
// argument, two Newton steps y <- y (3 - x y^2) / 2 in FP64.
__device__ inline double rsqrt_fp64(double x) {
  const double s = pow2_inv_of(x);                  // x s in [1, 2)
  const double xs = x * s;
  double y = (double)rsqrtf((float)xs);
  y = y * fma(-0.5 * xs, y * y, 1.5);
  y = y * fma(-0.5 * xs, y * y, 1.5);
  // 1/sqrt(x) = (1/sqrt(x s)) sqrt(s); s is a power of two
  const long long sb = __double_as_longlong(s);
  const int es = (int)((sb >> 52) & 0x7FF) - 1023;
  double root_s = (es & 1) ? 1.4142135623730951 : 1.0;
  root_s *= __longlong_as_double((long long)(1023 + (es >> 1)) << 52);
  return y * root_s;
}

// Number of row chunks whose partial Gram matrices gram64 writes (m x m doubles
// each, at most kGramChunks per problem).
constexpr int kGramChunks = 256;
// out0 = A^T B0 and (optional) out1 = A^T B1 (m x m, symmetrised; A, B n x m
// column-major).  part: kGramChunks m x m slots of problem z.
cudaError_t gram64(PSet A, PSet B0, PSet out0, const PSet *B1, const PSet *out1, int n, int m, PSet part, int P,
                   cudaStream_t s, long long *launches);
// out = sum of `chunks` m x m partials of A^T B, symmetrised.
cudaError_t gram_reduce(PSet part, PSet out, int chunks, int m, int P, cudaStream_t s, long long *launches);

// W = diag(d) R^-1 (column-major, upper triangular) with R^T R = diag(d) C diag(d)
// + shift I, d_j = 1 / sqrt(C_jj), in FP32: Y W is orthonormal to FP32 accuracy.
// A factorisation that breaks down is repeated with a larger shift; a second
// breakdown sets *flag to 1.  From the block Y itself, with C = Y^T Y:
cudaError_t cholqr32_factor(PSet Y, int n, int m, float shift, PSet W, int *flag, int P, cudaStream_t s,
                            long long *launches);
// ... or from a given C:
cudaError_t chol32(PSet C, int m, float shift, PSet W, int *flag, int P, cudaStream_t s, long long *launches);

// The same in FP64 (W to FP64 accuracy); for problem z only if only_if.at(z)[2] != 0,
// and without a shift at first if it is 1 (only_if.b0 null: always, shifted).
cudaError_t chol64(PSet C, int m, double shift, PSet W, int *flag, PSet only_if, int P, cudaStream_t s,
                   long long *launches);

// H (m x m, symmetric) scaled by the power of two that brings its largest
// entry into [1, 2), plus kLrShift I, = L L^T to ~2^-44 sqrt(h_ii h_jj): L (column-major, zeros above the
// diagonal) and B = L.  A pivot below kLrPivot (H is not positive semidefinite to
// rounding) makes L = I and B = H of that problem: L^T B is similar to H either way,
// up to the scale and the shift.
constexpr double kLrShift = 0x1p-28;
constexpr float kLrPivot = 0x1p-30f;
cudaError_t lr_factor(PSet H, int m, PSet L, PSet B, int P, cudaStream_t s, long long *launches);

// Out0 = A0 W and (optional) Out1 = A1 W (A, Out n x m column-major, W m x m
// column-major; tri: W upper triangular)
cudaError_t rotate_basis(PSet A0, PSet Out0, const PSet *A1, const PSet *Out1, PSet W, int n, int m, bool tri, int P,
                         cudaStream_t s, long long *launches);

}  // namespace hotrg
