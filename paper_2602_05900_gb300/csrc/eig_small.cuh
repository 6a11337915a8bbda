// Batched eigensolver for small symmetric matrices (4 <= m <= 96, m even): the
// Rayleigh-Ritz problems of the subspace iteration, the whole environments of
// small bond dimensions and iTEBD's bond density matrices.  FP32 two-sided
// Jacobi (Sec. II.B, Eqs. 5-6), then an FP64 refinement (see eig_small.cu).
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace hotrg {

constexpr int kErrEig = 4;          // in a context's device error flag: a direct solve did not finish
constexpr int kSmallEigSlots = 7;   // m x m scratch matrices per problem

struct SmallEig {
  int P, m;              // problems, matrix size
  PSet H;                // m x m matrix of problem z, symmetric to the last bit (of the products
                         // with it only one triangle is computed)
  PSet scratch;          // kSmallEigSlots consecutive m x m slots of problem z
  bool full;             // resolve every pair to FP64 rounding of H (direct solves); else to
                         // 2^-44 of the largest eigenvalue (Rayleigh-Ritz steps, whose H
                         // carries that much rounding)
  bool graded;           // full only: H is positive semidefinite to rounding and already nearly
                         // diagonal (a warm start); a hint, the result does not depend on it
  PSet out;              // leading eigenvectors: rows x cols, column-major, ld = rows
  int rows, cols;        // rows, cols <= m
  PSet theta;            // m eigenvalues, descending
  int *flag;             // set to 2 if the last stage did not finish
  int *err;              // (optional) raised to kErrEig then
  int *rounds, *sweeps;  // maxima over problems: FP64 rounds, FP32 sweeps
};

// Enqueues the solve on stream s; `launches` is incremented.
cudaError_t small_eig(const SmallEig &a, cudaStream_t s, long long *launches);

// theta[0] = G, X[0] = 1 for 1 x 1 matrices (theta padded with zeros to m entries)
cudaError_t eig_one(PSet G, PSet X, PSet theta, int m, int P, cudaStream_t s, long long *launches);

}  // namespace hotrg
