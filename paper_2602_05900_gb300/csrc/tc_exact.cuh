// Exact-slice GEMM: FP64-grade products on the BF16 tensor cores (sm_103a).
//
// GB300 executes FP64 at a few flops per clock per SM, BF16 tensor-core MMAs at
// thousands.  An FP64 operand row is written as 2^e (a_1 2^-6 + a_2 2^-12 + ...
// + a_S 2^-6S) with integers |a_1| <= 64, |a_s| <= 32 (round-to-nearest
// digits of the row scaled below 1); each digit times its power of two is an
// exact BF16 value (a "slice").  The product of two rows is then the sum over
// slice pairs (s, t) of exact BF16 x BF16 products; pairs with s + t <= S + 1
// are kept (the rest lie below 2^-6(S+1) of the leading term).  Pairs with the
// same s + t = d share one FP32 accumulator in tensor memory, an integer
// multiple of 2^-6d.  For d <= 6 its partial sums stay below 2^24 of that unit
// as long as K <= kXsMaxK (the d = 6 sum has five terms of at most 2^11, 2^10,
// 2^10, 2^10, 2^11 per k), so those accumulators are exact whatever the order of
// summation; the d >= 7 ones are 2^-30 smaller and exact but for saturated
// digits at the longest K.  The epilogue combines the accumulators into one
// 64-bit integer in units of 2^-50 (below the rounding of the digits), sums the
// K parts of a tile exactly (a cluster of CTAs, through distributed shared
// memory), and converts and scales once.  With
// S slices the result is within about 2^-(6S-1) of max|A_i.| max|B_j.| per
// term; the eigensolver's products G X use S = 8 (about 2^-47: FP64-grade).
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace hotrg {

constexpr int kXsBits = 6;        // bits per slice digit
constexpr int kXsMaxK = 2336;     // longest K part of one CTA (multiple of 32) with 7 2^10 K < 2^24
constexpr int kXsMaxBatch = 65535;  // instances of one launch (grid limit)
// Longest K of one launch.  A scaled element can round up to exactly 1, so a term
// reaches 2^50 units (its dropped digit pairs add at most 2^-24 of that) and the
// sum of 8192 of them 2^63: K stays below.  31 256, so that the parts of a
// launch divide into 1, 2, 4 or 8 of whole K blocks and never cover more.
constexpr int kXsMaxSumK = 7936;
constexpr int kXsMaxSlices = 8;
constexpr int kXsStagedK = 128;  // strided-K operands up to this K are sliced through shared memory

// Sliced operand: S planes of rows x pitch BF16 values (plane stride
// rows * pitch elements, K contiguous) and one power-of-two scale per row, for
// `batch` instances at fixed strides.
struct XsOperand {
  void *slices;        // __nv_bfloat16
  double *scale;
  int rows, K, pitch, S;
  int batch;
  long long bstride;   // BF16 elements between instances
  long long sstride;   // doubles between instances' scales
};

// Row pitch (elements) with a 16-byte multiple byte pitch.
inline int xs_pitch(int K) { return (K + 7) / 8 * 8; }
// BF16 elements of one instance's slices.
inline long long xs_elems(int rows, int K, int S) { return (long long)S * rows * xs_pitch(K); }

// Slices row r of instance z, whose element k is src.at(z)[rm(r) + km(k)].
cudaError_t xs_split(PSet src, IdxMap rm, IdxMap km, const XsOperand &dst, cudaStream_t s);

// The same with element k multiplied (kmode 1) or divided (kmode 2) by
// kscale.at(z)[k], a power of two (exact).  A product A B^T with A's columns
// and B's columns scaled inversely is unchanged, but the row slicing then
// sees balanced rows: used where the columns of A differ by many orders of
// magnitude (a column-normalising basis change).
cudaError_t xs_split_scaled(PSet src, IdxMap rm, IdxMap km, PSet kscale, int kmode,
                            const XsOperand &dst, cudaStream_t s);

// Optional addition of a product's launch: C += sig[1] X (X laid out like C), and
// sig[0] <- sig[1].
struct XsShift {
  bool on = false;
  PSet X{nullptr, nullptr, 0}, sig{nullptr, nullptr, 0};
};

// C(m, n) = sum_k A(m, k) B(n, k) in FP64 for every instance z, written to
// C + z * cstride + cm(m) + cn(n).  The K range is cut into `ksplit` equal
// parts (each <= kXsMaxSumK); part p is written at C + p * pstride (the caller
// sums the parts).  A.S == B.S, A.batch == B.batch.  err_flag receives 2 if a
// bounded wait runs out.
cudaError_t xs_gemm(const XsOperand &A, const XsOperand &B, int M, int N, int K, double *C,
                    IdxMap cm, IdxMap cn, long long cstride, int ksplit, long long pstride,
                    int *err_flag, cudaStream_t s, const XsShift &shift = XsShift{});

// C[m * ldc + n] = sum_p parts[p * pstride + m * N + n] (row-major parts).
cudaError_t xs_sum_parts(const double *parts, int nparts, long long pstride, int M, int N,
                         double *C, long long ldc, cudaStream_t s);

// Smallest number of launch parts with each part <= kXsMaxSumK.
inline int xs_min_split(int K) { return (K + kXsMaxSumK - 1) / kXsMaxSumK; }

}  // namespace hotrg

namespace hotrg {

// Scratch of gemm_xs: slices and row scales of both operands (for all
// instances of a batch) and the FP64 partial products of a split K.
struct XsWork {
  void *sa, *sb;              // BF16 slices
  double *sca, *scb;          // row scales
  double *parts;              // K-part results (dense [part][instance][M][N])
  long long cap_a, cap_b;     // BF16 elements
  long long cap_sa, cap_sb;   // doubles
  long long cap_parts;        // doubles
};

// Elements gemm_xs needs for one GEMM (A slices, B slices, A scales, B
// scales, parts), for `batch` instances.
void xs_gemm_needs(int M, int N, int K, int S, int batch, long long need[5]);

// The mapped GEMM of `g` (C(m, n) = sum_k A(m, k) B(n, k) through index maps,
// batched) as an exact-slice tensor-core GEMM with S digits: the operands are
// gathered and sliced, K is split into exact parts, the result is written in
// FP64 through g's output maps.  `launches` is incremented.
cudaError_t gemm_xs(const MappedGemm &g, int S, const XsWork &w, int *err_flag, cudaStream_t s, long long *launches);

// Whether gemm_xs of that size fits the scratch.
bool xs_fits(int M, int N, int K, int S, int batch, const XsWork &w);

// `count` products C_v(m, n) = sum_k A_v(m, k) A_v(n, k) of the same sizes and output
// maps (g[v].B is not read), C_v = g[0].C + v * batch * bC: every operand is sliced
// once and all products are one launch.  The scratch has to fit count * batch
// instances of A (syrk_xs_fits with that batch; K <= kXsMaxSumK).
bool syrk_xs_fits(int M, int K, int batch, int S, const XsWork &w);
cudaError_t syrk_xs(const MappedGemm *g, int count, int S, const XsWork &w, int *err_flag, cudaStream_t s,
                    long long *launches);

}  // namespace hotrg
