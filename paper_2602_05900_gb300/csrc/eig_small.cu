// Batched eigensolver for small symmetric matrices (see eig_small.cuh).
//
// GB300 runs FP64 at two FMAs per clock per SM and 64 cycles of latency, FP32 at
// 64 times that rate, so the rotations are done in FP32 and FP64 is kept for a
// few dense m x m products spread over many CTAs:
//
//   1. k_rr_jacobi32: FP32 cyclic Jacobi, one CTA per problem.  Its V
//      diagonalises H to FP32 relative accuracy.
//   2. (full solves) X = V made orthonormal to ~1e-12 by one Newton-Schulz step,
//      S = X^T H X in FP64, and a second FP32 pass on S: the first one sees the
//      small eigenvalues of a dense H only through the FP32 rounding of the
//      large entries; S is graded, and its small block is resolved at its own
//      scale.
//      Warm starts (from kLrMinSize rows) take another way to
//      X: H + shift = L L^T, FP32 passes on L^T L, which is similar to it and far
//      nearer to diagonal where the spectrum is graded (Rutishauser's LR step; the
//      preconditioning of Veselic and Hari's one-sided Jacobi method), and
//      X = L V, made orthonormal by a refinement pass that normalises the columns
//      and a Newton-Schulz step.  An FP32 rotation contaminates a column
//      with ~1e-13 of the leading eigenvalue, so the shift is 2^-28 of it: with 2^-48
//      columns belonging to eigenvalues of 1e-18 lost their orthogonality.  Over
//      graded, rank-deficient, degenerate and random environments of 34 to 96 rows
//      both passes together took 1445 sweeps without the factor and take 617 in a CPU model.
//   3. Two refinement passes (one after the factored route) X <- X (I + E) (Ogita and Aishima's iteration):
//      with G = X^T X, S = X^T H X and lambda_i = s_ii / g_ii,
//      E_ij = (s_ij - lambda_j g_ij) / (lambda_j - lambda_i) for separated pairs
//      and -g_ij / 2 inside clusters and for couplings at rounding level:
//      quadratic convergence of the vectors and of their orthonormality at once;
//      then two Newton-Schulz steps for the orthonormality the last pass left.
//   4. S = X^T H X once more, and exact 2 x 2 rotations (k_rr_sparse_jacobi) of
//      the pairs that still need one: those in clusters of near-equal values.
//
// Measured against the FP64 two-sided Jacobi on an 8-CTA cluster that this
// replaced (its rounds cost 4 us, half of it FP64 arithmetic): an iTEBD update
// of one chain at n = 60 took 3.63 ms and takes 0.37 ms, of 64 chains at n = 32
// 3.39 ms and 0.36 ms, a D = 8 FP64 step (n = 64) 2.88 ms and 0.43 ms.
//
// A CPU model of the four stages (dense, graded, rank-deficient and degenerate
// matrices, m = 16 to 96) leaves residuals and orthonormality at 1e-15 and at
// most a few rotations for stage 4.
#include <math.h>
#include <stdlib.h>

#include <type_traits>
#include <utility>

#include "eig_orth.cuh"
#include "kernel_attr.cuh"
#include "launch.cuh"
#include "eig_si.cuh"
#include "eig_small.cuh"

namespace hotrg {
namespace {

// Couplings, gaps and quotients of the FP64 stages are judged in FP32, relative
// to the largest diagonal entry: its exponent field (kept within the range in which
// every product below stays normal; that of 1 for a zero diagonal) is the bias of
// their conversions, so that a matrix of any scale is treated alike.
__device__ inline unsigned abs_hi(double h) { return (unsigned)__double2hiint(h) & 0x7FFFFFFFu; }
__device__ inline int scale_bias(unsigned hi) { return hi >> 20 ? min(max((int)(hi >> 20), 200), 1900) : 1023; }
__device__ inline unsigned warp_max(unsigned v) { return __reduce_max_sync(0xffffffffu, v); }

// |h| 2^(1023 - bias) truncated to FP32 with integer arithmetic (FP64 conversions
// run at the FP64 rate); values below the FP32 range give 0
__device__ inline float mag32(unsigned hi, unsigned lo, int bias) {
  const int e = (int)(hi >> 20) - (bias - 127);
  if (e <= 0) return 0.0f;
  if (e >= 255) return INFINITY;
  return __uint_as_float(((unsigned)e << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
}
__device__ inline float mag32(double h, int bias) { return mag32(abs_hi(h), (unsigned)__double2loint(h), bias); }

__device__ inline void jacobi_angle(double hpp, double hqq, double hpq, double &c, double &s) {
  // solve h_pq t^2 + (h_qq - h_pp) t - h_pq = 0 for the smaller root (Golub &
  // Van Loan's symmetric Schur decomposition) on a power-of-two scaled copy:
  // FP32 estimate, then two Newton steps whose residual is evaluated in FP64
  const double sc = pow2_inv_of(fmax(fabs(hpq), fmax(fabs(hpp), fabs(hqq))));
  const double a = hpp * sc, b = hqq * sc, g = hpq * sc, diff = b - a;
  const float fg = (float)g, fd = (float)diff;
  float t32;
  if (fabsf(fd) > 1e6f * fabsf(fg)) {
    t32 = fg / fd;                                  // 1/(2 tau), tau = diff / (2 g)
  } else {
    const float tau = fd / (2.0f * fg);
    t32 = copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
  }
  double t = (double)t32;
  // seed of c = (1 + t^2)^(-1/2) from the FP32 root, computed while t is refined
  const float c32 = rsqrtf(fmaf(t32, t32, 1.0f));
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const double F = fma(fma(g, t, diff), t, -g);   // g t^2 + diff t - g
    const double dF = fma(2.0 * g, t, diff);
    t -= F * (double)__frcp_rn((float)dF);
  }
  // |t| <= 1 (the smaller root), so x = 1 + t^2 lies in [1, 2] and needs no
  // power-of-two scaling: two Newton steps y <- y (3 - x y^2) / 2 in FP64
  const double x = fma(t, t, 1.0);
  double y = (double)c32;
  y = y * fma(-0.5 * x, y * y, 1.5);
  y = y * fma(-0.5 * x, y * y, 1.5);
  c = y;
  s = t * c;
}

// ---- stage 1: FP32 cyclic Jacobi ---------------------------------------------

constexpr int kJ32MaxSweeps = 30;
// Warm starts of at least this size are factored: 30 iTEBD updates, ms without and
// with the factor, one chain n = 8 3.09 / 3.16, 14 3.69 / 3.78, 16 4.31 / 4.05,
// 32 6.72 / 5.83, 60 15.2 / 11.0, 96 37.9 / 26.6; 64 chains n = 8 3.90 / 4.03,
// 16 5.58 / 5.45, 32 11.3 / 10.8, 60 38.8 / 36.5.  Cold environments save three
// sweeps, which the six additional launches cost again (D = 8 run 8.46 / 8.44 ms, in
// TF32 9.15 / 9.64).
constexpr int kLrMinSize = 16;

// Where the first pass of a factored matrix stops: between the columns of length
// sqrt(kLrShift), 2^-12 of it leaves couplings of 2e-4 in X^T X, which the
// refinement squares.  Without a floor FP32 noise between equal small entries was
// rotated up to the sweep limit.
constexpr float kLrFloor = 0x1p-40f;


constexpr float kJ32Rel2 = 1e-12f;   // a pair is rotated while h_pq^2 > this h_pp h_qq

// Layout of the kernel for up to HM pairs (h = m / 2 <= HM): tops of the slots at
// rows and columns 0..h-1, bottoms HM further on, so that the four entries of a
// block and the two buffers are compile-time offsets apart.  A warp takes 4 x 8
// blocks, and the row pitch is 8 or 24 modulo the 32 banks: its four rows of
// eight neighbours fall on different banks.  The angles of a whole sweep are
// kept, of two sweeps in turn.
template <int HM, int SPL>
struct J32Cfg {
  static constexpr int kLd = 2 * HM + 8;                     // row pitch
  static constexpr int kA = 2 * HM * kLd;                    // floats of one matrix buffer
  static constexpr int kRound = 16 * SPL;                    // slots of a round's angles (float2: c, s), >= HM
  static constexpr int kSweep = (2 * HM - 1) * kRound;       // float2 of one sweep's angles
  static constexpr size_t kSmem = 2 * kA * sizeof(float) + (2 * kSweep + kRound) * sizeof(float2);
  static_assert(kSmem <= 200 * 1024, "shared memory");
  static_assert(kLd % 32 == 8 || kLd % 32 == 24, "bank layout");
};

__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// FP32 cyclic Jacobi on the symmetric m x m matrix of problem z, all disjoint
// pairs of a round at once (Eq. 6 per 2 x 2 block), Brent and Luk's systolic
// order (Fig. 3): slot I holds a top and a bottom index, a round rotates every
// slot's pair and then moves the tops one slot up and the bottoms one slot down
// (slot 0's top stays), so every pair meets once in the m - 1 rounds of a sweep
// and a sweep ends with every index back in its place.  The permutation is the
// same in every round: a thread reads and writes the same addresses all the
// time (two buffers in turn), with no index arithmetic.
//
// What bounds it: the chain from one round's angles to the next, then
// shared-memory wavefronts and issue slots.  So a round has one barrier: warps of
// their own compute the next round's angles from this round's matrix and angles
// (the two diagonal entries and the coupling that meet in a slot, rotated on the
// spot) while the others rotate the matrix.  The angles use the approximate
// reciprocal and square roots (an angle needs no more; c and s = t c keep
// c^2 + s^2 = 1 to FP32 rounding).  The matrix is kept as the blocks I <= J only,
// and V is off the chain: its rows sit in the registers of more warps (16 lanes a
// row, SPL slots a lane; a round is a rotation and one shuffle each way), which
// replay the angles of one sweep while the others run the next, and meet them
// once per sweep.  A round at m = 60 took 0.55 us with two barriers and V in
// shared memory, 0.42 us with V in registers, and takes 0.35 us (0.08 us of it the
// barrier and the loop; the angles alone end at 0.22, the matrix alone at 0.28).  RPG: rows per
// group of 16 lanes, IA: blocks of the matrix per thread.
//
// A pair is rotated while |h_pq| exceeds both floor_abs (of the largest
// diagonal entry, scaled to [1, 2)) and 1e-6 of sqrt|h_pp h_qq|: entries
// between two small diagonal entries are resolved to FP32 relative accuracy.
// Vout (FP64, column-major) receives the accumulated rotation, its columns in
// the order of the final diagonal (unsorted); *sweeps the largest sweep count.
template <int HM, int SPL, int RPG, int IA>
__global__ void __launch_bounds__(1024, 1)
    k_rr_jacobi32(PSet Hin, int m, float floor_abs, int nang, int nA, PSet Vout, int *sweeps) {
  pdl_enter();
  using C = J32Cfg<HM, SPL>;
  extern __shared__ __align__(16) float jsh[];
  float *Abuf = jsh;
  float2 *ring = reinterpret_cast<float2 *>(jsh + 2 * C::kA);   // [sweep parity][round][slot]
  float2 *spare = ring + 2 * C::kSweep;                         // angles nobody uses
  __shared__ double s_scale;
  __shared__ int s_rot[2];                                   // by sweep parity
  const int h = m / 2;
  constexpr int ld = C::kLd;
  const int z = blockIdx.z, tid = threadIdx.x, T = blockDim.x;
  const double *H = Hin.at(z);
  if (tid < 32) {
    double v = 0.0;
    for (int i = tid; i < m; i += 32) v = fmax(v, fabs(H[(size_t)i * m + i]));
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (tid == 0) s_scale = (v > 0.0 && isfinite(v)) ? pow2_inv_of(v) : 1.0;
  }
  for (int e = tid; e < 2 * C::kSweep; e += T) ring[e] = make_float2(1.0f, 0.0f);   // slots past h stay so
  __syncthreads();
  const double sc = s_scale;
  auto at = [&](int i) { return i < h ? i : HM + i - h; };   // row or column of index i
  // the symmetric part: two-sided rotations of a matrix whose triangles differ by
  // rounding (a product's, in a tile on the diagonal) do not settle
  for (int e = tid; e < m * m; e += T) {
    const int a = e / m, b = e % m;
    Abuf[at(a) * ld + at(b)] = to_f32(0.5 * (H[e] + H[(size_t)b * m + a]) * sc);
  }
  __syncthreads();
  if (tid < nA) {
    // ---- angles: first nang threads (thread k: slot k); the matrix: up to nA
    auto bar = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nA) : "memory"); };
    // where an index moves after a round (slot order), and the stored place of an entry
    auto next = [&](int x) {
      if (x < h) return x == 0 ? 0 : (x < h - 1 ? x + 1 : m - 1);
      return x == h ? 1 : x - 1;
    };
    auto place = [&](int r, int c) {
      const int br = r < h ? r : r - h, bc = c < h ? c : c - h;
      const bool swap = br > bc || (br == bc && r >= h && c < h);
      return swap ? at(c) * ld + at(r) : at(r) * ld + at(c);
    };
    auto angle = [&](float app, float aqq, float apq) {
      float c = 1.0f, sv = 0.0f;
      if (fabsf(apq) > floor_abs && apq * apq > kJ32Rel2 * fabsf(app * aqq)) {
        // half-angle form of the smaller rotation: with r = hypot(d, 2 g),
        // c^2 = (1 + |d| / r) / 2 and s = sign(d) g / (r c)
        const float d = aqq - app, ir = rsqrt_approx(fmaf(d, d, 4.0f * apq * apq));
        const float w = fmaf(0.5f * fabsf(d), ir, 0.5f), ic = rsqrt_approx(w);
        c = w * ic;
        sv = copysignf(apq * ir, d) * (apq < 0.0f ? -ic : ic);
      }
      return make_float2(c, sv);
    };
    // the indices that meet in slot k after a round: their slots and kinds now
    const bool is_angle = tid < nang;
    const int k0 = tid < h ? tid : 0;
    const int tS = k0 == 0 ? 0 : k0 == 1 ? 0 : k0 - 1, qS = k0 == h - 1 ? h - 1 : k0 + 1;
    const bool t_top = k0 != 1, q_top = k0 == h - 1;
    const int lo = tS < qS ? tS : qS, hi = tS < qS ? qS : tS;
    const bool lo_top = tS < qS ? t_top : q_top, hi_top = tS < qS ? q_top : t_top;
    // this thread's blocks: tiles of 4 x 8 blocks that reach above the diagonal,
    // one per warp and k, their 32 blocks over the lanes
    int aI[IA], aJ[IA], at0[IA], ab0[IA], aw[IA][4];
    bool aok[IA];
#pragma unroll
    for (int k = 0; k < IA; ++k) {
      int left = (tid - nang) / 32 + k * ((nA - nang) / 32), ti = 0;
      while (left >= (h + 7) / 8 - ti / 2 && 4 * ti < h) left -= (h + 7) / 8 - ti / 2, ++ti;
      const int I = 4 * ti + ((tid & 31) >> 3), J = 8 * (ti / 2 + left) + (tid & 7);
      aok[k] = !is_angle && I <= J && J < h;
      aI[k] = aok[k] ? I : 0;
      aJ[k] = aok[k] ? J : 0;
      const int tI = next(aI[k]), bI = next(h + aI[k]), tJ = next(aJ[k]), bJ = next(h + aJ[k]);
      at0[k] = aI[k] * ld + aJ[k];
      ab0[k] = (HM + aI[k]) * ld + aJ[k];
      aw[k][0] = place(tI, tJ);
      aw[k][1] = place(tI, bJ);
      aw[k][2] = place(bI, tJ);
      aw[k][3] = place(bI, bJ);
    }
    // rotates the matrix by the angles cs into the other buffer, and computes the
    // next round's angles into cs_next
    auto do_round = [&](auto cur, const float2 *cs, float2 *cs_next) {
      constexpr int CUR = decltype(cur)::value;
      const float *A = Abuf + CUR * C::kA;
      float *B = Abuf + (CUR ^ 1) * C::kA;
      if (is_angle) {
        if (tid < h) {
          // row of the rotation that makes a slot's new top (c, -s) or bottom (s, c)
          const float2 gl = cs[lo], gh = cs[hi];
          const float ul = lo_top ? gl.x : gl.y, vl = lo_top ? -gl.y : gl.x;
          const float uh = hi_top ? gh.x : gh.y, vh = hi_top ? -gh.y : gh.x;
          const float *dl = A + lo * ld + lo, *dh = A + hi * ld + hi, *x = A + lo * ld + hi;
          const float l00 = dl[0], l01 = dl[HM], l11 = dl[HM * ld + HM];
          const float h00 = dh[0], h01 = dh[HM], h11 = dh[HM * ld + HM];
          const float x00 = x[0], x01 = x[HM], x10 = x[HM * ld], x11 = x[HM * ld + HM];
          const float nl = ul * (ul * l00 + vl * l01) + vl * (ul * l01 + vl * l11);
          const float nh = uh * (uh * h00 + vh * h01) + vh * (uh * h01 + vh * h11);
          const float nx = ul * (uh * x00 + vh * x01) + vl * (uh * x10 + vh * x11);
          cs_next[tid] = tS < qS ? angle(nl, nh, nx) : angle(nh, nl, nx);
        }
        bar();
        return;
      }
#pragma unroll
      for (int k = 0; k < IA; ++k)
        if (aok[k]) {
          const bool own = aI[k] == aJ[k];
          const float2 gI = cs[aI[k]], gJ = cs[aJ[k]];
          const float a00 = A[at0[k]], a01 = A[at0[k] + HM], a11 = A[ab0[k] + HM];
          const float a10 = own ? a01 : A[ab0[k]];
          const float b00 = gJ.x * a00 - gJ.y * a01, b01 = gJ.y * a00 + gJ.x * a01;
          const float b10 = gJ.x * a10 - gJ.y * a11, b11 = gJ.y * a10 + gJ.x * a11;
          const float n00 = gI.x * b00 - gI.y * b10, n11 = gI.y * b01 + gI.x * b11;
          float n01 = gI.x * b01 - gI.y * b11, n10 = gI.y * b00 + gI.x * b10;
          // a rotated slot's own coupling is zero; one left alone keeps it
          if (own) n01 = n10 = gI.y != 0.0f ? 0.0f : a01;
          B[aw[k][0]] = n00;
          B[aw[k][1]] = n01;
          B[aw[k][2]] = n10;
          B[aw[k][3]] = n11;
        }
      bar();
    };
    int cur = 0, sweep = 0;
    for (; sweep <= kJ32MaxSweeps; ++sweep) {
      // a sweep that would find nothing to rotate is not run
      float2 *cs = ring + (sweep & 1) * C::kSweep;
      if (tid == 0) s_rot[sweep & 1] = 0;
      bar();
      if (sweep < kJ32MaxSweeps) {
        const float *A = Abuf + cur * C::kA;
        bool any = false;
#pragma unroll
        for (int k = 0; k < IA; ++k)
          if (aok[k]) {
            const int I = aI[k], J = aJ[k];
            const float dI[2] = {A[I * ld + I], A[(HM + I) * ld + HM + I]};
            const float dJ[2] = {A[J * ld + J], A[(HM + J) * ld + HM + J]};
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
              for (int b = 0; b < 2; ++b) {
                if (I == J && !(a == 0 && b == 1)) continue;
                const float v = A[(a ? ab0[k] : at0[k]) + b * HM];
                any = any || (fabsf(v) > floor_abs && v * v > kJ32Rel2 * fabsf(dI[a] * dJ[b]));
              }
          }
        if (any) s_rot[sweep & 1] = 1;
      }
      __syncthreads();     // the last sweep's angles are ready; V has used up those of the one before
      if (!s_rot[sweep & 1]) break;
      if (tid < h) {
        const float *A = Abuf + cur * C::kA;
        cs[tid] = angle(A[tid * ld + tid], A[(HM + tid) * ld + HM + tid], A[tid * ld + HM + tid]);
      }
      bar();
      for (int r = 0; r < m - 1; ++r, cs += C::kRound) {
        // the last round's successor is the next sweep's first: computed there
        float2 *nx = r < m - 2 ? cs + C::kRound : spare;
        if (cur == 0) do_round(std::integral_constant<int, 0>{}, cs, nx);
        else do_round(std::integral_constant<int, 1>{}, cs, nx);
        cur ^= 1;
      }
    }
    if (tid == 0) atomicMax(sweeps, sweep);
  } else {
    // ---- V: RPG rows per group of 16 lanes, slots SPL l .. SPL l + SPL - 1 of a row in lane l
    const int l = tid & 15, row0 = (tid - nA) / 16 * RPG;
    float t[RPG][SPL], b[RPG][SPL];
    bool last[SPL];
#pragma unroll
    for (int q = 0; q < SPL; ++q) {
      const int sl = l * SPL + q;
      last[q] = sl == h - 1;
#pragma unroll
      for (int r = 0; r < RPG; ++r) {
        t[r][q] = row0 + r == sl ? 1.0f : 0.0f;
        b[r][q] = row0 + r == h + sl ? 1.0f : 0.0f;
      }
    }
    const bool l0 = l == 0;
    for (int sweep = 0;; ++sweep) {
      __syncthreads();
      const bool more = s_rot[sweep & 1] != 0;
      if (sweep > 0) {
        const float2 *cs = ring + ((sweep - 1) & 1) * C::kSweep + l * SPL;
        float2 g[SPL];
#pragma unroll
        for (int q = 0; q < SPL; ++q) g[q] = cs[q];
        for (int r = 0; r < m - 1; ++r) {
          float2 gn[SPL];
          cs += r < m - 2 ? C::kRound : 0;          // the next round's angles, ahead of their use
#pragma unroll
          for (int q = 0; q < SPL; ++q) gn[q] = cs[q];
#pragma unroll
          for (int i = 0; i < RPG; ++i) {
#pragma unroll
            for (int q = 0; q < SPL; ++q) {
              const float x = t[i][q], y = b[i][q];
              t[i][q] = g[q].x * x - g[q].y * y;
              b[i][q] = g[q].y * x + g[q].x * y;
            }
            // tops one slot up (slot 0's stays, slot 0's bottom follows into slot 1),
            // bottoms one slot down (the last top turns round)
            const float up = __shfl_up_sync(0xffffffffu, SPL == 1 && l0 ? b[i][0] : t[i][SPL - 1], 1, 16);
            const float dn = __shfl_down_sync(0xffffffffu, b[i][0], 1, 16);
            float nt[SPL], nb[SPL];
#pragma unroll
            for (int q = 0; q < SPL; ++q) {
              nt[q] = q == 0 ? (l0 ? t[i][0] : up) : (q == 1 && l0 ? b[i][0] : t[i][q > 0 ? q - 1 : 0]);
              nb[q] = last[q] ? t[i][q] : q == SPL - 1 ? dn : b[i][q < SPL - 1 ? q + 1 : q];
            }
#pragma unroll
            for (int q = 0; q < SPL; ++q) {
              t[i][q] = nt[q];
              b[i][q] = nb[q];
            }
          }
#pragma unroll
          for (int q = 0; q < SPL; ++q) g[q] = gn[q];
        }
      }
      if (!more) break;
    }
    double *out = Vout.at(z);
#pragma unroll
    for (int i = 0; i < RPG; ++i)
#pragma unroll
      for (int q = 0; q < SPL; ++q) {
        const int sl = l * SPL + q, row = row0 + i;
        if (row < m && sl < h) {
          out[row + (size_t)sl * m] = to_f64(t[i][q]);             // out[j + c m] = V[j][c]
          out[row + (size_t)(h + sl) * m] = to_f64(b[i][q]);
        }
      }
  }
}

// ---- FP64 m x m products -------------------------------------------------------

constexpr double kSfsCluster = 1e3;   // a pair is separated if |gap| > kSfsCluster |coupling|

// Out = op(A) B' with op(A) = A^T if ta, and B' = bs B + bd I, or (refine) I + E
// of the refinement pass built from S and G while the tile is staged.  Output
// truncated to rows x cols, column-major with ld = rows.
struct MmOp {
  PSet A, B, S, G, Out;
  int ta, refine;        // refine: 1, or 2 where A's columns still have to be normalised
  int sym;               // the product is symmetric: only its upper tiles are computed, and mirrored
  double bs, bd;
  int rows, cols;
};

// One or two products of every problem (blockIdx.z = op P + problem), one CTA
// per 8 x 8 output tile; the sum over k is split four ways across the CTA's
// threads and combined in a fixed order.  At m = 48 a tile is 1536 FP64 FMA
// cycles of one SM, about the launch's own latency: smaller tiles would only
// re-read more, larger ones leave SMs idle.
__global__ void __launch_bounds__(256) k_se_mm(MmOp op0, MmOp op1, int P, int m, float noise) {
  pdl_enter();
  __shared__ double As[8][kSiMaxBlock + 1];   // op(A) rows i0..i0+7, all k
  __shared__ double Bs[8][kSiMaxBlock + 1];   // B' columns j0..j0+7, all k
  __shared__ double part[4][8][9];
  __shared__ double lam[kSiMaxBlock], rn[kSiMaxBlock];
  __shared__ unsigned s_mx;
  const bool second = (int)blockIdx.z >= P;
  const MmOp &o = second ? op1 : op0;
  const int z = second ? (int)blockIdx.z - P : (int)blockIdx.z;
  const int i0 = blockIdx.x * 8, j0 = blockIdx.y * 8;
  if (i0 >= o.rows || j0 >= o.cols || (o.sym && i0 > j0)) return;
  const double *a = o.A.at(z);
  if (o.ta) {
    for (int e = threadIdx.x; e < 8 * m; e += blockDim.x) {
      const int r = e / m, k = e % m, i = i0 + r;
      As[r][k] = (i < m) ? a[(size_t)i * m + k] : 0.0;
    }
  } else {
    for (int e = threadIdx.x; e < 8 * m; e += blockDim.x) {
      const int r = e & 7, k = e >> 3, i = i0 + r;
      As[r][k] = (i < m) ? a[(size_t)k * m + i] : 0.0;
    }
  }
  if (!o.refine) {
    const double *b = o.B.at(z);
    for (int e = threadIdx.x; e < 8 * m; e += blockDim.x) {
      const int r = e / m, k = e % m, j = j0 + r;
      Bs[r][k] = (j < m) ? o.bs * b[(size_t)j * m + k] + (k == j ? o.bd : 0.0) : 0.0;
    }
  } else {
    const double *S = o.S.at(z), *G = o.G.at(z);
    // lambda = s / g to first order in g - 1 (V is orthonormal to 1e-5 or better)
    // or exactly, for columns of any length: then A diag(rn) is what is refined
    const bool norm = o.refine == 2;
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
      const double s = S[(size_t)k * m + k], g = G[(size_t)k * m + k];
      if (norm) {
        const double r = g > 0.0 ? rsqrt_fp64(g) : 1.0;
        rn[k] = r;
        lam[k] = s * r * r;
      } else {
        lam[k] = s * (2.0 - g);
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      unsigned v = 0;
      for (int k = threadIdx.x; k < m; k += 32) v = max(v, abs_hi(lam[k]));
      v = warp_max(v);
      if (threadIdx.x == 0) s_mx = v;
    }
    __syncthreads();
    const int bias = scale_bias(s_mx);
    const float fl = noise * mag32(s_mx, 0, bias);
    for (int e = threadIdx.x; e < 8 * m; e += blockDim.x) {
      const int r = e / m, k = e % m, j = j0 + r;
      double v = 0.0;
      if (j < m) {
        double g = G[(size_t)j * m + k];
        if (k == j) {
          v = norm ? rn[k] : 1.5 - 0.5 * g;                   // 1 + (1 - g) / 2
        } else {
          double s = S[(size_t)j * m + k];
          if (norm) {
            const double w = rn[k] * rn[j];
            g *= w;
            s *= w;
          }
          const double gap = lam[j] - lam[k];
          const double num = fma(-lam[j], g, s);
          const float off = mag32(fma(0.5 * gap, g, num), bias);    // s - (lam_j + lam_k) g / 2
          // the quotient needs FP32 accuracy only: what it misses is of the
          // order of 1e-7 of a coupling that the next pass sees
          if (mag32(gap, bias) > (float)kSfsCluster * off && off > fl)
            v = to_f64(to_f32(num, bias) / to_f32(gap, bias));
          else v = -0.5 * g;
          if (norm) v *= rn[k];
        }
      }
      Bs[r][k] = v;
    }
  }
  __syncthreads();
  const int ti = threadIdx.x & 7, tj = (threadIdx.x >> 3) & 7, ks = threadIdx.x >> 6;
  double acc = 0.0;
  for (int k = ks; k < m; k += 4) acc = fma(As[ti][k], Bs[tj][k], acc);
  part[ks][ti][tj] = acc;
  __syncthreads();
  if (threadIdx.x < 64) {
    const int i = i0 + ti, j = j0 + tj;
    if (i < o.rows && j < o.cols) {
      const double v = (part[0][ti][tj] + part[1][ti][tj]) + (part[2][ti][tj] + part[3][ti][tj]);
      o.Out.at(z)[(size_t)j * o.rows + i] = v;
      if (o.sym && i0 != j0) o.Out.at(z)[(size_t)i * o.rows + j] = v;
    }
  }
}

// ---- stage 4: rotations that are still needed ----------------------------------

// Classical-order ("largest first") two-sided Jacobi on the nearly diagonal
// symmetric m x m matrix Hin (one CTA per problem): each round, every row
// finds the partner with the largest entry that needs rotating (above
// 2^-floor_exp of the largest diagonal entry and not negligible against its
// own diagonal pair), the mutually largest pairs -- disjoint by construction,
// and always including the largest entry of the matrix -- are rotated at once
// (Eq. 6), and the accumulated rotation W follows.  Stops when nothing needs
// rotating; *rounds receives the round count (maximum over problems), flag is
// set to 2, and *err (if given) raised to kErrEig, if max_rounds do not suffice.  Eigenvalues descending
// in theta, Wout columns in the same order.  The search compares FP32
// magnitudes taken from the bits (an FP64 comparison of every entry would cost
// more than the rotations: m^2 of them at two per clock).
constexpr int kSparseRounds = 32;
constexpr int kSparseThreads = 1024;

// Rounds before a solve is given up: many times what any matrix has been seen to
// take.  The bounds-checked build lets a test lower them.
int sparse_rounds(int m) {
  if constexpr (kChecked)
    if (const char *v = getenv("HOTRG_TEST_SPARSE_ROUNDS")) return atoi(v);
  return kSparseRounds * m;
}

size_t sparse_smem(int m) {
  return (size_t)2 * m * (m + 1) * sizeof(double) + (size_t)m * (sizeof(int) + sizeof(float)) +
         (size_t)(m / 2 + 1) * (2 * sizeof(int) + 2 * sizeof(double)) + 64;
}

__global__ void __launch_bounds__(kSparseThreads, 1)
    k_rr_sparse_jacobi(PSet Hin, int m, int floor_exp, int max_rounds, PSet Wout, PSet theta, int *flag, int *err,
                       int *rounds_out) {
  pdl_enter();
  extern __shared__ double ssh[];
  const int ld = m + 1, maxsel = m / 2 + 1;
  double *H = ssh;                                  // row-major, symmetric part of Hin
  double *W = H + (size_t)m * ld;                   // W[r * ld + c]
  double *sc = W + (size_t)m * ld;                  // rotation c of selected pair k
  double *ss = sc + maxsel;                         // rotation s
  int *best = reinterpret_cast<int *>(ss + maxsel); // per row: partner with the largest entry, -1
  int *selp = best + m, *selq = selp + maxsel;
  float *rt = reinterpret_cast<float *>(selq + maxsel);   // sqrt|h_pp|
  __shared__ int nsel;
  const int z = blockIdx.z;
  const double *hin = Hin.at(z);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
    const int r = e % m, c = e / m;                 // column-major input: coalesced reads
    H[r * ld + c] = 0.5 * (hin[(size_t)c * m + r] + hin[(size_t)r * m + c]);
    W[r * ld + c] = r == c ? 1.0 : 0.0;
  }
  __syncthreads();
  unsigned mx = 0;                                  // every warp on its own: no barrier
  for (int i = lane; i < m; i += 32) mx = max(mx, abs_hi(H[i * ld + i]));
  mx = warp_max(mx);
  const int bias = scale_bias(mx);
  const float fl = ldexpf(mag32(mx, 0, bias), -floor_exp);
  int round = 0;
  bool done = false;
  for (; round < max_rounds; ++round) {
    for (int p = threadIdx.x; p < m; p += blockDim.x) rt[p] = sqrtf(mag32(H[p * ld + p], bias));
    if (threadIdx.x == 0) nsel = 0;
    __syncthreads();
    // (1) each row's best partner (one warp per row); rows p and q both read the
    // entry above the diagonal, so they agree on it
    for (int p = warp; p < m; p += nwarps) {
      float bv = 0.0f;
      int bq = -1;
      const float rp = 1e-15f * rt[p];
      for (int q = lane; q < m; q += 32) {
        const float hv = mag32(q > p ? H[p * ld + q] : H[q * ld + p], bias);
        if (q != p && hv > fl && hv > rp * rt[q] && hv > bv) {
          bv = hv;
          bq = q;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oq = __shfl_xor_sync(0xffffffffu, bq, o);
        if (ov > bv || (ov == bv && oq > bq)) {
          bv = ov;
          bq = oq;
        }
      }
      if (lane == 0) best[p] = bq;
    }
    __syncthreads();
    // (2) mutually best pairs, their angles
    for (int p = threadIdx.x; p < m; p += blockDim.x) {
      const int q = best[p];
      if (q > p && best[q] == p) {
        const int k = atomicAdd(&nsel, 1);
        double c, sv;
        jacobi_angle(H[p * ld + p], H[q * ld + q], H[p * ld + q], c, sv);
        selp[k] = p;
        selq[k] = q;
        sc[k] = c;
        ss[k] = sv;
      }
    }
    __syncthreads();
    const int ns = nsel;
    if (ns == 0) {
      done = true;
      break;
    }
    // (3) right factor: columns p, q of H and W
    for (int e = threadIdx.x; e < ns * m; e += blockDim.x) {
      const int k = e / m, r = e % m, p = selp[k], q = selq[k];
      const double c = sc[k], sv = ss[k];
      const double x = H[r * ld + p], y = H[r * ld + q];
      H[r * ld + p] = c * x - sv * y;
      H[r * ld + q] = sv * x + c * y;
      const double wx = W[r * ld + p], wy = W[r * ld + q];
      W[r * ld + p] = c * wx - sv * wy;
      W[r * ld + q] = sv * wx + c * wy;
    }
    __syncthreads();
    // (4) left factor: rows p, q; the rotated pair's own entries are zero
    for (int e = threadIdx.x; e < ns * m; e += blockDim.x) {
      const int k = e / m, col = e % m, p = selp[k], q = selq[k];
      const double c = sc[k], sv = ss[k];
      const double x = H[p * ld + col], y = H[q * ld + col];
      H[p * ld + col] = (col == q) ? 0.0 : c * x - sv * y;
      H[q * ld + col] = (col == p) ? 0.0 : sv * x + c * y;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (!done) {
      atomicExch(flag, 2);
      if (err) atomicMax(err, kErrEig);
    }
    atomicMax(rounds_out, round);
  }
  // sort descending (rank of each diagonal entry, ties by index); best[] now
  // holds the column of each rank
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const double ti = H[i * ld + i];
    int rk = 0;
    for (int j = 0; j < m; ++j) {
      const double tj = H[j * ld + j];
      rk += (tj > ti) || (tj == ti && j < i);
    }
    theta.at(z)[rk] = ti;
    best[rk] = i;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
    const int row = e % m, rk = e / m;
    Wout.at(z)[e] = W[row * ld + best[rk]];
  }
}

__global__ void k_eig_one(PSet G, PSet X, PSet theta, int m, int P) {
  pdl_enter();
  const int z = blockIdx.x * blockDim.x + threadIdx.x;
  if (z >= P) return;
  X.at(z)[0] = 1.0;
  theta.at(z)[0] = G.at(z)[0];
  for (int i = 1; i < m; ++i) theta.at(z)[i] = 0.0;
}

template <int HM, int SPL, int RPG, int IA>
cudaError_t run_j32(PSet H, int m, float floor_abs, PSet V, int *sweeps, int P, cudaStream_t s) {
  const auto kern = k_rr_jacobi32<HM, SPL, RPG, IA>;
  static SmemLimit limit;
  if (cudaError_t e = limit.raise(reinterpret_cast<const void *>(kern), (int)J32Cfg<HM, SPL>::kSmem)) return e;
  // threads of the angles, of the matrix (4 x 8 blocks per warp, IA of them in turn) and of V
  const int h = m / 2, nang = (h + 31) / 32 * 32;
  int tiles = 0;
  for (int ti = 0; 4 * ti < h; ++ti) tiles += (h + 7) / 8 - ti / 2;
  const int nA = nang + (tiles + IA - 1) / IA * 32;
  const int nV = ((m + RPG - 1) / RPG + 1) / 2 * 32;
  const size_t smem = J32Cfg<HM, SPL>::kSmem;
  launch_pdl(kern, dim3(1, 1, P), nA + nV, smem, s, H, m, floor_abs, nang, nA, V, sweeps);
  return cudaGetLastError();
}

cudaError_t launch_j32(PSet H, int m, float floor_abs, PSet V, int *sweeps, int P, cudaStream_t s) {
  if (m <= 32) return run_j32<16, 1, 2, 1>(H, m, floor_abs, V, sweeps, P, s);
  if (m <= 48) return run_j32<24, 2, 3, 1>(H, m, floor_abs, V, sweeps, P, s);
  if (m <= 64) return run_j32<32, 2, 3, 1>(H, m, floor_abs, V, sweeps, P, s);
  return run_j32<48, 3, 5, 3>(H, m, floor_abs, V, sweeps, P, s);
}

cudaError_t small_attrs() {
  static SmemLimit limit;
  return limit.raise(reinterpret_cast<const void *>(k_rr_sparse_jacobi), 200 * 1024);
}

}  // namespace

cudaError_t small_eig(const SmallEig &a, cudaStream_t s, long long *launches) {
  cudaError_t e = small_attrs();
  if (e) return e;
  const int P = a.P, m = a.m;
  if (m < 4 || (m & 1) || m > kSiMaxBlock || P < 1 || P > 65535) return cudaErrorInvalidValue;
  const long long mm = (long long)m * m;
  auto slot = [&](int i) { return PSet{a.scratch.b0 + i * mm, a.scratch.b1 + i * mm, a.scratch.stride}; };
  PSet X = slot(0), Xn = slot(1);
  const PSet Y = slot(2), G = slot(3), S = slot(4), V = slot(5), W = slot(6);
  // couplings below this share of the largest eigenvalue are rounding of the
  // products (full: of H itself), and are left alone
  const int floor_exp = a.full ? 51 : 44;
  const float noise = ldexpf(1.0f, -(floor_exp + 1));
  const int t = (m + 7) / 8;
  auto op = [&](PSet A, int ta, PSet B, double bs, double bd, PSet Out) {
    return MmOp{A, B, B, B, Out, ta, 0, 0, bs, bd, m, m};
  };
  auto sym = [&](PSet A, PSet B, PSet Out) { return MmOp{A, B, B, B, Out, 1, 0, 1, 1.0, 0.0, m, m}; };   // A^T B
  auto mm1 = [&](const MmOp &o) {
    launch_pdl(k_se_mm, dim3(t, t, P), 256, 0, s, o, o, P, m, noise);
    *launches += 1;
  };
  auto mm2 = [&](const MmOp &o, const MmOp &q) {
    if (2 * P > 65535) {              // grid.z holds both products of every problem
      mm1(o);
      mm1(q);
      return;
    }
    launch_pdl(k_se_mm, dim3(t, t, 2 * P), 256, 0, s, o, q, P, m, noise);
    *launches += 1;
  };
  // H is symmetric: H^T Y is read along its rows
  auto refine = [&](int kind) {
    mm2(sym(X, X, G), op(a.H, 1, X, 1.0, 0.0, Y));
    mm1(sym(X, Y, S));
    mm1(MmOp{X, X, S, G, Xn, 0, kind, 0, 1.0, 0.0, m, m});
    std::swap(X, Xn);
  };
  auto newton_schulz = [&]() {
    mm1(sym(X, X, G));
    mm1(op(X, 0, G, -0.5, 1.5, Xn));
    std::swap(X, Xn);
  };
  const bool lr = a.full && a.graded && m >= kLrMinSize;
  if (lr) {
    // L^T L in place of H = L L^T (see the file comment)
    if ((e = lr_factor(a.H, m, Y, G, P, s, launches))) return e;
    mm1(sym(Y, G, S));
    if ((e = launch_j32(S, m, kLrFloor, V, a.sweeps, P, s))) return e;
    mm1(op(Y, 0, V, 1.0, 0.0, X));
    refine(2);
    newton_schulz();
    mm1(op(a.H, 1, X, 1.0, 0.0, Y));
    mm1(sym(X, Y, S));
    if ((e = launch_j32(S, m, ldexpf(1.0f, -56), V, a.sweeps, P, s))) return e;
    mm1(op(X, 0, V, 1.0, 0.0, Xn));
    std::swap(X, Xn);
    *launches += 2;
  } else if (a.full) {
    // a dense H: the first FP32 pass stops at its rounding (2^-24), the second
    // one resolves what lies below; a graded H is resolved by the first
    if ((e = launch_j32(a.H, m, ldexpf(1.0f, a.graded ? -56 : -24), X, a.sweeps, P, s))) return e;
    mm1(sym(X, X, G));
    mm1(op(X, 0, G, -0.5, 1.5, Xn));
    mm1(op(a.H, 1, Xn, 1.0, 0.0, Y));
    mm1(sym(Xn, Y, S));
    if ((e = launch_j32(S, m, ldexpf(1.0f, -56), V, a.sweeps, P, s))) return e;
    mm1(op(Xn, 0, V, 1.0, 0.0, X));
    *launches += 2;
  } else {
    // pairs are resolved down to 2^-46 of the largest eigenvalue here (entries
    // between small diagonal entries keep FP32 relative accuracy): stopping at
    // 2^-30 costs no fewer sweeps and left hundreds of rotations to the last stage
    if ((e = launch_j32(a.H, m, ldexpf(1.0f, -46), X, a.sweeps, P, s))) return e;
    *launches += 1;
  }
  refine(1);
  if (!lr) refine(1);
  // orthonormal to rounding: barely separated pairs take E up to 1 / kSfsCluster,
  // whose square is what a pass leaves
  newton_schulz();
  newton_schulz();
  mm1(op(a.H, 1, X, 1.0, 0.0, Y));
  mm1(sym(X, Y, S));
  launch_pdl(k_rr_sparse_jacobi, dim3(1, 1, P), kSparseThreads, sparse_smem(m), s, S, m, floor_exp, sparse_rounds(m), W,
             a.theta, a.flag, a.err, a.rounds);
  *launches += 1;
  mm1(MmOp{X, W, W, W, a.out, 0, 0, 0, 1.0, 0.0, a.rows, a.cols});
  return cudaGetLastError();
}

cudaError_t eig_one(PSet G, PSet X, PSet theta, int m, int P, cudaStream_t s, long long *launches) {
  launch_pdl(k_eig_one, (P + 127) / 128, 128, 0, s, G, X, theta, m, P);
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace hotrg
