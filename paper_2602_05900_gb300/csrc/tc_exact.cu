// Exact-slice GEMM kernels (see tc_exact.cuh).
//
// k_xs_split*  one warp or one block per row: row max, power-of-two scale, S
//              digits, in integer arithmetic.
// k_xs_gemm    one CTA per 128 x BN output tile and K part; the parts of a tile
//              form a cluster:
//   warp 0 / lane 0   TMA producer: the S slices of A and of B of a K block in
//                     two copies (the slice index is a dimension of the box)
//                     into a shared-memory ring;
//   warp 1 / lane 0   MMA issuer: the slices of B lie behind each other in
//                     shared memory, so slice s of A times several slices
//                     t, t + 1, ... of B is one MMA with N = BN per slice whose
//                     columns fall on the accumulators d = s + t, s + t + 1, ...
//                     (tensor memory, BN columns each);
//   all warps         epilogue: accumulators -> one 64-bit integer per output
//                     in shared memory, summed over the cluster's K parts
//                     (exactly, in any order), converted and scaled once.
//
// Why this shape (GB300, 36 digit products at S = 8): an MMA with N = 48 reads
// its A slice (4 KB) from shared memory for 24 cycles of arithmetic, so one MMA
// per digit product is bound by those reads; with the slices of B stacked 11
// MMAs do the work of 36.  The epilogue used to do five FP32 -> int64
// conversions and four FP64 operations per output and K part at two FP64
// operations per clock and SM; now it adds a magic number per accumulator
// (or, for long K parts, converts to 32 bits) and converts once per output.
// Measured (kernel times with a cold L2): G X at n = 1024, m = 48, two problems
// 45.8 -> 30.3 us with the K-part sum included (5.8 us in a pass of its own
// before); n = 2304, m = 64 111 -> 48 us; slicing 96 rows of 1024 11.5 -> 6.5 us;
// hotrg_dgemm_emu of 3001 x 2777 x 3203 3.73 -> 2.28 ms (1.72 ms with its scratch from
// the memory pool).
// Waits are bounded as in the other tcgen05 kernels: on timeout the kernel sets
// *err_flag, lets its own TMA copies land, frees tensor memory and returns.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "tc_exact.cuh"
#include "kernel_attr.cuh"
#include "launch.cuh"
#include "tcgen05.cuh"

namespace cg = cooperative_groups;

namespace hotrg {
namespace {

using namespace tc;

constexpr int kXsThreads = 256;
constexpr int kXsUnit = 50;           // results are summed as integers in units of 2^-50
// Longest K part whose digit sums stay below 2^22 (ten units of 2^10 per k at
// most: eight digit pairs, two of them with the top digit), so that adding
// 1.5 2^23 units leaves the integer in the mantissa.
constexpr int kXsMagicK = 408;

template <int S, int BN>
struct XsCfg {
  // K block: 32 BF16 (64-byte rows, 64-byte swizzle) while two such stages of
  // all slices fit in shared memory, else 16 BF16 (32-byte rows and swizzle)
  static constexpr int BM = 128;
  static constexpr int ROW = (2 * S * (BM + BN) * 64 <= 200 * 1024) ? 64 : 32;
  static constexpr int BK = ROW / 2;
  static constexpr int A_BYTES = BM * ROW, B_BYTES = BN * ROW;
  static constexpr int STAGE_BYTES = S * (A_BYTES + B_BYTES);
  static constexpr int STAGES_RAW = (200 * 1024) / STAGE_BYTES;
  static constexpr int STAGES = STAGES_RAW > 4 ? 4 : STAGES_RAW;
  static constexpr int OUT_BYTES = BM * (BN + 1) * 8;      // integer outputs, after the main loop
  static constexpr int SMEM = (STAGES * STAGE_BYTES > OUT_BYTES ? STAGES * STAGE_BYTES : OUT_BYTES) + 1024;
  static constexpr int STACK = 256 / BN;                    // slices of B in one MMA
  static constexpr int COLS_RAW = S * BN;
  static constexpr int TMEM_COLS = COLS_RAW <= 128 ? 128 : COLS_RAW <= 256 ? 256 : 512;
  static_assert(STAGES >= 2, "pipeline needs two stages");
  static_assert(COLS_RAW <= 512, "accumulators exceed tensor memory");
  static_assert(BN % 16 == 0 && BN >= 32 && BN <= 96, "BN");
};

struct XsOut {
  double *C;
  IdxMap cm, cn;
  long long cstride, pstride;
  const double *sa, *sb;
  long long ssa, ssb;
  int rowmajor;          // lanes run along columns (unit column stride), else along rows
  XsShift shift;
};

// ---- slicing ------------------------------------------------------------------
//
// The row maximum is taken on the bit patterns (|x| of a double orders like its
// bits as an unsigned integer), the scaled row is rounded once (to nearest even)
// to a 6S-bit fixed-point integer N, and its digits are those of
// N + 32 (1 + 64 + ... + 64^(S-2)) less 32 each: d_S..d_2 in [-32, 31], then the
// top digit d_1 = what is left, |d_1| <= 64 because |row| < 2^e.  All in integer
// arithmetic and FP32: GB300's FP64 units would take a clock per element and SM.

// x 2^(6S - e) rounded to an integer, |x| < 2^e
template <int S>
__device__ __forceinline__ long long xs_fixed(double x, int e) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
  const int ef = (int)(bits >> 52) & 0x7FF;
  const unsigned long long mant = (bits & 0xFFFFFFFFFFFFFull) | (ef ? 1ull << 52 : 0ull);
  const int sh = 1075 - (ef ? ef : 1) - kXsBits * S + e;     // >= 53 - 6S >= 5 but for subnormal rows
  if (sh > 54) return 0;
  if (sh <= 0) return (long long)bits < 0 ? -(long long)(mant << -sh) : (long long)(mant << -sh);
  const unsigned long long half = (1ull << (sh - 1)) - 1;
  const long long n = static_cast<long long>((mant + half + ((mant >> sh) & 1)) >> sh);
  return (long long)bits < 0 ? -n : n;
}

// digits of two neighbouring elements k, k + 1 (k even) of a row, one 32-bit
// store per plane
template <int S>
__device__ __forceinline__ void xs_store2(__nv_bfloat16 *out, long long plane, int k, long long N0,
                                          long long N1) {
  constexpr long long kBias = 32ll * (((1ll << (kXsBits * (S - 1))) - 1) / 63);
  const unsigned long long M0 = static_cast<unsigned long long>(N0 + kBias);
  const unsigned long long M1 = static_cast<unsigned long long>(N1 + kBias);
#pragma unroll
  for (int p = 0; p < S; ++p) {
    const float unit = 1.0f / (float)(1ull << (kXsBits * (p + 1)));
    float f0, f1;
    if (p == 0) {
      f0 = (float)(int)((long long)M0 >> (kXsBits * (S - 1))) * unit;
      f1 = (float)(int)((long long)M1 >> (kXsBits * (S - 1))) * unit;
    } else {
      // (2^23 + u) unit - (2^23 + 32) unit, exact
      const int j = S - 1 - p;
      const unsigned u0 = (unsigned)(M0 >> (kXsBits * j)) & 63u, u1 = (unsigned)(M1 >> (kXsBits * j)) & 63u;
      f0 = fmaf(__uint_as_float(0x4B000000u | u0), unit, -8388640.0f * unit);
      f1 = fmaf(__uint_as_float(0x4B000000u | u1), unit, -8388640.0f * unit);
    }
    // digits fit a BF16: the upper halves of the FP32 patterns
    *reinterpret_cast<unsigned *>(out + p * plane + k) =
        __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
  }
}

constexpr unsigned long long kXsAbs = 0x7FFFFFFFFFFFFFFFull, kXsInf = 0x7FF0000000000000ull;
__device__ __forceinline__ unsigned long long xs_mag(double x) {
  const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(x)) & kXsAbs;
  return u > kXsInf ? kXsInf : u;                           // NaN poisons the row like +inf
}

// Slices one row with nt threads (thread t); elem(k) reads an element, reduce
// combines the threads' maxima.  The first 8 nt elements stay in registers.
template <int S, class Elem, class Reduce>
__device__ __forceinline__ void xs_slice_row(Elem elem, Reduce reduce, int K, int t, int nt,
                                             __nv_bfloat16 *out, long long plane, double *scale) {
  constexpr int CH = 4;
  double v[2 * CH];
  unsigned long long mb = 0;
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int k = 2 * (t + c * nt);
    v[2 * c] = k < K ? elem(k) : 0.0;
    v[2 * c + 1] = k + 1 < K ? elem(k + 1) : 0.0;
    const unsigned long long a = xs_mag(v[2 * c]), b = xs_mag(v[2 * c + 1]);
    mb = a > mb ? a : mb;
    mb = b > mb ? b : mb;
  }
  for (int k = 2 * CH * nt + t; k < K; k += nt) {
    const unsigned long long a = xs_mag(elem(k));
    mb = a > mb ? a : mb;
  }
  mb = reduce(mb);
  const bool finite = mb < kXsInf;
  int e = 0;
  if (finite && mb != 0) (void)frexp(__longlong_as_double(static_cast<long long>(mb)), &e);   // max < 2^e
  if (t == 0) *scale = finite ? ldexp(1.0, e) : NAN;
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int k = 2 * (t + c * nt);
    if (k < K)
      xs_store2<S>(out, plane, k, finite ? xs_fixed<S>(v[2 * c], e) : 0,
                   finite ? xs_fixed<S>(v[2 * c + 1], e) : 0);
  }
  for (int k = 2 * (t + CH * nt); k < K; k += 2 * nt) {
    const double a = elem(k), b = k + 1 < K ? elem(k + 1) : 0.0;
    xs_store2<S>(out, plane, k, finite ? xs_fixed<S>(a, e) : 0, finite ? xs_fixed<S>(b, e) : 0);
  }
}

__device__ __forceinline__ unsigned long long xs_warp_max(unsigned long long mb) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, mb, o);
    mb = t > mb ? t : mb;
  }
  return mb;
}

// element k of a row, with the optional power-of-two column factor
__device__ __forceinline__ double xs_elem(const double *a, long long ro, const IdxMap &km, const double *ks,
                                          int kmode, int k) {
  const double v = a[ro + map_off32(km, k)];
  if (kmode == 1) return v * ks[k];
  if (kmode == 2) return v / ks[k];
  return v;
}

// one warp per row
template <int S>
__global__ void __launch_bounds__(256) k_xs_split(PSet src, int R, int K, IdxMap rm, IdxMap km,
                                                  __nv_bfloat16 *dst, int pitch, long long bstride,
                                                  double *scale, long long sstride, PSet kscale,
                                                  int kmode) {
  pdl_enter();
  const int z = blockIdx.z;
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= R) return;
  const double *a = src.at(z), *ks = kmode ? kscale.at(z) : nullptr;
  const long long ro = map_off32(rm, r);
  xs_slice_row<S>([&](int k) { return xs_elem(a, ro, km, ks, kmode, k); }, xs_warp_max, K, lane, 32,
                  dst + z * bstride + (long long)r * pitch, (long long)R * pitch, scale + z * sstride + r);
}

// One 128-thread block per row, for long rows (K >= 256): the warp-per-row
// kernel leaves most of the GPU idle when there are few rows (the n-long columns
// of a basis: 2m rows) and walks each row serially.  Same digits.
constexpr int kXsRowThreads = 128;
template <int S>
__global__ void __launch_bounds__(kXsRowThreads) k_xs_split_row(PSet src, int R, int K, IdxMap rm, IdxMap km,
                                                                __nv_bfloat16 *dst, int pitch,
                                                                long long bstride, double *scale,
                                                                long long sstride, PSet kscale, int kmode) {
  pdl_enter();
  const int z = blockIdx.z, r = blockIdx.x;
  const double *a = src.at(z), *ks = kmode ? kscale.at(z) : nullptr;
  const long long ro = map_off32(rm, r);
  __shared__ unsigned long long part[kXsRowThreads / 32];
  auto reduce = [&](unsigned long long mb) {
    mb = xs_warp_max(mb);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = mb;
    __syncthreads();
    mb = 0;
#pragma unroll
    for (int w = 0; w < kXsRowThreads / 32; ++w) mb = part[w] > mb ? part[w] : mb;
    return mb;
  };
  xs_slice_row<S>([&](int k) { return xs_elem(a, ro, km, ks, kmode, k); }, reduce, K, threadIdx.x, kXsRowThreads,
                  dst + z * bstride + (long long)r * pitch, (long long)R * pitch, scale + z * sstride + r);
}

// The same slicing for operands whose rows are contiguous but whose K index is
// strided (the basis of a rotation X W, column-major X as the A operand): a
// block stages 32 rows x K (K <= kXsStagedK) through shared memory with loads
// that run along the rows, then each warp slices its rows along K as above.
template <int S>
__global__ void __launch_bounds__(256) k_xs_split_staged(PSet src, int R, int K, IdxMap rm,
                                                         IdxMap km, __nv_bfloat16 *dst, int pitch,
                                                         long long bstride, double *scale,
                                                         long long sstride, PSet kscale, int kmode) {
  pdl_enter();
  __shared__ double tile[32][kXsStagedK + 1];
  const int z = blockIdx.z;
  const int r0 = blockIdx.x * 32;
  const double *a = src.at(z), *ks = kmode ? kscale.at(z) : nullptr;
  // load: thread t reads row r0 + (t & 31) of column k = t / 32, + 8 per pass
  for (int e = threadIdx.x; e < 32 * K; e += blockDim.x) {
    const int rl = e & 31, k = e >> 5, r = r0 + rl;
    tile[rl][k] = r < R ? xs_elem(a, map_off32(rm, r), km, ks, kmode, k) : 0.0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int rl = threadIdx.x >> 5; rl < 32; rl += blockDim.x >> 5) {
    const int r = r0 + rl;
    if (r >= R) break;
    xs_slice_row<S>([&](int k) { return tile[rl][k]; }, xs_warp_max, K, lane, 32,
                    dst + z * bstride + (long long)r * pitch, (long long)R * pitch, scale + z * sstride + r);
  }
}

// ---- product -------------------------------------------------------------------

// binary exponent of a row scale (a power of two), or a sentinel for a NaN row
constexpr int kXsNanExp = 1 << 20;
__device__ __forceinline__ int xs_exp(double s) {
  if (!(s == s)) return kXsNanExp;
  return s > 1.7e308 ? 1024 : ilogb(s);
}
// T 2^e; T = 0 and results outside the normal range take the slow way
__device__ __forceinline__ double xs_scaled(long long T, int e) {
  if (e >= kXsNanExp / 2) return NAN;
  const double v = (double)T;
  const int hi = __double2hiint(v), ne = ((hi >> 20) & 0x7FF) + e;
  if (T != 0 && ne > 0 && ne < 0x7FF) return __hiloint2double(hi + e * (1 << 20), __double2loint(v));
  return ldexp(v, e);
}

template <int S, int BN>
__global__ void __launch_bounds__(kXsThreads, 1)
    k_xs_gemm(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
              int M, int N, int K, int kb_per_part, int ntn, int csplit, XsOut o, int *err_flag,
              long long wait, int stall) {
  using C = XsCfg<S, BN>;
  constexpr int STAGES = C::STAGES;

  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], acc_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int s_fail, s_issued, s_consumed;
  __shared__ long long s_roff[C::BM], s_coff[BN];
  __shared__ int s_ea[C::BM], s_eb[BN];

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // blockIdx.x = (outer part, N tile, K part of the cluster)
  const int rank = blockIdx.x % csplit, tile = blockIdx.x / csplit;
  const int ntile = tile % ntn, opart = tile / ntn;
  const int m0 = blockIdx.y * C::BM, n0 = ntile * BN, z = blockIdx.z;
  const int nkb = (K + C::BK - 1) / C::BK;
  const int kb0 = (opart * csplit + rank) * kb_per_part;
  const int kb1 = min(nkb, kb0 + kb_per_part);
  const int nk = max(0, kb1 - kb0);

  auto a_tile = [&](int s) { return smem_base + s * C::STAGE_BYTES; };
  auto b_tile = [&](int s) { return smem_base + s * C::STAGE_BYTES + S * C::A_BYTES; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    mbar_init(smem_u32(&acc_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
    s_issued = 0;
    s_consumed = 0;
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base_sh)),
                 "r"(C::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_base_sh;
  // the operands are the kernel before's: everything above needs none of them
  pdl_enter();

  if (warp == 0 && lane == 0) {
    int i = 0;
    for (; i < (stall ? 0 : nk); ++i) {    // a stalled launch issues nothing
      const int s = i % STAGES;
      const uint32_t ph = (i / STAGES) & 1;
      if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1, wait)) {
        atomicExch(&s_fail, 1);
        break;
      }
      const uint32_t fb = smem_u32(&full_bar[s]);
      mbar_expect_tx(fb, C::STAGE_BYTES);
      const int kx = (kb0 + i) * C::BK;
      tma_load_4d(a_tile(s), &ta, fb, kx, m0, 0, z);
      tma_load_4d(b_tile(s), &tb, fb, kx, n0, 0, z);
    }
    s_issued = i;
  } else if (warp == 1 && lane == 0) {
    int i = 0;
    for (; i < nk; ++i) {
      const int s = i % STAGES;
      const uint32_t ph = (i / STAGES) & 1;
      if (!mbar_wait(smem_u32(&full_bar[s]), ph, wait)) {
        atomicExch(&s_fail, 1);
        break;
      }
      fence_after();
      // descriptors differ only in their start-address field (address >> 4,
      // 14 bits, no carry for shared-memory addresses): base + offset >> 4
      const uint64_t adesc = sw_desc<C::ROW>(a_tile(s)), bdesc = sw_desc<C::ROW>(b_tile(s));
#pragma unroll 1
      for (int k = 0; k < C::BK / 16; ++k) {
        const uint32_t first = (i == 0 && k == 0) ? 0u : 1u;   // slice 0 of A opens every accumulator
#pragma unroll
        for (int a = 0; a < S; ++a)
#pragma unroll
          for (int t = 0; t < S - a; t += C::STACK) {
            const int cnt = (S - a - t) < C::STACK ? (S - a - t) : C::STACK;
            mma_bf16(tmem + (a + t) * BN, adesc + ((a * C::A_BYTES + k * 32) >> 4),
                     bdesc + ((t * C::B_BYTES + k * 32) >> 4), make_idesc(false, C::BM, cnt * BN),
                     a == 0 ? first : 1u);
          }
      }
      mma_commit(smem_u32(&empty_bar[s]));
    }
    s_consumed = i;
    mma_commit(smem_u32(&acc_bar));
  } else if (warp >= 2) {
    // output offsets and scale exponents of the tile's rows and columns
    for (int e = threadIdx.x - 64; e < C::BM + BN; e += kXsThreads - 64) {
      if (e < C::BM) {
        const int row = m0 + e;
        s_roff[e] = row < M ? map_off32(o.cm, row) : 0;
        s_ea[e] = row < M ? xs_exp(o.sa[z * o.ssa + row]) : 0;
      } else {
        const int c = e - C::BM, col = n0 + c;
        s_coff[c] = col < N ? map_off32(o.cn, col) : 0;
        s_eb[c] = col < N ? xs_exp(o.sb[z * o.ssb + col]) : 0;
      }
    }
  }
  __syncwarp();

  // ---- epilogue 1: thread (warp w, lane l) owns accumulator row 32 (w % 4) + l
  // and every other group of 16 columns
  const bool acc_ok = mbar_wait(smem_u32(&acc_bar), 0, wait);
  fence_after();
  if (!acc_ok) atomicExch(&s_fail, 1);
  const bool ok = acc_ok && (*(volatile int *)&s_fail == 0);
  // integer outputs in the (now free) ring: [row][BN + 1] or [column][128]
  long long *outb = reinterpret_cast<long long *>(smem_raw + (smem_base - smem_u32(smem_raw)));
  const int rp = o.rowmajor ? BN + 1 : 1, cp = o.rowmajor ? 1 : C::BM;
  if (ok) {
    const int rl = (warp & 3) * 32 + lane;
    const uint32_t trow = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const bool magic = kb_per_part * C::BK <= kXsMagicK;
#pragma unroll 1
    for (int c = warp >> 2; c < BN / 16; c += 2) {
      long long acc[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) acc[j] = 0;
      if (nk > 0) {
#pragma unroll
        for (int d = 0; d < S; ++d) {
          uint32_t r[16];
          tmem_ld16(tmem + trow + d * BN + c * 16, r);
          // accumulator d holds integers in units of 2^-6(d+2)
          constexpr int kTop = kXsUnit - 2 * kXsBits;          // shift of d = 0
          const int sh = kTop - kXsBits * d;
          int n[16];
          if (magic) {
            const float mg = 1.5f * 8388608.0f / (float)(1ull << (kXsBits * (d + 2)));
#pragma unroll
            for (int j = 0; j < 16; ++j)
              n[j] = __float_as_int(__uint_as_float(r[j]) + mg) - __float_as_int(mg);
          } else {
            const float up = (float)(1ull << (kXsBits * (d + 2)));
#pragma unroll
            for (int j = 0; j < 16; ++j) n[j] = __float2int_rn(__uint_as_float(r[j]) * up);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            if (sh >= 31) acc[j] += (long long)n[j] << (sh < 0 ? 0 : sh);
            else if (sh >= 0) acc[j] += (long long)n[j] * (1 << (sh < 0 ? 0 : sh > 30 ? 30 : sh));
            else acc[j] += (n[j] + (1 << (sh < 0 ? -sh - 1 : 0))) >> (sh < 0 ? -sh : 0);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) outb[rl * rp + (c * 16 + j) * cp] = acc[j];
    }
  }
  fence_before();
  __syncthreads();
  cg::cluster_group cluster = cg::this_cluster();
  if (csplit > 1) cluster.sync();

  // ---- epilogue 2: every CTA of the cluster finishes its share of the rows
  // (rowmajor) or columns
  if (ok) {
    double *Cz = o.C + z * o.cstride + opart * o.pstride;
    const double sg = o.shift.on ? o.shift.sig.at(z)[1] : 0.0;
    const double *add = o.shift.on ? o.shift.X.at(z) : nullptr;
    const int share = (o.rowmajor ? C::BM : BN) / csplit;
    const int inner = o.rowmajor ? BN : C::BM;
    for (int e = threadIdx.x; e < share * inner; e += kXsThreads) {
      const int a = rank * share + e / inner, b = e % inner;
      const int rl = o.rowmajor ? a : b, cl = o.rowmajor ? b : a;
      if (m0 + rl >= M || n0 + cl >= N) continue;
      long long T = 0;
      if (csplit == 1) {
        T = outb[rl * rp + cl * cp];
      } else {
        long long v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          v[q] = q < csplit ? *cluster.map_shared_rank(outb + rl * rp + cl * cp, q) : 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) T += v[q];
      }
      const long long off = s_roff[rl] + s_coff[cl];
      double v = xs_scaled(T, s_ea[rl] + s_eb[cl] - kXsUnit);
      if (o.shift.on) v = fma(sg, add[off], v);
      Cz[off] = v;
    }
    if (o.shift.on && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) o.shift.sig.at(z)[0] = sg;
  }
  if (csplit > 1) cluster.sync();      // no CTA leaves while others may still read its sums
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_fail) atomicMax(err_flag, 2);   // a timeout outranks the non-finite flag (1) it may cause
    for (int i = s_consumed; i < s_issued; ++i)
      (void)mbar_wait(smem_u32(&full_bar[i % STAGES]), (i / STAGES) & 1);
    // the MMAs (acc_bar tracks all of them) finish before the dealloc
    (void)mbar_wait(smem_u32(&acc_bar), 0);
  }
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(C::TMEM_COLS)
                 : "memory");
  }
}

// ---- host side ----------------------------------------------------------

bool make_xs_map(CUtensorMap *m, const XsOperand &op, int box_rows, int row_bytes) {
  auto enc = encode_fn();
  if (!enc) return false;
  const long long bs = op.batch > 1 ? op.bstride : (long long)op.pitch * op.rows * op.S;
  cuuint64_t dims[4] = {(cuuint64_t)op.K, (cuuint64_t)op.rows, (cuuint64_t)op.S,
                        (cuuint64_t)(op.batch < 1 ? 1 : op.batch)};
  cuuint64_t strides[3] = {(cuuint64_t)op.pitch * 2, (cuuint64_t)op.pitch * 2 * op.rows,
                           (cuuint64_t)bs * 2};
  // all slices of a K block in one copy: [slice][row][k] in shared memory
  cuuint32_t box[4] = {(cuuint32_t)(row_bytes / 2), (cuuint32_t)box_rows, (cuuint32_t)op.S, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, op.slices, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE,
                   row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <int S, int BN>
cudaError_t launch_xs(const XsOperand &A, const XsOperand &B, int M, int N, int K,
                      const XsOut &o, int osplit, int *err, cudaStream_t s) {
  using C = XsCfg<S, BN>;
  static SmemLimit limit;
  if (cudaError_t e = limit.raise(reinterpret_cast<const void *>(k_xs_gemm<S, BN>), C::SMEM)) return e;
  CUtensorMap ta, tb;
  if (!make_xs_map(&ta, A, C::BM, C::ROW) || !make_xs_map(&tb, B, BN, C::ROW))
    return cudaErrorInvalidValue;
  const int nkb = (K + C::BK - 1) / C::BK;
  const int ntn = (N + BN - 1) / BN, ntm = (M + C::BM - 1) / C::BM;
  const int batch = A.batch < 1 ? 1 : A.batch;
  // K parts of a cluster: as many as the exactness of a part needs, and more
  // (each at least 64 long) while the tiles do not fill the 152 SMs (one CTA
  // each): a part's copies and MMAs are what a small product waits for
  const int kpart = (nkb + osplit - 1) / osplit * C::BK;
  int csplit = 1;
  while (csplit < 8 && (kpart > csplit * kXsMaxK ||
                        ((long long)ntn * ntm * batch * osplit * csplit * 2 <= 152 && kpart >= 128 * csplit)))
    csplit *= 2;
  const int kbp = (nkb + osplit * csplit - 1) / (osplit * csplit);
  if (kbp * C::BK > kXsMaxK || csplit * kbp * C::BK > kXsMaxSumK || ntm > 65535 || batch > 65535) return cudaErrorInvalidValue;
  const int stall = take_stall(kStallGemm) ? 1 : 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)csplit * ntn * osplit, ntm, batch);
  cfg.blockDim = dim3(kXsThreads, 1, 1);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csplit;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_xs_gemm<S, BN>, ta, tb, M, N, K, kbp, ntn, csplit, o, err, wait_limit(),
                            stall);
}

// Tile width: the accumulators (S x BN columns) fill tensor memory at most, and
// of the widths that fit, the one with the least padded work (16 columns' worth
// per tile for the copies of A).
template <int S>
cudaError_t dispatch_xs(const XsOperand &A, const XsOperand &B, int M, int N, int K,
                        const XsOut &o, int osplit, int *err, cudaStream_t s) {
  constexpr int kMax = 512 / S >= 96 ? 96 : 512 / S >= 80 ? 80 : 64;
  int best = 32;
  long long cost = 0;
  for (int bn : {32, 48, 64, 80, 96}) {
    if (bn > kMax) break;
    const long long c = (long long)((N + bn - 1) / bn) * (bn + 16);
    if (bn == 32 || c < cost) {
      best = bn;
      cost = c;
    }
  }
  switch (best) {
    case 32: return launch_xs<S, 32>(A, B, M, N, K, o, osplit, err, s);
    case 48: return launch_xs<S, 48>(A, B, M, N, K, o, osplit, err, s);
    case 64: return launch_xs<S, 64>(A, B, M, N, K, o, osplit, err, s);
  }
  if constexpr (kMax >= 80)
    if (best == 80) return launch_xs<S, 80>(A, B, M, N, K, o, osplit, err, s);
  if constexpr (kMax >= 96)
    if (best == 96) return launch_xs<S, 96>(A, B, M, N, K, o, osplit, err, s);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t xs_split(PSet src, IdxMap rm, IdxMap km, const XsOperand &d, cudaStream_t s) {
  return xs_split_scaled(src, rm, km, PSet{nullptr, nullptr, 0}, 0, d, s);
}

cudaError_t xs_split_scaled(PSet src, IdxMap rm, IdxMap km, PSet kscale, int kmode,
                            const XsOperand &d, cudaStream_t s) {
  if (d.rows <= 0 || d.K <= 0) return cudaSuccess;
  if (d.S < 1 || d.S > kXsMaxSlices || d.pitch < d.K) return cudaErrorInvalidValue;
  const dim3 g((d.rows + 7) / 8, 1, d.batch < 1 ? 1 : d.batch);
  if (g.z > 65535u) return cudaErrorInvalidConfiguration;
  __nv_bfloat16 *dst = static_cast<__nv_bfloat16 *>(d.slices);
  if (rm.s0 == 1 && rm.n0 >= d.rows && km.s0 != 1 && d.K <= kXsStagedK) {
    const dim3 gs((d.rows + 31) / 32, 1, d.batch < 1 ? 1 : d.batch);
    switch (d.S) {
#define XS_STAGED_CASE(SS)                                                                    \
  case SS:                                                                                    \
    launch_pdl(k_xs_split_staged<SS>, gs, 256, 0, s, src, d.rows, d.K, rm, km, dst, d.pitch, d.bstride, \
                                             d.scale, d.sstride, kscale, kmode);              \
    break;
      XS_STAGED_CASE(1) XS_STAGED_CASE(2) XS_STAGED_CASE(3) XS_STAGED_CASE(4)
      XS_STAGED_CASE(5) XS_STAGED_CASE(6) XS_STAGED_CASE(7) XS_STAGED_CASE(8)
#undef XS_STAGED_CASE
    }
    return cudaGetLastError();
  }
  if (d.K >= 256) {
    const dim3 gr(d.rows, 1, d.batch < 1 ? 1 : d.batch);
    switch (d.S) {
#define XS_ROW_CASE(SS)                                                                       \
  case SS:                                                                                    \
    launch_pdl(k_xs_split_row<SS>, gr, kXsRowThreads, 0, s, src, d.rows, d.K, rm, km, dst, d.pitch, d.bstride,  \
                                          d.scale, d.sstride, kscale, kmode);                 \
    break;
      XS_ROW_CASE(1) XS_ROW_CASE(2) XS_ROW_CASE(3) XS_ROW_CASE(4)
      XS_ROW_CASE(5) XS_ROW_CASE(6) XS_ROW_CASE(7) XS_ROW_CASE(8)
#undef XS_ROW_CASE
    }
    return cudaGetLastError();
  }
  switch (d.S) {
#define XS_SPLIT_CASE(SS)                                                                     \
  case SS:                                                                                    \
    launch_pdl(k_xs_split<SS>, g, 256, 0, s, src, d.rows, d.K, rm, km, dst, d.pitch, d.bstride,       \
                                     d.scale, d.sstride, kscale, kmode);                      \
    break;
    XS_SPLIT_CASE(1) XS_SPLIT_CASE(2) XS_SPLIT_CASE(3) XS_SPLIT_CASE(4)
    XS_SPLIT_CASE(5) XS_SPLIT_CASE(6) XS_SPLIT_CASE(7) XS_SPLIT_CASE(8)
#undef XS_SPLIT_CASE
  }
  return cudaGetLastError();
}

cudaError_t xs_gemm(const XsOperand &A, const XsOperand &B, int M, int N, int K, double *C,
                    IdxMap cm, IdxMap cn, long long cstride, int ksplit, long long pstride,
                    int *err_flag, cudaStream_t s, const XsShift &shift) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (K <= 0 || A.K != K || B.K != K || A.rows < M || B.rows < N || A.S != B.S || ksplit < 1)
    return cudaErrorInvalidValue;
  if ((A.batch < 1 ? 1 : A.batch) != (B.batch < 1 ? 1 : B.batch)) return cudaErrorInvalidValue;
  if (A.pitch != xs_pitch(A.pitch) || B.pitch != xs_pitch(B.pitch) || A.pitch < K || B.pitch < K)
    return cudaErrorInvalidValue;
  if ((A.batch > 1 && (A.bstride * 2) % 16) || (B.batch > 1 && (B.bstride * 2) % 16))
    return cudaErrorInvalidValue;
  if ((reinterpret_cast<uintptr_t>(A.slices) & 15) || (reinterpret_cast<uintptr_t>(B.slices) & 15))
    return cudaErrorInvalidValue;
  if (ksplit < xs_min_split(K) || (shift.on && ksplit > 1)) return cudaErrorInvalidValue;
  XsOut o{C, cm, cn, cstride, pstride, A.scale, B.scale, A.sstride, B.sstride,
          cn.s0 == 1 && cm.s0 != 1 ? 1 : 0, shift};
  switch (A.S) {
    case 4: return dispatch_xs<4>(A, B, M, N, K, o, ksplit, err_flag, s);
    case 5: return dispatch_xs<5>(A, B, M, N, K, o, ksplit, err_flag, s);
    case 6: return dispatch_xs<6>(A, B, M, N, K, o, ksplit, err_flag, s);
    case 7: return dispatch_xs<7>(A, B, M, N, K, o, ksplit, err_flag, s);
    case 8: return dispatch_xs<8>(A, B, M, N, K, o, ksplit, err_flag, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hotrg

namespace hotrg {
namespace {

__global__ void k_xs_sum_parts(const double *parts, int nparts, long long pstride, int M, int N,
                               double *C, long long ldc) {
  pdl_enter();
  const long long total = (long long)M * N;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int p = 0; p < nparts; ++p) v += parts[p * pstride + e];
    C[(e / N) * ldc + e % N] = v;
  }
}

}  // namespace

cudaError_t xs_sum_parts(const double *parts, int nparts, long long pstride, int M, int N,
                         double *C, long long ldc, cudaStream_t s) {
  const long long total = (long long)M * N;
  long long b = (total + 255) / 256;
  if (b > 152 * 8) b = 152 * 8;
  launch_pdl(k_xs_sum_parts, (int)(b < 1 ? 1 : b), 256, 0, s, parts, nparts, pstride, M, N, C, ldc);
  return cudaGetLastError();
}

}  // namespace hotrg

namespace hotrg {
namespace {

// C(cm(m) + cn(n)) of instance z = sum_p parts[((p * batch + z) * M + m) * N + n]
__global__ void k_xs_scatter_parts(const double *parts, int nparts, int batch, int M, int N,
                                   double *C, IdxMap cm, IdxMap cn, long long bC) {
  pdl_enter();
  const int z = blockIdx.y;
  const long long mn = (long long)M * N;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < mn;
       e += (long long)gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int p = 0; p < nparts; ++p) v += parts[((long long)p * batch + z) * mn + e];
    const long long m = e / N, n = e % N;
    C[z * bC + map_off(cm, m) + map_off(cn, n)] = v;
  }
}

}  // namespace

void xs_gemm_needs(int M, int N, int K, int S, int batch, long long need[5]) {
  const int ks = xs_min_split(K);
  need[0] = xs_elems(M, K, S) * batch;
  need[1] = xs_elems(N, K, S) * batch;
  need[2] = (long long)M * batch;
  need[3] = (long long)N * batch;
  need[4] = ks > 1 ? (long long)ks * batch * M * N : 0;
}

bool xs_fits(int M, int N, int K, int S, int batch, const XsWork &w) {
  long long need[5];
  xs_gemm_needs(M, N, K, S, batch, need);
  return need[0] <= w.cap_a && need[1] <= w.cap_b && need[2] <= w.cap_sa && need[3] <= w.cap_sb &&
         need[4] <= w.cap_parts;
}

bool syrk_xs_fits(int M, int K, int batch, int S, const XsWork &w) {
  return M > 0 && K > 0 && batch <= kXsMaxBatch && xs_min_split(K) == 1 && xs_fits(M, 0, K, S, batch, w);
}

cudaError_t syrk_xs(const MappedGemm *g, int count, int S, const XsWork &w, int *err_flag, cudaStream_t s,
                    long long *launches) {
  const int M = g[0].M, K = g[0].K, G = g[0].batch < 1 ? 1 : g[0].batch;
  if (count < 1 || !syrk_xs_fits(M, K, count * G, S, w))
    return cudaErrorInvalidValue;
  const long long ea = xs_elems(M, K, S);
  cudaError_t e;
  for (int v = 0; v < count; ++v) {
    const MappedGemm &q = g[v];
    if (q.M != M || q.N != M || q.K != K || q.C != g[0].C + v * G * g[0].bC) return cudaErrorInvalidValue;
    const PSet pa{const_cast<double *>(q.A), const_cast<double *>(q.A) + q.bA, 2 * q.bA};
    const XsOperand a{static_cast<__nv_bfloat16 *>(w.sa) + v * G * ea, w.sca + (long long)v * G * M, M, K, xs_pitch(K), S,
                      G, ea, M};
    if ((e = xs_split(pa, q.am, q.ak, a, s))) return e;
  }
  const XsOperand all{w.sa, w.sca, M, K, xs_pitch(K), S, count * G, ea, M};
  *launches += count + 1;
  return xs_gemm(all, all, M, M, K, g[0].C, g[0].cm, g[0].cn, g[0].bC, 1, 0, err_flag, s);
}

cudaError_t gemm_xs(const MappedGemm &g, int S, const XsWork &w, int *err_flag, cudaStream_t s, long long *launches) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  const int batch = g.batch < 1 ? 1 : g.batch;
  if (!xs_fits(g.M, g.N, g.K, S, batch, w)) return cudaErrorInvalidValue;
  const long long ea = xs_elems(g.M, g.K, S), eb = xs_elems(g.N, g.K, S);
  XsOperand a{w.sa, w.sca, g.M, g.K, xs_pitch(g.K), S, batch, ea, g.M};
  XsOperand b{w.sb, w.scb, g.N, g.K, xs_pitch(g.K), S, batch, eb, g.N};
  // a batch of instances at stride bA is the PSet "problem z at A + z bA"
  const PSet pa{const_cast<double *>(g.A), const_cast<double *>(g.A) + g.bA, 2 * g.bA};
  const PSet pb{const_cast<double *>(g.B), const_cast<double *>(g.B) + g.bB, 2 * g.bB};
  cudaError_t e;
  if ((e = xs_split(pa, g.am, g.ak, a, s)) || (e = xs_split(pb, g.bn, g.bk, b, s))) return e;
  const int ks = xs_min_split(g.K);
  *launches += ks == 1 ? 3 : 4;
  if (ks == 1) return xs_gemm(a, b, g.M, g.N, g.K, g.C, g.cm, g.cn, g.bC, 1, 0, err_flag, s);
  const long long mn = (long long)g.M * g.N;
  if ((e = xs_gemm(a, b, g.M, g.N, g.K, w.parts, map1(g.N), map1(1), mn, ks, mn * batch,
                   err_flag, s)))
    return e;
  long long blocks = (mn + 255) / 256;
  const long long cap = (152LL * 8 + batch - 1) / batch;
  if (blocks > cap) blocks = cap;
  launch_pdl(k_xs_scatter_parts, dim3((unsigned)(blocks < 1 ? 1 : blocks), batch), 256, 0, s, 
      w.parts, ks, batch, g.M, g.N, g.C, g.cm, g.cn, g.bC);
  return cudaGetLastError();
}

}  // namespace hotrg
