// FP64 products on the tensor cores: C = A . B^T from exact integer slices.
//
// The FP64 pipe of this GPU gives 1.1 TFLOP/s, its BF16 tensor cores 1900. The
// scheme is that of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59 (2012) 95),
// with fixed-point slices as in Ootomo, Ozaki and Yokota (IJHPCA 38 (2024) 297):
// every row of an operand gets one power-of-two scale 2^E above its largest
// magnitude and each value becomes a 56-bit fixed-point number, cut into seven
// signed base-256 digits d_1 .. d_7 in [-128, 128], exact in BF16:
//     x = 2^E sum_i d_i 2^{1 - 8i},   |error| <= 2^{E - 56}.
// A product of two digits is at most 2^14, so sums of up to seven of them over 128
// K values stay below 2^24 and the FP32 accumulator of the tensor cores holds them
// exactly, whatever the order (its truncation never acts). Digit products with the
// same weight i + j = g share an accumulator; g = 2 .. 9 are kept (34 products, the
// first dropped weight is 2^-78 of the scales). After every 128 K values the
// epilogue takes the eight integer sums out of TMEM and adds them into a 96-bit
// integer per element; one conversion and one rounding to FP64 end the tile. The
// result does not depend on the order of anything.
//
// Error. A value is off by at most 2^-56 of its row's scale, so with x_k = |a_k| / 2^Ea and
// y_k = |b_k| / 2^Eb the digits give c within 2^-56 2^{Ea+Eb} (sum x + sum y), whatever the
// size of the products (and the dropped weights within K 2^-61.6): much is lost where a row
// of A is large where the row of B is small (badly scaled auxiliary functions, orbitals on
// different fragments). A chain of FP64 FMAs gives c within K 2^-53 2^{Ea+Eb} S, S = sum x y.
// So every element is checked: an extra product of the leading eight bits of the magnitudes
// gives S from below (oz_check_kernel), and elements with 8 K S < sum x + sum y + K / 50 are
// formed by FP64 FMAs (oz_fma_kernel). So are those of rows with a NaN or an infinity, which
// have no scale. S = 0 is exact (no K index has both factors). Up to the rounding to
// FP64 the bound is then no larger than that of the FMA chain, for any element of any input. On N(0, 1) e^{-0.02 Q}
// factors no element fails the check, on the products of the Fock and DF steps 1e-3 and
// fewer; with an unnormalised auxiliary basis (metric diagonal over 1e11) 9 in 10 of the
// product with the inverse factor do, and it runs at the FP64 pipe's rate.
//
// Kernel (one CTA per SM, persistent, tiles 128 x 64):
//   warp 0      producer: bulk copies of the seven slices of 128 A rows (56 KB, one
//               copy) and of 64 B rows (28 KB, seven copies), 32 K values; 2 stages
//   warp 1      TMEM allocator and MMA issuer: 2 x 34 MMAs (N = 64) per stage; the
//               products of one A slice run back to back on the collector buffer
//   warps 2-9   epilogue (32 columns each): TMEM -> integers -> FP64 stores
// TMEM: 8 accumulators x 64 columns = all 512. Every wait is bounded (about 2 s).
// The slices lie in memory as the MMAs want them in shared memory, [row / 128][K / 32]
// [slice][row % 128][64 bytes, swizzled]: as K-major planes behind a tensor map a stage
// was 1344 rows of 64 bytes and took 4400 clocks to arrive, twice what its MMAs take.
#include <cuda_bf16.h>

#include <climits>

#include "internal.cuh"
#include "oz_gemm.cuh"
#include "tc_common.cuh"

namespace dsrg {

constexpr int OZ_BM = 128, OZ_BN = 64;
constexpr int OZ_KB = 32;                     // K values per stage (64 bytes: one swizzle span)
constexpr int OZ_CHUNK = 4;                   // stages per exact accumulation (128 K values)
constexpr int OZ_STAGES = 2;
constexpr int OZ_A_SLICE = OZ_BM * 64, OZ_B_SLICE = OZ_BN * 64;
constexpr int OZ_A_BYTES = OZ_S * OZ_A_SLICE, OZ_B_BYTES = OZ_S * OZ_B_SLICE;
constexpr int OZ_STAGE_BYTES = OZ_A_BYTES + OZ_B_BYTES;
constexpr int OZ_THREADS = 320, OZ_EPI_WARPS = 8;
constexpr int OZ_EXP_INF = 0x7ff;             // exponent field of a row with an infinity or a NaN
constexpr unsigned long long OZ_SUM_INF = 1ull << 46;  // its sum (others: at most K (2^24 + 1) < 2^46)
constexpr long long OZ_TINY = LLONG_MIN;      // a value that is not 0 but is as a fixed-point number

// ------------------------------- row scales -------------------------------
// Biased exponent of the largest magnitude of every row, by atomicMax (rexp starts
// at 0). One CTA: 64 rows x 64 K values; lanes run along the contiguous index.
template <bool KCONT>
__global__ void __launch_bounds__(256) oz_rowmax_kernel(OzRows s, int* __restrict__ rexp) {
  __shared__ int mx[64];
  const int r0 = blockIdx.x * 64, l0 = blockIdx.y * 64, K = s.L1 * s.L2;
  if (threadIdx.x < 64) mx[threadIdx.x] = 0;
  __syncthreads();
  const int f = threadIdx.x & 63, g = threadIdx.x >> 6;
  int m = 0;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int rr = KCONT ? g + 4 * k : f, l = l0 + (KCONT ? f : g + 4 * k);
    long long off;
    int e = 0;
    if (oz_row(s, r0 + rr, off) && l < K) {
      const double x = s.p[off + oz_k(s, l)];
      e = (__double2hiint(x) >> 20) & 0x7ff;
    }
    if (KCONT) {
      for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
      if ((threadIdx.x & 31) == 0) atomicMax(&mx[rr], e);
    } else {
      m = max(m, e);
    }
  }
  if (!KCONT) atomicMax(&mx[f], m);
  __syncthreads();
  if (threadIdx.x < 64 && r0 + threadIdx.x < s.total) atomicMax(&rexp[r0 + threadIdx.x], mx[threadIdx.x]);
}

// ------------------------------- slices -------------------------------
// x as a fixed-point integer of the row scale: round(x 2^{55 - E}), |.| <= 2^55, or OZ_TINY.
__device__ __forceinline__ long long oz_fixed(double x, int rowexp) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(u >> 52) & 0x7ff;
  if (rowexp == OZ_EXP_INF || (u << 1) == 0) return 0;
  if (e == 0) return OZ_TINY;                           // below 2^-1022
  unsigned long long m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
  const int sh = rowexp - e - 2;  // right shift of the 53-bit significand
  if (sh <= 0)
    m <<= -sh;  // 0, 1 or 2 places (e <= rowexp)
  else if (sh < 64)
    m = (m + (1ull << (sh - 1))) >> sh;
  else
    m = 0;
  if (m == 0) return OZ_TINY;
  return (u >> 63) ? -(long long)m : (long long)m;
}

// Byte offset of the 8 values (16 bytes) from K index l (a multiple of 8) of a slice of a
// plane row: 64-byte rows with the 64-byte swizzle (16-byte chunk ^= row bits 1-2).
__device__ __forceinline__ size_t oz_off(int row, int l, int sl, int nkb) {
  const int r = row & 127;
  const size_t blk = ((size_t)(row >> 7) * nkb + (l >> 5)) * OZ_S + sl;
  return (blk * 128 + r) * 64 + (size_t)((((l >> 3) & 3) ^ ((r >> 1) & 3)) * 16);
}

// ... and of a row of the check plane (one slice).
__device__ __forceinline__ size_t oz_check_off(int row, int l, int nkb) {
  const int r = row & 127;
  return (((size_t)(row >> 7) * nkb + (l >> 5)) * 128 + r) * 64 +
         (size_t)((((l >> 3) & 3) ^ ((r >> 1) & 3)) * 16);
}

// 64 rows x 64 K values per CTA through shared memory. The check plane (after the slices)
// holds the leading eight bits of |x| / 2^E (2^-60 where they are all 0, but x is not); rsum
// the sum of |x| / 2^E over the row in 2^-24 units, rounded up (integers: the order of the atomics does not matter).
template <bool KCONT>
__global__ void __launch_bounds__(256) oz_slice_kernel(OzRows s, const int* __restrict__ rexp,
                                                       unsigned long long* __restrict__ rsum,
                                                       __nv_bfloat16* __restrict__ planes, int Kp) {
  __shared__ long long t[64][65];
  const int r0 = blockIdx.x * 64, l0 = blockIdx.y * 64, K = s.L1 * s.L2;
  const int f = threadIdx.x & 63, g = threadIdx.x >> 6;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int rr = KCONT ? g + 4 * k : f, ll = KCONT ? f : g + 4 * k;
    long long off, v = 0;
    if (oz_row(s, r0 + rr, off) && l0 + ll < K) v = oz_fixed(s.p[off + oz_k(s, l0 + ll)], rexp[r0 + rr]);
    t[rr][ll] = v;
  }
  __syncthreads();
  const int rr = threadIdx.x >> 2, c0 = (threadIdx.x & 3) * 16;
  const bool on = r0 + rr < s.total && l0 + c0 < Kp;
  const int nkb = Kp / OZ_KB;
  long long v[16];
  uint32_t sum = 0;  // below 2^29
  uint32_t cw[8];
#pragma unroll
  for (int k = 0; k < 16; k += 2) {
    float x[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const long long w = t[rr][c0 + k + i];
      v[k + i] = w == OZ_TINY ? 0 : w;
      // |x| in 2^-24 units, rounded down (by up to 2 units): the complement of a negative
      const int hi = (int)(v[k + i] >> 31), m = hi ^ (hi >> 31);
      sum += m + (w != 0);
      x[i] = w == 0 ? 0.0f : fmaxf((float)m * 0x1p-24f, 0x1p-60f);
    }
    cw[k / 2] = __byte_perm(__float_as_uint(x[0]), __float_as_uint(x[1]), 0x7632);  // upper halves
  }
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  sum += __shfl_xor_sync(0xffffffffu, sum, 2);
  if (!on) return;
  if ((threadIdx.x & 3) == 0) {
    const bool inf = l0 == 0 && rexp[r0 + rr] == OZ_EXP_INF;
    if (inf || sum) atomicAdd(&rsum[r0 + rr], inf ? OZ_SUM_INF : (unsigned long long)sum);
  }
  {
    uint8_t* o = (uint8_t*)planes + (size_t)OZ_S * s.total * Kp * sizeof(__nv_bfloat16);
    *(uint4*)(o + oz_check_off(r0 + rr, l0 + c0, nkb)) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
    *(uint4*)(o + oz_check_off(r0 + rr, l0 + c0 + 8, nkb)) = make_uint4(cw[4], cw[5], cw[6], cw[7]);
  }
#pragma unroll
  for (int sl = OZ_S - 1; sl >= 0; --sl) {
    uint32_t w[8];
#pragma unroll
    for (int k = 0; k < 16; k += 2) {
      const int d0 = sl ? (int)(signed char)v[k] : (int)v[k];
      const int d1 = sl ? (int)(signed char)v[k + 1] : (int)v[k + 1];
      v[k] = (v[k] - d0) >> 8;
      v[k + 1] = (v[k + 1] - d1) >> 8;
      const __nv_bfloat162 h = __floats2bfloat162_rn((float)d0, (float)d1);
      w[k / 2] = *(const uint32_t*)&h;
    }
    uint8_t* o = (uint8_t*)planes;
    *(uint4*)(o + oz_off(r0 + rr, l0 + c0, sl, nkb)) = make_uint4(w[0], w[1], w[2], w[3]);
    *(uint4*)(o + oz_off(r0 + rr, l0 + c0 + 8, sl, nkb)) = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// ------------------------------- the product -------------------------------
__device__ __forceinline__ void oz_bulk(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          su32(dst)),
      "l"(src), "r"(bytes), "r"(su32(bar))
      : "memory");
}

// The products of digit i of A (descriptor low word a) with the digits 1 .. JN of B (from
// b), into the accumulators from d on; the leader lane of a converged warp issues. MODE 0:
// `acc` is for all of them, 1: for the last, the others accumulate, 2: all accumulate. A
// stays in the collector buffer. One block per digit: see tc_mma3_if.
template <int JN, int MODE>
__device__ __forceinline__ void oz_row(uint32_t leader, uint32_t d, uint32_t a, uint32_t b, uint32_t acc) {
  constexpr uint32_t idesc = idesc_128xn<true>(OZ_BN);
  static_assert((MODE == 2 && JN >= 2 && JN <= 6) || (MODE < 2 && JN == 7), "the rows of oz_kstep");
  if constexpr (JN == 7 && MODE == 0) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .b64 a, b0, b1, b2, b3, b4, b5, b6;\n"
        " setp.ne.b32 p, %16, 0;\n setp.ne.b32 q, %17, 0;\n mov.b64 a, {%14, %18};\n"
        " mov.b64 b0, {%7, %18};\n"
        " mov.b64 b1, {%8, %18};\n"
        " mov.b64 b2, {%9, %18};\n"
        " mov.b64 b3, {%10, %18};\n"
        " mov.b64 b4, {%11, %18};\n"
        " mov.b64 b5, {%12, %18};\n"
        " mov.b64 b6, {%13, %18};\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], a, b0, %15, p;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%1], a, b1, %15, p;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%2], a, b2, %15, p;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%3], a, b3, %15, p;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%4], a, b4, %15, p;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%5], a, b5, %15, p;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%6], a, b6, %15, p;\n"
        "}\n" ::"r"(d + 0 * OZ_BN), "r"(d + 1 * OZ_BN), "r"(d + 2 * OZ_BN), "r"(d + 3 * OZ_BN),
        "r"(d + 4 * OZ_BN), "r"(d + 5 * OZ_BN), "r"(d + 6 * OZ_BN),
        "r"(b + 0 * OZ_B_SLICE / 16), "r"(b + 1 * OZ_B_SLICE / 16), "r"(b + 2 * OZ_B_SLICE / 16),
        "r"(b + 3 * OZ_B_SLICE / 16), "r"(b + 4 * OZ_B_SLICE / 16), "r"(b + 5 * OZ_B_SLICE / 16),
        "r"(b + 6 * OZ_B_SLICE / 16),
        "r"(a), "r"(idesc), "r"(acc), "r"(leader), "r"(DESC_SW64_HI)
        : "memory");
  } else if constexpr (JN == 7 && MODE == 1) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .b64 a, b0, b1, b2, b3, b4, b5, b6;\n"
        " setp.ne.b32 p, %16, 0;\n setp.ne.b32 q, %17, 0;\n mov.b64 a, {%14, %18};\n"
        " mov.b64 b0, {%7, %18};\n"
        " mov.b64 b1, {%8, %18};\n"
        " mov.b64 b2, {%9, %18};\n"
        " mov.b64 b3, {%10, %18};\n"
        " mov.b64 b4, {%11, %18};\n"
        " mov.b64 b5, {%12, %18};\n"
        " mov.b64 b6, {%13, %18};\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], a, b0, %15, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%1], a, b1, %15, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%2], a, b2, %15, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%3], a, b3, %15, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%4], a, b4, %15, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%5], a, b5, %15, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%6], a, b6, %15, p;\n"
        "}\n" ::"r"(d + 0 * OZ_BN), "r"(d + 1 * OZ_BN), "r"(d + 2 * OZ_BN), "r"(d + 3 * OZ_BN),
        "r"(d + 4 * OZ_BN), "r"(d + 5 * OZ_BN), "r"(d + 6 * OZ_BN),
        "r"(b + 0 * OZ_B_SLICE / 16), "r"(b + 1 * OZ_B_SLICE / 16), "r"(b + 2 * OZ_B_SLICE / 16),
        "r"(b + 3 * OZ_B_SLICE / 16), "r"(b + 4 * OZ_B_SLICE / 16), "r"(b + 5 * OZ_B_SLICE / 16),
        "r"(b + 6 * OZ_B_SLICE / 16),
        "r"(a), "r"(idesc), "r"(acc), "r"(leader), "r"(DESC_SW64_HI)
        : "memory");
  } else if constexpr (JN == 6 && MODE == 2) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .b64 a, b0, b1, b2, b3, b4, b5;\n"
        " setp.ne.b32 p, %14, 0;\n setp.ne.b32 q, %15, 0;\n mov.b64 a, {%12, %16};\n"
        " mov.b64 b0, {%6, %16};\n"
        " mov.b64 b1, {%7, %16};\n"
        " mov.b64 b2, {%8, %16};\n"
        " mov.b64 b3, {%9, %16};\n"
        " mov.b64 b4, {%10, %16};\n"
        " mov.b64 b5, {%11, %16};\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], a, b0, %13, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%1], a, b1, %13, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%2], a, b2, %13, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%3], a, b3, %13, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%4], a, b4, %13, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%5], a, b5, %13, q;\n"
        "}\n" ::"r"(d + 0 * OZ_BN), "r"(d + 1 * OZ_BN), "r"(d + 2 * OZ_BN), "r"(d + 3 * OZ_BN),
        "r"(d + 4 * OZ_BN), "r"(d + 5 * OZ_BN),
        "r"(b + 0 * OZ_B_SLICE / 16), "r"(b + 1 * OZ_B_SLICE / 16), "r"(b + 2 * OZ_B_SLICE / 16),
        "r"(b + 3 * OZ_B_SLICE / 16), "r"(b + 4 * OZ_B_SLICE / 16), "r"(b + 5 * OZ_B_SLICE / 16),
        "r"(a), "r"(idesc), "r"(acc), "r"(leader), "r"(DESC_SW64_HI)
        : "memory");
  } else if constexpr (JN == 5 && MODE == 2) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .b64 a, b0, b1, b2, b3, b4;\n"
        " setp.ne.b32 p, %12, 0;\n setp.ne.b32 q, %13, 0;\n mov.b64 a, {%10, %14};\n"
        " mov.b64 b0, {%5, %14};\n"
        " mov.b64 b1, {%6, %14};\n"
        " mov.b64 b2, {%7, %14};\n"
        " mov.b64 b3, {%8, %14};\n"
        " mov.b64 b4, {%9, %14};\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], a, b0, %11, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%1], a, b1, %11, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%2], a, b2, %11, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%3], a, b3, %11, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%4], a, b4, %11, q;\n"
        "}\n" ::"r"(d + 0 * OZ_BN), "r"(d + 1 * OZ_BN), "r"(d + 2 * OZ_BN), "r"(d + 3 * OZ_BN),
        "r"(d + 4 * OZ_BN),
        "r"(b + 0 * OZ_B_SLICE / 16), "r"(b + 1 * OZ_B_SLICE / 16), "r"(b + 2 * OZ_B_SLICE / 16),
        "r"(b + 3 * OZ_B_SLICE / 16), "r"(b + 4 * OZ_B_SLICE / 16),
        "r"(a), "r"(idesc), "r"(acc), "r"(leader), "r"(DESC_SW64_HI)
        : "memory");
  } else if constexpr (JN == 4 && MODE == 2) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .b64 a, b0, b1, b2, b3;\n"
        " setp.ne.b32 p, %10, 0;\n setp.ne.b32 q, %11, 0;\n mov.b64 a, {%8, %12};\n"
        " mov.b64 b0, {%4, %12};\n"
        " mov.b64 b1, {%5, %12};\n"
        " mov.b64 b2, {%6, %12};\n"
        " mov.b64 b3, {%7, %12};\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], a, b0, %9, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%1], a, b1, %9, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%2], a, b2, %9, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%3], a, b3, %9, q;\n"
        "}\n" ::"r"(d + 0 * OZ_BN), "r"(d + 1 * OZ_BN), "r"(d + 2 * OZ_BN), "r"(d + 3 * OZ_BN),
        "r"(b + 0 * OZ_B_SLICE / 16), "r"(b + 1 * OZ_B_SLICE / 16), "r"(b + 2 * OZ_B_SLICE / 16),
        "r"(b + 3 * OZ_B_SLICE / 16),
        "r"(a), "r"(idesc), "r"(acc), "r"(leader), "r"(DESC_SW64_HI)
        : "memory");
  } else if constexpr (JN == 3 && MODE == 2) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .b64 a, b0, b1, b2;\n"
        " setp.ne.b32 p, %8, 0;\n setp.ne.b32 q, %9, 0;\n mov.b64 a, {%6, %10};\n"
        " mov.b64 b0, {%3, %10};\n"
        " mov.b64 b1, {%4, %10};\n"
        " mov.b64 b2, {%5, %10};\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], a, b0, %7, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%1], a, b1, %7, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%2], a, b2, %7, q;\n"
        "}\n" ::"r"(d + 0 * OZ_BN), "r"(d + 1 * OZ_BN), "r"(d + 2 * OZ_BN),
        "r"(b + 0 * OZ_B_SLICE / 16), "r"(b + 1 * OZ_B_SLICE / 16), "r"(b + 2 * OZ_B_SLICE / 16),
        "r"(a), "r"(idesc), "r"(acc), "r"(leader), "r"(DESC_SW64_HI)
        : "memory");
  } else if constexpr (JN == 2 && MODE == 2) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .b64 a, b0, b1;\n"
        " setp.ne.b32 p, %6, 0;\n setp.ne.b32 q, %7, 0;\n mov.b64 a, {%4, %8};\n"
        " mov.b64 b0, {%2, %8};\n"
        " mov.b64 b1, {%3, %8};\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], a, b0, %5, q;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%1], a, b1, %5, q;\n"
        "}\n" ::"r"(d + 0 * OZ_BN), "r"(d + 1 * OZ_BN),
        "r"(b + 0 * OZ_B_SLICE / 16), "r"(b + 1 * OZ_B_SLICE / 16),
        "r"(a), "r"(idesc), "r"(acc), "r"(leader), "r"(DESC_SW64_HI)
        : "memory");
  }
}

// One K step (16 values) from the descriptor low words of the first slices: digit pairs
// (i, j), i + j <= 9 (accumulator i + j - 2), the j of one i back to back. The first product
// of a weight starts its accumulator: those of i = 1, and (2, 7).
__device__ __forceinline__ void oz_kstep(uint32_t leader, uint32_t d, uint32_t a, uint32_t b, bool first) {
  static_assert(OZ_S == 7 && OZ_G == 8, "the rows below");
  constexpr uint32_t A = OZ_A_SLICE / 16;
  const uint32_t acc = first ? 0u : 1u;
  oz_row<7, 0>(leader, d, a, b, acc);
  oz_row<7, 1>(leader, d + OZ_BN, a + A, b, acc);
  oz_row<6, 2>(leader, d + 2 * OZ_BN, a + 2 * A, b, 1u);
  oz_row<5, 2>(leader, d + 3 * OZ_BN, a + 3 * A, b, 1u);
  oz_row<4, 2>(leader, d + 4 * OZ_BN, a + 4 * A, b, 1u);
  oz_row<3, 2>(leader, d + 5 * OZ_BN, a + 5 * A, b, 1u);
  oz_row<2, 2>(leader, d + 6 * OZ_BN, a + 6 * A, b, 1u);
}

__device__ __forceinline__ void oz_tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "r"(taddr));
}

struct OzTile {
  int arow, brow;       // first plane rows
  int i0, j0;           // first row and column of C
  long long coff;       // its problem's offset in C
};
__device__ __forceinline__ OzTile oz_tile(const OzArgs& a, int it) {
  const int per = a.mt * a.nt, pr = it / per, r = it % per;
  OzTile t;
  // row blocks of `band` tiles with the columns inside: the CTAs running at one time
  // share operand slabs in L2
  const int mb = r / (a.band * a.nt), rem = r % (a.band * a.nt);
  const int rows = min(a.band, a.mt - mb * a.band);
  const int n = rem / rows, m = mb * a.band + rem % rows;
  t.i0 = m * OZ_BM;
  t.j0 = n * OZ_BN;
  const int2 ij = a.pairs ? a.pairs[a.p0 + pr * a.pstep] : make_int2(pr, pr);
  t.arow = a.arow0 + ij.x * a.astep + t.i0;
  t.brow = a.brow0 + ij.y * a.bstep + t.j0;
  t.coff = (long long)pr * a.sc;
  return t;
}

// The mask words [128 rows][2 x 32 columns] of an item, and the bytes that say whether the
// epilogue warps of the check set any.
__device__ __forceinline__ uint32_t* oz_mask(const OzArgs& a, int it) {
  return (uint32_t*)a.mask + (size_t)it * 256;
}
__device__ __forceinline__ uint8_t* oz_mask_any(const OzArgs& a, int it) {
  return (uint8_t*)a.mask + (size_t)a.n_items * 1024 + (size_t)it * 8;
}

__global__ void __launch_bounds__(OZ_THREADS, 1)
    oz_gemm_kernel(const uint8_t* __restrict__ pa, const uint8_t* __restrict__ pb,
                   const __grid_constant__ OzArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + OZ_STAGES * OZ_STAGE_BYTES);
  uint64_t* empty = full + OZ_STAGES;
  uint64_t* tfull = empty + OZ_STAGES;
  uint64_t* tempty = tfull + 1;
  uint64_t* drain = tempty + 1;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < OZ_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, OZ_EPI_WARPS);
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    const uint32_t leader = tc_elect();
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int it = blockIdx.x; ok && it < a.n_items; it += gridDim.x) {
      const OzTile t = oz_tile(a, it);
      const uint8_t* ga = pa + (size_t)(t.arow >> 7) * a.kstages * OZ_A_BYTES;
      const uint8_t* gb = pb + (size_t)(t.brow >> 7) * a.kstages * OZ_A_BYTES + (t.brow & 64) * 64;
      for (int kb = 0; kb < a.kstages; ++kb) {
        if (!TC_WARP_WAIT(&empty[stage], phase ^ 1u, abort_flag, a.status)) {
          ok = false;
          break;
        }
        uint8_t* st = smem + stage * OZ_STAGE_BYTES;
        mbar_expect_tx_if(leader, &full[stage], (uint32_t)OZ_STAGE_BYTES);
        if (leader) {
          // A: a whole 128-row block; B: a 64-row half of every slice of its block
          oz_bulk(st, ga + (size_t)kb * OZ_A_BYTES, OZ_A_BYTES, &full[stage]);
#pragma unroll
          for (int sl = 0; sl < OZ_S; ++sl)
            oz_bulk(st + OZ_A_BYTES + sl * OZ_B_SLICE, gb + (size_t)kb * OZ_A_BYTES + sl * OZ_A_SLICE,
                    OZ_B_SLICE, &full[stage]);
        }
        __syncwarp();
        if (++stage == OZ_STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok && leader) {
      int s = stage;
      uint32_t ph = phase;
      for (int k = 0; k < OZ_STAGES; ++k) {
        if (--s < 0) {
          s = OZ_STAGES - 1;
          ph ^= 1u;
        }
        const unsigned long long t0 = gtimer();
        while (!mbar_try(&full[s], ph) && gtimer() - t0 < TC_WAIT_NS) {
        }
      }
    }
  } else if (warp == 1) {
    const uint32_t leader = tc_elect();
    const uint32_t tm = tc_uniform(tmem), base_lo = tc_uniform(desc_sw64_lo(su32(smem)));
    int stage = 0;
    uint32_t phase = 0, tphase = 0;
    bool ok = true, issued = false;
    for (int it = blockIdx.x; ok && it < a.n_items; it += gridDim.x) {
      for (int kb = 0; kb < a.kstages; ++kb) {
        if (kb % OZ_CHUNK == 0) {
          if (!TC_WARP_WAIT(tempty, tphase ^ 1u, abort_flag, a.status)) {
            ok = false;
            break;
          }
          tphase ^= 1u;
        }
        if (!TC_WARP_WAIT(&full[stage], phase, abort_flag, a.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = base_lo + (uint32_t)(stage * (OZ_STAGE_BYTES / 16)), sb = sa + OZ_A_BYTES / 16;
        oz_kstep(leader, tm, sa, sb, kb % OZ_CHUNK == 0);
        oz_kstep(leader, tm, sa + 32 / 16, sb + 32 / 16, false);
        issued = true;
        tc_commit_if(leader, &empty[stage]);
        if (++stage == OZ_STAGES) {
          stage = 0;
          phase ^= 1u;
        }
        if (kb % OZ_CHUNK == OZ_CHUNK - 1 || kb == a.kstages - 1) tc_commit_if(leader, tfull);
      }
    }
    if (!ok && issued && leader) {
      tc_commit(drain);
      const unsigned long long t0 = gtimer();
      while (!mbar_try(drain, 0) && gtimer() - t0 < TC_WAIT_NS) {
      }
    }
  } else {
    const int quarter = warp & 3, ch = (warp - 2) >> 2;  // TMEM lanes and column half
    const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(ch * 32);
    uint32_t tphase = 0;
    const int nchunks = (a.kstages + OZ_CHUNK - 1) / OZ_CHUNK;
    for (int it = blockIdx.x; it < a.n_items; it += gridDim.x) {
      const OzTile t = oz_tile(a, it);
      // 96-bit sums in units of 2^-70 of the scales: hi 2^32 + lo
      long long hi[32];
      uint32_t lo[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        hi[c] = 0;
        lo[c] = 0;
      }
      bool ok = true;
      for (int ck = 0; ck < nchunks; ++ck) {
        ok = mbar_wait(tfull, tphase, abort_flag, a.status) && ok;
        tphase ^= 1u;
        tc_fence_after();
        if (ok) {
#pragma unroll
          for (int c8 = 0; c8 < 4; ++c8) {
            uint32_t r[4][8];
            // weights 6 .. 9 (2^-70 units: 2^24, 2^16, 2^8, 1)
#pragma unroll
            for (int g = 0; g < 4; ++g) oz_tmem_ld8(tb + (uint32_t)((4 + g) * OZ_BN + 8 * c8), r[g]);
            tmem_ld_wait();
            int carry[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const int k = 8 * c8 + c;
              long long v = (long long)lo[k] + __float2int_rn(__uint_as_float(r[3][c]));
              v += (long long)__float2int_rn(__uint_as_float(r[2][c])) << 8;
              v += (long long)__float2int_rn(__uint_as_float(r[1][c])) << 16;
              v += (long long)__float2int_rn(__uint_as_float(r[0][c])) << 24;
              lo[k] = (uint32_t)v;
              carry[c] = (int)(v >> 32);
            }
            // weights 2 .. 5 (2^-38 units)
#pragma unroll
            for (int g = 0; g < 4; ++g) oz_tmem_ld8(tb + (uint32_t)(g * OZ_BN + 8 * c8), r[g]);
            tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const int k = 8 * c8 + c;
              long long v = hi[k] + carry[c] + __float2int_rn(__uint_as_float(r[3][c]));
              v += (long long)__float2int_rn(__uint_as_float(r[2][c])) << 8;
              v += (long long)__float2int_rn(__uint_as_float(r[1][c])) << 16;
              v += (long long)__float2int_rn(__uint_as_float(r[0][c])) << 24;
              hi[k] = v;
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty);
      }
      if (!ok) continue;
      const int i = t.i0 + quarter * 32 + lane;
      if (i < a.M) {
        // value = (hi + lo 2^-32) 2^-38 2^{Ea + Eb}, E = exponent field - 1022
        const int ra = t.arow + quarter * 32 + lane, ea = a.aexp[ra];
        // elements of oz_fma_kernel
        const uint32_t skip = oz_mask(a, it)[(quarter * 32 + lane) * 2 + ch];
        double* crow = a.C + t.coff + (long long)i * a.ci;
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          const int j = t.j0 + ch * 32 + c;
          if (j < a.N && !(skip >> c & 1u)) {
            double d = fma((double)lo[c], 2.3283064365386962890625e-10, (double)hi[c]);
            const int rb = t.brow + ch * 32 + c, eb = a.bexp[rb];
            const int e = ea + eb - 2 * 1022 - 38;
            const int hw = __double2hiint(d), ef = (hw >> 20) & 0x7ff;
            if (ef != 0) {
              if (ef + e > 0 && ef + e < 0x7ff)
                d = __hiloint2double(hw + (e << 20), __double2loint(d));
              else
                d = scalbn(d, e);
            }
            if (a.alpha != 1.0) d *= a.alpha;
            double* p = crow + (long long)j * a.cj;
            *p = a.accumulate ? *p + d : d;
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
  }
}

// ------------------------------- the check -------------------------------
// S of every element (see the head of the file) in one FP32 accumulation over all of K, and
// its mask bit. One BF16 product against the 34 of the slices, bound by its operands' copies
// and the epilogue: 4 stages of up to 128 K values. 33 us beside 780 us for the products of
// 86 pairs at 24/2/372/1200, 17 beside 190 us (K = 398) in the DF transform.
constexpr int OC_KB = 4;  // blocks of 32 K values per stage
constexpr int OC_STAGES = 4;
constexpr int OC_STAGE_BYTES = OC_KB * (OZ_A_SLICE + OZ_B_SLICE);

__global__ void __launch_bounds__(OZ_THREADS, 1)
    oz_check_kernel(const uint8_t* __restrict__ pa, const uint8_t* __restrict__ pb,
                    const __grid_constant__ OzArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + OC_STAGES * OC_STAGE_BYTES);
  uint64_t* empty = full + OC_STAGES;
  uint64_t* tfull = empty + OC_STAGES;  // [2]
  uint64_t* tempty = tfull + 2;         // [2]
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < OC_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&tfull[t], 1);
      mbar_init(&tempty[t], OZ_EPI_WARPS);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tmem_slot)),
                 "r"(128u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int nst = (a.kstages + OC_KB - 1) / OC_KB;

  if (warp == 0) {
    const uint32_t leader = tc_elect();
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int it = blockIdx.x; ok && it < a.n_items; it += gridDim.x) {
      const OzTile t = oz_tile(a, it);
      const uint8_t* ga = pa + (size_t)(t.arow >> 7) * a.kstages * OZ_A_SLICE;
      const uint8_t* gb = pb + (size_t)(t.brow >> 7) * a.kstages * OZ_A_SLICE + (t.brow & 64) * 64;
      for (int ks = 0; ks < nst; ++ks) {
        if (!TC_WARP_WAIT(&empty[stage], phase ^ 1u, abort_flag, a.status)) {
          ok = false;
          break;
        }
        uint8_t* st = smem + stage * OC_STAGE_BYTES;
        const int k0 = ks * OC_KB, nk = min(OC_KB, a.kstages - k0);
        mbar_expect_tx_if(leader, &full[stage], (uint32_t)(nk * (OZ_A_SLICE + OZ_B_SLICE)));
        if (leader) {
          oz_bulk(st, ga + (size_t)k0 * OZ_A_SLICE, (uint32_t)(nk * OZ_A_SLICE), &full[stage]);
          for (int k = 0; k < nk; ++k)
            oz_bulk(st + OC_KB * OZ_A_SLICE + k * OZ_B_SLICE, gb + (size_t)(k0 + k) * OZ_A_SLICE, OZ_B_SLICE,
                    &full[stage]);
        }
        __syncwarp();
        if (++stage == OC_STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok && leader) {
      int s = stage;
      uint32_t ph = phase;
      for (int k = 0; k < OC_STAGES; ++k) {
        if (--s < 0) {
          s = OC_STAGES - 1;
          ph ^= 1u;
        }
        const unsigned long long t0 = gtimer();
        while (!mbar_try(&full[s], ph) && gtimer() - t0 < TC_WAIT_NS) {
        }
      }
    }
  } else if (warp == 1) {
    const uint32_t leader = tc_elect();
    const uint32_t tm = tc_uniform(tmem), base_lo = tc_uniform(desc_sw64_lo(su32(smem)));
    constexpr uint32_t idesc = idesc_128xn<true>(OZ_BN);
    int stage = 0, tb = 0;
    uint32_t phase = 0, tphase = 0;
    bool ok = true, issued = false;
    for (int it = blockIdx.x; ok && it < a.n_items; it += gridDim.x) {
      if (!TC_WARP_WAIT(&tempty[tb], tphase ^ 1u, abort_flag, a.status)) {
        ok = false;
        break;
      }
      tc_fence_after();
      for (int ks = 0; ks < nst; ++ks) {
        if (!TC_WARP_WAIT(&full[stage], phase, abort_flag, a.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = base_lo + (uint32_t)(stage * (OC_STAGE_BYTES / 16));
        const uint32_t sb = sa + OC_KB * OZ_A_SLICE / 16;
        const int nk = min(OC_KB, a.kstages - ks * OC_KB);
        for (int k = 0; k < nk; ++k)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            tc_mma_if<true>(leader, tm + (uint32_t)(tb * OZ_BN), sa + k * (OZ_A_SLICE / 16) + 2 * h,
                            sb + k * (OZ_B_SLICE / 16) + 2 * h, idesc, (ks | k | h) ? 1u : 0u);
        issued = true;
        tc_commit_if(leader, &empty[stage]);
        if (++stage == OC_STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok) break;
      tc_commit_if(leader, &tfull[tb]);
      if (++tb == 2) {
        tb = 0;
        tphase ^= 1u;
      }
    }
    if (!ok && issued && leader) {
      tc_commit(drain);
      const unsigned long long t0 = gtimer();
      while (!mbar_try(drain, 0) && gtimer() - t0 < TC_WAIT_NS) {
      }
    }
  } else {
    const int quarter = warp & 3, ch = (warp - 2) >> 2;  // TMEM lanes and column half
    const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(ch * 32);
    const unsigned long long* asum = (const unsigned long long*)(a.aexp + a.a.total);
    const unsigned long long* bsum = (const unsigned long long*)(a.bexp + a.b.total);
    const float K = (float)(a.a.L1 * a.a.L2), K8 = 8.0f * K;
    int tb = 0;
    uint32_t tphase = 0;
    for (int it = blockIdx.x; it < a.n_items; it += gridDim.x) {
      const OzTile t = oz_tile(a, it);
      const bool ok = mbar_wait(&tfull[tb], tphase, abort_flag, a.status);
      tc_fence_after();
      uint32_t r[2][16];
      if (ok) {
        tmem_ld16(tl + (uint32_t)(tb * OZ_BN), r[0]);
        tmem_ld16(tl + (uint32_t)(tb * OZ_BN + 16), r[1]);
        tmem_ld_wait();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[tb]);
      if (++tb == 2) {
        tb = 0;
        tphase ^= 1u;
      }
      const int row = quarter * 32 + lane, i = t.i0 + row;
      uint32_t word = 0;
      if (ok && i < a.M) {
        // (sums in 2^-9 units, rounded up: a conversion from 64 bits would be one of the FP64 pipe)
        const float sa = (float)(uint32_t)(asum[t.arow + row] >> 15) * 0x1p-9f + 0x1p-8f + 0.02f * K;
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          const int j = ch * 32 + c;
          if (t.j0 + j < a.N) {
            const float S = __uint_as_float(r[c >> 4][c & 15]);
            const float sums = sa + (float)(uint32_t)(bsum[t.brow + j] >> 15) * 0x1p-9f;
            if ((S > 0.0f && K8 * S < sums) || sums >= (float)(OZ_SUM_INF >> 24)) word |= 1u << c;
          }
        }
      }
      oz_mask(a, it)[row * 2 + ch] = word;
      const bool any = __any_sync(0xffffffffu, word != 0);
      if (lane == 0) oz_mask_any(a, it)[warp - 2] = any;
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(128u)
                 : "memory");
  }
}

// The elements the check set, from the FP64 operands, in units of 16 rows x 64 columns (as
// 64 x 64 ones, few products filled the chip: 110, 72 and 105 us in the triangular inverse
// at naux = 1200, 35, 53 and 84 us now): a warp each, its lanes along K, where an eighth of a
// unit or less is set, else the unit in chunks of 16 K values (the chain of
// gemm_fp64_kernel in grad.cu). Bound by the FP64 pipe where much is set: the DF transform at
// 398 functions and naux = 1200 takes 33 ms with auxiliary functions scaled by 2^-20 .. 2^20
// (8.5 ms as drawn; 143 ms with FP64 FMAs alone). With none set the launch takes 4 us.
constexpr int OF_ROWS = 16, OF_UNITS = OZ_BM / OF_ROWS, OF_FEW = 128;
__global__ void __launch_bounds__(256) oz_fma_kernel(const __grid_constant__ OzArgs a) {
  __shared__ double sA[16][OF_ROWS + 1], sB[16][OZ_BN + 1];
  __shared__ uint32_t sm[2 * OF_ROWS];  // the unit's mask words
  __shared__ unsigned short list[OF_FEW];
  __shared__ unsigned char work[256];
  __shared__ int cnt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int L1 = a.a.L1, L2 = a.a.L2, K = L1 * L2;
  auto put = [&](double* p, double d) { *p = a.accumulate ? fma(a.alpha, d, *p) : a.alpha * d; };
  const long long units = (long long)a.n_items * OF_UNITS;
  for (long long base = blockIdx.x; base < units; base += 256ll * gridDim.x) {
    // 256 units at a time: which of them may have any
    const long long mine = base + (long long)tid * gridDim.x;
    bool any = false;
    if (mine < units) {
      // bytes of the warps that had the rows' TMEM quarter: q = warp & 3, warps 2 to 9
      const int b = (((int)(mine % OF_UNITS) >> 1) + 2) & 3;
      const uint8_t* m = oz_mask_any(a, (int)(mine / OF_UNITS));
      any = m[b] | m[b + 4];
    }
    work[tid] = any;
    if (!__syncthreads_or(any)) continue;
    for (int w = 0; w < 256; ++w) {
      if (!work[w]) continue;
      const long long u = base + (long long)w * gridDim.x;
      const int it = (int)(u / OF_UNITS), r0 = (int)(u % OF_UNITS) * OF_ROWS;
      __syncthreads();  // the previous unit is done
      if (tid == 0) cnt = 0;
      if (tid < 2 * OF_ROWS) sm[tid] = oz_mask(a, it)[r0 * 2 + tid];
      __syncthreads();
      if (tid < 2 * OF_ROWS)
        for (uint32_t m = sm[tid]; m; m &= m - 1) {
          const int k = atomicAdd(&cnt, 1);
          if (k < OF_FEW) list[k] = (unsigned short)((tid >> 1) << 6 | (tid & 1) << 5 | (__ffs(m) - 1));
        }
      __syncthreads();
      const int n = cnt;
      if (n == 0) continue;
      const OzTile t = oz_tile(a, it);
      const int i0 = t.i0 + r0, ar = t.arow + r0;
      double* C = a.C + t.coff;
      if (n <= OF_FEW) {
        for (int e = warp; e < n; e += 8) {  // (whatever the order of the list)
          const int r = list[e] >> 6, c = list[e] & 63;
          long long oa, ob;
          oz_row(a.a, ar + r, oa);
          oz_row(a.b, t.brow + c, ob);
          double d = 0.0;
#pragma unroll 4
          for (int l = lane; l < K; l += 32)
            d = fma(a.a.p[oa + oz_k(a.a, l)], a.b.p[ob + oz_k(a.b, l)], d);
          for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
          if (lane == 0) put(C + (long long)(i0 + r) * a.ci + (long long)(t.j0 + c) * a.cj, d);
        }
        continue;
      }
      const int r = tid >> 4, cx = tid & 15;  // columns cx, + 16, + 32, + 48 of row r
      double acc[4] = {};
      for (int l0 = 0; l0 < K; l0 += 16) {
        {
          const int l = l0 + cx;  // K along 16 lanes, a row each
          long long o;
          sA[cx][r] = l < K && i0 + r < a.M && oz_row(a.a, ar + r, o) ? a.a.p[o + oz_k(a.a, l)] : 0.0;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int c = r + 16 * k;
            sB[cx][c] = l < K && t.j0 + c < a.N && oz_row(a.b, t.brow + c, o) ? a.b.p[o + oz_k(a.b, l)] : 0.0;
          }
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < 16; ++l)
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[k] = fma(sA[l][r], sB[l][cx + 16 * k], acc[k]);
        __syncthreads();
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int c = cx + 16 * k;
        if (sm[r * 2 + (c >> 5)] >> (c & 31) & 1u)
          put(C + (long long)(i0 + r) * a.ci + (long long)(t.j0 + c) * a.cj, acc[k]);
      }
    }
    __syncthreads();
  }
}

// ------------------------------- host side -------------------------------
cudaError_t oz_pack(cudaStream_t st, const OzRows& s, __nv_bfloat16* planes, int* rexp) {
  const int Kp = oz_kpad((long long)s.L1 * s.L2);
  const dim3 grid((unsigned)((s.total + 63) / 64), (unsigned)((Kp + 63) / 64));
  cudaError_t e = cudaMemsetAsync(rexp, 0, (size_t)s.total * OZ_ROW_INFO, st);
  if (e != cudaSuccess) return e;
  unsigned long long* rsum = (unsigned long long*)(rexp + s.total);
  // lanes along K when K is the unit-stride index, else along the rows
  if ((s.L2 == 1 ? s.k1 : s.k2) == 1 && s.ri != 1) {
    oz_rowmax_kernel<true><<<grid, 256, 0, st>>>(s, rexp);
    oz_slice_kernel<true><<<grid, 256, 0, st>>>(s, rexp, rsum, planes, Kp);
  } else {
    oz_rowmax_kernel<false><<<grid, 256, 0, st>>>(s, rexp);
    oz_slice_kernel<false><<<grid, 256, 0, st>>>(s, rexp, rsum, planes, Kp);
  }
  return cudaGetLastError();
}

cudaError_t oz_multiply(cudaStream_t st, const __nv_bfloat16* pa, const __nv_bfloat16* pb, OzArgs a,
                        int n_prob) {
  const int Kp = oz_kpad((long long)a.a.L1 * a.a.L2);
  a.mt = (a.M + OZ_BM - 1) / OZ_BM;
  a.nt = (a.N + OZ_BN - 1) / OZ_BN;
  a.band = 12;
  a.kstages = Kp / OZ_KB;
  const long long items = (long long)a.mt * a.nt * n_prob;
  if (items <= 0 || items > 0x7fffffff) return cudaErrorInvalidValue;
  a.n_items = (int)items;
  const int nsm = sm_count();
  const unsigned grid = (unsigned)(items < nsm ? items : nsm);
  const size_t smc = (size_t)OC_STAGES * OC_STAGE_BYTES + 1024 + 256;
  raise_smem_limit((const void*)oz_check_kernel, smc);
  oz_check_kernel<<<grid, OZ_THREADS, smc, st>>>((const uint8_t*)(pa + (size_t)OZ_S * a.a.total * Kp),
                                                 (const uint8_t*)(pb + (size_t)OZ_S * a.b.total * Kp), a);
  const size_t sm = (size_t)OZ_STAGES * OZ_STAGE_BYTES + 1024 + 256;
  raise_smem_limit((const void*)oz_gemm_kernel, sm);
  oz_gemm_kernel<<<grid, OZ_THREADS, sm, st>>>((const uint8_t*)pa, (const uint8_t*)pb, a);
  const long long units = items * OF_UNITS;
  oz_fma_kernel<<<(unsigned)(units < 4ll * nsm ? units : 4ll * nsm), 256, 0, st>>>(a);
  return cudaGetLastError();
}

// ------------------------------- generic GEMM -------------------------------
static long long oz_up(long long x, long long m) { return (x + m - 1) / m * m; }
static size_t oz_row_bytes(long long K) { return oz_plane_bytes(1, K) + OZ_ROW_INFO; }

size_t oz_work_bytes(long long M, long long N, long long K, long long nb, bool shared_a, bool shared_b) {
  const long long mp = oz_up(M, OZ_ROW_PAD), np = oz_up(N, OZ_ROW_PAD);
  const size_t mask = oz_mask_bytes(mp, np, 1);  // (rows padded to whole blocks: either side may be M)
  const size_t need = ((shared_a ? mp : mp * nb) + (shared_b ? np : np * nb)) * oz_row_bytes(K) + nb * mask;
  const size_t one = (mp + np) * oz_row_bytes(K) + mask;
  const size_t cap = need < OZ_WS_CAP ? need : OZ_WS_CAP;
  return (cap > one ? cap : (one < 4 * OZ_WS_CAP ? one : 4 * OZ_WS_CAP)) + 4096;
}

// The tensor-core form is seven launches, 100 to 130 us for the smallest products; the FP64
// pipe does 1.1 TFLOP/s on tiles that fill the chip, and less on others. Whole DF calls whose
// last product alone is past the line, digits against FMAs: 1128 / 1090 us at 1.0e8 operations,
// 1488 / 1500 at 1.8e8, 1811 / 1884 at 2.4e8; with three products of 1.1e8 to 2.2e8 of
// which two have a side of 8: 1038 / 2619 us. So the line lies where full tiles lose 40 us.
static bool oz_worthwhile(double flops) { return flops >= 1e8; }

cudaError_t launch_gemm(cudaStream_t st, const GemmArgs& g0, const OzWork& w, int* launches) {
  GemmArgs g = g0;
  if (g.M <= 0 || g.N <= 0 || g.nb <= 0) return cudaSuccess;
  int none = 0, &count = launches ? *launches : none;
  // batches that are one matrix: the shared operand's problems follow one another
  if (g.nb > 1 && g.sb == 0 && g.sa == (long long)g.M * g.ai && g.sc == (long long)g.M * g.ci &&
      (long long)g.M * g.nb < (1ll << 30)) {
    g.M *= g.nb;
    g.nb = 1;
  } else if (g.nb > 1 && g.sa == 0 && g.sb == (long long)g.N * g.bj && g.sc == (long long)g.N * g.cj &&
             (long long)g.N * g.nb < (1ll << 30)) {
    g.N *= g.nb;
    g.nb = 1;
  }
  const long long K = (long long)g.L1 * g.L2;
  const double flops = 2.0 * g.M * g.N * (double)K * g.nb;
  if (!w.mem || !oz_worthwhile(flops) || K > OZ_MAX_K) {
    ++count;
    return launch_gemm_fp64(st, g0);
  }
  // the operand on the 128-row side: the one that wastes less of the tiles
  auto tiles = [](long long m, long long n) {
    return oz_up(m, OZ_BM) * oz_up(n, OZ_BN);
  };
  const bool swap = tiles(g.N, g.M) < tiles(g.M, g.N);
  const int m = swap ? g.N : g.M, n = swap ? g.M : g.N;
  const double *pm = swap ? g.Bm : g.A, *pn = swap ? g.A : g.Bm;
  const long long rm = swap ? g.bj : g.ai, m1 = swap ? g.b1 : g.a1, m2 = swap ? g.b2 : g.a2,
                  zm = swap ? g.sb : g.sa;
  const long long rn = swap ? g.ai : g.bj, n1 = swap ? g.a1 : g.b1, n2 = swap ? g.a2 : g.b2,
                  zn = swap ? g.sa : g.sb;
  const long long cm = swap ? g.cj : g.ci, cn = swap ? g.ci : g.cj;
  const bool share_m = g.nb > 1 && zm == 0, share_n = g.nb > 1 && zn == 0;
  const size_t rb = oz_row_bytes(K);
  const size_t avail = w.bytes > 2048 ? w.bytes - 2048 : 0;
  const size_t mb128 = oz_mask_bytes(OZ_BM, n, 1);  // mask of 128 rows
  const long long np = oz_up(n, OZ_ROW_PAD);
  long long mb = oz_up(m, OZ_ROW_PAD);  // rows of the 128-row side at a time
  // problems at a time
  const size_t fixed = ((share_m ? mb : 0) + (share_n ? np : 0)) * rb;
  const size_t per = ((share_m ? 0 : mb) + (share_n ? 0 : np)) * rb + mb / OZ_BM * mb128;
  long long zb = fixed + per <= avail ? (long long)((avail - fixed) / per) : 0;
  if (zb > g.nb) zb = g.nb;
  if (zb < 1) {
    // not even one problem: a problem's rows in blocks
    const size_t left = avail > np * rb ? avail - np * rb : 0;
    mb = (long long)(left / (OZ_ROW_PAD * rb + mb128)) * OZ_ROW_PAD;
    if (mb < OZ_ROW_PAD) {
      ++count;
      return launch_gemm_fp64(st, g0);
    }
    zb = 1;
  }
  uint8_t* base = (uint8_t*)w.mem;
  const long long m_rows = mb * (share_m ? 1 : zb), n_rows = np * (share_n ? 1 : zb);
  __nv_bfloat16* plm = (__nv_bfloat16*)base;
  __nv_bfloat16* pln = (__nv_bfloat16*)(base + oz_up(oz_plane_bytes(m_rows, K), 256));
  int* xm = (int*)((uint8_t*)pln + oz_up(oz_plane_bytes(n_rows, K), 256));
  int* xn = (int*)((uint8_t*)xm + m_rows * OZ_ROW_INFO);
  void* mask = (uint8_t*)xn + n_rows * OZ_ROW_INFO;  // (row counts are multiples of 128)
  cudaError_t e;
  for (long long z0 = 0; z0 < g.nb; z0 += zb) {
    const int nz = (int)(g.nb - z0 < zb ? g.nb - z0 : zb);
    OzArgs a;
    a.b = oz_rows(pn + z0 * zn, share_n ? 1 : nz, n, (int)np, rn, zn, g.L1, g.L2, n1, n2);
    if (z0 == 0 || !share_n) {
      if ((e = oz_pack(st, a.b, pln, xn)) != cudaSuccess) return e;
      count += OZ_PACK_LAUNCHES;
    }
    for (long long r0 = 0; r0 < m; r0 += mb) {
      const int mr = (int)(m - r0 < mb ? m - r0 : mb);
      a.a = oz_rows(pm + z0 * zm + r0 * rm, share_m ? 1 : nz, mr, (int)(mb < m ? oz_up(mr, OZ_ROW_PAD) : mb),
                    rm, zm, g.L1, g.L2, m1, m2);
      if (z0 == 0 || !share_m || mb < m) {
        if ((e = oz_pack(st, a.a, plm, xm)) != cudaSuccess) return e;
        count += OZ_PACK_LAUNCHES;
      }
      a.aexp = xm;
      a.bexp = xn;
      a.status = w.status;
      a.C = g.C + z0 * g.sc + r0 * cm;
      a.ci = cm;
      a.cj = cn;
      a.sc = g.sc;
      a.M = mr;
      a.N = n;
      a.pairs = nullptr;
      a.p0 = 0;
      a.pstep = 1;
      a.arow0 = a.brow0 = 0;
      a.astep = share_m ? 0 : a.a.rpad;
      a.bstep = share_n ? 0 : a.b.rpad;
      a.alpha = g.alpha;
      a.accumulate = g.accumulate;
      a.mask = mask;
      if ((e = oz_multiply(st, plm, pln, a, nz)) != cudaSuccess) return e;
      count += OZ_MULTIPLY_LAUNCHES;
    }
  }
  return cudaSuccess;
}

}  // namespace dsrg
