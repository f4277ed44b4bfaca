// tcgen05 / TMA / mbarrier building blocks shared by the tensor-core kernels
// (inline PTX for sm_103a).
#pragma once

#include <cuda.h>
#include <stdint.h>

namespace dsrg {

constexpr unsigned long long TC_WAIT_NS = 2000000000ull;  // bound of every device-side wait

// The first TAIL_Q auxiliary functions (with decaying factors the largest
// terms) are contracted on CUDA cores in FP32 with round-to-nearest; the
// tensor cores, whose FP32 accumulator truncates toward zero at every
// instruction, take Q >= TAIL_Q.
constexpr int TAIL_Q = 32;
constexpr int TAIL_PAD = 256;  // zero rows after the last plane row of the FP32 tail rows

// ------------------------------- PTX helpers -------------------------------
__device__ __forceinline__ uint32_t su32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait on phase `parity`; false if it ran out or another role aborted.
static __device__ __noinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag,
                                       int* status) {
  if (mbar_try(b, parity)) return true;
  const unsigned long long t0 = gtimer();
  while (true) {
    if (mbar_try(b, parity)) return true;
    if (*abort_flag) return false;
    if (gtimer() - t0 > TC_WAIT_NS) {
      *abort_flag = 1;
      atomicExch(status, 1);
      return false;
    }
  }
}
// Expected bytes and a TMA load of a whole converged warp, by its leader lane (tc_elect).
__device__ __forceinline__ void mbar_expect_tx_if(uint32_t leader, uint64_t* b, uint32_t bytes) {
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n"
               " @q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}\n" ::"r"(su32(b)),
               "r"(bytes), "r"(leader)
               : "memory");
}
__device__ __forceinline__ void tma_load_2d_if(uint32_t leader, void* dst, const CUtensorMap* map,
                                               uint64_t* bar, int c0, int c1) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n"
      " @q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, "
      "%4}], [%2];\n}\n" ::"r"(su32(dst)),
      "l"((unsigned long long)map), "r"(su32(bar)), "r"(c0), "r"(c1), "r"(leader)
      : "memory");
}
// Bring a box of the tensor into L2 ahead of its load (no shared-memory write).
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int c0, int c1) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(
                   (unsigned long long)map),
               "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// One lane of a converged warp (the same one every time); 1 there, 0 elsewhere. An MMA
// issuer runs with its whole warp and predicates the MMAs and commits on this: its
// descriptors are then warp-uniform values the compiler keeps in uniform registers, where
// the MMA reads them. Issued from inside `if (lane == 0)`, every operand is first moved
// there, about 90 clocks an MMA, more than a 128 x 64 one takes.
__device__ __forceinline__ uint32_t tc_elect() {
  uint32_t p;
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
  return p;
}
// A value that is the same in every lane, as a warp-uniform one.
__device__ __forceinline__ uint32_t tc_uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }
// Bounded wait of a whole warp (uniform result): one test in line, the rest in a call.
#define TC_WARP_WAIT(bar, ...)                     \
  (__all_sync(0xffffffffu, mbar_try(bar, FIRST_ARG(__VA_ARGS__))) || \
   __all_sync(0xffffffffu, mbar_wait(bar, __VA_ARGS__)))
#define FIRST_ARG(x, ...) (x)
__device__ __forceinline__ void tc_commit_if(uint32_t leader, uint64_t* bar) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(
          su32(bar)),
      "r"(leader)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   su32(bar))
               : "memory");
}
// Shared-memory matrix descriptor: K-major operand, 64-byte swizzle, rows at a 64-byte
// pitch. Low word: address / 16 (offsets add as offset / 16: shared memory ends below
// 2^18 bytes) and the leading byte offset (unused for swizzled K-major); high word: stride
// byte offset of 8 rows x 64 B, the descriptor version of tcgen05, the swizzle.
constexpr uint32_t DESC_SW64_HI = (512u >> 4) | 1u << 14 | 4u << 29;
__device__ __forceinline__ uint32_t desc_sw64_lo(uint32_t saddr) { return (saddr >> 4) | 1u << 16; }
// The products of a split K step, D (+)= [A_lo B_lo +] A_lo B_hi + A_hi B_lo + A_hi B_hi, by
// the leader lane (tc_elect) of a whole converged warp; descriptors by their low words
// (desc_sw64_lo). `acc` 0: D starts at the first product. A_hi stays in the collector
// buffer between its products. One block for all of them: an MMA takes 64 clocks, and the
// issuing warp, at 4 to 6 clocks an instruction, is what limits short stages (every MMA
// with its own predicates and 64-bit descriptors: 65 clocks each and 575 a stage).
template <bool BF16, bool LOLO>
__device__ __forceinline__ void tc_mma3_if(uint32_t leader, uint32_t d, uint32_t al, uint32_t ah,
                                           uint32_t bl, uint32_t bh, uint32_t idesc, uint32_t acc) {
#define DSRG_MMA3(KIND, FIRST, P2)                                                              \
  asm volatile("{\n .reg .pred p, q;\n .reg .b64 xl, xh, yl, yh;\n"                            \
               " setp.ne.b32 p, %6, 0;\n setp.ne.b32 q, %7, 0;\n"                              \
               " mov.b64 xl, {%1, %8};\n mov.b64 xh, {%2, %8};\n"                              \
               " mov.b64 yl, {%3, %8};\n mov.b64 yh, {%4, %8};\n" FIRST                        \
               " @q tcgen05.mma.cta_group::1.kind::" KIND " [%0], xl, yh, %5, " P2 ";\n"        \
               " @q tcgen05.mma.cta_group::1.kind::" KIND ".collector::a::fill [%0], xh, yl, %5, q;\n"    \
               " @q tcgen05.mma.cta_group::1.kind::" KIND ".collector::a::lastuse [%0], xh, yh, %5, q;\n" \
               "}\n" ::"r"(d),                                                                  \
               "r"(al), "r"(ah), "r"(bl), "r"(bh), "r"(idesc), "r"(acc), "r"(leader),           \
               "r"(DESC_SW64_HI)                                                                \
               : "memory")
#define DSRG_LL(KIND) " @q tcgen05.mma.cta_group::1.kind::" KIND " [%0], xl, yl, %5, p;\n"
  if (BF16 && LOLO) DSRG_MMA3("f16", DSRG_LL("f16"), "q");
  else if (BF16) DSRG_MMA3("f16", "", "p");
  else if (LOLO) DSRG_MMA3("tf32", DSRG_LL("tf32"), "q");
  else DSRG_MMA3("tf32", "", "p");
#undef DSRG_LL
#undef DSRG_MMA3
}
// One MMA D (+)= A B by the leader lane of a whole converged warp.
template <bool BF16>
__device__ __forceinline__ void tc_mma_if(uint32_t leader, uint32_t d, uint32_t a, uint32_t b,
                                          uint32_t idesc, uint32_t acc) {
#define DSRG_MMA1(KIND)                                                                      \
  asm volatile("{\n .reg .pred p, q;\n .reg .b64 x, y;\n"                                    \
               " setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"                            \
               " mov.b64 x, {%1, %6};\n mov.b64 y, {%2, %6};\n"                              \
               " @q tcgen05.mma.cta_group::1.kind::" KIND " [%0], x, y, %3, p;\n}\n" ::"r"(d), \
               "r"(a), "r"(b), "r"(idesc), "r"(acc), "r"(leader), "r"(DESC_SW64_HI)          \
               : "memory")
  if (BF16) DSRG_MMA1("f16");
  else DSRG_MMA1("tf32");
#undef DSRG_MMA1
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15},"
      " [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// 32 TMEM lanes x 16 columns as 16 x 8 fragments: lane l of the warp gets, in
// r[8h + 4g + 2v + e], row 16 h + l / 4 + 8 v and column 8 g + 2 (l % 4) + e.
__device__ __forceinline__ void tmem_ld_frag16(uint32_t taddr, uint32_t (&r)[16]) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[8 * h]), "=r"(r[8 * h + 1]), "=r"(r[8 * h + 2]), "=r"(r[8 * h + 3]),
                   "=r"(r[8 * h + 4]), "=r"(r[8 * h + 5]), "=r"(r[8 * h + 6]), "=r"(r[8 * h + 7])
                 : "r"(taddr + ((uint32_t)(16 * h) << 16)));
}
// 16 columns of the warp's 32 lanes, one register per column
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void named_bar(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
// The FP32 tail rows: fl32(B) of the first TAIL_Q auxiliary functions of every
// plane row, in blocks of 8 rows, [row / 8][q / 4][row % 8][q % 4]. The four
// values of 8 consecutive rows are one 128-byte line, so a warp's load of any 8
// rows at one q / 4 meets every shared-memory/L1 bank once (as 128-byte rows they
// met the same 32 bytes of banks: 25 cycles of the data path per load, which the
// MMAs' operand reads share).
__host__ __device__ __forceinline__ size_t tail_off(size_t row) {
  return (row >> 3) * (8 * TAIL_Q) + (row & 7) * 4;
}

// x_ab += sum_{q < TAIL_Q} T_a[q] T_b[q] for the 16 columns b of one chunk, in
// FP32 with round-to-nearest, q from the last to the first. `ra`: this thread's
// tail row, `rb`: the first of the chunk's 16 rows (a multiple of 8; the same for
// every lane of the warp, so each load is a broadcast).
__device__ __forceinline__ void tail_add16(const float* __restrict__ ra,
                                           const float* __restrict__ rb, uint32_t (&r)[16]) {
  float t[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) t[k] = 0.f;
#pragma unroll 2
  for (int q4 = TAIL_Q / 4 - 1; q4 >= 0; --q4) {
    const float4 a = __ldg((const float4*)(ra + 32 * q4));
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float4 b = __ldg((const float4*)(rb + (k >> 3) * (8 * TAIL_Q) + (k & 7) * 4 + 32 * q4));
      t[k] = fmaf(a.w, b.w, t[k]);
      t[k] = fmaf(a.z, b.z, t[k]);
      t[k] = fmaf(a.y, b.y, t[k]);
      t[k] = fmaf(a.x, b.x, t[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < 16; ++k) r[k] = __float_as_uint(__uint_as_float(r[k]) + t[k]);
}

// The same sums for a block of 32 rows x 16 NC columns in the fragment layout of
// tmem_ld_frag16: a thread's 16 NC elements are 4 rows (`ra`, 8 apart) x 4 NC
// columns (`rb`, pairs 8 apart), so a loaded value feeds 4 NC or 4 FMAs instead of
// one: a load fills registers at 128 bytes a clock and SM, which the row-per-lane
// form above, with 17 loads for 16 FMAs, is bound by. Same FMA order per element.
template <int NC>
__device__ __forceinline__ void tail_frag(const float* __restrict__ ra,
                                          const float* __restrict__ rb, float (&t)[NC][16]) {
#pragma unroll
  for (int n = 0; n < NC; ++n)
#pragma unroll
    for (int k = 0; k < 16; ++k) t[n][k] = 0.f;
#pragma unroll 2
  for (int q4 = TAIL_Q / 4 - 1; q4 >= 0; --q4) {
    float4 a[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) a[v] = __ldg((const float4*)(ra + 8 * TAIL_Q * v + 32 * q4));
#pragma unroll
    for (int c = 0; c < 4 * NC; ++c) {  // column 8 (c / 2) + c % 2 from rb
      const float4 b = __ldg((const float4*)(rb + 8 * TAIL_Q * (c >> 1) + 4 * (c & 1) + 32 * q4));
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        float& s = t[c >> 2][8 * (v >> 1) + 4 * ((c >> 1) & 1) + 2 * (v & 1) + (c & 1)];
        s = fmaf(a[v].w, b.w, s);
        s = fmaf(a[v].z, b.z, s);
        s = fmaf(a[v].y, b.y, s);
        s = fmaf(a[v].x, b.x, s);
      }
    }
  }
}

// Add the tensor cores' rest of the same block from TMEM.
template <int NC>
__device__ __forceinline__ void tmem_add_frag(uint32_t taddr, float (&t)[NC][16]) {
#pragma unroll
  for (int n = 0; n < NC; ++n) {
    uint32_t r[16];
    tmem_ld_frag16(taddr + 16 * n, r);
    tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < 16; ++k) t[n][k] = __uint_as_float(r[k]) + t[n][k];
  }
}

// Instruction descriptor: D = F32, A/B = TF32 (2) or BF16 (1), both K-major, M = 128, N given
// (a multiple of 16, 16..256).
template <bool BF16>
__host__ __device__ constexpr uint32_t idesc_128xn(uint32_t n) {
  return (1u << 4) | ((BF16 ? 1u : 2u) << 7) | ((BF16 ? 1u : 2u) << 10) | ((n >> 3) << 17) |
         ((128u >> 4) << 24);
}
// Instruction descriptor: D = F32, A/B = TF32 (2) or BF16 (1), both K-major, M = N = 128.
template <bool BF16>
__host__ __device__ constexpr uint32_t idesc_128x128() {
  return (1u << 4) | ((BF16 ? 1u : 2u) << 7) | ((BF16 ? 1u : 2u) << 10) | ((128u >> 3) << 17) |
         ((128u >> 4) << 24);
}

}  // namespace dsrg
