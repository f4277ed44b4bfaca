// Split-precision CAVV (diagram F2), CCAV (diagram F3) and the integrals of
// the active block from one tensor-core GEMM over the hi/lo planes of CCVV.
//
// Every one of these quantities is a product of two rows of the hole x
// particle factors B: (ge|uf), (ge|hx), (hx|h'y) with g, h holes, u an
// active hole, e, f virtuals and x, y active particles. The planes already
// hold the rows (g, e) for every hole g and virtual e (K-major over Q); the
// rows (h, x) of the active particles are appended to them (nH*nA rows,
// padded to 64). One GEMM
//     Y = P[(g,e)] . P[(u,f) ; (h,x)]^T       (hi.hi + hi.lo + lo.hi, FP32 accumulation,
//                                              + lo.lo on tiles where the rows overlap;
//                                              the first 32 auxiliary functions are added
//                                              in the epilogue in FP32 round-to-nearest)
// then holds, at row (g, e):
//     columns u*nVpad + f   ->  (ge|uf) = X_u[e,f] of F2 for g = m core,
//                               M_xu[e,f] = (xe|uf) for g = x active
//     columns XC + h*nA + x ->  (ge|hx): Z_u[m,n,e] = (me|nu) of F3, and the
//                               virtual parts of (ia|ux), (ix|ua)
// (Sec. III step 4: the integrals with active indices are formed explicitly,
// then contracted). CUDA-core kernels then evaluate the F2 and F3 energies, with
// regulators and sums in pairs of FP32 numbers away from D = 0 and in FP64 near it, and
// gather the active-block integrals; (hx|h'y), which has no virtual index, is
// formed in FP64 from B directly.
//
// The GEMM kernel (one CTA per SM, persistent, tiles 128 x 256):
//   warp 0      TMA producer (the whole warp runs the loop, an elected lane issues)
//   warp 1      TMEM allocator and MMA issuer (likewise)
//   warps 2-5   epilogue: TMEM -> registers -> FP32 stores of Y
// Shared memory: 4 stages x (A 128 rows + B 256 rows) x 2 planes x 64 B, 64-byte
// swizzle. TMEM: 2 buffers x 256 columns. Every wait is bounded (about 2 s).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include "ff.cuh"
#include "index.cuh"
#include "internal.cuh"
#include "regulators.cuh"
#include "tc_common.cuh"

namespace dsrg {

constexpr int G_BM = 128, G_BN = 256;
constexpr int G_KB = 64;                              // K bytes per row per stage
constexpr int G_STAGES = 4;
constexpr int G_A_BYTES = G_BM * G_KB;                // 8 KB per plane
constexpr int G_B_BYTES = G_BN * G_KB;                // 16 KB per plane
constexpr int G_STAGE_BYTES = 2 * (G_A_BYTES + G_B_BYTES);
constexpr int G_THREADS = 192;
constexpr uint32_t G_TMEM_COLS = 512;
constexpr int XROW_ALIGN = 64;
constexpr int F2_T = 32;                              // F2 epilogue tile edge

struct TcGemmArgs {
  int a_row0;        // row r of Y is plane row a_row0 + r
  int b_row0;        // column c of Y is plane row b_row0 + c
  int m_tiles, n_tiles;
  int kblocks;        // K stages on the tensor cores: Q from kq0 to the padded end
  int kq0;            // = TAIL_Q: Q < kq0 is added in the epilogue from `tail`
  const float* tail;  // [plane rows + TAIL_PAD][TAIL_Q] fl32(B) of Q < TAIL_Q (tail_off)
  float* Y;
  long long ldy;
  int* status;
};

__host__ __device__ constexpr uint32_t idesc_mn(bool bf16, uint32_t m, uint32_t n) {
  return (1u << 4) | ((bf16 ? 1u : 2u) << 7) | ((bf16 ? 1u : 2u) << 10) | ((n >> 3) << 17) |
         ((m >> 4) << 24);
}

// The MMAs of one K stage of one tile (two K steps). K runs from the last
// auxiliary function to the first and the cross products go before hi*hi: the
// FP32 accumulator truncates toward zero at every instruction, and with
// factors that decrease along Q this keeps it small until the largest terms
// arrive. GRAM (the tile's A rows and B rows overlap, so its diagonal holds
// squares sum_Q P_r^2) also keeps lo*lo, whose omission would bias them low.
template <bool BF16, bool GRAM>
__device__ __forceinline__ void gemm_stage_mmas(uint32_t leader, uint32_t d, uint32_t sa, uint32_t sb,
                                                int kb) {
  constexpr uint32_t idesc = idesc_mn(BF16, G_BM, G_BN);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const uint32_t off = (1 - k) * 32 / 16;
    const uint32_t acc0 = (kb > 0 || k > 0) ? 1u : 0u;
    tc_mma3_if<BF16, GRAM>(leader, d, sa + off + G_A_BYTES / 16, sa + off, sb + off + G_B_BYTES / 16,
                           sb + off, idesc, acc0);
  }
}

template <bool BF16>
__global__ void __launch_bounds__(G_THREADS, 1)
    split_gemm_kernel(const __grid_constant__ CUtensorMap map_hi,
                      const __grid_constant__ CUtensorMap map_lo, const TcGemmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* tiles = smem;
  uint64_t* full = (uint64_t*)(smem + G_STAGES * G_STAGE_BYTES);
  uint64_t* empty = full + G_STAGES;
  uint64_t* tfull = empty + G_STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_items = a.m_tiles * a.n_tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < G_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 4);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tmem_slot)),
                 "r"(G_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    const uint32_t leader = tc_elect();
    if (leader) {
      asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&map_hi) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&map_lo) : "memory");
    }
    __syncwarp();
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x) {
      const int arow = a.a_row0 + (it / a.n_tiles) * G_BM;
      const int brow = a.b_row0 + (it % a.n_tiles) * G_BN;
      for (int kb = 0; kb < a.kblocks; ++kb) {
        if (!TC_WARP_WAIT(&empty[stage], phase ^ 1u, abort_flag, a.status)) {
          ok = false;
          break;
        }
        uint8_t* st = tiles + stage * G_STAGE_BYTES;
        mbar_expect_tx_if(leader, &full[stage], (uint32_t)G_STAGE_BYTES);
        // the last auxiliary functions first (see the K order of the MMA issuer)
        const int kq = a.kq0 + (a.kblocks - 1 - kb) * (G_KB / (BF16 ? 2 : 4));
        tma_load_2d_if(leader, st, &map_hi, &full[stage], kq, arow);
        tma_load_2d_if(leader, st + G_A_BYTES, &map_lo, &full[stage], kq, arow);
        uint8_t* sb = st + 2 * G_A_BYTES;
        tma_load_2d_if(leader, sb, &map_hi, &full[stage], kq, brow);
        tma_load_2d_if(leader, sb + G_A_BYTES, &map_hi, &full[stage], kq, brow + G_BM);
        tma_load_2d_if(leader, sb + G_B_BYTES, &map_lo, &full[stage], kq, brow);
        tma_load_2d_if(leader, sb + G_B_BYTES + G_A_BYTES, &map_lo, &full[stage], kq, brow + G_BM);
        if (++stage == G_STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok && leader) {
      int s = stage;
      uint32_t ph = phase;
      for (int k = 0; k < G_STAGES; ++k) {
        if (--s < 0) {
          s = G_STAGES - 1;
          ph ^= 1u;
        }
        const unsigned long long t0 = gtimer();
        while (!mbar_try(&full[s], ph) && gtimer() - t0 < TC_WAIT_NS) {
        }
      }
    }
  } else if (warp == 1) {
    const uint32_t leader = tc_elect(), tmem_u = tc_uniform(tmem_base);
    const uint32_t tiles_lo = tc_uniform(desc_sw64_lo(su32(tiles)));
    int stage = 0;
    uint32_t phase = 0;
    int tbuf = 0;
    uint32_t tphase = 0;
    bool ok = true, issued = false;
    for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x) {
      if (!TC_WARP_WAIT(&tempty[tbuf], tphase ^ 1u, abort_flag, a.status)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t d = tmem_u + (uint32_t)(tbuf * G_BN);
      const int arow = a.a_row0 + (it / a.n_tiles) * G_BM;
      const int brow = a.b_row0 + (it % a.n_tiles) * G_BN;
      const bool gram = arow < brow + G_BN && brow < arow + G_BM;
      for (int kb = 0; kb < a.kblocks; ++kb) {
        if (!TC_WARP_WAIT(&full[stage], phase, abort_flag, a.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = tiles_lo + (uint32_t)(stage * (G_STAGE_BYTES / 16));
        const uint32_t sb = sa + 2 * G_A_BYTES / 16;
        if (gram)
          gemm_stage_mmas<BF16, true>(leader, d, sa, sb, kb);
        else
          gemm_stage_mmas<BF16, false>(leader, d, sa, sb, kb);
        issued = true;
        tc_commit_if(leader, &empty[stage]);
        if (++stage == G_STAGES) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok) break;
      tc_commit_if(leader, &tfull[tbuf]);
      if (++tbuf == 2) {
        tbuf = 0;
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
    // epilogue: warp w reads TMEM lanes 32*(w%4).. (its rows of the tile)
    const int quarter = warp & 3;
    int tbuf = 0;
    uint32_t tphase = 0;
    for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
      const bool ok = mbar_wait(&tfull[tbuf], tphase, abort_flag, a.status);
      tc_fence_after();
      if (ok) {
        const uint32_t t = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(tbuf * G_BN);
        // fragments of 32 rows x 32 columns (tail_frag): this thread holds the rows
        // r0, + 8, + 16, + 24 and the column pairs cl, cl + 8
        const int r0 = quarter * 32 + (lane >> 2), cl = 2 * (lane & 3);
        float* y = a.Y + (size_t)((it / a.n_tiles) * G_BM + r0) * a.ldy + (it % a.n_tiles) * G_BN + cl;
        const float* ta = a.tail + tail_off(a.a_row0 + (it / a.n_tiles) * G_BM + r0);
        const float* tb = a.tail + tail_off(a.b_row0 + (it % a.n_tiles) * G_BN + cl);
        for (int c0 = 0; c0 < G_BN; c0 += 32) {
          // the first TAIL_Q auxiliary functions in FP32 round-to-nearest
          float x[2][16];
          tail_frag<2>(ta, tb + (size_t)c0 * TAIL_Q, x);
          tmem_add_frag<2>(t + c0, x);
#pragma unroll
          for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
              float* o = y + (long long)(16 * (k >> 3) + 8 * ((k >> 1) & 1)) * a.ldy + c0 + 16 * n +
                         8 * ((k >> 2) & 1);
              *(float2*)o = make_float2(x[n][k], x[n][k + 1]);
            }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[tbuf]);
      if (++tbuf == 2) {
        tbuf = 0;
        tphase ^= 1u;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(G_TMEM_COLS)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// Active-particle rows of the planes and their FP64 copy.
//   plane row xrow0 + h*nA + x  =  B[Q][h][x]  (split like the main rows)
//   Xq[(h*nA + x) * Q + q]      =  B[q][h][x]  (FP64)
// ---------------------------------------------------------------------------
template <bool BF16>
__global__ void xrows_kernel(const double* __restrict__ B, Sizes z, long long xrow0, int Qld,
                             void* __restrict__ hi, void* __restrict__ lo, double* __restrict__ Xq,
                             float* __restrict__ tail) {
  const int T = z.nH * z.nA;
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= (size_t)T * z.Q) return;
  const int t = (int)(k / z.Q), q = (int)(k % z.Q);
  const int h = t / z.nA, x = t % z.nA;
  const double v = B[bidx(z, q, h, x)];
  Xq[k] = v;
  const size_t o = (size_t)(xrow0 + t) * Qld + q;
  // the same split of fl32(B) as the main plane rows
  const float vf = (float)v;
  if (q < TAIL_Q) tail[tail_off(xrow0 + t) + 32 * (q >> 2) + (q & 3)] = vf;
  if (BF16) {
    const __nv_bfloat16 vh = __float2bfloat16_rn(vf);
    ((__nv_bfloat16*)hi)[o] = vh;
    ((__nv_bfloat16*)lo)[o] = __float2bfloat16_rn(vf - __bfloat162float(vh));
  } else {
    uint32_t u = __float_as_uint(vf);
    if ((u & 0x7f800000u) != 0x7f800000u) u = (u + 0xfffu + ((u >> 13) & 1u)) & 0xffffe000u;
    const float vh = __uint_as_float(u);
    uint32_t w = __float_as_uint(vf - vh);
    if ((w & 0x7f800000u) != 0x7f800000u) w = (w + 0xfffu + ((w >> 13) & 1u)) & 0xffffe000u;
    ((float*)hi)[o] = vh;
    ((float*)lo)[o] = __uint_as_float(w);
  }
}

// (hx|h'y) in FP64: one warp per pair t1 <= t2 of active-particle rows.
__global__ void xx_gram_kernel(const double* __restrict__ Xq, int T, int Q, double* __restrict__ Gxx) {
  const int w = (int)(((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  const int npair = T * (T + 1) / 2;
  if (w >= npair) return;
  int t1 = 0, r = w;
  while (r >= T - t1) {
    r -= T - t1;
    ++t1;
  }
  const int t2 = t1 + r;
  const double* a = Xq + (size_t)t1 * Q;
  const double* b = Xq + (size_t)t2 * Q;
  double acc = 0.0;
  for (int q = lane; q < Q; q += 32) acc = fma(a[q], b[q], acc);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) {
    Gxx[(size_t)t1 * T + t2] = acc;
    Gxx[(size_t)t2 * T + t1] = acc;
  }
}

// ---------------------------------------------------------------------------
// F2 (CAVV), spin-adapted (closed-shell spin sum of Table 2's F2):
//   F2 = sum_m sum_{u,v} G_uv sum_ef X_u[e,f] (2 X_v[e,f] - X_v[f,e]) Rv_u Rt_v,
//   X_u[e,f] = (me|uf), D_u = e_m + e_u - e_e - e_f,
//   Rv_u = 1 + exp(-s D_u^2) (Eq. (15)), Rt_v = (1 - exp(-s D_v^2)) / D_v (Eq. (13)).
// One CTA per (m, 32 x 32 tile pair E <= F); for E < F each position (e,f) also
// adds its mirror (f,e), whose X_u[f,e] is the same CTA's transposed tile.
// Away from D = 0 the regulators and sums are pairs of FP32 numbers (ff.cuh);
// |D_u| < 1/4 (or a pair without the flag of pair_info_kernel) takes expm1 and an FP64
// divide.
//
// Bound by FP32 issue: about 120 FP32 instructions per position and active orbital.
// cc-pV5Z size (24/2/1214/3400): 386 us; with the FP64 regulator from factor tables
// 1099 us (FP64 pipe); size 31/5/467/1609: 258 us, 891 us before.
// ---------------------------------------------------------------------------
template <int NA>
__global__ void __launch_bounds__(256) cavv_f2_kernel(const float* __restrict__ Y, long long ldy,
                                                      int nVpad, const double* __restrict__ eps,
                                                      const double* __restrict__ G, double s, Sizes z,
                                                      const int2* __restrict__ tps, int n_tp,
                                                      const double2* __restrict__ pinfo,
                                                      double* __restrict__ partials,
                                                      unsigned long long* __restrict__ counts) {
  extern __shared__ float f2s[];
  float* sX = f2s;                              // [NA][32][33]   X_u[e,f]
  float* sXt = sX + NA * F2_T * (F2_T + 1);     // [NA][32][33]   X_u[f,e]
  __shared__ double sEe[F2_T], sEf[F2_T], sE[NA];
  // e_e, e_f and E_u as FP32 pairs; G as FP32 head + FP32 remainder for FP32 sums
  __shared__ ff sEeP[F2_T], sEfP[F2_T], sEP[NA], sTab[8];
  __shared__ float sGh[NA * NA], sGl[NA * NA];
  __shared__ int sFact, sFar;
  __shared__ double red[8];
  const int m = blockIdx.x / n_tp;
  const int2 ab = tps[blockIdx.x % n_tp];
  const int E0 = ab.x * F2_T, F0 = ab.y * F2_T;
  const int ve = z.nC + z.nA;
  const float* Ym = Y + (size_t)m * nVpad * ldy;
  for (int k = threadIdx.x; k < NA * F2_T * F2_T; k += 256) {
    const int u = k / (F2_T * F2_T), r = (k / F2_T) % F2_T, c = k % F2_T;
    sX[(u * F2_T + r) * (F2_T + 1) + c] = Ym[(size_t)(E0 + r) * ldy + u * nVpad + F0 + c];
    sXt[(u * F2_T + c) * (F2_T + 1) + r] = Ym[(size_t)(F0 + r) * ldy + u * nVpad + E0 + c];
  }
  if (threadIdx.x < F2_T) {  // warp 0
    const int t = threadIdx.x;
    const int e = E0 + t, f = F0 + t;
    const double xe = e < z.nV ? eps[ve + e] : 0.0, xf = f < z.nV ? eps[ve + f] : 0.0;
    sEe[t] = xe;
    sEf[t] = xf;
    sEeP[t] = ff_from(xe);
    sEfP[t] = ff_from(xf);
    // whether every D_u of the tile pair is so far from 0 that exp(-s D_u^2) < 2^-63
    // (then Rv = 1 and Rt = 1/D_u; FP32 with a margin: it only picks a path)
    float elo = e < z.nV ? (float)xe : 3.0e38f, ehi = e < z.nV ? (float)xe : -3.0e38f;
    float flo = f < z.nV ? (float)xf : 3.0e38f, fhi = f < z.nV ? (float)xf : -3.0e38f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      elo = fminf(elo, __shfl_xor_sync(0xffffffffu, elo, o));
      ehi = fmaxf(ehi, __shfl_xor_sync(0xffffffffu, ehi, o));
      flo = fminf(flo, __shfl_xor_sync(0xffffffffu, flo, o));
      fhi = fmaxf(fhi, __shfl_xor_sync(0xffffffffu, fhi, o));
    }
    if (t == 0) {
      int fact = 1, far = 1;
      for (int u = 0; u < NA; ++u) {
        const double E = pinfo[m * z.nA + u].x;
        sE[u] = E;
        sEP[u] = ff_from(E);
        // a pair whose energies leave the range of the FP32 pairs counts as one
        // whose factors overflow
        const float dhi = (float)E - elo - flo, dlo = (float)E - ehi - fhi;
        fact = fact && pinfo[m * z.nA + u].y != 0.0 &&
               fmaxf(fabsf(dhi), fabsf(dlo)) < 1e15f;
        const float dn = dhi <= 0.0f ? dhi : (dlo >= 0.0f ? dlo : 0.0f);
        far = far && (dhi <= -0.25f || dlo >= 0.25f) && dn * dn > 46.0f / (float)s;
      }
      sFact = fact;
      sFar = far && fact;
    }
  }
  if (threadIdx.x < NA * NA) {
    const double g = G[threadIdx.x];
    sGh[threadIdx.x] = (float)g;
    sGl[threadIdx.x] = (float)(g - (double)(float)g);
  }
  if (threadIdx.x >= 248) sTab[threadIdx.x - 248] = ff_exp_entry(threadIdx.x - 248);
  __syncthreads();
  const bool mirror = ab.x < ab.y;
  const bool fact = sFact != 0;
  const bool tile_far = sFar != 0;
  const int c = threadIdx.x & 31;
  const int f = F0 + c;
  const ff kreg = ff_reg_scale(s);
  double acc = 0.0;
  ff accf = {0.f, 0.f};
  unsigned long long near = 0;  // positions of this thread on the expm1 path
  if (threadIdx.x == 0 && !fact) atomicAdd(&counts[DSRG_COUNT_CAVV_UNFACTORABLE], 1ull);
  if (f < z.nV) {
    for (int r = threadIdx.x >> 5; r < F2_T; r += 8) {
      const int e = E0 + r;
      if (e >= z.nV) break;
      const ff eef = ff_add(sEeP[r], sEfP[c]);
      float X[NA], Xt[NA];
      bool far = fact;
#pragma unroll
      for (int u = 0; u < NA; ++u) {
        X[u] = sX[(u * F2_T + r) * (F2_T + 1) + c];
        Xt[u] = sXt[(u * F2_T + r) * (F2_T + 1) + c];
        // the path test, whose threshold is not sharp (both paths are accurate near it)
        far = far && fabsf(sEP[u].h - eef.h) >= 0.25f;
      }
      if (far || tile_far) {
        // every D_u away from 0 (|D_u| >= 1/4): Rt_u = (1 - g_u) / D_u, g_u =
        // exp(-s D_u^2). The exchange
        // combination Q_uv = X_u (2 X_v - Xt_v) [+ mirror], the smooth factor
        // Rv_u = 1 + g_u in [1, 2) and the u sums with G_uv run in FP32 with
        // round-to-nearest (unbiased; G as head + remainder, so its own rounding
        // is not a systematic error); each v sum meets Rt_v as a pair. The
        // remainder sums take Rt in FP32 (they are 2^-24 of the head sums).
        ff Rt[NA];
        float a[NA], at[NA];
#pragma unroll
        for (int u = 0; u < NA; ++u) {
          const ff D = ff_diff(sEP[u], eef);
          Rt[u] = ff_inv(D);
          float w = 1.0f;
          if (!tile_far) {
            const ff om = ff_one_minus_exp(D, kreg, sTab);
            Rt[u] = ff_mul(om, Rt[u]);
            w = 1.0f + ((1.0f - om.h) - om.l);
          }
          a[u] = w * X[u];
          at[u] = w * Xt[u];
        }
        // sum_u G_uv Rv_u Q_uv = (2 X_v - Xt_v) sum_u G_uv Rv_u X_u
        //                       [+ (2 Xt_v - X_v) sum_u G_uv Rv_u Xt_u for the mirror]
        float tl = 0.0f;
#pragma unroll
        for (int v = 0; v < NA; ++v) {
          float zh = 0.0f, zl = 0.0f, zth = 0.0f, ztl = 0.0f;
#pragma unroll
          for (int u = 0; u < NA; ++u) {
            // volatile: reloaded per position instead of held in 2 NA^2 registers
            const float gh = ((volatile float*)sGh)[u * NA + v];
            const float gl = ((volatile float*)sGl)[u * NA + v];
            zh = fmaf(gh, a[u], zh);
            zl = fmaf(gl, a[u], zl);
            if (mirror) {
              zth = fmaf(gh, at[u], zth);
              ztl = fmaf(gl, at[u], ztl);
            }
          }
          const float dv = 2.0f * X[v] - Xt[v], dtv = 2.0f * Xt[v] - X[v];
          const float ch = mirror ? fmaf(dv, zh, dtv * zth) : dv * zh;
          const float cl = mirror ? fmaf(dv, zl, dtv * ztl) : dv * zl;
          ff_acc(accf, ff_mul(ch, Rt[v]));
          tl = fmaf(cl, Rt[v].h, tl);
        }
        ff_acc(accf, ff{tl, 0.f});
      } else {
        // a D_u near 0 (or a pair whose factors could overflow): expm1 regulators
        // and the exchange combination in FP64
        ++near;
        const double ee = sEe[r] + sEf[c];
        double Rv[NA], Rt[NA];
#pragma unroll
        for (int u = 0; u < NA; ++u) {
          const double D = sE[u] - ee;
          Rt[u] = reg_t(D, s);
          Rv[u] = reg_v(D, s);
        }
        double t1 = 0.0, t2 = 0.0;
#pragma unroll
        for (int v = 0; v < NA; ++v) {
          double c1 = 0.0, c2 = 0.0;
#pragma unroll
          for (int u = 0; u < NA; ++u) {
            const double w = G[u * NA + v] * Rv[u];
            c1 = fma(w, (double)X[u], c1);
            c2 = fma(w, (double)Xt[u], c2);
          }
          t1 = fma(c1, (2.0 * (double)X[v] - (double)Xt[v]) * Rt[v], t1);
          t2 = fma(c2, (2.0 * (double)Xt[v] - (double)X[v]) * Rt[v], t2);
        }
        acc += mirror ? (t1 + t2) : t1;
      }
    }
  }
  if (near) atomicAdd(&counts[DSRG_COUNT_CAVV_NEAR], near);
  const double tot = block_sum<256>(acc + ff_to(accf), red);
  if (threadIdx.x == 0) partials[blockIdx.x] = tot;
}

// ---------------------------------------------------------------------------
// Adjoint of F2 for the gradient of split plans: X_u from the GEMM output Y of
// the energy call just made (its error, about 1e-8 relative, is far below the
// gradient's). Per position (e, f) (and its mirror (f, e) for E < F), with
// P_v = 2 X_v[e,f] - X_v[f,e]:
//   dE/dX_u[e,f] = Rv_u s1_u + Rt_u s2_u,
//   s1_u = sum_v G_uv Rt_v P_v,  s2_u = sum_v G_vu Rv_v P_v,
// and the derivative of the summand with respect to D_u,
//   X_u Rv_u' s1_u + (sum_w G_wu Rv_w X_w) P_u Rt_u',
// goes to e_m and e_u (+) and to e_e, e_f (-); the s derivative likewise.
// Away from D = 0 (the paths of the energy kernel) regulators and sums are pairs of
// FP32 numbers (ff.cuh); near it RegD and FP64. In FP64 throughout, with the
// exponentials from tables and an atomic per position for e_e, the kernel was bound by
// the FP64 pipe: 682 us at 24/2/372/1200, 178 us now.
// ---------------------------------------------------------------------------
// a warp's sum of pairs, the same in every lane
__device__ __forceinline__ ff ff_warp_sum(ff v) {
  for (int o = 16; o > 0; o >>= 1)
    v = ff_add(v, ff{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
  return v;
}
__device__ __forceinline__ ff ff_fma(ff a, ff b, ff c) { return ff_add(c, ff_mul(a, b)); }
__device__ __forceinline__ ff ff_neg(ff a) { return ff{-a.h, -a.l}; }

template <int NA>
__global__ void __launch_bounds__(256) cavv_adj_tc_kernel(
    const float* __restrict__ Y, long long ldy, int nVpad, const double* __restrict__ eps,
    const double* __restrict__ G, double s, Sizes z, const int2* __restrict__ tps, int n_tp,
    const double2* __restrict__ pinfo, double* __restrict__ dX, double* __restrict__ deps,
    double* __restrict__ ds) {
  extern __shared__ float f2s[];
  float* sX = f2s;                              // [NA][32][33]   X_u[e,f]
  float* sXt = sX + NA * F2_T * (F2_T + 1);     // [NA][32][33]   X_u[f,e]
  __shared__ double sEe[F2_T], sEf[F2_T], sE[NA];
  __shared__ ff sEeP[F2_T], sEfP[F2_T], sEP[NA], sG[NA * NA], sTab[8];
  __shared__ int sFact, sFar;
  __shared__ double rowacc[F2_T], colacc[F2_T];
  __shared__ double red[8];
  const int m = blockIdx.x / n_tp;
  const int2 ab = tps[blockIdx.x % n_tp];
  const int E0 = ab.x * F2_T, F0 = ab.y * F2_T;
  const int ve = z.nC + z.nA;
  const float* Ym = Y + (size_t)m * nVpad * ldy;
  for (int k = threadIdx.x; k < NA * F2_T * F2_T; k += 256) {
    const int u = k / (F2_T * F2_T), r = (k / F2_T) % F2_T, c = k % F2_T;
    sX[(u * F2_T + r) * (F2_T + 1) + c] = Ym[(size_t)(E0 + r) * ldy + u * nVpad + F0 + c];
    sXt[(u * F2_T + c) * (F2_T + 1) + r] = Ym[(size_t)(F0 + r) * ldy + u * nVpad + E0 + c];
  }
  if (threadIdx.x < F2_T) {  // warp 0: the paths of cavv_f2_kernel
    const int t = threadIdx.x;
    const int e = E0 + t, f = F0 + t;
    const double xe = e < z.nV ? eps[ve + e] : 0.0, xf = f < z.nV ? eps[ve + f] : 0.0;
    sEe[t] = xe;
    sEf[t] = xf;
    sEeP[t] = ff_from(xe);
    sEfP[t] = ff_from(xf);
    colacc[t] = 0.0;
    float elo = e < z.nV ? (float)xe : 3.0e38f, ehi = e < z.nV ? (float)xe : -3.0e38f;
    float flo = f < z.nV ? (float)xf : 3.0e38f, fhi = f < z.nV ? (float)xf : -3.0e38f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      elo = fminf(elo, __shfl_xor_sync(0xffffffffu, elo, o));
      ehi = fmaxf(ehi, __shfl_xor_sync(0xffffffffu, ehi, o));
      flo = fminf(flo, __shfl_xor_sync(0xffffffffu, flo, o));
      fhi = fmaxf(fhi, __shfl_xor_sync(0xffffffffu, fhi, o));
    }
    if (t == 0) {
      int fact = 1, far = 1;
      for (int u = 0; u < NA; ++u) {
        const double E = pinfo[m * z.nA + u].x;
        sE[u] = E;
        sEP[u] = ff_from(E);
        const float dhi = (float)E - elo - flo, dlo = (float)E - ehi - fhi;
        fact = fact && pinfo[m * z.nA + u].y != 0.0 && fmaxf(fabsf(dhi), fabsf(dlo)) < 1e15f;
        const float dn = dhi <= 0.0f ? dhi : (dlo >= 0.0f ? dlo : 0.0f);
        far = far && (dhi <= -0.25f || dlo >= 0.25f) && dn * dn > 46.0f / (float)s;
      }
      sFact = fact;
      sFar = far && fact;
    }
  }
  if (threadIdx.x < NA * NA) sG[threadIdx.x] = ff_from(G[threadIdx.x]);
  if (threadIdx.x >= 248) sTab[threadIdx.x - 248] = ff_exp_entry(threadIdx.x - 248);
  __syncthreads();
  const bool mirror = ab.x < ab.y;
  const bool fact = sFact != 0;
  const bool tile_far = sFar != 0;
  const int c = threadIdx.x & 31;
  const int f = F0 + c;
  const ff kreg = ff_reg_scale(s), s2 = ff_from(2.0 * s);
  const ff zero = {0.f, 0.f};
  ff dss = zero, cacc = zero, du[NA];
#pragma unroll
  for (int u = 0; u < NA; ++u) du[u] = zero;
  for (int r = threadIdx.x >> 5; r < F2_T; r += 8) {
    const int e = E0 + r;
    if (e >= z.nV) break;
    ff gsum = zero;
    if (f < z.nV) {
      const ff eef = ff_add(sEeP[r], sEfP[c]);
      float X[NA], Xt[NA];
      bool far = fact;
#pragma unroll
      for (int u = 0; u < NA; ++u) {
        X[u] = sX[(u * F2_T + r) * (F2_T + 1) + c];
        Xt[u] = sXt[(u * F2_T + r) * (F2_T + 1) + c];
        far = far && fabsf(sEP[u].h - eef.h) >= 0.25f;
      }
      double* dxp = dX + ((size_t)m * NA * z.nV + e) * z.nV + f;        // (e, f), then (f, e)
      if (far || tile_far) {
        // Rt = (1 - g)/D, Rt' = 2 s g - Rt/D, dRt/ds = D g; Rv = 1 + g, Rv' = -2 s D g,
        // dRv/ds = -D^2 g
        ff Rt[NA], Rd[NA], Rs[NA], Rv[NA];
#pragma unroll
        for (int u = 0; u < NA; ++u) {
          const ff D = ff_diff(sEP[u], eef), inv = ff_inv(D);
          Rt[u] = inv;
          Rs[u] = zero;
          Rv[u] = ff{1.f, 0.f};
          if (!tile_far) {
            const ff om = ff_one_minus_exp(D, kreg, sTab), g = ff_diff(ff{1.f, 0.f}, om);
            Rt[u] = ff_mul(om, inv);
            Rs[u] = ff_mul(D, g);
            Rv[u] = ff_add(ff{1.f, 0.f}, g);
            Rd[u] = ff_diff(ff_mul(g, s2), ff_mul(Rt[u], inv));
          } else {
            Rd[u] = ff_neg(ff_mul(inv, inv));
          }
        }
        // one side per pass: (e, f) with X, then its mirror with X and Xt exchanged
#pragma unroll 1
        for (int side = 0; side < (mirror ? 2 : 1); ++side) {
          ff b[NA], w[NA], x[NA];
#pragma unroll
          for (int v = 0; v < NA; ++v) {
            const ff P = ff_two_sum(2.0f * X[v], -Xt[v]);
            b[v] = ff_mul(Rt[v], P);
            w[v] = ff_mul(Rv[v], P);
            x[v] = ff_mul(X[v], Rv[v]);
          }
#pragma unroll
          for (int u = 0; u < NA; ++u) {
            ff s1 = zero, sw = zero, cw = zero;
#pragma unroll
            for (int v = 0; v < NA; ++v) {
              // volatile: reloaded instead of held in 4 NA^2 registers
              volatile const ff& g1 = sG[u * NA + v];
              volatile const ff& g2 = sG[v * NA + u];
              const ff guv = {g1.h, g1.l}, gvu = {g2.h, g2.l};
              s1 = ff_fma(guv, b[v], s1);
              sw = ff_fma(gvu, w[v], sw);
              cw = ff_fma(gvu, x[v], cw);
            }
            dxp[(size_t)u * z.nV * z.nV] = ff_to(ff_fma(Rt[u], sw, ff_mul(Rv[u], s1)));
            const ff xs = ff_mul(X[u], s1), cp = ff_mul(cw, ff_two_sum(2.0f * X[u], -Xt[u]));
            // X Rv' s1 + cw P Rt' and the same by s: Rv' = -2 s Rs, dRv/ds = -D Rs
            const ff gD = ff_diff(ff_mul(cp, Rd[u]), ff_mul(xs, ff_mul(s2, Rs[u])));
            ff_acc(du[u], gD);
            ff_acc(gsum, gD);
            if (!tile_far) {
              const ff D = ff_diff(sEP[u], eef);
              ff_acc(dss, ff_mul(Rs[u], ff_diff(cp, ff_mul(D, xs))));
            }
          }
#pragma unroll
          for (int v = 0; v < NA; ++v) {
            const float t = X[v];
            X[v] = Xt[v];
            Xt[v] = t;
          }
          dxp = dX + ((size_t)m * NA * z.nV + f) * z.nV + e;
        }
      } else {
        // a D_u near 0 (or a pair whose factors could overflow) in FP64
        const double ee = sEe[r] + sEf[c];
        RegD Rv[NA], Rt[NA];
#pragma unroll
        for (int u = 0; u < NA; ++u) rtv_d(sE[u] - ee, s, Rt[u], Rv[u]);
#pragma unroll 1
        for (int side = 0; side < (mirror ? 2 : 1); ++side) {
#pragma unroll
          for (int u = 0; u < NA; ++u) {
            double s1 = 0.0, sw = 0.0, cw = 0.0;
#pragma unroll
            for (int v = 0; v < NA; ++v) {
              const double P = 2.0 * (double)X[v] - (double)Xt[v], gv = G[v * NA + u] * Rv[v].v;
              s1 = fma(G[u * NA + v] * Rt[v].v, P, s1);
              sw = fma(gv, P, sw);
              cw = fma(gv, (double)X[v], cw);
            }
            const double P = 2.0 * (double)X[u] - (double)Xt[u], xs = (double)X[u] * s1, cp = cw * P;
            dxp[(size_t)u * z.nV * z.nV] = Rv[u].v * s1 + Rt[u].v * sw;
            const ff gD = ff_from(xs * Rv[u].dD + cp * Rt[u].dD);
            ff_acc(du[u], gD);
            ff_acc(gsum, gD);
            ff_acc(dss, ff_from(xs * Rv[u].ds + cp * Rt[u].ds));
          }
#pragma unroll
          for (int v = 0; v < NA; ++v) {
            const float t = X[v];
            X[v] = Xt[v];
            Xt[v] = t;
          }
          dxp = dX + ((size_t)m * NA * z.nV + f) * z.nV + e;
        }
      }
      ff_acc(cacc, gsum);
    }
    __syncwarp();
    const ff t = ff_warp_sum(gsum);  // row r is this warp's alone
    if (c == 0) rowacc[r] = ff_to(t);
  }
  atomicAdd(&colacc[c], ff_to(cacc));
  double tm = 0.0;
  const double ts = block_sum<256>(ff_to(dss), red);
#pragma unroll
  for (int u = 0; u < NA; ++u) {
    const double t = block_sum<256>(ff_to(du[u]), red);
    tm += t;
    if (threadIdx.x == 0) atomicAdd(&deps[z.nC + u], t);
  }
  if (threadIdx.x == 0) {
    atomicAdd(&deps[m], tm);
    atomicAdd(ds, ts);
  }
  if (threadIdx.x < F2_T) {
    const int e = E0 + threadIdx.x, ff_ = F0 + threadIdx.x;
    if (e < z.nV) atomicAdd(&deps[ve + e], -rowacc[threadIdx.x]);
    if (ff_ < z.nV) atomicAdd(&deps[ve + ff_], -colacc[threadIdx.x]);
  }
}

// ---------------------------------------------------------------------------
// F3 (CCAV), spin-adapted:
//   F3 = sum_{u,v} Hh_uv sum_{m,n,e} Z_v[m,n,e] (2 Z_u[m,n,e] - Z_u[n,m,e])
//        (1 + exp(-s D_v^2)) (1 - exp(-s D_u^2))/D_u,
//   Z_u[m,n,e] = (me|nu) = Y[(m,e), XC + n*nA + u], D_u = e_m + e_n - e_e - e_u,
//   Hh = 2 I - G. One CTA per virtual e. Regulators and sums are pairs of FP32
//   numbers (ff.cuh) where every |D_u| >= 1/4, FP64 elsewhere: 31 us against 120 us
//   (FP64 throughout) at the cc-pV5Z size.
// ---------------------------------------------------------------------------
template <int NA>
__global__ void __launch_bounds__(256) ccav_f3_kernel(const float* __restrict__ Y, long long ldy,
                                                      int nVpad, long long xc,
                                                      const double* __restrict__ eps,
                                                      const double* __restrict__ G, double s, Sizes z,
                                                      double* __restrict__ partials) {
  extern __shared__ float f3s[];  // [nC][nC*NA]: Z_u[m,n,e] at m*(nC*NA) + n*NA + u
  __shared__ double sH[NA * NA];
  __shared__ ff sHp[NA * NA], sTab[8];
  __shared__ double red[8];
  const int e = blockIdx.x, nC = z.nC, w = nC * NA;
  for (int k = threadIdx.x; k < nC * w; k += 256) {
    const int m = k / w, r = k % w;
    f3s[k] = Y[(size_t)(m * nVpad + e) * ldy + xc + r];
  }
  if (threadIdx.x < NA * NA) {
    const int u = threadIdx.x / NA, v = threadIdx.x % NA;
    const double h = (u == v ? 2.0 : 0.0) - G[threadIdx.x];
    sH[threadIdx.x] = h;
    sHp[threadIdx.x] = ff_from(h);
  }
  if (threadIdx.x >= 248) sTab[threadIdx.x - 248] = ff_exp_entry(threadIdx.x - 248);
  __syncthreads();
  const double ee = eps[nC + z.nA + e];
  const ff kreg = ff_reg_scale(s);
  double acc = 0.0;
  ff accf = {0.f, 0.f};
  for (int mn = threadIdx.x; mn < nC * nC; mn += 256) {
    const int m = mn / nC, n = mn % nC;
    const double base = eps[m] + eps[n] - ee;
    float Zmn[NA], Znm[NA];
    ff D[NA];
    bool away = true;  // every |D_u| >= 1/4 and within the range of the FP32 pairs
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      Zmn[u] = f3s[m * w + n * NA + u];
      Znm[u] = f3s[n * w + m * NA + u];
      D[u] = ff_from(base - eps[nC + u]);
      away = away && fabsf(D[u].h) >= 0.25f && fabsf(D[u].h) < 1e15f;
    }
    if (away && s <= 1e3) {
      ff Rt[NA], W[NA];  // Rt_u and Rv_u Z_u[m,n,e]
#pragma unroll
      for (int u = 0; u < NA; ++u) {
        const ff om = ff_one_minus_exp(D[u], kreg, sTab);
        Rt[u] = ff_mul(om, ff_inv(D[u]));
        const ff rv = ff_fast_sum(2.0f, -om.h);
        W[u] = ff_mul(Zmn[u], ff{rv.h, rv.l - om.l});
      }
#pragma unroll
      for (int u = 0; u < NA; ++u) {
        const ff zu = ff_two_sum(2.0f * Zmn[u], -Znm[u]);
        ff cc = {0.f, 0.f};
#pragma unroll
        for (int v = 0; v < NA; ++v) ff_acc(cc, ff_mul(sHp[u * NA + v], W[v]));
        ff_acc(accf, ff_mul(cc, ff_mul(zu, Rt[u])));
      }
    } else {
      double Rv[NA], Rt[NA];
#pragma unroll
      for (int u = 0; u < NA; ++u) {
        const double Du = base - eps[nC + u];
        // one exponential for both regulators: for s D^2 > 1/2, 1 - exp(-s D^2) > 0.39
        // has no cancellation; below, expm1
        const double x = s * Du * Du;
        const double g = exp(-x);
        const double em = x > 0.5 ? g - 1.0 : expm1(-x);
        Rv[u] = (1.0 + g) * (double)Zmn[u];
        Rt[u] = Du == 0.0 ? 0.0 : -em / Du;
      }
#pragma unroll
      for (int u = 0; u < NA; ++u) {
        const double zu = 2.0 * (double)Zmn[u] - (double)Znm[u];
        double cc = 0.0;
#pragma unroll
        for (int v = 0; v < NA; ++v) cc = fma(sH[u * NA + v], Rv[v], cc);
        acc = fma(cc, zu * Rt[u], acc);
      }
    }
  }
  const double tot = block_sum<256>(acc + ff_to(accf), red);
  if (threadIdx.x == 0) partials[e] = tot;
}

// ---------------------------------------------------------------------------
// Active-block integrals from Y (virtual indices) and Gxx (active particles):
//   K1[i][u][x][a] = (ia|ux), K2[i][u][x][a] = (ix|ua)   [nH][nA][nA][nP]
//   K3[i][x][j][y] = (ix|jy)                              [nH][nA][nH][nA]
//   M[x][u][e][f]  = (xe|uf)                              [nA][nA][nV][nV]
// ---------------------------------------------------------------------------
__global__ void act_gather_kernel(const float* __restrict__ Y, long long ldy, int nVpad,
                                  long long xc, const double* __restrict__ Gxx, Sizes z,
                                  double* __restrict__ K1, double* __restrict__ K2,
                                  double* __restrict__ K3, double* __restrict__ M) {
  const int nA = z.nA, nC = z.nC, T = z.nH * nA;
  const size_t n12 = (size_t)z.nH * nA * nA * z.nP;
  const size_t n3 = (size_t)T * T;
  const size_t nm = (size_t)nA * nA * z.nV * z.nV;
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < 2 * n12) {
    const bool second = k >= n12;
    const size_t r = second ? k - n12 : k;
    const unsigned r32 = (unsigned)r;  // nH nA^2 nP < 2^31
    const int a = (int)(r32 % z.nP);
    const int x = (int)((r32 / z.nP) % nA);
    const int u = (int)((r32 / (unsigned)(z.nP * nA)) % nA);
    const int i = (int)(r32 / (unsigned)(z.nP * nA * nA));
    double v;
    if (!second) {  // (ia|ux)
      v = (a < nA) ? Gxx[(size_t)(i * nA + a) * T + (nC + u) * nA + x]
                   : (double)Y[(size_t)(i * nVpad + a - nA) * ldy + xc + (nC + u) * nA + x];
      K1[r] = v;
    } else {        // (ix|ua)
      v = (a < nA) ? Gxx[(size_t)(i * nA + x) * T + (nC + u) * nA + a]
                   : (double)Y[(size_t)((nC + u) * nVpad + a - nA) * ldy + xc + i * nA + x];
      K2[r] = v;
    }
  } else if (k < 2 * n12 + n3) {
    const size_t r = k - 2 * n12;  // [i][x][j][y] = Gxx[(i,x)][(j,y)]
    K3[r] = Gxx[r];
  } else if (k < 2 * n12 + n3 + nm) {
    const size_t r = k - 2 * n12 - n3;
    int xu, e, f;
    split_xu_ef(r, z.nV, xu, e, f);
    const int u = xu % nA, x = xu / nA;
    M[r] = (double)Y[(size_t)((nC + x) * nVpad + e) * ldy + (size_t)u * nVpad + f];
  }
}

// ------------------------------- host side -------------------------------
struct RestState {
  int nVpad = 0, XR = 0, ncols = 0, n_tiles = 0, m_tiles = 0, grid = 0;
  long long ldy = 0, xc = 0;
  float* Y = nullptr;
  double* Xq = nullptr;
  double* Gxx = nullptr;
  double2* pinfo = nullptr;  // [nC nA]  E_m + E_u, factorisable flag (pair_info_kernel)
  int2* d_tp = nullptr;
  int n_tp = 0;
};

int rest_xrows(const Sizes& z) {
  if (z.nA == 0) return 0;
  return (z.nH * z.nA + XROW_ALIGN - 1) / XROW_ALIGN * XROW_ALIGN;
}

static void rest_dims(const Sizes& z, RestState* st) {
  st->nVpad = (z.nV + G_BM - 1) / G_BM * G_BM;
  st->XR = rest_xrows(z);
  st->ncols = z.nA * st->nVpad + st->XR;
  st->n_tiles = (st->ncols + G_BN - 1) / G_BN;
  st->m_tiles = z.nH * st->nVpad / G_BM;
  st->ldy = (long long)st->n_tiles * G_BN;
  st->xc = (long long)z.nA * st->nVpad;
  const int nt = (z.nV + F2_T - 1) / F2_T;
  st->n_tp = nt * (nt + 1) / 2;
}

size_t rest_y_bytes(const Sizes& z) {
  if (z.nA == 0) return 0;
  RestState st;
  rest_dims(z, &st);
  return (size_t)z.nH * st.nVpad * st.ldy * sizeof(float);
}

int rest_cavv_blocks(const dsrg_plan* p) {
  RestState st;
  rest_dims(p->z, &st);
  return p->z.nC * st.n_tp;
}

int rest_ccav_blocks(const dsrg_plan* p) { return p->z.nV; }

static size_t gemm_smem_bytes() { return (size_t)G_STAGES * G_STAGE_BYTES + 1024 + 256; }
static size_t f2_smem_bytes(int na) { return (size_t)2 * na * F2_T * (F2_T + 1) * sizeof(float); }
static size_t f3_smem_bytes(const Sizes& z) { return (size_t)z.nC * z.nC * z.nA * sizeof(float); }

bool rest_supported(const Sizes& z) {
  return z.nA <= NA_MAX && f3_smem_bytes(z) <= 200 * 1024;
}

bool rest_alloc(dsrg_plan* p, float* shared_y) {
  const Sizes& z = p->z;
  RestState* st = new RestState();
  p->rest = st;
  rest_dims(z, st);
  int nsm = 148;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->device);
  const int items = st->m_tiles * st->n_tiles;
  st->grid = items < nsm ? items : nsm;
  const int T = z.nH * z.nA;
  bool ok = true;
  if (shared_y)
    st->Y = shared_y;
  else
    ok = plan_alloc(p, (void**)&st->Y, rest_y_bytes(z));
  ok = ok && plan_alloc(p, (void**)&st->Xq, (size_t)T * z.Q * 8) &&
       plan_alloc(p, (void**)&st->Gxx, (size_t)T * T * 8) &&
       plan_alloc(p, (void**)&st->pinfo, (size_t)z.nC * z.nA * sizeof(double2)) &&
       plan_alloc(p, (void**)&st->d_tp, (size_t)st->n_tp * sizeof(int2));
  if (!ok) return false;
  const int nt = (z.nV + F2_T - 1) / F2_T;
  std::vector<int2> tp;
  for (int A = 0; A < nt; ++A)
    for (int B = A; B < nt; ++B) tp.push_back(make_int2(A, B));
  return cudaMemcpy(st->d_tp, tp.data(), tp.size() * sizeof(int2), cudaMemcpyHostToDevice) ==
         cudaSuccess;
}

void rest_free(dsrg_plan* p) {
  delete p->rest;
  p->rest = nullptr;
}

// CAVV and CCAV partials and the active-block integrals K1, K2, K3, M of this
// call (requires the planes staged by the CCVV launch of the same call).
cudaError_t launch_split_rest(dsrg_plan* p, const double* B, const double* eps, const double* G,
                              double s) {
  RestState* st = p->rest;
  const Sizes& z = p->z;
  const bool bf16 = p->prec == DSRG_PREC_BF16X3;
  cudaStream_t stream = p->stream, side = side_stream(p);
  const int T = z.nH * z.nA;
  const long long xrow0 = (long long)z.nH * st->nVpad;
  {
    const size_t n = (size_t)T * z.Q;
    void* hi = split_plane_ptr(p, true);
    void* lo = split_plane_ptr(p, false);
    float* tail = (float*)split_tail_ptr(p);
    const int Qld = split_qld(p);
    if (bf16)
      xrows_kernel<true><<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(B, z, xrow0, Qld, hi, lo,
                                                                         st->Xq, tail);
    else
      xrows_kernel<false><<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(B, z, xrow0, Qld, hi, lo,
                                                                          st->Xq, tail);
    DSRG_LAUNCH_CHECK(p);
  }
  {
    TcGemmArgs a;
    a.a_row0 = 0;
    a.b_row0 = z.nC * st->nVpad;
    a.m_tiles = st->m_tiles;
    a.n_tiles = st->n_tiles;
    a.kq0 = TAIL_Q;
    a.kblocks = (split_qpad(p) - TAIL_Q) / (G_KB / (bf16 ? 2 : 4));
    a.tail = split_tail_ptr(p);
    a.Y = st->Y;
    a.ldy = st->ldy;
    a.status = p->d_status;
    const size_t sm = gemm_smem_bytes();
    const CUtensorMap* mh = split_map(p, true);
    const CUtensorMap* ml = split_map(p, false);
    if (bf16) {
      raise_smem_limit((const void*)split_gemm_kernel<true>, sm);
      split_gemm_kernel<true><<<st->grid, G_THREADS, sm, stream>>>(*mh, *ml, a);
    } else {
      raise_smem_limit((const void*)split_gemm_kernel<false>, sm);
      split_gemm_kernel<false><<<st->grid, G_THREADS, sm, stream>>>(*mh, *ml, a);
    }
    DSRG_LAUNCH_CHECK(p);
  }
  {
    // F2 and F3 read Y only: beside the active block where the call has forked
    if (p->forked) {
      const cudaError_t e = plan_link(stream, p->ev_gemm, p->caller);
      if (e != cudaSuccess) return e;
    }
    pair_info_kernel<<<1, 1024, 0, side>>>(eps, s, z, nullptr, z.nC * z.nA, st->pinfo);
    DSRG_LAUNCH_CHECK(p);
  }
  {
    const Segment& sg = p->segs[p->seg_cavv];
    const size_t sm = f2_smem_bytes(z.nA);
#define F2_LAUNCH(NA_)                                                                             \
  case NA_:                                                                                        \
    raise_smem_limit((const void*)cavv_f2_kernel<NA_>, sm); \
    cavv_f2_kernel<NA_><<<sg.count, 256, sm, side>>>(st->Y, st->ldy, st->nVpad, eps, G, s, z,       \
                                                      st->d_tp, st->n_tp, st->pinfo,              \
                                                      p->d_partials + sg.begin, p->d_counts);     \
    break;
    switch (z.nA) {
      F2_LAUNCH(1) F2_LAUNCH(2) F2_LAUNCH(3) F2_LAUNCH(4)
      F2_LAUNCH(5) F2_LAUNCH(6) F2_LAUNCH(7) F2_LAUNCH(8)
      default: return cudaErrorInvalidValue;
    }
#undef F2_LAUNCH
    DSRG_LAUNCH_CHECK(p);
  }
  {
    const Segment& sg = p->segs[p->seg_ccav];
    const size_t sm = f3_smem_bytes(z);
#define F3_LAUNCH(NA_)                                                                             \
  case NA_:                                                                                        \
    raise_smem_limit((const void*)ccav_f3_kernel<NA_>, sm); \
    ccav_f3_kernel<NA_><<<sg.count, 256, sm, side>>>(st->Y, st->ldy, st->nVpad, st->xc, eps, G, s, \
                                                      z, p->d_partials + sg.begin);              \
    break;
    switch (z.nA) {
      F3_LAUNCH(1) F3_LAUNCH(2) F3_LAUNCH(3) F3_LAUNCH(4)
      F3_LAUNCH(5) F3_LAUNCH(6) F3_LAUNCH(7) F3_LAUNCH(8)
      default: return cudaErrorInvalidValue;
    }
#undef F3_LAUNCH
    DSRG_LAUNCH_CHECK(p);
  }
  {
    const int npair = T * (T + 1) / 2;
    xx_gram_kernel<<<(npair + 7) / 8, 256, 0, stream>>>(st->Xq, T, z.Q, st->Gxx);
    DSRG_LAUNCH_CHECK(p);
  }
  {
    const size_t n = 2 * (size_t)z.nH * z.nA * z.nA * z.nP + (size_t)T * T +
                     (size_t)z.nA * z.nA * z.nV * z.nV;
    act_gather_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(
        st->Y, st->ldy, st->nVpad, st->xc, st->Gxx, z, p->act.K1, p->act.K2, p->act.K3, p->act.M);
    DSRG_LAUNCH_CHECK(p);
  }
  return cudaSuccess;
}

// Adjoint of F2 for split plans (the gradient), after the energy call on the
// same stream: writes dX [nC][nA][nV][nV] and adds to deps, ds.
cudaError_t launch_split_cavv_adjoint(dsrg_plan* p, const double* eps, const double* G, double s,
                                      double* dX, double* deps, double* ds) {
  RestState* st = p->rest;
  const Sizes& z = p->z;
  const size_t sm = f2_smem_bytes(z.nA);
  const unsigned grid = (unsigned)(z.nC * st->n_tp);
  if (grid == 0) return cudaSuccess;
#define F2A_LAUNCH(NA_)                                                                     \
  case NA_:                                                                                 \
    raise_smem_limit((const void*)cavv_adj_tc_kernel<NA_>, sm);                             \
    cavv_adj_tc_kernel<NA_><<<grid, 256, sm, p->stream>>>(st->Y, st->ldy, st->nVpad, eps, G, s, z, \
                                                        st->d_tp, st->n_tp, st->pinfo, dX,  \
                                                        deps, ds);                          \
    break;
  switch (z.nA) {
    F2A_LAUNCH(1) F2A_LAUNCH(2) F2A_LAUNCH(3) F2A_LAUNCH(4)
    F2A_LAUNCH(5) F2A_LAUNCH(6) F2A_LAUNCH(7) F2A_LAUNCH(8)
    default: return cudaErrorInvalidValue;
  }
#undef F2A_LAUNCH
  DSRG_LAUNCH_CHECK(p);
  return cudaSuccess;
}

}  // namespace dsrg
