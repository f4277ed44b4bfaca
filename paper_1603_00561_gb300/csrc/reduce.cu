// Deterministic compensated reduction of the per-CTA partial sums into the
// block energies, and the pair energies of diagram F1 (Eq. (23)).
#include "internal.cuh"

namespace dsrg {

// Neumaier's compensated sum: (s, c) += x.
__device__ __forceinline__ void neumaier_add(double& s, double& c, double x) {
  const double t = s + x;
  if (fabs(s) >= fabs(x))
    c += (s - t) + x;
  else
    c += (x - t) + s;
  s = t;
}

// (a, ca) += (b, cb) of the lane o away; the lower lane's sum comes first in both, so
// both get the same operands in the same order.
__device__ __forceinline__ void neumaier_xor(double& S, double& C, int o) {
  const double oS = __shfl_xor_sync(0xffffffffu, S, o);
  const double oC = __shfl_xor_sync(0xffffffffu, C, o);
  const bool low = (threadIdx.x & o) == 0;
  double a = low ? S : oS;
  const double b = low ? oS : S;
  double cc = (low ? C : oC) + (low ? oC : C);
  neumaier_add(a, cc, b);
  S = a;
  C = cc;
}

// Level 1: one CTA of RED_THREADS threads per chunk of RED_CHUNK partials of one
// segment. Each thread sums a fixed strided subset with Neumaier compensation, the
// lanes of a warp meet in a fixed butterfly, thread 0 adds the warps in order. Small
// chunks on many SMs: a compensated add is 7 FP64 instructions, each 64 clocks of a
// scheduler's FP64 pipe (chunks of 4096 on 256 threads took 16 us, of which the
// partials' reads are under 1).
__global__ void __launch_bounds__(RED_THREADS) reduce_chunks_kernel(
    const double* __restrict__ partials, const Segment* __restrict__ segs,
    const int2* __restrict__ chunks, double* __restrict__ red) {
  __shared__ double sh_s[RED_THREADS / 32], sh_c[RED_THREADS / 32];
  const int2 ch = chunks[blockIdx.x];
  const Segment sg = segs[ch.x];
  const int k0 = ch.y * RED_CHUNK;
  const int k1 = min(sg.count, k0 + RED_CHUNK);
  const double* p = partials + sg.begin;
  double s = 0.0, c = 0.0;
  for (int k = k0 + threadIdx.x; k < k1; k += RED_THREADS) neumaier_add(s, c, p[k]);
  for (int o = 1; o < 32; o <<= 1) neumaier_xor(s, c, o);
  if ((threadIdx.x & 31) == 0) {
    sh_s[threadIdx.x >> 5] = s;
    sh_c[threadIdx.x >> 5] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < RED_THREADS / 32; ++w) {
      neumaier_add(s, c, sh_s[w]);
      c += sh_c[w];
    }
    red[2 * blockIdx.x] = s;
    red[2 * blockIdx.x + 1] = c;
  }
}

// Level 2 (one CTA): warp b folds the chunk pairs of block b, lanes in chunk order
// and then a fixed butterfly. out[0..3] = blocks, out[4] = their total.
__global__ void __launch_bounds__(128) reduce_blocks_kernel(const Segment* __restrict__ segs,
                                                            const int2* __restrict__ chunks,
                                                            int nchunks,
                                                            const double* __restrict__ red,
                                                            double* __restrict__ out) {
  __shared__ double blk[4];
  const int b = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double S = 0.0, C = 0.0;
  for (int k = lane; k < nchunks; k += 32) {
    if (segs[chunks[k].x].block != b) continue;
    neumaier_add(S, C, red[2 * k]);
    C += red[2 * k + 1];
  }
  for (int o = 1; o < 32; o <<= 1) neumaier_xor(S, C, o);
  if (lane == 0) blk[b] = S + C;
  __syncthreads();
  if (threadIdx.x != 0) return;
  double T = 0.0, TC = 0.0;
  for (int k = 0; k < 4; ++k) {
    out[k] = blk[k];
    neumaier_add(T, TC, blk[k]);
  }
  out[4] = T + TC;
}

cudaError_t launch_final_reduce(dsrg_plan* p, double* out) {
  if (p->n_chunks > 0) {
    reduce_chunks_kernel<<<p->n_chunks, RED_THREADS, 0, p->stream>>>(p->d_partials, p->d_segs, p->d_chunks,
                                                            p->d_red);
    DSRG_LAUNCH_CHECK(p);
  }
  reduce_blocks_kernel<<<1, 128, 0, p->stream>>>(p->d_segs, p->d_chunks, p->n_chunks, p->d_red, out);
  DSRG_LAUNCH_CHECK(p);
  return cudaSuccess;
}

// Pair energies e[i][j] from the CCVV partials: items are pair-major, n_tp per
// pair; a pair i<j carries e_ij + e_ji = 2 e_ij.
__global__ void pair_energies_kernel(const double* __restrict__ part, const int2* __restrict__ pairs,
                                     int n_pairs, int n_tp, int nC, double* __restrict__ out) {
  const int pidx = blockIdx.x * blockDim.x + threadIdx.x;
  if (pidx >= n_pairs) return;
  double s = 0.0, c = 0.0;
  for (int k = 0; k < n_tp; ++k) neumaier_add(s, c, part[(size_t)pidx * n_tp + k]);
  const double tot = s + c;
  const int2 ij = pairs[pidx];
  if (ij.x == ij.y) {
    out[ij.x * nC + ij.y] = tot;
  } else {
    out[ij.x * nC + ij.y] = 0.5 * tot;
    out[ij.y * nC + ij.x] = 0.5 * tot;
  }
}

cudaError_t launch_pair_energies(dsrg_plan* p, double* pairs) {
  const Segment& sg = p->segs[p->seg_ccvv];
  const int n_tp = sg.count / p->n_pairs;
  pair_energies_kernel<<<(p->n_pairs + 127) / 128, 128, 0, p->stream>>>(
      p->d_partials + sg.begin, p->d_pairs, p->n_pairs, n_tp, p->z.nC, pairs);
  DSRG_LAUNCH_CHECK(p);
  return cudaSuccess;
}

}  // namespace dsrg
