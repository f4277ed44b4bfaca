// The integral factorisations of Sec. II.C, in FP64.
//
// Density fitting in the MO basis:
//   (pq|P) = sum_{mu nu} C_{mu p} (mu nu|P) C_{nu q}             (two GEMMs per P)
//   B^Q_pq = sum_P [W]_QP (pq|P),  W W^T = J^{-1}
// The paper writes W = J^{-1/2}; any W with W W^T = J^{-1} gives the same
// integrals (pq|rs) = sum_Q B^Q_pq B^Q_rs and hence the same energy, and this
// code takes W = L^{-1} from the Cholesky factor J = L L^T (one forward
// elimination instead of an eigendecomposition of the metric). The factors
// then differ from the J^{-1/2} ones by an orthogonal rotation of Q.
//
// Cholesky decomposition of the integrals: the matrix M[(pq),(rs)] = (pq|rs)
// is given implicitly by factors F^k_pq (M = sum_k F^k (F^k)^T); the pivoted
// incomplete Cholesky decomposition (outer-product form with diagonal
// pivoting, Golub & Van Loan) picks at step k the pair p with the largest
// remaining diagonal d_p, forms L[:,k] = (M[:,p] - sum_{j<k} L[:,j] L[p,j]) /
// sqrt(d_p) and subtracts L[:,k]^2 from d, until max d < tau. The whole loop
// runs on the device (a flag stops the remaining steps); the host reads the
// rank at the end.
#include <cmath>
#include <new>
#include <vector>

#include "coop.cuh"
#include "internal.cuh"
#include "oz_gemm.cuh"

namespace dsrg {
namespace {

// ---------------------------- Cholesky of the metric ----------------------------
// Blocked right-looking Cholesky on the lower triangle of A, CB columns at a time:
// the diagonal block in one CTA, the panel below it with one warp per row, the trailing
// update in CB x CB tiles. An SM does two FP64 FMAs a clock, so what counts is that
// every step spreads over all of them: 3 launches per CB columns and small tiles
// (one column per step, 2 naux launches, took 60 ms at naux = 1200; 2.6 ms now). A
// non-positive pivot sets *bad.
constexpr int CB = 32;

__global__ void __launch_bounds__(256) chol_diag_kernel(double* __restrict__ A, int n, int k0,
                                                        int* __restrict__ bad) {
  __shared__ double t[CB][CB + 1];
  const int nb = min(CB, n - k0);
  for (int e = threadIdx.x; e < CB * CB; e += 256) {
    const int i = e / CB, j = e % CB;
    t[i][j] = (i < nb && j <= i) ? A[(size_t)(k0 + i) * n + k0 + j] : (i == j ? 1.0 : 0.0);
  }
  __syncthreads();
  for (int k = 0; k < nb; ++k) {
    const double akk = t[k][k];
    if (!(akk > 0.0)) {  // the same value in every thread
      if (threadIdx.x == 0) atomicExch(bad, 1);
      return;
    }
    const double r = 1.0 / sqrt(akk);
    __syncthreads();
    if (threadIdx.x >= k && threadIdx.x < nb) t[threadIdx.x][k] *= r;
    __syncthreads();
    for (int e = threadIdx.x; e < CB * CB; e += 256) {
      const int i = e / CB, j = e % CB;
      if (j > k && i >= j) t[i][j] = fma(-t[i][k], t[j][k], t[i][j]);
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < CB * CB; e += 256) {
    const int i = e / CB, j = e % CB;
    if (i < nb && j <= i) A[(size_t)(k0 + i) * n + k0 + j] = t[i][j];
  }
}

// Rows i >= k0 + CB of the panel: x L_kk^T = a, one warp per row, lane j holds x_j.
__global__ void __launch_bounds__(128) chol_panel_kernel(double* __restrict__ A, int n, int k0) {
  __shared__ double t[CB][CB + 1], rd[CB];
  for (int e = threadIdx.x; e < CB * CB; e += 128) {
    const int i = e / CB, j = e % CB;
    t[i][j] = j <= i ? A[(size_t)(k0 + i) * n + k0 + j] : 0.0;
  }
  __syncthreads();
  if (threadIdx.x < CB) rd[threadIdx.x] = 1.0 / t[threadIdx.x][threadIdx.x];
  __syncthreads();
  const int lane = threadIdx.x & 31, i = k0 + CB + blockIdx.x * 4 + (threadIdx.x >> 5);
  if (i >= n) return;
  double a = A[(size_t)i * n + k0 + lane];
#pragma unroll 4
  for (int k = 0; k < CB; ++k) {
    const double x = __shfl_sync(0xffffffffu, a, k) * rd[k];
    if (lane == k) a = x;
    if (lane > k) a = fma(-x, t[lane][k], a);
  }
  A[(size_t)i * n + k0 + lane] = a;
}

// A[i][j] -= sum_k L[i][k] L[j][k] over the panel's CB columns, tiles on or below the diagonal.
__global__ void __launch_bounds__(256) chol_update_kernel(double* __restrict__ A, int n, int k0) {
  if (blockIdx.x > blockIdx.y) return;
  __shared__ double si[CB][CB + 1], sj[CB][CB + 1];
  const int i0 = k0 + CB + blockIdx.y * CB, j0 = k0 + CB + blockIdx.x * CB;
  for (int e = threadIdx.x; e < CB * CB; e += 256) {
    const int r = e / CB, c = e % CB;
    si[r][c] = i0 + r < n ? A[(size_t)(i0 + r) * n + k0 + c] : 0.0;
    sj[r][c] = j0 + r < n ? A[(size_t)(j0 + r) * n + k0 + c] : 0.0;
  }
  __syncthreads();
  const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 8
  for (int k = 0; k < CB; ++k) {
    const double b = sj[c][k];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = fma(si[r0 + 8 * q][k], b, acc[q]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = i0 + r0 + 8 * q, j = j0 + c;
    if (i < n && j <= i) A[(size_t)i * n + j] -= acc[q];
  }
}

// L^{-1} (lower triangular, Li zeroed before), the diagonal blocks of CB columns: one warp
// per block, lane c its column c, Li[i][c] = (delta_ic - sum_{k<i} L[i][k] Li[k][c]) / L[i][i].
__global__ void __launch_bounds__(32) tri_diag_kernel(const double* __restrict__ L, int n,
                                                      double* __restrict__ Li) {
  __shared__ double t[CB][CB + 1], rd[CB];
  const int lane = threadIdx.x, k0 = blockIdx.x * CB, nb = min(CB, n - k0);
  for (int i = 0; i < CB; ++i)
    t[i][lane] = (i < nb && lane <= i) ? L[(size_t)(k0 + i) * n + k0 + lane] : (i == lane ? 1.0 : 0.0);
  __syncwarp();
  rd[lane] = 1.0 / t[lane][lane];
  __syncwarp();
  double x[CB];
#pragma unroll
  for (int i = 0; i < CB; ++i) {
    double v = i == lane ? 1.0 : 0.0;
#pragma unroll
    for (int k = 0; k < i; ++k) v = fma(-t[i][k], x[k], v);
    x[i] = v * rd[i];
    if (i < nb && lane <= i) Li[(size_t)(k0 + i) * n + k0 + lane] = x[i];
  }
}

// ... and the rest by doubling: with the inverses of two neighbouring diagonal blocks of
// sizes w and w2 <= w, the block below the first is -Li_22 (L_21 Li_11), all pairs of a
// size at once. L_21 Li_11 waits, transposed, in the upper triangle of L, which nothing
// reads. (By forward substitution, a warp per column: 3.9 ms at naux = 1200, 0.9 ms now.)
cudaError_t tri_inverse(cudaStream_t st, double* L, int n, double* Li, const OzWork& ow) {
  cudaError_t e = cudaMemsetAsync(Li, 0, (size_t)n * n * 8, st);
  if (e != cudaSuccess) return e;
  tri_diag_kernel<<<(n + CB - 1) / CB, 32, 0, st>>>(L, n, Li);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  for (long long w = CB; w < n; w *= 2) {
    const int full = (int)(n / (2 * w));                 // pairs of two whole blocks
    const long long at = 2 * w * full, last = n - at - w;  // and one with a shorter second
    for (int ragged = 0; ragged < 2; ++ragged) {
      const int nb = ragged ? (last > 0 ? 1 : 0) : full;
      if (nb == 0) continue;
      const long long o = ragged ? at : 0, step = 2 * w * (n + 1);
      const int w1 = (int)w, w2 = (int)(ragged ? last : w);
      const double* L21 = L + (o + w) * n + o;
      double* T = L + o * n + o + w;  // T[i][j] at [j][i]
      double *L11 = Li + o * (n + 1), *L22 = Li + (o + w) * (n + 1), *X = Li + (o + w) * n + o;
      GemmArgs g = batched(mk(w2, w1, w1, 1, L21, n, 1, 0, L11, n, 0, 1, T, 1, n, 1.0), nb, step, step, step);
      g.accumulate = 0;
      if ((e = launch_gemm(st, g, ow)) != cudaSuccess) return e;
      g = batched(mk(w2, w1, w2, 1, L22, n, 1, 0, T, 1, 0, n, X, n, 1, -1.0), nb, step, step, step);
      g.accumulate = 0;
      if ((e = launch_gemm(st, g, ow)) != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// A second stream beside st for the scope: work queued on it starts after st's so far.
struct SideStream {
  cudaStream_t s = nullptr;
  cudaEvent_t ev = nullptr;
  bool open(cudaStream_t st) {
    int lo = 0, hi = 0;
    return cudaDeviceGetStreamPriorityRange(&lo, &hi) == cudaSuccess &&
           cudaStreamCreateWithPriority(&s, cudaStreamNonBlocking, hi) == cudaSuccess &&
           cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) == cudaSuccess &&
           cudaEventRecord(ev, st) == cudaSuccess && cudaStreamWaitEvent(s, ev, 0) == cudaSuccess;
  }
  bool join(cudaStream_t st) {
    return cudaEventRecord(ev, s) == cudaSuccess && cudaStreamWaitEvent(st, ev, 0) == cudaSuccess;
  }
  ~SideStream() {
    if (s) cudaStreamSynchronize(s);  // (an error left it unjoined)
    if (ev) cudaEventDestroy(ev);
    if (s) cudaStreamDestroy(s);
  }
};

// ------------------------------ pivoted Cholesky ------------------------------
struct CdState {
  int rank;     // vectors accepted
  GridBar bar;
};
struct CdSlot {
  double v;
  long long i;
};
constexpr int CD_SLOTS = 2048;  // CTAs of the decomposition, at most
constexpr size_t CD_MIN_EXTRA = 88;  // bytes a work array has beyond the diagonal, at least
static_assert(sizeof(CdState) <= CD_MIN_EXTRA, "the state lies there");

// Stream-ordered memory for the scope.
struct StreamAlloc {
  cudaStream_t st;
  void* p = nullptr;
  explicit StreamAlloc(cudaStream_t s) : st(s) {}
  void* get(size_t bytes) {
    if (cudaMallocAsync(&p, bytes, st) != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
    return p;
  }
  ~StreamAlloc() {
    if (p) cudaFreeAsync(p, st);
  }
};

// d[p] = M_pp = sum_k F[k][p]^2 (p over the N = n^2 pairs)
__global__ void cd_diag_kernel(const double* __restrict__ F, int K0, size_t N, double* __restrict__ d) {
  const size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N) return;
  double acc = 0.0;
  for (int k = 0; k < K0; ++k) {
    const double f = F[(size_t)k * N + p];
    acc = fma(f, f, acc);
  }
  d[p] = acc;
}

// The whole decomposition in one cooperative launch, one barrier per vector. Step k:
// every CTA knows the largest remaining diagonal of its elements (ties: the lowest
// index) and reads the others'; the column of the winner p,
//   L[:, k] = (M[:, p] - sum_{j<k} L[:, j] L[p, j]) / sqrt(d_p), M[:, p] = sum_kk F_kk F_kk[p],
// is formed by tiles of 32 elements with 8 warps sharing the sum over kk and j (in
// fixed parts, added in order), then d -= L[:, k]^2. Stops at max d < tau or max_rank.
// (As three launches per step up to max_rank, n^2 by default, most of them after the
// end: 31.9 ms for n = 56 and 240 vectors; 3.1 ms now, and 3.9 ms with 16 warps a CTA.)
constexpr int CD_T = 32, CD_W = 8;
__global__ void __launch_bounds__(CD_T * CD_W) cd_run_kernel(const double* __restrict__ F, int K0,
                                                             long long N, double tau, int max_rank,
                                                             double* __restrict__ L,
                                                             double* __restrict__ d,
                                                             CdSlot* __restrict__ slots,
                                                             CdState* __restrict__ st) {
  __shared__ double part[CD_W][CD_T];
  __shared__ double sv[CD_W];
  __shared__ long long si[CD_W];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tid = threadIdx.x;
  const long long ntile = (N + CD_T - 1) / CD_T;
  unsigned gen = 0;
  // the larger of (v, i) and another pair, ties to the lower index
  auto take = [](double& v, long long& i, double w, long long j) {
    if (w > v || (w == v && j < i)) {
      v = w;
      i = j;
    }
  };
  auto warp_max = [&](double& v, long long& i) {
    for (int o = 16; o > 0; o >>= 1)
      take(v, i, __shfl_xor_sync(0xffffffffu, v, o), __shfl_xor_sync(0xffffffffu, i, o));
  };
  double best = -1.0;  // over this thread's elements of d (threads of warp 0)
  long long bi = 0;
  if (warp == 0)
    for (long long t = blockIdx.x; t < ntile; t += gridDim.x) {
      const long long q = t * CD_T + lane;
      if (q < N && d[q] > best) {
        best = d[q];
        bi = q;
      }
    }
  int rank = 0;
  for (;; ++rank) {
    if (warp == 0) {  // the other warps hold no elements of d
      warp_max(best, bi);
      if (lane == 0) slots[(rank & 1) * gridDim.x + blockIdx.x] = CdSlot{best, bi};
    }
    if (!grid_barrier(&st->bar, gen)) return;
    double v = -1.0;
    long long vi = 0;
    for (int c = tid; c < gridDim.x; c += CD_T * CD_W) {
      const CdSlot* sl = &slots[(rank & 1) * gridDim.x + c];
      take(v, vi, __ldcg(&sl->v), __ldcg(&sl->i));
    }
    warp_max(v, vi);
    if (lane == 0) {
      sv[warp] = v;
      si[warp] = vi;
    }
    __syncthreads();
    double dmax = sv[0];
    long long p = si[0];
#pragma unroll
    for (int w = 1; w < CD_W; ++w) take(dmax, p, sv[w], si[w]);
    if (dmax < tau || rank >= max_rank) break;
    const double rs = sqrt(dmax);
    best = -1.0;
    bi = 0;
    for (long long t = blockIdx.x; t < ntile; t += gridDim.x) {
      const long long q = t * CD_T + lane;
      double m = 0.0;
      if (q < N) {
#pragma unroll 16
        for (int kk = warp; kk < K0; kk += CD_W) m = fma(F[(size_t)kk * N + q], F[(size_t)kk * N + p], m);
#pragma unroll 16
        for (int j = warp; j < rank; j += CD_W)
          m = fma(-__ldcg(&L[(size_t)j * N + q]), __ldcg(&L[(size_t)j * N + p]), m);
      }
      part[warp][lane] = m;
      __syncthreads();
      if (warp == 0 && q < N) {
        double sum = part[0][lane];
#pragma unroll
        for (int w = 1; w < CD_W; ++w) sum += part[w][lane];
        const double x = sum / rs;
        L[(size_t)rank * N + q] = x;
        const double nd = q == p ? 0.0 : d[q] - x * x;
        d[q] = nd;
        if (nd > best) {
          best = nd;
          bi = q;
        }
      }
      __syncthreads();
    }
  }
  if (blockIdx.x == 0 && tid == 0) st->rank = rank;
}

// Workspace of the products on the tensor cores (the largest of them; 0 where they
// are too small for it).
size_t df_gemm_bytes(int nbf, int naux, int np, int nq) {
  size_t a = oz_work_bytes(np, nbf, nbf, naux, true, false);
  const size_t b = oz_work_bytes((long long)np * naux, nq, nbf, 1, false, false);
  const size_t c = oz_work_bytes(naux, (long long)np * nq, naux, 1, false, false);
  a = a > b ? a : b;
  a = a > c ? a : c;
  for (long long w = CB; w < naux; w *= 2) {  // tri_inverse
    const long long nb = naux / (2 * w) > 0 ? naux / (2 * w) : 1;
    const size_t t = oz_work_bytes(w, w, w, nb, false, false);
    a = a > t ? a : t;
  }
  return a;
}

}  // namespace
}  // namespace dsrg

using namespace dsrg;

extern "C" {

dsrg_status_t dsrg_df_mo_transform(const double* ao3, const double* C, const double* metric,
                                   int32_t nbf, int32_t nmo, int32_t naux, int32_t p0, int32_t np,
                                   int32_t q0, int32_t nq, double* B_out, double* work,
                                   size_t work_bytes, void* cuda_stream) {
  if (!ao3 || !C || !metric || !B_out || !work) return DSRG_ERR_INVALID_ARG;
  if (nbf < 1 || nmo < 1 || naux < 1 || np < 1 || nq < 1 || p0 < 0 || q0 < 0 || p0 + np > nmo ||
      q0 + nq > nmo)
    return DSRG_ERR_INVALID_ARG;
  if (((uintptr_t)ao3 | (uintptr_t)C | (uintptr_t)metric | (uintptr_t)B_out | (uintptr_t)work) & 7u)
    return DSRG_ERR_INVALID_ARG;
  if (work_bytes < dsrg_df_mo_transform_min_work_bytes(nbf, naux, np, nq)) return DSRG_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  double* Y = work;                                        // [naux][np][nbf]
  double* Z = Y + (size_t)naux * np * nbf;                 // [naux][np][nq]
  double* Lm = Z + (size_t)naux * np * nq;                 // [naux][naux] metric -> L
  double* Li = Lm + (size_t)naux * naux;                   // [naux][naux] L^{-1}
  int* bad = (int*)(Li + (size_t)naux * naux);             // and the waits' status word
  OzWork ow;
  // what is left of the work array holds the digits of the products; FP64 FMAs where it is short
  uint8_t* end = (uint8_t*)work + work_bytes;
  uint8_t* mem = (uint8_t*)(((uintptr_t)(bad + 8) + 255) & ~(uintptr_t)255);
  if (mem < end) {
    const size_t left = (size_t)(end - mem), most = df_gemm_bytes(nbf, naux, np, nq);
    ow.mem = mem;
    ow.bytes = left < most ? left : most;
  }
  ow.status = bad + 1;
  if (cudaMemsetAsync(bad, 0, 2 * sizeof(int), st) != cudaSuccess) return DSRG_ERR_CUDA;
  cudaError_t e;
  // J = L L^T: a chain of short launches, beside the two products that do not need it
  SideStream side;
  if (!side.open(st)) return DSRG_ERR_CUDA;
  if (cudaMemcpyAsync(Lm, metric, (size_t)naux * naux * 8, cudaMemcpyDeviceToDevice, side.s) != cudaSuccess)
    return DSRG_ERR_CUDA;
  for (int k = 0; k < naux; k += CB) {
    chol_diag_kernel<<<1, 256, 0, side.s>>>(Lm, naux, k, bad);
    const int left = naux - k - CB;
    if (left > 0) {
      chol_panel_kernel<<<(left + 3) / 4, 128, 0, side.s>>>(Lm, naux, k);
      const unsigned nt = (unsigned)((left + CB - 1) / CB);
      chol_update_kernel<<<dim3(nt, nt), 256, 0, side.s>>>(Lm, naux, k);
    }
  }
  if (cudaGetLastError() != cudaSuccess) return DSRG_ERR_CUDA;
  // Y[P][p][nu] = sum_mu C[mu][p0 + p] ao3[P][mu][nu]
  GemmArgs g1 = batched(mk(np, nbf, nbf, 1, C + p0, 1, nmo, 0, ao3, nbf, 0, 1, Y, nbf, 1, 1.0), naux,
                        0, (long long)nbf * nbf, (long long)np * nbf);
  g1.accumulate = 0;
  // Z[P][p][q] = sum_nu Y[P][p][nu] C[nu][q0 + q]
  GemmArgs g2 = batched(mk(np, nq, nbf, 1, Y, nbf, 1, 0, C + q0, nmo, 0, 1, Z, nq, 1, 1.0), naux,
                        (long long)np * nbf, 0, (long long)np * nq);
  g2.accumulate = 0;
  if ((e = launch_gemm(st, g1, ow)) != cudaSuccess || (e = launch_gemm(st, g2, ow)) != cudaSuccess)
    return DSRG_ERR_CUDA;
  if (!side.join(st) || tri_inverse(st, Lm, naux, Li, ow) != cudaSuccess) return DSRG_ERR_CUDA;
  // B[Q][pq] = sum_P Li[Q][P] Z[P][pq]  (Li lower triangular; the GEMM reads it whole)
  const long long npq = (long long)np * nq;
  GemmArgs g3 = mk(naux, (int)npq, naux, 1, Li, naux, 1, 0, Z, npq, 0, 1, B_out, npq, 1, 1.0);
  g3.accumulate = 0;
  if ((e = launch_gemm(st, g3, ow)) != cudaSuccess) return DSRG_ERR_CUDA;
  int hbad[2] = {0, 0};
  if (cudaMemcpyAsync(hbad, bad, sizeof(hbad), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return DSRG_ERR_CUDA;
  if (hbad[1]) return DSRG_ERR_TIMEOUT;
  return hbad[0] ? DSRG_ERR_INVALID_ARG : DSRG_OK;
}

size_t dsrg_df_mo_transform_min_work_bytes(int32_t nbf, int32_t naux, int32_t np, int32_t nq) {
  return ((size_t)naux * np * nbf + (size_t)naux * np * nq + 2 * (size_t)naux * naux) * 8 + 64;
}

size_t dsrg_df_mo_transform_work_bytes(int32_t nbf, int32_t naux, int32_t np, int32_t nq) {
  return dsrg_df_mo_transform_min_work_bytes(nbf, naux, np, nq) + 448 + df_gemm_bytes(nbf, naux, np, nq);
}

dsrg_status_t dsrg_cd_factors(const double* F, int32_t nfac, int32_t n, double tau,
                              int32_t max_rank, double* L_out, int32_t* rank_out, double* work,
                              size_t work_bytes, void* cuda_stream) {
  if (!F || !L_out || !rank_out || !work || nfac < 1 || n < 1 || max_rank < 1 || !(tau > 0.0))
    return DSRG_ERR_INVALID_ARG;
  if (((uintptr_t)F | (uintptr_t)L_out | (uintptr_t)work) & 7u) return DSRG_ERR_INVALID_ARG;
  const size_t N = (size_t)n * n;
  if (work_bytes < N * 8 + CD_MIN_EXTRA) return DSRG_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  double* d = work;
  CdState* cs = (CdState*)(d + N);
  CdSlot* slots = (CdSlot*)(((uintptr_t)(cs + 1) + 15) & ~(uintptr_t)15);
  StreamAlloc own(st);  // the slots, for a work array that has no room for them
  if (work_bytes < dsrg_cd_factors_work_bytes(n) && !(slots = (CdSlot*)own.get(2 * CD_SLOTS * sizeof(CdSlot))))
    return DSRG_ERR_OOM;
  if (cudaMemsetAsync(cs, 0, sizeof(CdState), st) != cudaSuccess) return DSRG_ERR_CUDA;
  cd_diag_kernel<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(F, nfac, N, d);
  if (cudaGetLastError() != cudaSuccess) return DSRG_ERR_CUDA;
  const long long nt = ((long long)N + CD_T - 1) / CD_T;
  int grid = coop_grid(cd_run_kernel, CD_T * CD_W, 0, (int)(nt < CD_SLOTS ? nt : CD_SLOTS));
  if (grid < 1) return DSRG_ERR_CUDA;
  long long NN = (long long)N;
  int K0 = nfac;
  void* args[] = {(void*)&F, &K0, &NN, &tau, &max_rank, &L_out, &d, &slots, &cs};
  if (cudaLaunchCooperativeKernel((const void*)cd_run_kernel, dim3(grid), dim3(CD_T * CD_W), args, 0,
                                  st) != cudaSuccess)
    return DSRG_ERR_CUDA;
  CdState h{};
  if (cudaMemcpyAsync(&h, cs, sizeof(CdState), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return DSRG_ERR_CUDA;
  if (h.bar.abort) return DSRG_ERR_TIMEOUT;
  *rank_out = h.rank;
  return DSRG_OK;
}

size_t dsrg_cd_factors_work_bytes(int32_t n) {
  return (size_t)n * n * 8 + sizeof(CdState) + 64 + 2 * CD_SLOTS * sizeof(CdSlot);
}

}  // extern "C"
