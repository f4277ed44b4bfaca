// Generalized Fock matrix and semicanonical orbitals (Sec. II.B, Eq. (8);
// Sec. III, steps 2-3 of the procedure), all FP64.
//
//   f_pq = h_pq + sum_rs D_rs [(pq|rs) - 1/2 (ps|rq)],  (pq|rs) = sum_Q B^Q_pq B^Q_rs
//
// with D the spin-summed density of the reference (2 on the core diagonal, G on
// the active block, 0 on the virtuals): Eq. (8) summed over spin for a
// spin-free density. The Coulomb part is a contraction of the factors with
// w_Q = sum_rs B^Q_rs D_rs; the exchange part K_pq = sum_{Q, r in H}
// X^Q_pr B^Q_rq, X^Q_pr = sum_{s in H} B^Q_ps D_sr, is one GEMM over the
// composite index (Q, r).
//
// The core, active and virtual blocks of f are then diagonalised separately by
// a parallel cyclic Jacobi method (round-robin pairing, m/2 disjoint rotations
// per step; the rotation of each pair as in Golub & Van Loan, Matrix
// Computations, Sec. 8.5, "symmetric Schur decomposition" of a 2 x 2 block).
// Eigenvalues are sorted ascending within each block and each eigenvector's
// largest component is made positive. U = blockdiag(U_C, U_A, U_V) gives
//   eps = diag(U^T f U), f^(1) = hole x particle block of U^T f U (its active x
//   active part, which belongs to the diagonal block, set to 0),
//   B'^Q = U_H^T B^Q_HP U_P, G' = U_A^T G U_A, lambda2' and lambda3' rotated
//   on every active index.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <new>
#include <numeric>
#include <vector>

#include "coop.cuh"
#include "internal.cuh"
#include "oz_gemm.cuh"

namespace dsrg {
struct JacState {
  GridBar bar;
  int sweeps;  // of the slowest block so far
  // status word of the products' bounded waits: kept until a call reports it (the Fock
  // build alone is asynchronous and cannot)
  int wait;
};
}  // namespace dsrg

struct dsrg_sc_plan {
  dsrg::Sizes z{};
  int device = 0;
  cudaStream_t stream = nullptr;
  std::string last_error;
  std::vector<void*> allocs;
  size_t ws_bytes = 0;
  double *w = nullptr;      // [naux]
  double *J = nullptr;      // [n][n]
  double *K = nullptr;      // [nk][n][n]
  double *X = nullptr;      // [naux][n][nH]
  double *f = nullptr;      // [n][n]
  double *U = nullptr;      // [n][n]
  double *T = nullptr;      // [n][n]; the other copy of A during the Jacobi sweeps
  double *A = nullptr;      // [mmax][mmax] Jacobi work matrix
  double *V = nullptr;      // [mmax][mmax] Jacobi eigenvectors
  double *diag = nullptr;   // [mmax] eigenvalues in matrix order
  double2 *slots = nullptr; // [JAC_SLOTS] partial norms
  dsrg::JacState *jac = nullptr;
  int nk = 1;               // partial exchange matrices (parts of the sum over Q)
  dsrg::OzWork oz;          // workspace of the tensor-core products
  double *Bhp = nullptr;    // [naux][nH][nP] gathered hole x particle factors
  double *Bt = nullptr;     // [naux][nH][nP] after the particle rotation
  double *L3t = nullptr;    // [(2 nA)^6] intermediate of the lambda3 rotation
  int mmax = 0;
  int sweeps_last = 0;
};

namespace dsrg {
namespace {

bool sc_alloc(dsrg_sc_plan* p, void** ptr, size_t bytes) {
  *ptr = nullptr;
  if (cudaMalloc(ptr, bytes ? bytes : 8) != cudaSuccess) {
    cudaGetLastError();
    *ptr = nullptr;
    return false;
  }
  p->allocs.push_back(*ptr);
  p->ws_bytes += bytes;
  return true;
}

// ... of at most 2/5 of the free memory.
bool sc_alloc_spare(dsrg_sc_plan* p, void** ptr, size_t bytes) {
  *ptr = nullptr;
  return bytes <= digits_limit() && sc_alloc(p, ptr, bytes);
}

// w_Q = sum_rs B^Q_rs D_rs = 2 sum_m B^Q_mm + sum_uv B^Q_{nC+u, nC+v} G_uv (one warp per Q).
__global__ void fock_w_kernel(const double* __restrict__ B, const double* __restrict__ G, Sizes z,
                              double* __restrict__ w) {
  const int q = (int)(((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (q >= z.Q) return;
  const size_t n = (size_t)z.n;
  const double* Bq = B + (size_t)q * n * n;
  double acc = 0.0;
  for (int m = lane; m < z.nC; m += 32) acc += 2.0 * Bq[(size_t)m * n + m];
  for (int k = lane; k < z.nA * z.nA; k += 32) {
    const int u = k / z.nA, v = k % z.nA;
    acc = fma(Bq[(size_t)(z.nC + u) * n + z.nC + v], G[k], acc);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) w[q] = acc;
}

// J_pq = sum_Q B^Q_pq w_Q: one thread per (p, q), Q outer (coalesced along q).
__global__ void fock_j_kernel(const double* __restrict__ B, const double* __restrict__ w, Sizes z,
                              double* __restrict__ J) {
  const size_t nn = (size_t)z.n * z.n;
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nn) return;
  double acc = 0.0;
  for (int q = 0; q < z.Q; ++q) acc = fma(B[(size_t)q * nn + k], w[q], acc);
  J[k] = acc;
}

// X^Q_pr = sum_{s in H} B^Q_ps D_sr for r in H: 2 B^Q_pm (core m), sum_u B^Q_{p,nC+u} G_uv.
__global__ void fock_x_kernel(const double* __restrict__ B, const double* __restrict__ G, Sizes z,
                              double* __restrict__ X) {
  const size_t total = (size_t)z.Q * z.n * z.nH;
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= total) return;
  const int r = (int)(k % z.nH);
  const size_t qp = k / z.nH;  // q * n + p
  const double* row = B + qp * z.n;
  double v;
  if (r < z.nC) {
    v = 2.0 * row[r];
  } else {
    const int vv = r - z.nC;
    v = 0.0;
    for (int u = 0; u < z.nA; ++u) v = fma(row[z.nC + u], G[u * z.nA + vv], v);
  }
  X[k] = v;
}

// f = h + J - K / 2 (K in nk parts), symmetrised (the two halves round differently only in
// K); NaN if a wait of the product that forms K ran out (its tiles are then not written)
__global__ void fock_sum_kernel(const double* __restrict__ h, const double* __restrict__ J,
                                const double* __restrict__ K, int nk, int n,
                                const int* __restrict__ wait, double* __restrict__ f) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x, nn = (size_t)n * n;
  if (k >= nn) return;
  const int p = (int)(k / n), q = (int)(k % n);
  const size_t kt = (size_t)q * n + p;
  double ka = 0.0, kb = 0.0;
  for (int z = 0; z < nk; ++z) {
    ka += K[z * nn + k];
    kb += K[z * nn + kt];
  }
  const double a = fma(-0.5, ka, h[k] + J[k]);
  const double b = fma(-0.5, kb, h[kt] + J[kt]);
  f[k] = *wait ? __longlong_as_double(0x7ff8000000000000ll) : 0.5 * (a + b);
}

// ---------------------------- Jacobi eigensolver ----------------------------
// Round-robin pairing of mp (even) positions: at step t position 0 stays and
// the others rotate; pair k couples slots k and mp-1-k.
__device__ __forceinline__ int rr_slot(int k, int t, int mp) {
  return k == 0 ? 0 : 1 + (k - 1 + t) % (mp - 1);
}

__global__ void jac_copy_kernel(const double* __restrict__ f, int n, int lo, int m,
                                double* __restrict__ A, double* __restrict__ V) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m * m) return;
  const int i = k / m, j = k % m;
  A[k] = f[(size_t)(lo + i) * n + lo + j];
  V[k] = (i == j) ? 1.0 : 0.0;
}

// The whole diagonalisation in one cooperative launch, one barrier per step (a step is
// 2 us of FP64 work at m = 372; as three launches per step, 11 000 in all, it was the
// launches that took the 90 ms: 20.6 ms of it now). A tile is 16 x 16 pairs of pairs: with
// the (c, s) of its 32 pairs, formed in the CTA from the current diagonal blocks, each
// thread turns one 2 x 2 block A[P][R] -> J_P^T A[P][R] J_R from one copy of A into the
// other, so no CTA waits for another within a step; the same CTA turns 32 rows of V by
// its 16 column pairs in place.
// The angle comes from FP32 and two Newton-Raphson steps; c^2 + s^2 = 1 holds to FP64.
constexpr int JT = 16;
constexpr int JAC_SLOTS = 2048;  // CTAs, at most

__device__ __forceinline__ double2 jac_rotation(double app, double aqq, double apq) {
  if (apq == 0.0) return make_double2(1.0, 0.0);
  // tan of the angle, |t| <= 1; scaled so that the FP32 quotient neither under- nor overflows
  const double num = aqq - app, den = 2.0 * apq;
  const double sc = fmax(fabs(num), fabs(den));
  const int e = ((__double2hiint(sc) >> 20) & 0x7ff) - 1023;
  const double f = __hiloint2double((1023 - (e < -1000 ? -1000 : (e > 1000 ? 1000 : e))) << 20, 0);
  const double nf = num * f, df = den * f, h = 0.5 * df;
  const float tau = (float)nf / (float)df;
  float tf = 1.0f / (fabsf(tau) + sqrtf(fmaf(tau, tau, 1.0f)));
  if (tau < 0.0f) tf = -tf;
  // two Newton-Raphson steps on h t^2 + nf t - h = 0 (slope |nf + df t| >= 1)
  double t = (double)tf;
  const float slope = (float)fma(df, t, nf);
  const double is = (double)(1.0f / slope);
  t = fma(-fma(fma(h, t, nf), t, -h), is, t);
  t = fma(-fma(fma(h, t, nf), t, -h), is, t);
  const double w = fma(t, t, 1.0);
  double c = (double)rsqrtf((float)w);
  c = c * fma(-0.5 * w * c, c, 1.5);
  // both by what is left of c^2 + s^2 = 1: one rounding each, so that thousands of
  // rotations do not shrink or stretch a vector
  double s = t * c;
  const double u = 0.5 * fma(-s, s, fma(-c, c, 1.0));
  c = fma(u, c, c);
  s = fma(u, s, s);
  return make_double2(c, s);
}

__global__ void __launch_bounds__(JT * JT) jac_run_kernel(double* __restrict__ A0,
                                                          double* __restrict__ A1,
                                                          double* __restrict__ V, int m, int mp,
                                                          int max_sweeps, double2* __restrict__ slots,
                                                          double* __restrict__ diag,
                                                          JacState* __restrict__ st) {
  __shared__ double2 rot[2][JT];
  __shared__ double sh0[JT * JT], sh1[JT * JT];
  const int K = mp / 2, nt = (K + JT - 1) / JT, tid = threadIdx.x;
  const int tx = tid % JT, ty = tid / JT;
  unsigned gen = 0;
  double *Ac = A0, *An = A1;
  int sweep = 0;
  for (;; ++sweep) {
    // off-diagonal and whole squared norm, in a fixed order
    double o = 0.0, w = 0.0;
    for (size_t k = (size_t)blockIdx.x * (JT * JT) + tid; k < (size_t)m * m; k += (size_t)gridDim.x * JT * JT) {
      const double x = __ldcg(&Ac[k]);
      w = fma(x, x, w);
      if (k / m != k % m) o = fma(x, x, o);
    }
    sh0[tid] = o;
    sh1[tid] = w;
    __syncthreads();
    for (int h = JT * JT / 2; h > 0; h >>= 1) {
      if (tid < h) {
        sh0[tid] += sh0[tid + h];
        sh1[tid] += sh1[tid + h];
      }
      __syncthreads();
    }
    if (tid == 0) slots[blockIdx.x] = make_double2(sh0[0], sh1[0]);
    if (!grid_barrier(&st->bar, gen)) return;
    o = w = 0.0;
    for (int c = tid; c < gridDim.x; c += JT * JT) {
      const double2 x = __ldcg(&slots[c]);
      o += x.x;
      w += x.y;
    }
    sh0[tid] = o;
    sh1[tid] = w;
    __syncthreads();
    for (int h = JT * JT / 2; h > 0; h >>= 1) {
      if (tid < h) {
        sh0[tid] += sh0[tid + h];
        sh1[tid] += sh1[tid + h];
      }
      __syncthreads();
    }
    const double off = sh0[0], all = sh1[0];
    __syncthreads();
    // (an infinite norm is no convergence)
    if ((off <= 1e-30 * all && all < INFINITY) || off == 0.0 || sweep >= max_sweeps) break;
    for (int t = 0; t < mp - 1; ++t) {
      for (int tile = blockIdx.x; tile < nt * nt; tile += gridDim.x) {
        const int tp = tile / nt, tr = tile % nt;
        // this thread's pairs and, before the rotations are known, its elements: the loads
        // and the rotations' arithmetic overlap
        auto pair = [&](int k, int& i, int& j) {
          i = k < K ? rr_slot(k, t, mp) : m;  // m: no such index
          j = k < K ? rr_slot(mp - 1 - k, t, mp) : m;
        };
        int p, q, r, s;
        pair(tp * JT + ty, p, q);
        pair(tr * JT + tx, r, s);
        auto get = [&](int i, int j) { return i < m && j < m ? __ldcg(&Ac[(size_t)i * m + j]) : 0.0; };
        const double pr = get(p, r), ps = get(p, s), qr = get(q, r), qs = get(q, s);
        double vx[2], vy[2];  // V rows 32 tp .. by the column pairs of this tile
        const bool cols = r < m && s < m;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = 2 * JT * tp + ty + JT * h;
          vx[h] = i < m && cols ? __ldcg(&V[(size_t)i * m + r]) : 0.0;
          vy[h] = i < m && cols ? __ldcg(&V[(size_t)i * m + s]) : 0.0;
        }
        __syncthreads();  // the previous tile's reads of rot
        if (tid < 2 * JT) {
          int i, j;
          pair((tid < JT ? tp : tr) * JT + tid % JT, i, j);
          rot[tid / JT][tid % JT] = i < m && j < m ? jac_rotation(get(i, i), get(j, j), get(i, j))
                                                   : make_double2(1.0, 0.0);
        }
        __syncthreads();
        const double2 a = rot[0][ty], b = rot[1][tx];
        const double pr1 = a.x * pr - a.y * qr, qr1 = a.y * pr + a.x * qr;
        const double ps1 = a.x * ps - a.y * qs, qs1 = a.y * ps + a.x * qs;
        auto put = [&](int i, int j, double v) {
          if (i < m && j < m) An[(size_t)i * m + j] = v;
        };
        put(p, r, b.x * pr1 - b.y * ps1);
        put(p, s, b.y * pr1 + b.x * ps1);
        put(q, r, b.x * qr1 - b.y * qs1);
        put(q, s, b.y * qr1 + b.x * qs1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = 2 * JT * tp + ty + JT * h;
          if (i < m && cols) {
            V[(size_t)i * m + r] = b.x * vx[h] - b.y * vy[h];
            V[(size_t)i * m + s] = b.y * vx[h] + b.x * vy[h];
          }
        }
      }
      if (!grid_barrier(&st->bar, gen)) return;
      double* x = Ac;
      Ac = An;
      An = x;
    }
  }
  for (int k = blockIdx.x * (JT * JT) + tid; k < m; k += gridDim.x * JT * JT)
    diag[k] = __ldcg(&Ac[(size_t)k * m + k]);
  if (blockIdx.x == 0 && tid == 0) st->sweeps = max(st->sweeps, sweep);
}

// Whether eigenvalue x of index i comes before dc of index c: ascending, a NaN above every
// number, equal values and NaNs by index. A total order: the places of m eigenvalues are a
// permutation whatever they are, so that every column is written, by one CTA.
__device__ __forceinline__ bool jac_before(double x, int i, double dc, int c) {
  const bool xn = isnan(x), cn = isnan(dc);
  if (xn || cn) return xn == cn ? i < c : cn;
  return x < dc || (x == dc && i < c);
}

// U block and eps from the eigenvalues diag and V, one CTA per column: column c of V
// becomes column lo + rank of U, rank = its place in ascending order (jac_before),
// with its largest-magnitude component made positive (first one on ties).
__global__ void __launch_bounds__(128) jac_store_kernel(const double* __restrict__ diag,
                                                        const double* __restrict__ V, int m, int n,
                                                        int lo, double* __restrict__ U,
                                                        double* __restrict__ eps) {
  __shared__ int cnt;
  __shared__ double sv[128];
  __shared__ int si[128];
  const int c = blockIdx.x, tid = threadIdx.x;
  const double dc = diag[c];
  if (tid == 0) cnt = 0;
  __syncthreads();
  int below = 0, imax = 0;
  double vmax = -1.0;
  for (int i = tid; i < m; i += 128) {
    below += jac_before(diag[i], i, dc, c);
    const double a = fabs(V[(size_t)i * m + c]);
    if (a > vmax) {
      vmax = a;
      imax = i;
    }
  }
  atomicAdd(&cnt, below);
  sv[tid] = vmax;
  si[tid] = imax;
  __syncthreads();
  for (int o = 64; o > 0; o >>= 1) {
    if (tid < o && (sv[tid + o] > sv[tid] || (sv[tid + o] == sv[tid] && si[tid + o] < si[tid]))) {
      sv[tid] = sv[tid + o];
      si[tid] = si[tid + o];
    }
    __syncthreads();
  }
  const int k = cnt;
  const double sg = V[(size_t)si[0] * m + c] < 0.0 ? -1.0 : 1.0;
  for (int i = tid; i < m; i += 128) U[(size_t)(lo + i) * n + lo + k] = sg * V[(size_t)i * m + c];
  if (tid == 0) eps[lo + k] = dc;
}

// ------------------------------ transformations ------------------------------
// Bhp[Q][i][a] = B^Q[i][nC + a] (hole rows, particle columns)
__global__ void gather_hp_kernel(const double* __restrict__ B, Sizes z, double* __restrict__ Bhp) {
  const size_t total = (size_t)z.Q * z.nH * z.nP;
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= total) return;
  const int a = (int)(k % z.nP);
  const size_t qi = k / z.nP;
  const int i = (int)(qi % z.nH);
  const size_t q = qi / z.nH;
  Bhp[k] = B[(q * z.n + i) * z.n + z.nC + a];
}

// f1 = hole x particle block of T = U^T f U with the active x active part 0
__global__ void f1_kernel(const double* __restrict__ T, Sizes z, double* __restrict__ f1) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= z.nH * z.nP) return;
  const int i = k / z.nP, a = k % z.nP;
  f1[k] = (i >= z.nC && a < z.nA) ? 0.0 : T[(size_t)i * z.n + z.nC + a];
}

// G' = UA^T G UA and lambda2' = L rotated on every index (one thread per output)
__global__ void rot_active_kernel(const double* __restrict__ U, const double* __restrict__ G,
                                  const double* __restrict__ L, Sizes z, double* __restrict__ Go,
                                  double* __restrict__ Lo) {
  const int nA = z.nA, nA2 = nA * nA, nA4 = nA2 * nA2;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  auto ua = [&](int a, int u) { return U[(size_t)(z.nC + a) * z.n + z.nC + u]; };
  if (k < nA2) {
    const int u = k / nA, v = k % nA;
    double acc = 0.0;
    for (int a = 0; a < nA; ++a)
      for (int b = 0; b < nA; ++b) acc = fma(ua(a, u) * ua(b, v), G[a * nA + b], acc);
    Go[k] = acc;
  } else if (k < nA2 + nA4) {
    const int r = k - nA2;
    const int y = r % nA, x = (r / nA) % nA, v = (r / nA2) % nA, u = r / (nA2 * nA);
    double acc = 0.0;
    for (int a = 0; a < nA; ++a)
      for (int b = 0; b < nA; ++b)
        for (int c = 0; c < nA; ++c)
          for (int d = 0; d < nA; ++d)
            acc = fma(ua(a, u) * ua(b, v) * ua(c, x) * ua(d, y), L[((a * nA + b) * nA + c) * nA + d],
                      acc);
    Lo[r] = acc;
  }
}

// One index of the spin-orbital three-body cumulant rotated by Us = UA (x) I2:
// out[..., X_ax, ...] = sum_a Us[a][X] in[..., a, ...] on axis `ax` (0..5).
__global__ void rot_l3_axis_kernel(const double* __restrict__ U, Sizes z, int ax,
                                   const double* __restrict__ in, double* __restrict__ out) {
  const int n2 = 2 * z.nA;
  size_t total = 1;
  for (int d = 0; d < 6; ++d) total *= (size_t)n2;
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= total) return;
  size_t stride = 1;
  for (int d = 5; d > ax; --d) stride *= (size_t)n2;
  const int X = (int)((k / stride) % n2);
  const size_t base = k - (size_t)X * stride;
  double acc = 0.0;
  for (int a = X & 1; a < n2; a += 2) {  // spin conserved: a and X of the same spin
    const double us = U[(size_t)(z.nC + (a >> 1)) * z.n + z.nC + (X >> 1)];
    acc = fma(us, in[base + (size_t)a * stride], acc);
  }
  out[k] = acc;
}

cudaError_t sc_check(dsrg_sc_plan* p) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) p->last_error = cudaGetErrorString(e);
  return e;
}

// Waits for the plan's stream, reads its words and reports a wait that ran out since the
// last report (the barrier's word is that of the last semicanonicalisation alone).
dsrg_status_t sc_wait(dsrg_sc_plan* p, JacState* js) {
  cudaStream_t st = p->stream;
  if (cudaMemcpyAsync(js, p->jac, sizeof(*js), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return DSRG_ERR_CUDA;
  if (!js->bar.abort && !js->wait) return DSRG_OK;
  p->last_error = "a device-side wait ran out";
  if (cudaMemsetAsync(&p->jac->bar.abort, 0, sizeof(int), st) != cudaSuccess ||
      cudaMemsetAsync(&p->jac->wait, 0, sizeof(int), st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return DSRG_ERR_CUDA;
  return DSRG_ERR_TIMEOUT;
}

// Diagonalise the block [lo, lo + m) of f (symmetric); writes U and eps there.
cudaError_t jacobi_block(dsrg_sc_plan* p, int lo, int m, double* eps) {
  if (m == 0) return cudaSuccess;
  cudaStream_t st = p->stream;
  const int n = p->z.n;
  cudaError_t e;
  jac_copy_kernel<<<(m * m + 255) / 256, 256, 0, st>>>(p->f, n, lo, m, p->A, p->V);
  if ((e = sc_check(p)) != cudaSuccess) return e;
  int mp = m + (m & 1);
  const int nt = (mp / 2 + JT - 1) / JT;
  int grid = coop_grid(jac_run_kernel, JT * JT, 0, nt * nt < JAC_SLOTS ? nt * nt : JAC_SLOTS);
  if (grid < 1) return cudaErrorInvalidConfiguration;
  int max_sweeps = m > 1 ? 30 : 0;
  e = cudaMemsetAsync(&p->jac->bar.count, 0, sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  void* args[] = {&p->A, &p->T, &p->V, &m, &mp, &max_sweeps, &p->slots, &p->diag, &p->jac};
  e = cudaLaunchCooperativeKernel((const void*)jac_run_kernel, dim3(grid), dim3(JT * JT), args, 0, st);
  if (e != cudaSuccess) return e;
  jac_store_kernel<<<m, 128, 0, st>>>(p->diag, p->V, m, n, lo, p->U, eps);
  return sc_check(p);
}

cudaError_t build_fock(dsrg_sc_plan* p, const double* h, const double* B, const double* G) {
  const Sizes& z = p->z;
  cudaStream_t st = p->stream;
  cudaError_t e;
  const size_t nn = (size_t)z.n * z.n;
  fock_w_kernel<<<(unsigned)(((size_t)z.Q * 32 + 255) / 256), 256, 0, st>>>(B, G, z, p->w);
  if ((e = sc_check(p)) != cudaSuccess) return e;
  fock_j_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, st>>>(B, p->w, z, p->J);
  if ((e = sc_check(p)) != cudaSuccess) return e;
  const size_t nx = (size_t)z.Q * z.n * z.nH;
  fock_x_kernel<<<(unsigned)((nx + 255) / 256), 256, 0, st>>>(B, G, z, p->X);
  if ((e = sc_check(p)) != cudaSuccess) return e;
  // K[p][q] = sum_{Q, r in H} X[Q][p][r] B[Q][r][q]
  const int qc = (z.Q + p->nk - 1) / p->nk, full = z.Q / qc, rest = z.Q - full * qc;
  auto part = [&](int q0, int nq, double* K) {
    GemmArgs g = mk(z.n, z.n, nq, z.nH, p->X + (size_t)q0 * z.n * z.nH, z.nH, (long long)z.n * z.nH, 1,
                    B + (size_t)q0 * nn, (long long)nn, z.n, 1, K, z.n, 1, 1.0);
    g.accumulate = 0;
    return g;
  };
  if ((e = launch_gemm(st, batched(part(0, qc, p->K), full, (long long)qc * z.n * z.nH, (long long)qc * nn,
                                   (long long)nn), p->oz)) != cudaSuccess)
    return e;
  if (rest && (e = launch_gemm(st, part(full * qc, rest, p->K + (size_t)full * nn), p->oz)) != cudaSuccess)
    return e;
  fock_sum_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, st>>>(h, p->J, p->K, full + (rest ? 1 : 0), z.n,
                                                               &p->jac->wait, p->f);
  return sc_check(p);
}

}  // namespace
}  // namespace dsrg

using namespace dsrg;

extern "C" {

dsrg_status_t dsrg_sc_plan_create(dsrg_sc_plan_t** out, const dsrg_sizes_t* sz, void* cuda_stream) {
  if (!out) return DSRG_ERR_INVALID_ARG;
  *out = nullptr;
  if (!sz || sz->ncore < 0 || sz->nactive < 0 || sz->nvirt < 0 || sz->naux < 1 ||
      sz->ncore + sz->nactive + sz->nvirt < 1)
    return DSRG_ERR_INVALID_ARG;
  if (sz->nactive > NA_MAX) return DSRG_ERR_UNSUPPORTED;
  const long long n = (long long)sz->ncore + sz->nactive + sz->nvirt;
  if (n > (1 << 15) || (long long)sz->naux * n * n > (1ll << 36)) return DSRG_ERR_UNSUPPORTED;
  dsrg_sc_plan* p = new (std::nothrow) dsrg_sc_plan();
  if (!p) return DSRG_ERR_OOM;
  Sizes& z = p->z;
  z.nC = sz->ncore;
  z.nA = sz->nactive;
  z.nV = sz->nvirt;
  z.Q = sz->naux;
  z.nH = z.nC + z.nA;
  z.nP = z.nA + z.nV;
  z.n = z.nC + z.nA + z.nV;
  p->stream = (cudaStream_t)cuda_stream;
  cudaGetDevice(&p->device);
  p->mmax = std::max(z.nC, std::max(z.nA, z.nV));
  const size_t nn = (size_t)z.n * z.n, mm = (size_t)p->mmax * p->mmax;
  const size_t nhp = (size_t)z.Q * z.nH * z.nP;
  {
    // the exchange matrix has few tiles and a long sum: parts of it over Q, so that about
    // two tiles per SM run, each part at least 512 long
    const long long tiles = ((z.n + 127) / 128) * (long long)((z.n + 63) / 64);
    long long nk = 2 * sm_count() / tiles, most = (long long)z.Q * z.nH / 512;
    nk = nk > 16 ? 16 : nk;
    nk = nk > most ? most : nk;
    p->nk = nk < 1 ? 1 : (int)(nk > z.Q ? z.Q : nk);
    const long long qc = (z.Q + p->nk - 1) / p->nk;
    size_t b = oz_work_bytes(z.n, z.n, qc * z.nH, p->nk, false, false);
    b = std::max(b, oz_work_bytes(z.n, z.n, z.n, 1, false, false));
    b = std::max(b, oz_work_bytes((long long)z.Q * z.nH, z.nP, z.nP, 1, false, false));
    b = std::max(b, oz_work_bytes(z.nH, z.nP, z.nH, z.Q, true, false));
    p->oz.bytes = b;
  }
  bool ok = sc_alloc(p, (void**)&p->w, (size_t)z.Q * 8) && sc_alloc(p, (void**)&p->J, nn * 8) &&
            sc_alloc(p, (void**)&p->K, nn * 8) &&
            sc_alloc(p, (void**)&p->X, (size_t)z.Q * z.n * z.nH * 8) &&
            sc_alloc(p, (void**)&p->f, nn * 8) && sc_alloc(p, (void**)&p->U, nn * 8) &&
            sc_alloc(p, (void**)&p->T, nn * 8) && sc_alloc(p, (void**)&p->A, mm * 8) &&
            sc_alloc(p, (void**)&p->V, mm * 8) &&
            sc_alloc(p, (void**)&p->diag, (size_t)p->mmax * 8) &&
            sc_alloc(p, (void**)&p->slots, JAC_SLOTS * sizeof(double2)) &&
            sc_alloc(p, (void**)&p->jac, sizeof(JacState)) && sc_alloc(p, (void**)&p->Bhp, nhp * 8) &&
            sc_alloc(p, (void**)&p->Bt, nhp * 8);
  ok = ok && cudaMemset(p->jac, 0, sizeof(JacState)) == cudaSuccess;
  if (ok) p->oz.status = &p->jac->wait;
  size_t n3 = 1;
  for (int d = 0; d < 6; ++d) n3 *= (size_t)(2 * z.nA);
  ok = ok && (z.nA == 0 || sc_alloc(p, (void**)&p->L3t, n3 * 8));
  if (!ok) {
    for (void* a : p->allocs) cudaFree(a);
    delete p;
    return DSRG_ERR_OOM;
  }
  // what the plan can do without: the digits of the products (FP64 FMAs then) and the
  // partial exchange matrices (one then)
  if (!sc_alloc_spare(p, &p->oz.mem, p->oz.bytes)) p->oz.bytes = 0;
  void* parts = nullptr;
  if (p->nk > 1 && sc_alloc_spare(p, &parts, p->nk * nn * 8))
    p->K = (double*)parts;
  else
    p->nk = 1;
  *out = p;
  return DSRG_OK;
}

dsrg_status_t dsrg_sc_plan_destroy(dsrg_sc_plan_t* p) {
  if (!p) return DSRG_OK;
  cudaStreamSynchronize(p->stream);
  for (void* a : p->allocs) cudaFree(a);
  delete p;
  return DSRG_OK;
}

const char* dsrg_sc_last_error(const dsrg_sc_plan_t* p) { return p ? p->last_error.c_str() : "no plan"; }

int32_t dsrg_sc_last_sweeps(const dsrg_sc_plan_t* p) { return p ? p->sweeps_last : -1; }

dsrg_status_t dsrg_generalized_fock(dsrg_sc_plan_t* p, const double* h, const double* Bfull,
                                   const double* gamma1, double* f_dev) {
  if (!p || !h || !Bfull || !f_dev || (p->z.nA > 0 && !gamma1)) return DSRG_ERR_INVALID_ARG;
  if (((uintptr_t)h | (uintptr_t)Bfull | (uintptr_t)gamma1 | (uintptr_t)f_dev) & 7u)
    return DSRG_ERR_INVALID_ARG;
  if (build_fock(p, h, Bfull, gamma1) != cudaSuccess) return DSRG_ERR_CUDA;
  const size_t nn = (size_t)p->z.n * p->z.n;
  if (cudaMemcpyAsync(f_dev, p->f, nn * 8, cudaMemcpyDeviceToDevice, p->stream) != cudaSuccess)
    return DSRG_ERR_CUDA;
  return DSRG_OK;
}

dsrg_status_t dsrg_semicanonicalize(dsrg_sc_plan_t* p, const double* h, const double* Bfull,
                                    const double* gamma1, const double* lambda2,
                                    const double* lambda3, double* eps_out, double* B_out,
                                    double* f1_out, double* gamma1_out, double* lambda2_out,
                                    double* lambda3_out, double* U_out) {
  if (!p || !h || !Bfull || !eps_out || !B_out || !f1_out) return DSRG_ERR_INVALID_ARG;
  const Sizes& z = p->z;
  if (z.nA > 0 && (!gamma1 || !lambda2 || !gamma1_out || !lambda2_out)) return DSRG_ERR_INVALID_ARG;
  if (lambda3 && z.nA > 0 && !lambda3_out) return DSRG_ERR_INVALID_ARG;
  const uintptr_t mis = (uintptr_t)h | (uintptr_t)Bfull | (uintptr_t)gamma1 | (uintptr_t)lambda2 |
                        (uintptr_t)lambda3 | (uintptr_t)eps_out | (uintptr_t)B_out |
                        (uintptr_t)f1_out | (uintptr_t)gamma1_out | (uintptr_t)lambda2_out |
                        (uintptr_t)lambda3_out | (uintptr_t)U_out;
  if (mis & 7u) return DSRG_ERR_INVALID_ARG;
  cudaStream_t st = p->stream;
  const size_t nn = (size_t)z.n * z.n;
  p->sweeps_last = 0;
  if (cudaMemsetAsync(p->jac, 0, offsetof(JacState, wait), st) != cudaSuccess) return DSRG_ERR_CUDA;
  if (build_fock(p, h, Bfull, gamma1) != cudaSuccess) return DSRG_ERR_CUDA;
  if (cudaMemsetAsync(p->U, 0, nn * 8, st) != cudaSuccess) return DSRG_ERR_CUDA;
  if (jacobi_block(p, 0, z.nC, eps_out) != cudaSuccess ||
      jacobi_block(p, z.nC, z.nA, eps_out) != cudaSuccess ||
      jacobi_block(p, z.nH, z.nV, eps_out) != cudaSuccess)
    return DSRG_ERR_CUDA;
  cudaError_t e;
  // T = f U, then T <- U^T T (written to K): U^T f U
  GemmArgs g1 = mk(z.n, z.n, z.n, 1, p->f, z.n, 1, 0, p->U, z.n, 0, 1, p->T, z.n, 1, 1.0);
  g1.accumulate = 0;
  GemmArgs g2 = mk(z.n, z.n, z.n, 1, p->U, 1, z.n, 0, p->T, z.n, 0, 1, p->K, z.n, 1, 1.0);
  g2.accumulate = 0;
  if ((e = launch_gemm(st, g1, p->oz)) != cudaSuccess || (e = launch_gemm(st, g2, p->oz)) != cudaSuccess)
    return DSRG_ERR_CUDA;
  f1_kernel<<<(z.nH * z.nP + 255) / 256, 256, 0, st>>>(p->K, z, f1_out);
  if (sc_check(p) != cudaSuccess) return DSRG_ERR_CUDA;
  // B' = U_H^T B_HP U_P: gather, particle rotation over all (Q, i) rows, hole rotation per Q
  const size_t nhp = (size_t)z.Q * z.nH * z.nP;
  gather_hp_kernel<<<(unsigned)((nhp + 255) / 256), 256, 0, st>>>(Bfull, z, p->Bhp);
  if (sc_check(p) != cudaSuccess) return DSRG_ERR_CUDA;
  const double* UP = p->U + (size_t)z.nC * z.n + z.nC;  // U[nC + a'][nC + a], row pitch n
  GemmArgs g3 = mk(z.Q * z.nH, z.nP, z.nP, 1, p->Bhp, z.nP, 1, 0, UP, z.n, 0, 1, p->Bt, z.nP, 1, 1.0);
  g3.accumulate = 0;
  // B'[Q][i][a] = sum_i' U[i'][i] Bt[Q][i'][a]
  GemmArgs g4 = batched(mk(z.nH, z.nP, z.nH, 1, p->U, 1, z.n, 0, p->Bt, z.nP, 0, 1, B_out, z.nP, 1,
                           1.0),
                        z.Q, 0, (long long)z.nH * z.nP, (long long)z.nH * z.nP);
  g4.accumulate = 0;
  if ((e = launch_gemm(st, g3, p->oz)) != cudaSuccess || (e = launch_gemm(st, g4, p->oz)) != cudaSuccess)
    return DSRG_ERR_CUDA;
  if (z.nA > 0) {
    const int n4 = z.nA * z.nA * z.nA * z.nA + z.nA * z.nA;
    rot_active_kernel<<<(n4 + 127) / 128, 128, 0, st>>>(p->U, gamma1, lambda2, z, gamma1_out,
                                                        lambda2_out);
    if (sc_check(p) != cudaSuccess) return DSRG_ERR_CUDA;
    if (lambda3) {
      // six one-index rotations, alternating between the scratch and lambda3_out
      size_t total = 1;
      for (int d = 0; d < 6; ++d) total *= (size_t)(2 * z.nA);
      const double* src = lambda3;
      for (int ax = 0; ax < 6; ++ax) {
        double* dst = (ax % 2 == 0) ? p->L3t : lambda3_out;
        rot_l3_axis_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(p->U, z, ax, src, dst);
        if (sc_check(p) != cudaSuccess) return DSRG_ERR_CUDA;
        src = dst;
      }
    }
  }
  if (U_out && cudaMemcpyAsync(U_out, p->U, nn * 8, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
    return DSRG_ERR_CUDA;
  JacState js{};
  const dsrg_status_t status = sc_wait(p, &js);
  p->sweeps_last = js.sweeps;
  return status;
}

dsrg_status_t dsrg_sc_sync(dsrg_sc_plan_t* p) {
  if (!p) return DSRG_ERR_INVALID_ARG;
  JacState js{};
  return sc_wait(p, &js);
}

dsrg_status_t dsrg_sc_selftest_wait_timeout(dsrg_sc_plan_t* p) {
  if (!p) return DSRG_ERR_INVALID_ARG;
  return launch_wait_selftest(p->stream, &p->jac->wait) == cudaSuccess ? DSRG_OK : DSRG_ERR_CUDA;
}

}  // extern "C"
