// The FP64 plans' pair contractions on the tensor cores (oz_gemm.cu: exact integer
// slices, elements checked against the error bound of FP64 FMAs) with FP64 regulators
// and sums.
//
// Plane rows as in the split plans: (h, e) for every hole h and virtual e (nVpad rows
// per hole), then (h, x) for every hole and active particle.
//   CCVV  v^{ij}[a,b] = (ia|jb) for a group of core pairs into a buffer, then one CTA
//         per (pair, 64 x 64 virtual tile pair) adds (x^2 - x y + y^2) R, R = (1 -
//         exp(-2 s D^2))/D (Eq. (23)); the same partial slots as ccvv_fp64_kernel.
//   rest  Y = P . P[(u,f); (h',x)]^T holds (ge|uf), (ge|h'x), (hx|uf), (hx|h'y): CAVV
//         (F2), CCAV (F3) and the active block's integrals read it.
//
// The FP64 CUDA-core kernels these replace ran at the FP64 pipe's rate: 101.6 ms for
// CCVV and 16 ms for CAVV at the cc-pVTZ size (24/2/372/1200); here 4.7 ms (products 3.3,
// their check 0.1, regulators 1.4) and 0.35 ms, and 0.65 ms for the product of the rest. Regulators beside
// the next group's product would need registers that its kernel leaves no room for.
// The regulators are what is left on that pipe: about 25 FP64 instructions each.
#include <new>

#include "internal.cuh"
#include "oz_gemm.cuh"
#include "regulators.cuh"

namespace dsrg {

struct Fp64Tc {
  int nVpad = 0, xrow0 = 0, XR = 0;
  OzRows rows{};               // p (B) is filled per call
  __nv_bfloat16* planes = nullptr;
  int* rexp = nullptr;
  void* mask = nullptr;        // of the products of a group, or of Y
  int group = 0;               // core pairs per buffer
  double* V = nullptr;         // [group][nV][nV]
  double* Y = nullptr;         // [xrow0 + nH nA][ldy]
  long long ldy = 0, xc = 0;
};

// 1/D to FP64 rounding: a 20-bit seed and two Newton-Raphson steps.
__device__ __forceinline__ double inv_fp64(double D) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(D));
  r = fma(fma(-D, r, 1.0), r, r);
  return fma(fma(-D, r, 1.0), r, r);
}

// (1 - e^{-x}) / D and e^{-x} for x = c D^2: one exponential where 1 - e^{-x} has no
// cancellation (x > 1/2), none where e^{-x} is below FP64 precision, expm1 elsewhere.
__device__ __forceinline__ double reg_one(double D, double x, double& g) {
  if (x > 0.5 && x < 1e300) {
    g = x > 44.0 ? 0.0 : exp(-x);
    return (1.0 - g) * inv_fp64(D);
  }
  g = exp(-x);
  return D == 0.0 ? 0.0 : -expm1(-x) / D;
}

constexpr int RT = 64;

__global__ void __launch_bounds__(256) ccvv_reg_fp64_kernel(
    const double* __restrict__ V, const double* __restrict__ eps, double s, Sizes z,
    const int2* __restrict__ pairs, int p0, int pstep, const int2* __restrict__ tps, int n_tp,
    double* __restrict__ partials) {
  __shared__ double sy[RT][RT + 1], se[2][RT];
  __shared__ double red[8];
  const int k = blockIdx.x / n_tp, tp = blockIdx.x % n_tp, pair = p0 + k * pstep;
  const int2 ij = pairs[pair], ab = tps[tp];
  const int a0 = ab.x * RT, b0 = ab.y * RT, ve = z.nC + z.nA;
  const double* v = V + (size_t)k * z.nV * z.nV;
  for (int e = threadIdx.x; e < RT * RT; e += 256) {
    const int r = e / RT, c = e % RT;  // y_ab = v_ba
    sy[c][r] = (b0 + r < z.nV && a0 + c < z.nV) ? v[(size_t)(b0 + r) * z.nV + a0 + c] : 0.0;
  }
  if (threadIdx.x < 2 * RT) {
    const int o = (threadIdx.x < RT ? a0 : b0) + (threadIdx.x & (RT - 1));
    se[threadIdx.x / RT][threadIdx.x & (RT - 1)] = o < z.nV ? eps[ve + o] : 0.0;
  }
  __syncthreads();
  const double E = eps[ij.x] + eps[ij.y], s2 = 2.0 * s;
  const int c = threadIdx.x & (RT - 1), b = b0 + c;
  double acc = 0.0;
  if (b < z.nV) {
    const double eb = se[1][c];
#pragma unroll 4
    for (int r = threadIdx.x / RT; r < RT; r += 256 / RT) {
      const int a = a0 + r;
      if (a >= z.nV) break;
      const double x = v[(size_t)a * z.nV + b], y = sy[r][c];
      const double D = E - se[0][r] - eb;
      double g;
      const double R = reg_one(D, s2 * D * D, g);
      acc = fma(fma(x, x - y, y * y), R, acc);
    }
  }
  const double w = (ij.x == ij.y ? 1.0 : 2.0) * (ab.x < ab.y ? 2.0 : 1.0);
  const double tot = block_sum<256>(acc, red);
  if (threadIdx.x == 0) partials[(size_t)pair * n_tp + tp] = w * tot;
}

// F1 adjoint of one (pair, 64 x 64 tile pair): W^{ij}_ab = dE/dv^{ij}_ab = (4x - 2y) R,
// W^{ij}_ba = (4y - 2x) R with x = v_ab, y = v_ba, and W^{ji} the transpose, into W[i][j]
// and W[j][i] (pitch nVp, rows through shared memory); the eps and s derivatives of
// both orders of the pair (see ccvv_adj_kernel in grad.cu for one order).
__global__ void __launch_bounds__(256) ccvv_adj_v_kernel(
    const double* __restrict__ V, const double* __restrict__ eps, double s, Sizes z,
    const int2* __restrict__ pairs, int p0, const int2* __restrict__ tps, int n_tp, int nVp,
    double* __restrict__ W, double* __restrict__ deps, double* __restrict__ ds) {
  extern __shared__ double adj_sm[];
  double* sp = adj_sm;                 // [64][65]: y, then (4x - 2y) R
  double* sq = sp + RT * (RT + 1);     // [64][65]: (4y - 2x) R
  __shared__ double se[2][RT], rowacc[RT], colacc[RT], red[8];
  const int k = blockIdx.x / n_tp, tp = blockIdx.x % n_tp, pair = p0 + k;
  const int2 ij = pairs[pair], ab = tps[tp];
  const int a0 = ab.x * RT, b0 = ab.y * RT, ve = z.nC + z.nA;
  const double* v = V + (size_t)k * z.nV * z.nV;
  for (int e = threadIdx.x; e < RT * RT; e += 256) {
    const int r = e / RT, c = e % RT;
    sp[c * (RT + 1) + r] = (b0 + r < z.nV && a0 + c < z.nV) ? v[(size_t)(b0 + r) * z.nV + a0 + c] : 0.0;
  }
  if (threadIdx.x < 2 * RT) {
    const int o = (threadIdx.x < RT ? a0 : b0) + (threadIdx.x & (RT - 1));
    se[threadIdx.x / RT][threadIdx.x & (RT - 1)] = o < z.nV ? eps[ve + o] : 0.0;
  }
  if (threadIdx.x < RT) rowacc[threadIdx.x] = colacc[threadIdx.x] = 0.0;
  __syncthreads();
  const double E = eps[ij.x] + eps[ij.y];
  const bool mirror = ab.x < ab.y, two = ij.x != ij.y;
  const double wt = mirror ? 2.0 : 1.0, f = two ? 2.0 : 1.0;
  const int c = threadIdx.x & (RT - 1), b = b0 + c;
  double* Wij = W + ((size_t)ij.x * z.nC + ij.y) * nVp * nVp;
  double* Wji = W + ((size_t)ij.y * z.nC + ij.x) * nVp * nVp;
  double dk = 0.0, dss = 0.0, cacc = 0.0;
  if (b < z.nV) {
    for (int r = threadIdx.x / RT; r < RT; r += 256 / RT) {
      const int a = a0 + r;
      if (a >= z.nV) break;
      const double x = v[(size_t)a * z.nV + b], y = sp[r * (RT + 1) + c];
      const RegD R = rf1_d(E - se[0][r] - se[1][c], s);
      const double wp = (4.0 * x - 2.0 * y) * R.v, wq = (4.0 * y - 2.0 * x) * R.v;
      sp[r * (RT + 1) + c] = wp;
      sq[r * (RT + 1) + c] = wq;
      Wij[(size_t)a * nVp + b] = wp;
      if (two && mirror) Wji[(size_t)a * nVp + b] = wq;
      const double q = fma(x, x - y, y * y);
      dk = fma(2.0 * wt * q, R.dD, dk);
      dss = fma(wt * q, R.ds, dss);
      const double gv = -2.0 * f * q * R.dD;
      atomicAdd(&rowacc[r], gv);
      cacc += gv;
    }
  }
  if (mirror) atomicAdd(&colacc[c], cacc);
  const double tk = block_sum<256>(dk, red);
  const double ts = block_sum<256>(f * dss, red);
  if (threadIdx.x == 0) {
    atomicAdd(&deps[ij.x], tk);
    if (two) atomicAdd(&deps[ij.y], tk);
    atomicAdd(ds, ts);
  }
  __syncthreads();
  // the transposed positions (b, a)
  for (int e = threadIdx.x; e < RT * RT; e += 256) {
    const int cc = e / RT, rr = e % RT;  // b = b0 + cc, a = a0 + rr
    if (b0 + cc >= z.nV || a0 + rr >= z.nV) continue;
    const size_t o = (size_t)(b0 + cc) * nVp + a0 + rr;
    if (mirror) Wij[o] = sq[rr * (RT + 1) + cc];
    if (two) Wji[o] = sp[rr * (RT + 1) + cc];
  }
  if (threadIdx.x < RT) {
    if (a0 + threadIdx.x < z.nV) atomicAdd(&deps[ve + a0 + threadIdx.x], rowacc[threadIdx.x]);
    if (mirror && b0 + threadIdx.x < z.nV) atomicAdd(&deps[ve + b0 + threadIdx.x], colacc[threadIdx.x]);
  }
}

// F2 (CAVV) from X_u[e,f] = (me|uf) = Y[(m,e), u nVpad + f], one CTA per (m, 32 x 32
// tile pair E <= F) as cavv_f2_kernel, in FP64.
constexpr int FT = 32;
template <int NA>
__global__ void __launch_bounds__(256) cavv_y_fp64_kernel(
    const double* __restrict__ Y, long long ldy, int nVpad, const double* __restrict__ eps,
    const double* __restrict__ G, double s, Sizes z, const int2* __restrict__ tps, int n_tp,
    double* __restrict__ partials) {
  extern __shared__ double sXt[];  // [NA][32][33]  X_u[f,e]
  __shared__ double sG[NA * NA], red[8];
  const int m = blockIdx.x / n_tp;
  const int2 ab = tps[blockIdx.x % n_tp];
  const int E0 = ab.x * FT, F0 = ab.y * FT, ve = z.nC + z.nA;
  const double* Ym = Y + (size_t)m * nVpad * ldy;
  for (int k = threadIdx.x; k < NA * FT * FT; k += 256) {
    const int u = k / (FT * FT), r = (k / FT) % FT, c = k % FT;
    sXt[(u * FT + c) * (FT + 1) + r] =
        (F0 + r < z.nV && E0 + c < z.nV) ? Ym[(size_t)(F0 + r) * ldy + u * nVpad + E0 + c] : 0.0;
  }
  if (threadIdx.x < NA * NA) sG[threadIdx.x] = G[threadIdx.x];
  __syncthreads();
  const bool mirror = ab.x < ab.y;
  const int c = threadIdx.x & 31, f = F0 + c;
  double acc = 0.0;
  if (f < z.nV) {
    const double ef = eps[ve + f];
    for (int r = threadIdx.x >> 5; r < FT; r += 8) {
      const int e = E0 + r;
      if (e >= z.nV) break;
      const double base = eps[m] - eps[ve + e] - ef;
      double X[NA], Xt[NA], Rv[NA], Rt[NA];
#pragma unroll
      for (int u = 0; u < NA; ++u) {
        X[u] = Ym[(size_t)e * ldy + u * nVpad + f];
        Xt[u] = sXt[(u * FT + r) * (FT + 1) + c];
        const double D = base + eps[z.nC + u];
        double g;
        Rt[u] = reg_one(D, s * D * D, g);
        Rv[u] = 1.0 + g;
      }
      double t1 = 0.0, t2 = 0.0;
#pragma unroll
      for (int v = 0; v < NA; ++v) {
        double c1 = 0.0, c2 = 0.0;
#pragma unroll
        for (int u = 0; u < NA; ++u) {
          const double w = sG[u * NA + v] * Rv[u];
          c1 = fma(w, X[u], c1);
          c2 = fma(w, Xt[u], c2);
        }
        t1 = fma(c1, (2.0 * X[v] - Xt[v]) * Rt[v], t1);
        t2 = fma(c2, (2.0 * Xt[v] - X[v]) * Rt[v], t2);
      }
      acc += mirror ? (t1 + t2) : t1;
    }
  }
  const double tot = block_sum<256>(acc, red);
  if (threadIdx.x == 0) partials[blockIdx.x] = tot;
}

// F3 (CCAV) from Z_u[m,n,e] = (me|nu) = Y[(m,e), xc + n nA + u], one CTA per virtual e.
template <int NA>
__global__ void __launch_bounds__(256) ccav_y_fp64_kernel(
    const double* __restrict__ Y, long long ldy, int nVpad, long long xc,
    const double* __restrict__ eps, const double* __restrict__ G, double s, Sizes z,
    double* __restrict__ partials) {
  extern __shared__ double sZ[];  // [nC][nC*NA]
  __shared__ double sH[NA * NA], red[8];
  const int e = blockIdx.x, nC = z.nC, w = nC * NA;
  for (int k = threadIdx.x; k < nC * w; k += 256)
    sZ[k] = Y[(size_t)((k / w) * nVpad + e) * ldy + xc + k % w];
  if (threadIdx.x < NA * NA) {
    const int u = threadIdx.x / NA, v = threadIdx.x % NA;
    sH[threadIdx.x] = (u == v ? 2.0 : 0.0) - G[threadIdx.x];
  }
  __syncthreads();
  const double ee = eps[nC + z.nA + e];
  double acc = 0.0;
  for (int mn = threadIdx.x; mn < nC * nC; mn += 256) {
    const int m = mn / nC, n = mn % nC;
    const double base = eps[m] + eps[n] - ee;
    double W[NA], Rt[NA];
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      const double D = base - eps[nC + u];
      double g;
      Rt[u] = reg_one(D, s * D * D, g);
      W[u] = (1.0 + g) * sZ[m * w + n * NA + u];
    }
#pragma unroll
    for (int u = 0; u < NA; ++u) {
      double cc = 0.0;
#pragma unroll
      for (int v = 0; v < NA; ++v) cc = fma(sH[u * NA + v], W[v], cc);
      acc = fma(cc, (2.0 * sZ[m * w + n * NA + u] - sZ[n * w + m * NA + u]) * Rt[u], acc);
    }
  }
  const double tot = block_sum<256>(acc, red);
  if (threadIdx.x == 0) partials[e] = tot;
}

// The active block's integrals from Y: K1 = (ia|ux), K2 = (ix|ua) [nH][nA][nA][nP],
// K3 = (ix|jy) [nH][nA][nH][nA], M = (xe|uf) [nA][nA][nV][nV].
__global__ void gather_y_fp64_kernel(const double* __restrict__ Y, long long ldy, int nVpad,
                                     int xrow0, long long xc, Sizes z, double* __restrict__ K1,
                                     double* __restrict__ K2, double* __restrict__ K3,
                                     double* __restrict__ M) {
  const int nA = z.nA, nC = z.nC, T = z.nH * nA;
  const size_t n12 = (size_t)z.nH * nA * nA * z.nP, n3 = (size_t)T * T;
  const size_t nm = (size_t)nA * nA * z.nV * z.nV;
  size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  // Y row of the hole x particle pair (h, a)
  auto row = [&](int h, int a) {
    return (size_t)(a < nA ? xrow0 + h * nA + a : h * nVpad + a - nA) * ldy;
  };
  if (k < 2 * n12) {
    const size_t r = k >= n12 ? k - n12 : k;
    const int a = (int)(r % z.nP), x = (int)((r / z.nP) % nA);
    const int u = (int)((r / ((size_t)z.nP * nA)) % nA), i = (int)(r / ((size_t)z.nP * nA * nA));
    if (k < n12)
      K1[r] = Y[row(i, a) + xc + (nC + u) * nA + x];
    else
      K2[r] = Y[row(nC + u, a) + xc + i * nA + x];
    return;
  }
  k -= 2 * n12;
  if (k < n3) {
    K3[k] = Y[(size_t)(xrow0 + k / T) * ldy + xc + k % T];
    return;
  }
  k -= n3;
  if (k >= nm) return;
  const int f = (int)(k % z.nV), e = (int)((k / z.nV) % z.nV);
  const int xu = (int)(k / ((size_t)z.nV * z.nV));
  M[k] = Y[(size_t)((nC + xu / nA) * nVpad + e) * ldy + (size_t)(xu % nA) * nVpad + f];
}

// ------------------------------- host side -------------------------------
// Bytes of the pair buffer: about the L2, so that the regulator kernel reads what the
// product just wrote from it.
constexpr size_t V_BYTES = (size_t)96 << 20;

// The slices and the check plane take 16 bytes per value of B, Y one FP64 per (hole,
// virtual) and active pair, the pair buffer at least one pair's integrals. A plan takes them
// only where they are within `limit` and can be had: others run on the CUDA-core kernels,
// which need none of it (they run for hours there, but they run).
void fp64_tc_alloc(dsrg_plan* p, size_t limit) {
  const Sizes& z = p->z;
  if (z.Q > OZ_MAX_K) return;
  const long long nVpad = (z.nV + OZ_ROW_PAD - 1ll) / OZ_ROW_PAD * OZ_ROW_PAD;
  const long long XR = (z.nH * z.nA + OZ_ROW_PAD - 1ll) / OZ_ROW_PAD * OZ_ROW_PAD;
  const long long rows = z.nH * nVpad + XR;
  const size_t per = (size_t)z.nV * z.nV * sizeof(double);
  if (rows > 2000000000ll) return;
  Fp64Tc* w = new (std::nothrow) Fp64Tc();
  if (!w) return;
  w->nVpad = (int)nVpad;
  w->xrow0 = z.nH * w->nVpad;
  w->XR = (int)XR;
  OzRows& r = w->rows;
  // B[(q nH + h) nP + a], rows (h, nA + e) and then (h, x)
  r = oz_rows(nullptr, z.nH, z.nV, w->nVpad, 1, z.nP, 1, z.Q, 0, (long long)z.nH * z.nP);
  r.off0 = z.nA;
  r.total = w->xrow0 + w->XR;
  r.xrow0 = w->xrow0;
  r.xn = z.nA > 0 ? z.nA : 1;
  r.xrows = z.nH * z.nA;
  r.xsb = z.nP;
  r.xri = 1;
  w->xc = (long long)z.nA * w->nVpad;
  w->ldy = w->xc + (z.nH * z.nA + 7) / 8 * 8;
  const size_t mask_1 = oz_mask_bytes(z.nV, z.nV, 1);  // whole tiles: larger than `per` for a few virtuals
  const size_t fit = V_BYTES / (per > mask_1 ? per : mask_1);
  w->group = (int)(fit < 1 ? 1 : (fit > (size_t)p->n_pairs ? (size_t)p->n_pairs : fit));
  const size_t mask_v = oz_mask_bytes(z.nV, z.nV, w->group);
  const size_t mask_y = oz_mask_bytes(w->xrow0 + z.nH * z.nA, w->xc + z.nH * z.nA, 1);
  const size_t mask = mask_v > mask_y ? mask_v : mask_y;
  const size_t y = z.nA == 0 ? 0 : (size_t)(w->xrow0 + z.nH * z.nA) * w->ldy * sizeof(double);
  const size_t need = oz_plane_bytes(r.total, z.Q) + (size_t)r.total * OZ_ROW_INFO + mask + per * w->group + y;
  const size_t n_allocs = p->allocs.size(), ws = p->ws_bytes;
  if (need <= limit &&
      plan_alloc(p, (void**)&w->planes, oz_plane_bytes(r.total, z.Q)) &&
      plan_alloc(p, (void**)&w->rexp, (size_t)r.total * OZ_ROW_INFO) && plan_alloc(p, &w->mask, mask) &&
      plan_alloc(p, (void**)&w->V, per * w->group) && (y == 0 || plan_alloc(p, (void**)&w->Y, y))) {
    p->f64 = w;
    return;
  }
  plan_release(p, n_allocs, ws);
  delete w;
}

void fp64_tc_free(dsrg_plan* p) {
  delete p->f64;
  p->f64 = nullptr;
}

static OzRows rows_of(const dsrg_plan* p, const double* B) {
  OzRows r = p->f64->rows;
  r.p = B;
  return r;
}

// The pair products' arguments (the planes are packed).
static OzArgs pair_args(const dsrg_plan* p, const double* B) {
  const Fp64Tc* w = p->f64;
  OzArgs a;
  a.a = a.b = rows_of(p, B);
  a.aexp = a.bexp = w->rexp;
  a.status = p->d_status;
  a.C = w->V;
  a.ci = p->z.nV;
  a.cj = 1;
  a.sc = (long long)p->z.nV * p->z.nV;
  a.M = a.N = p->z.nV;
  a.pairs = p->d_pairs;
  a.p0 = 0;
  a.pstep = 1;
  a.arow0 = a.brow0 = 0;
  a.astep = a.bstep = w->nVpad;
  a.alpha = 1.0;
  a.accumulate = 0;
  a.mask = w->mask;
  return a;
}

cudaError_t launch_ccvv_fp64_tc(dsrg_plan* p, const double* B, const double* eps, double s) {
  Fp64Tc* w = p->f64;
  if (!w) return launch_ccvv_fp64(p, B, eps, s);
  const Sizes& z = p->z;
  cudaError_t e;
  OzArgs a = pair_args(p, B);
  if ((e = oz_pack(p->stream, a.a, w->planes, w->rexp)) != cudaSuccess) return e;
  p->launches += OZ_PACK_LAUNCHES;
  const Segment& sg = p->segs[p->seg_ccvv];
  a.pstep = p->shard_world;
  // (64 bits: a world may be as large as an int, and group times that is not)
  const long long world = p->shard_world;
  for (long long q0 = p->shard_rank; q0 < p->n_pairs; q0 += w->group * world) {
    const long long left = (p->n_pairs - q0 + world - 1) / world;
    const int p0 = (int)q0, n = (int)(left < w->group ? left : w->group);
    a.p0 = p0;
    if ((e = oz_multiply(p->stream, w->planes, w->planes, a, n)) != cudaSuccess) return e;
    p->launches += OZ_MULTIPLY_LAUNCHES;
    ccvv_reg_fp64_kernel<<<(unsigned)(n * p->n_tp_ccvv), 256, 0, p->stream>>>(
        w->V, eps, s, z, p->d_pairs, p0, p->shard_world, p->d_tp_ccvv, p->n_tp_ccvv,
        p->d_partials + sg.begin);
    DSRG_LAUNCH_CHECK(p);
  }
  return cudaSuccess;
}

// F1 adjoint of every pair (one rank): W [nC][nC][nVp][nVp], adds to deps and ds. The
// planes are those of the energy call just made on the stream (same B).
cudaError_t launch_ccvv_adj_fp64_tc(dsrg_plan* p, const double* B, const double* eps, double s, int nVp,
                                    double* W, double* deps, double* ds) {
  Fp64Tc* w = p->f64;
  const size_t sm = 2 * RT * (RT + 1) * sizeof(double);
  raise_smem_limit((const void*)ccvv_adj_v_kernel, sm);
  OzArgs a = pair_args(p, B);
  cudaError_t e;
  for (int p0 = 0; p0 < p->n_pairs; p0 += w->group) {
    const int n = p->n_pairs - p0 < w->group ? p->n_pairs - p0 : w->group;
    a.p0 = p0;
    if ((e = oz_multiply(p->stream, w->planes, w->planes, a, n)) != cudaSuccess) return e;
    p->launches += OZ_MULTIPLY_LAUNCHES;
    ccvv_adj_v_kernel<<<(unsigned)(n * p->n_tp_ccvv), 256, sm, p->stream>>>(
        w->V, eps, s, p->z, p->d_pairs, p0, p->d_tp_ccvv, p->n_tp_ccvv, nVp, W, deps, ds);
    DSRG_LAUNCH_CHECK(p);
  }
  return cudaSuccess;
}

const double* fp64_tc_y(const dsrg_plan* p, long long* ldy, int* nVpad, long long* xc) {
  if (!p->f64) return nullptr;
  *ldy = p->f64->ldy;
  *nVpad = p->f64->nVpad;
  *xc = p->f64->xc;
  return p->f64->Y;
}

// CAVV and CCAV partials and K1, K2, K3, M (the planes are those of the CCVV launch of
// the same call).
cudaError_t launch_rest_fp64_tc(dsrg_plan* p, const double* B, const double* eps, const double* G,
                                double s) {
  Fp64Tc* w = p->f64;
  const Sizes& z = p->z;
  if (z.nA == 0) return cudaSuccess;
  cudaStream_t st = p->stream;
  cudaError_t e;
  OzArgs a;
  a.a = a.b = rows_of(p, B);
  a.aexp = a.bexp = w->rexp;
  a.status = p->d_status;
  a.C = w->Y;
  a.ci = w->ldy;
  a.cj = 1;
  a.sc = 0;
  a.M = w->xrow0 + z.nH * z.nA;
  a.N = z.nA * w->nVpad + z.nH * z.nA;
  a.pairs = nullptr;
  a.p0 = 0;
  a.pstep = 1;
  a.arow0 = 0;
  a.brow0 = z.nC * w->nVpad;
  a.astep = a.bstep = 0;
  a.alpha = 1.0;
  a.accumulate = 0;
  a.mask = w->mask;
  if ((e = oz_multiply(st, w->planes, w->planes, a, 1)) != cudaSuccess) return e;
  p->launches += OZ_MULTIPLY_LAUNCHES;
  const Segment &s2 = p->segs[p->seg_cavv], &s3 = p->segs[p->seg_ccav];
  const size_t sm2 = (size_t)z.nA * FT * (FT + 1) * 8, sm3 = (size_t)z.nC * z.nC * z.nA * 8;
#define REST_CASE(NA_)                                                                            \
  case NA_:                                                                                       \
    raise_smem_limit((const void*)cavv_y_fp64_kernel<NA_>, sm2);                                  \
    cavv_y_fp64_kernel<NA_><<<s2.count, 256, sm2, st>>>(w->Y, w->ldy, w->nVpad, eps, G, s, z,     \
                                                        p->d_tp_cavv, p->n_tp_cavv,               \
                                                        p->d_partials + s2.begin);                \
    DSRG_LAUNCH_CHECK(p);                                                                         \
    raise_smem_limit((const void*)ccav_y_fp64_kernel<NA_>, sm3);                                  \
    ccav_y_fp64_kernel<NA_><<<s3.count, 256, sm3, st>>>(w->Y, w->ldy, w->nVpad, w->xc, eps, G, s, \
                                                        z, p->d_partials + s3.begin);             \
    DSRG_LAUNCH_CHECK(p);                                                                         \
    break;
  switch (z.nA) {
    REST_CASE(1) REST_CASE(2) REST_CASE(3) REST_CASE(4)
    REST_CASE(5) REST_CASE(6) REST_CASE(7) REST_CASE(8)
    default: return cudaErrorInvalidValue;
  }
#undef REST_CASE
  const size_t n = 2 * (size_t)z.nH * z.nA * z.nA * z.nP + (size_t)z.nH * z.nA * z.nH * z.nA +
                   (size_t)z.nA * z.nA * z.nV * z.nV;
  gather_y_fp64_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
      w->Y, w->ldy, w->nVpad, w->xrow0, w->xc, z, p->act.K1, p->act.K2, p->act.K3, p->act.M);
  DSRG_LAUNCH_CHECK(p);
  return cudaSuccess;
}

}  // namespace dsrg
