// FP64 products on the tensor cores from exact integer slices, checked element by element
// against the error of FP64 FMAs (oz_gemm.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace dsrg {

constexpr int OZ_S = 7;  // slices (base-256 digits) of a value
constexpr int OZ_G = 8;  // accumulators: digit pairs by weight i + j = 2 .. OZ_G + 1

// The rows of one operand. Plane row R < xrow0 is row r = R % rpad (valid: r < rows)
// of problem z = R / rpad; R >= xrow0 is an extra row t = R - xrow0 (valid: t < xrows).
// Its value at the K index (l1, l2), l = l1 L2 + l2, is p[off(R) + l1 k1 + l2 k2],
//   off = off0 + z sb + r ri,   extra rows: (t / xn) xsb + (t % xn) xri.
struct OzRows {
  const double* p;
  int total;  // plane rows
  int rpad, rows;
  long long off0, ri, sb;
  int xrow0, xn, xrows;
  long long xsb, xri;
  int L1, L2;
  long long k1, k2;
};
__device__ __forceinline__ bool oz_row(const OzRows& s, int R, long long& off) {
  if (R < s.xrow0) {
    const int z = R / s.rpad, r = R - z * s.rpad;
    off = s.off0 + (long long)z * s.sb + (long long)r * s.ri;
    return R < s.total && r < s.rows;
  }
  const int t = R - s.xrow0;
  off = (long long)(t / s.xn) * s.xsb + (long long)(t % s.xn) * s.xri;
  return t < s.xrows;
}
__device__ __forceinline__ long long oz_k(const OzRows& s, int l) {
  const int l1 = s.L1 == 1 ? 0 : l / s.L2;
  return (long long)l1 * s.k1 + (long long)(l - l1 * s.L2) * s.k2;
}
inline OzRows oz_rows(const double* p, int nb, int rows, int rpad, long long ri, long long sb, int L1,
                      int L2, long long k1, long long k2) {
  OzRows s;
  s.p = p;
  s.rows = rows;
  s.rpad = rpad;
  s.total = nb * rpad;
  s.off0 = 0;
  s.ri = ri;
  s.sb = sb;
  s.xrow0 = s.total;
  s.xn = 1;
  s.xrows = 0;
  s.xsb = s.xri = 0;
  s.L1 = L1;
  s.L2 = L2;
  s.k1 = k1;
  s.k2 = k2;
  return s;
}

// C[p][i*ci + j*cj] (+)= alpha sum_l A[a0 + i][l] B[b0 + j][l], i < M, j < N. Problem
// p multiplies the plane rows from a0 = arow0 + x * astep with those from b0 = brow0 +
// y * bstep, (x, y) = pairs[p0 + p * pstep] (pairs null: (p, p)); its C starts at p * sc.
struct OzArgs {
  OzRows a, b;
  const int* aexp;  // row scales and sums by plane row (oz_pack)
  const int* bexp;
  int* status;
  double* C;
  long long ci, cj, sc;
  int M, N;
  const int2* pairs;
  int p0, pstep;
  int arow0, astep, brow0, bstep;
  double alpha;
  int accumulate;
  void* mask;       // oz_mask_bytes(M, N, problems), 8-byte aligned: elements left to FP64 FMAs
  // filled by oz_multiply
  int mt, nt, band, kstages, n_items;
};

constexpr long long OZ_MAX_K = 1ll << 21;  // limit of oz_pack's grid and of the integer sums' headroom
constexpr int OZ_ROW_PAD = 128;  // plane rows of a problem are a multiple, so that tiles start in it
__host__ __device__ inline int oz_kpad(long long K) { return (int)((K + 31) / 32 * 32); }
// Seven slices and the plane of leading digits for the check.
inline size_t oz_plane_bytes(long long rows, long long K) {
  return (size_t)(OZ_S + 1) * rows * oz_kpad(K) * sizeof(__nv_bfloat16);
}
// Per plane row: exponent of its scale, and the sum of its scaled magnitudes (2^-24 units).
constexpr size_t OZ_ROW_INFO = sizeof(int) + sizeof(unsigned long long);
// A bit per element of every 128 x 64 tile, and a byte per epilogue warp of the check.
inline size_t oz_mask_bytes(long long M, long long N, long long problems) {
  return (size_t)((M + 127) / 128) * ((N + 63) / 64) * problems * (128 * 8 + 8);
}
// Row scales and sums (OZ_ROW_INFO * total bytes at rexp) and slices (oz_plane_bytes(total,
// K); oz_off) of one operand, total a multiple of OZ_ROW_PAD.
constexpr int OZ_PACK_LAUNCHES = 2, OZ_MULTIPLY_LAUNCHES = 3;
cudaError_t oz_pack(cudaStream_t st, const OzRows& s, __nv_bfloat16* planes, int* rexp);
// The product of two packed operands (a.a, a.b: their rows as packed; the FP64 values at
// a.a.p and a.b.p are read again where the check finds the slices short of bits).
cudaError_t oz_multiply(cudaStream_t st, const __nv_bfloat16* pa, const __nv_bfloat16* pb, OzArgs a,
                        int n_prob);


// A generic FP64 GEMM (GemmArgs) in a caller's workspace: on the tensor cores, or by the
// FP64 kernel where that is faster (see oz_worthwhile) or `bytes` is too small.
struct OzWork {
  void* mem = nullptr;
  size_t bytes = 0;
  int* status = nullptr;  // device status word of the bounded waits
};
struct GemmArgs;
// The kernels queued are added to *launches (may be null).
cudaError_t launch_gemm(cudaStream_t st, const GemmArgs& g, const OzWork& w, int* launches = nullptr);
// Workspace that lets launch_gemm run nb problems of M x N x K at once, at most OZ_WS_CAP
// (the problems then run in turns).
constexpr size_t OZ_WS_CAP = (size_t)512 << 20;
size_t oz_work_bytes(long long M, long long N, long long K, long long nb, bool shared_a, bool shared_b);

}  // namespace dsrg
