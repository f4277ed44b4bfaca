// Pairs of FP32 numbers (head + tail, 48 bits) for the regulator epilogues.
//
// Why: the FP64 pipe of this GPU retires 2 FMAs per SM and clock against 128
// on the FP32 pipe. The FP64 regulator (1 - exp(-k D^2))/D of one integral took
// 7 FP64 instructions and a conversion, 32 us for the 128 x 128 positions of a
// CCVV work item whose tensor-core work takes 18 us (cc-pVTZ size). The same
// regulator in FP32 pairs is about 90 FP32 instructions, under 6 us.
//
// Accuracy: a pair carries 48 bits; 1/D and 1 - exp(-k D^2) below have relative
// errors under 2^-40 (at most 2^-40.8 in tests/test_ff.py, which compares them with
// FP64 over the range of arguments), as had the FP64 form, whose 1/D came from a 20-bit
// seed and one Newton-Raphson step.
//
// The error-free sums and products are Knuth's and Dekker's (T. J. Dekker,
// Numer. Math. 18 (1971) 224), with an FMA for the product's error.
#pragma once

#include <cuda_runtime.h>

namespace dsrg {

struct ff {
  float h, l;
};

#ifdef __CUDA_ARCH__
// round-to-nearest operations that the compiler may not contract or reorder
#define FF_ADD(a, b) __fadd_rn(a, b)
#define FF_SUB(a, b) __fsub_rn(a, b)
#define FF_MUL(a, b) __fmul_rn(a, b)
#define FF_FMA(a, b, c) __fmaf_rn(a, b, c)
#else
#define FF_ADD(a, b) ((a) + (b))
#define FF_SUB(a, b) ((a) - (b))
#define FF_MUL(a, b) ((a) * (b))
#define FF_FMA(a, b, c) fmaf(a, b, c)
#endif
#define FF_FN __host__ __device__ __forceinline__

FF_FN ff ff_from(double d) {
  ff r;
  r.h = (float)d;
  r.l = (float)(d - (double)r.h);
  return r;
}
FF_FN double ff_to(ff a) { return (double)a.h + (double)a.l; }

// a + b exactly, for any a and b
FF_FN ff ff_two_sum(float a, float b) {
  ff r;
  r.h = FF_ADD(a, b);
  const float bb = FF_SUB(r.h, a);
  r.l = FF_ADD(FF_SUB(a, FF_SUB(r.h, bb)), FF_SUB(b, bb));
  return r;
}
// a + b exactly, for |a| >= |b| or a = 0
FF_FN ff ff_fast_sum(float a, float b) {
  ff r;
  r.h = FF_ADD(a, b);
  r.l = FF_SUB(b, FF_SUB(r.h, a));
  return r;
}

// a - b
FF_FN ff ff_diff(ff a, ff b) {
  const ff t = ff_two_sum(a.h, -b.h);
  return ff_fast_sum(t.h, FF_ADD(t.l, FF_SUB(a.l, b.l)));
}

// a + b
FF_FN ff ff_add(ff a, ff b) {
  const ff t = ff_two_sum(a.h, b.h);
  return ff_fast_sum(t.h, FF_ADD(t.l, FF_ADD(a.l, b.l)));
}

// a += b: the heads exactly, the tails in FP32, renormalised
FF_FN void ff_acc(ff& a, ff b) {
  const ff t = ff_two_sum(a.h, b.h);
  a = ff_fast_sum(t.h, FF_ADD(a.l, FF_ADD(t.l, b.l)));
}

FF_FN ff ff_mul(ff a, ff b) {
  ff r;
  r.h = FF_MUL(a.h, b.h);
  r.l = FF_FMA(a.l, b.h, FF_FMA(a.h, b.l, FF_FMA(a.h, b.h, -r.h)));
  return r;
}
FF_FN ff ff_mul(float a, ff b) {
  ff r;
  r.h = FF_MUL(a, b.h);
  r.l = FF_FMA(a, b.l, FF_FMA(a, b.h, -r.h));
  return r;
}

// the pair rounded to FP32 (a product's head alone lacks its tail)
FF_FN float ff_round(ff a) { return FF_ADD(a.h, a.l); }

// 1/D: an FP32 seed r (error e < 2^-22) and r (1 + e + e^2), remainder e^3
FF_FN ff ff_inv(ff D) {
  ff r;
#ifdef __CUDA_ARCH__
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.h) : "f"(D.h));
#else
  r.h = 1.0f / D.h;
#endif
  const float e = FF_FMA(-D.l, r.h, FF_FMA(-D.h, r.h, 1.0f));
  r.l = FF_MUL(r.h, FF_FMA(e, e, e));
  return r;
}

// k = 8 log2(e) c for exp(-c D^2) (ff_reg_scale), the argument in eighths of a
// power of two
FF_FN ff ff_reg_scale(double c) { return ff_from(c * 11.541560327111707); }

// 2^{-m/8}, head and tail; `tab` of ff_one_minus_exp
FF_FN ff ff_exp_entry(int m) {
  const double t[8] = {1.0,
                       0.917004043204671231744,
                       0.840896415253714543031,
                       0.771105412703970411806,
                       0.707106781186547524401,
                       0.648419777325504832966,
                       0.594603557501360533359,
                       0.545253866332628829603};
  return ff_from(t[m]);
}

// 1 - exp(-c D^2) for k = ff_reg_scale(c), c >= 0. With x = k D^2 and n = rint(x)
// it is (1 - T) - T expm1(y), T = 2^{-n/8}, y = -(x - n) ln(2)/8, |y| <= 0.0434;
// expm1 by its Taylor series, the leading terms in pairs: y + y^2 (1/2 + y (1/6 +
// y (1/24 + ...))). For n = 0 it is -expm1(y) with no cancellation, so small
// c D^2 keep their relative accuracy. x > 700 (T < 2^-87) is cut off there.
FF_FN ff ff_one_minus_exp(ff D, ff k, const ff* tab) {
  // x = k D^2
  const float p = FF_MUL(D.h, D.h);
  const float pl = FF_FMA(FF_ADD(D.h, D.h), D.l, FF_FMA(D.h, D.h, -p));
  float xh = FF_MUL(p, k.h);
  float xl = FF_FMA(pl, k.h, FF_FMA(p, k.l, FF_FMA(p, k.h, -xh)));
  if (!(xh < 700.0f)) {
    xh = 700.0f;
    xl = 0.0f;
  }
  const float t = FF_ADD(xh, 12582912.0f);  // 1.5 * 2^23: rint(x) in the low bits
#ifdef __CUDA_ARCH__
  const int n = __float_as_int(t) - 0x4B400000;
#else
  const int n = (int)(t - 12582912.0f);
#endif
  const ff r = ff_two_sum(FF_SUB(xh, FF_SUB(t, 12582912.0f)), xl);
  // y = -r ln(2)/8
  const ff y = ff_mul(r, ff{-0.0866433978f, 2.38081777e-10f});
  const float z = FF_FMA(y.h, FF_FMA(y.h, FF_FMA(y.h, 1.0f / 5040.0f, 1.0f / 720.0f), 1.0f / 120.0f),
                         1.0f / 24.0f);
  // u = 1/6 + y z, w = 1/2 + y u (pairs)
  const float yz = FF_MUL(y.h, z);
  const ff u0 = ff_fast_sum(1.0f / 6.0f, yz);
  const ff u = {u0.h, FF_ADD(u0.l, -4.96705e-9f)};  // 1/6 - fl32(1/6)
  const ff v = ff_mul(y, u);
  const ff w0 = ff_fast_sum(0.5f, v.h);
  const ff w = {w0.h, FF_ADD(w0.l, v.l)};
  const ff q = ff_mul(ff_mul(y, y), w);
  const ff e0 = ff_fast_sum(y.h, q.h);
  const ff em = {e0.h, FF_ADD(e0.l, FF_ADD(y.l, q.l))};
  // T = 2^{-n/8}
  const ff tm = tab[n & 7];
#ifdef __CUDA_ARCH__
  const float sc = __int_as_float(0x3f800000 - ((n >> 3) << 23));
#else
  const float sc = ldexpf(1.0f, -(n >> 3));
#endif
  const ff T = {FF_MUL(tm.h, sc), FF_MUL(tm.l, sc)};
  const ff P = ff_mul(T, em);
  const ff a = ff_fast_sum(1.0f, -T.h);
  const ff g = ff_fast_sum(a.h, -P.h);
  return ff_fast_sum(g.h, FF_ADD(g.l, FF_SUB(FF_SUB(a.l, T.l), P.l)));
}

}  // namespace dsrg
