// Double-float ("double-word") arithmetic: a value is the unevaluated sum hi + lo of two FP32
// numbers with |lo| <= ulp(hi) / 2, about 48 significand bits.  The FP64 pipe of this GPU issues
// two fused multiply-adds per clock per SM against 128 for FP32, so element arithmetic that the
// FP64 pipe bounds runs faster as FP32 pairs at nearly FP64 accuracy.
//
// Building blocks (error-free transformations, round-to-nearest FP32):
//   TwoSum (Knuth 1969, Moller 1965): s + e = a + b exactly, 6 operations;
//   FastTwoSum (Dekker 1971): the same when |a| >= |b| (or a = 0), 3 operations;
//   TwoProd with FMA: p + e = a b exactly, 2 operations.
// Double-word operations from Joldes, Muller, Popescu, "Tight and rigorous error bounds for basic
// building blocks of double-word arithmetic", ACM TOMS 44 (2017):
//   addition "AccurateDWPlusDW" (their Algorithm 6), relative error <= 3u^2 + 13u^3;
//   multiplication "DWTimesDW3" (Algorithm 12, with FMA), relative error <= 4u^2;
// u = 2^-24.  Every operation is written out with the _rn intrinsics so that the compiler neither
// contracts nor reorders it.
//
// Conversions from and to binary64 use integer operations only (no FP64 instruction):
//   split: hi = the double truncated to 24 significand bits, lo = the remaining 29 bits rounded to
//   FP32 (exact integer-to-float tricks for 23 and 6 of them, one FMA), then FastTwoSum to restore
//   |lo| <= ulp(hi) / 2; relative error at most 2^-48.  Magnitudes below 2^-80 keep only hi, and values outside the FP32 exponent range
//   are not representable (the wedge operator's data are far inside both limits).
//   join: hi and lo widened exactly to binary64 (bit manipulation) and added with one FP64 add,
//   which is exact because hi + lo has at most 48 significant bits.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

namespace tn {

#if defined(__CUDA_ARCH__)
#define TN_DF_HD __device__ __forceinline__
#define TN_FADD(a, b) __fadd_rn(a, b)
#define TN_FSUB(a, b) __fsub_rn(a, b)
#define TN_FMUL(a, b) __fmul_rn(a, b)
#define TN_FFMA(a, b, c) __fmaf_rn(a, b, c)
#else
#define TN_DF_HD inline
#define TN_FADD(a, b) ((float)((a) + (b)))
#define TN_FSUB(a, b) ((float)((a) - (b)))
#define TN_FMUL(a, b) ((float)((a) * (b)))
#define TN_FFMA(a, b, c) std::fma((float)(a), (float)(b), (float)(c))
#endif

TN_DF_HD void two_sum(float a, float b, float& s, float& e) {
  s = TN_FADD(a, b);
  const float bb = TN_FSUB(s, a);
  e = TN_FADD(TN_FSUB(a, TN_FSUB(s, bb)), TN_FSUB(b, bb));
}
TN_DF_HD void fast_two_sum(float a, float b, float& s, float& e) {
  s = TN_FADD(a, b);
  e = TN_FSUB(b, TN_FSUB(s, a));
}

struct alignas(8) dfl {
  float hi, lo;
  dfl() = default;
  TN_DF_HD constexpr dfl(float h, float l) : hi(h), lo(l) {}
  // from a double known at compile time (constants of the element ops); folded by the compiler
  TN_DF_HD constexpr dfl(double x) : hi((float)x), lo((float)(x - (double)(float)x)) {}
};

TN_DF_HD dfl operator-(dfl a) { return dfl(-a.hi, -a.lo); }

// AccurateDWPlusDW
TN_DF_HD dfl operator+(dfl x, dfl y) {
  float sh, sl, th, tl, vh, vl, zh, zl;
  two_sum(x.hi, y.hi, sh, sl);
  two_sum(x.lo, y.lo, th, tl);
  const float c = TN_FADD(sl, th);
  fast_two_sum(sh, c, vh, vl);
  const float w = TN_FADD(tl, vl);
  fast_two_sum(vh, w, zh, zl);
  return dfl(zh, zl);
}
TN_DF_HD dfl operator-(dfl x, dfl y) { return x + (-y); }

// DWTimesDW3
TN_DF_HD dfl operator*(dfl x, dfl y) {
  const float ch = TN_FMUL(x.hi, y.hi);
  const float cl1 = TN_FFMA(x.hi, y.hi, -ch);
  const float tl0 = TN_FMUL(x.lo, y.lo);
  const float tl1 = TN_FFMA(x.hi, y.lo, tl0);
  const float cl2 = TN_FFMA(x.lo, y.hi, tl1);
  const float cl3 = TN_FADD(cl1, cl2);
  float zh, zl;
  fast_two_sum(ch, cl3, zh, zl);
  return dfl(zh, zl);
}

// Sum without the second TwoSum (the "sloppy" double-word addition): absolute error about
// 2u^2 (|x| + |y|), so it is kept for sums whose terms do not cancel; 11 operations.
TN_DF_HD dfl add_nc(dfl x, dfl y) {
  float sh, sl, zh, zl;
  two_sum(x.hi, y.hi, sh, sl);
  const float w = TN_FADD(sl, TN_FADD(x.lo, y.lo));
  fast_two_sum(sh, w, zh, zl);
  return dfl(zh, zl);
}
// x y + w in one pass: the exact product of the high parts (TwoProd), the cross terms by FMA,
// then the sloppy addition of w; absolute error about 3u^2 (|x y| + |w|), for the same use;
// 15 operations against 20 for a multiplication followed by an addition.
TN_DF_HD dfl fma_nc(dfl x, dfl y, dfl w) {
  const float ph = TN_FMUL(x.hi, y.hi);
  float pl = TN_FFMA(x.hi, y.hi, -ph);
  pl = TN_FFMA(x.hi, y.lo, pl);
  pl = TN_FFMA(x.lo, y.hi, pl);
  float sh, sl, zh, zl;
  two_sum(ph, w.hi, sh, sl);
  const float t = TN_FADD(sl, TN_FADD(pl, w.lo));
  fast_two_sum(sh, t, zh, zl);
  return dfl(zh, zl);
}

TN_DF_HD dfl& operator+=(dfl& a, dfl b) { return a = a + b; }
TN_DF_HD dfl& operator-=(dfl& a, dfl b) { return a = a - b; }

TN_DF_HD uint64_t df_bits_of(double x) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}
TN_DF_HD double df_double_of(uint64_t b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}
TN_DF_HD float df_float_of(uint32_t b) {
#if defined(__CUDA_ARCH__)
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, 4);
  return x;
#endif
}
TN_DF_HD uint32_t df_ubits_of(float x) {
#if defined(__CUDA_ARCH__)
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}

// binary64 -> double-float with integer operations (see the file comment)
TN_DF_HD dfl split(double x) {
  const uint64_t b = df_bits_of(x);
  const uint32_t bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  const uint32_t sign = bh & 0x80000000u;
  const int e = (int)((bh >> 20) & 0x7ffu);         // biased binary64 exponent
  if (e < 1023 - 126) return dfl(df_float_of(sign), 0.0f);  // zero or below the FP32 normal range
  const uint32_t m23 = ((bh & 0xfffffu) << 3) | (bl >> 29);  // top 23 stored significand bits
  const float hi = df_float_of(sign | ((uint32_t)(e - 1023 + 127) << 23) | m23);
  // the next 23 and the last 6 bits as exact integers (2^23 + n - 2^23), joined and rounded once, scaled by
  // 2^(e - 1023 - 46)
  const float t23 = TN_FSUB(df_float_of(0x4b000000u | ((bl >> 6) & 0x7fffffu)), 8388608.0f);
  const float t6 = TN_FSUB(df_float_of(0x4b000000u | (bl & 0x3fu)), 8388608.0f);
  const float t = TN_FFMA(t6, 0.015625f, t23);
  const int se = e - 1023 - 46 + 127;
  const float lo_mag = se >= 1 ? TN_FMUL(t, df_float_of((uint32_t)se << 23)) : 0.0f;
  const float lo = df_float_of(df_ubits_of(lo_mag) | sign);
  float zh, zl;
  fast_two_sum(hi, lo, zh, zl);
  return dfl(zh, zl);
}

// exact FP32 -> binary64 widening by bit manipulation (FP32 subnormals become 0)
TN_DF_HD double widen(float f) {
  const uint32_t u = df_ubits_of(f);
  const uint32_t e = (u >> 23) & 0xffu;
  if (e == 0) return df_double_of((uint64_t)(u & 0x80000000u) << 32);
  const uint64_t bits = ((uint64_t)(u & 0x80000000u) << 32) | ((uint64_t)(e + 1023 - 127) << 52) |
                        ((uint64_t)(u & 0x7fffffu) << 29);
  return df_double_of(bits);
}

// double-float -> binary64: one exact FP64 addition
TN_DF_HD double join(dfl a) { return widen(a.hi) + widen(a.lo); }

#if defined(__CUDACC__)
// Packed double-float: two independent values in the lanes of f32x2 registers (hi.x + lo.x,
// hi.y + lo.y), every operation the scalar one lane-wise with the packed FP32 instructions (one
// issue slot per pair).  Lanes never mix inside an operation and every packed instruction rounds
// each lane to nearest, so a lane follows the scalar formula step for step.  A kernel written with
// df2 may still group its sums differently from its scalar version: the two then agree to the
// double-float rounding level (about 2^-46 relative), not bitwise.
struct alignas(16) df2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 p2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a - b lane-wise, rounded to nearest: the packed subtraction of PTX (no intrinsic exists)
__device__ __forceinline__ float2 p2sub(float2 a, float2 b) {
  unsigned long long ra, rb, rd;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
  return d;
}
// A rounded product, as a fused multiply-add with 0: nvcc 13.0 contracts a packed multiplication and an addition
// of its result into one fused operation, also from PTX with explicit rounding (measured: the running sums
// below then lose 1e-7 where s cancels most of x y).  Same cost; a product of -0 becomes +0.
__device__ __forceinline__ float2 p2mul(float2 a, float2 b) { return p2fma(a, b, make_float2(0.f, 0.f)); }
__device__ __forceinline__ float2 p2neg(float2 a) { return make_float2(-a.x, -a.y); }

__device__ __forceinline__ df2 pack(dfl a, dfl b) { return df2{make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)}; }
__device__ __forceinline__ dfl lane_x(const df2& a) { return dfl(a.hi.x, a.lo.x); }
__device__ __forceinline__ dfl lane_y(const df2& a) { return dfl(a.hi.y, a.lo.y); }

__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = p2add(a, b);
  const float2 bb = p2sub(s, a);
  e = p2add(p2sub(a, p2sub(s, bb)), p2sub(b, bb));
}
__device__ __forceinline__ void fast_two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = p2add(a, b);
  e = p2sub(b, p2sub(s, a));
}
// AccurateDWPlusDW, lane-wise
__device__ __forceinline__ df2 add2(const df2& x, const df2& y) {
  float2 sh, sl, th, tl, vh, vl, zh, zl;
  two_sum2(x.hi, y.hi, sh, sl);
  two_sum2(x.lo, y.lo, th, tl);
  fast_two_sum2(sh, p2add(sl, th), vh, vl);
  fast_two_sum2(vh, p2add(tl, vl), zh, zl);
  return df2{zh, zl};
}
__device__ __forceinline__ df2 sub2(const df2& x, const df2& y) { return add2(x, df2{p2neg(y.hi), p2neg(y.lo)}); }
// DWTimesDW3, lane-wise
__device__ __forceinline__ df2 mul2(const df2& x, const df2& y) {
  const float2 ch = p2mul(x.hi, y.hi);
  const float2 cl1 = p2fma(x.hi, y.hi, p2neg(ch));
  const float2 tl1 = p2fma(x.hi, y.lo, p2mul(x.lo, y.lo));
  const float2 cl2 = p2fma(x.lo, y.hi, tl1);
  float2 zh, zl;
  fast_two_sum2(ch, p2add(cl1, cl2), zh, zl);
  return df2{zh, zl};
}
// Running sums of packed double-words, not renormalised between steps (acc2: value s + l, s the rounded sum
// of the high parts, l everything below it).  A contraction of three products costs 24 packed
// operations this way against 39 with a renormalised multiplication and two renormalised fused operations.  Errors: each
// step rounds l, which stays a few u |terms|, so a step adds about u^2 |terms|; the products drop l l.  That
// is the level at which the operands are rounded to double-words anyway (the accurate additions they
// replace keep no more digits of such operands).
//   acc_fma2 is TwoSum (Knuth, Moller) of s and the rounded product p; its second error term p - (s' - s) is
//   formed by FMA from x y itself, so it holds the product's rounding too.  (With s' = fma(x, y, s), one
//   operation less, TwoSum loses its exactness when s cancels most of x y: 1e-7 errors at single nodes.)
struct acc2 {
  float2 s, l;
};
__device__ __forceinline__ acc2 acc_of(const df2& x) { return acc2{x.hi, x.lo}; }
__device__ __forceinline__ df2 df_of(const acc2& a) { return df2{a.s, a.l}; }
__device__ __forceinline__ acc2 prod2(const df2& x, const df2& y) {
  const float2 p = p2mul(x.hi, y.hi);
  float2 l = p2fma(x.hi, y.hi, p2neg(p));
  l = p2fma(x.hi, y.lo, l);
  l = p2fma(x.lo, y.hi, l);
  return acc2{p, l};
}
__device__ __forceinline__ void acc_fma2(acc2& a, const df2& x, const df2& y) {
  const float2 s = p2add(a.s, p2mul(x.hi, y.hi));
  const float2 nb = p2sub(a.s, s);                 // -(s - a.s)
  const float2 ea = p2sub(a.s, p2add(s, nb));      // what a.s lost
  const float2 eb = p2fma(x.hi, y.hi, nb);         // what x y lost, the rounding of the product included
  float2 l = p2add(a.l, p2add(ea, eb));
  l = p2fma(x.hi, y.lo, l);
  a.l = p2fma(x.lo, y.hi, l);
  a.s = s;
}
__device__ __forceinline__ void acc_add2(acc2& a, const df2& x) {
  float2 s, e;
  two_sum2(a.s, x.hi, s, e);
  a.l = p2add(a.l, p2add(e, x.lo));
  a.s = s;
}
__device__ __forceinline__ acc2 sum2(const df2& x, const df2& y) {
  acc2 a = acc_of(x);
  acc_add2(a, y);
  return a;
}
__device__ __forceinline__ df2 norm2(const df2& a) {  // FastTwoSum of the two parts
  df2 r;
  fast_two_sum2(a.hi, a.lo, r.hi, r.lo);
  return r;
}
__device__ __forceinline__ df2 neg2(const df2& x) { return df2{p2neg(x.hi), p2neg(x.lo)}; }
__device__ __forceinline__ df2 diff2(const df2& x, const df2& y) { return df_of(sum2(x, neg2(y))); }
__device__ __forceinline__ df2 dot3(const df2& x0, const df2& y0, const df2& x1, const df2& y1, const df2& x2,
                                    const df2& y2) {
  acc2 a = prod2(x0, y0);
  acc_fma2(a, x1, y1);
  acc_fma2(a, x2, y2);
  return df_of(a);
}
__device__ __forceinline__ df2 both(const dfl& a) { return pack(a, a); }
#endif

}  // namespace tn
