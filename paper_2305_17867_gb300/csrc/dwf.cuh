// Double-word float ("float-float") arithmetic: a value is the unevaluated
// sum h + l of two floats with |l| <= ulp(h) / 2, about 48 significant bits.
// The mixed-precision modes run the M2M / L2L shifts of the upper tree in it
// instead of FP64: GB300 issues FP64 at 1/64 of the FP32 rate, and a
// double-word multiply-add takes about fifteen FP32 instructions.
//
// Building blocks (error-free transformations):
//  * TwoSum (Knuth, TAOCP vol. 2, 4.2.2; Moller 1965): s = fl(a + b) and the
//    exact rounding error e, a + b = s + e, in six additions;
//  * Fast2Sum (Dekker 1971): the same in three additions when |a| >= |b|;
//  * TwoProd by FMA: p = fl(a b), e = fma(a, b, -p), a b = p + e exactly.
// Sum of two double-words: TwoSum of the high parts, the low parts added to
// its error, renormalised by Fast2Sum (the "sloppy" double-word sum analysed
// by Joldes, Muller and Popescu, ACM TOMS 44(2), 2017).  Its error is at most
// about 4 u^2 (|x| + |y|) with u = 2^-24, i.e. 2^-46 (|x| + |y|): an absolute
// bound of the kind FP64 summation has (2^-53 (|x| + |y|)), with no relative
// bound when x and y cancel.  Product: TwoProd of the high parts plus the two
// cross terms by FMA, renormalised by Fast2Sum (the low x low term, below
// u^2 |x y|, is dropped): relative error at most about 4 u^2 = 2^-46.
// Every operation is written with the _rn intrinsics, which the compiler
// never contracts into an FMA or reorders: the transformations depend on each
// rounding taking place as written.
#pragma once

#include <cuda_runtime.h>

struct dwf {
  float h, l;
  __device__ __forceinline__ dwf() = default;
  __device__ __forceinline__ constexpr dwf(float hi, float lo) : h(hi), l(lo) {}
  __device__ __forceinline__ dwf(int v) : h((float)v), l(0.f) {}  // small integers (0, 1)
  __device__ __forceinline__ explicit dwf(double v) {
    h = __double2float_rn(v);
    l = __double2float_rn(__dsub_rn(v, (double)h));
  }
  __device__ __forceinline__ explicit operator double() const {
    return __dadd_rn((double)h, (double)l);
  }
};

__device__ __forceinline__ dwf dw_fast2sum(float a, float b) {  // |a| >= |b| (or a = 0)
  const float s = __fadd_rn(a, b);
  return dwf(s, __fsub_rn(b, __fsub_rn(s, a)));
}

__device__ __forceinline__ dwf operator+(dwf x, dwf y) {
  const float s = __fadd_rn(x.h, y.h);
  const float bp = __fsub_rn(s, x.h);
  const float e = __fadd_rn(__fsub_rn(x.h, __fsub_rn(s, bp)), __fsub_rn(y.h, bp));
  return dw_fast2sum(s, __fadd_rn(e, __fadd_rn(x.l, y.l)));
}
__device__ __forceinline__ dwf operator-(dwf x) { return dwf(-x.h, -x.l); }
__device__ __forceinline__ dwf operator-(dwf x, dwf y) { return x + (-y); }
__device__ __forceinline__ dwf operator*(dwf x, dwf y) {
  const float p = __fmul_rn(x.h, y.h);
  float e = __fmaf_rn(x.h, y.h, -p);
  e = __fmaf_rn(x.h, y.l, e);
  e = __fmaf_rn(x.l, y.h, e);
  return dw_fast2sum(p, e);
}
__device__ __forceinline__ dwf& operator+=(dwf& x, dwf y) { return x = x + y; }
__device__ __forceinline__ dwf& operator-=(dwf& x, dwf y) { return x = x - y; }
__device__ __forceinline__ dwf& operator*=(dwf& x, dwf y) { return x = x * y; }
__device__ __forceinline__ dwf fma(dwf a, dwf b, dwf c) { return a * b + c; }

// ---- conversions without the FP64 pipe ----------------------------------------
// GB300 converts double <-> float at two lanes a cycle and SM (a warp's
// instruction takes 16 cycles), like all FP64 work; these go through the bit
// patterns.  x = h + l as the conversions give them, h = fl(x), l = fl(x - h)
// (2^-49 of x; the same bits): round to nearest even at bit 29 of the
// significand, and the signed 29-bit rest converted as an integer.  False for
// what float exponents cannot hold with room for l (outside 2^-63 .. 2^117),
// infinities and NaN.
__device__ __forceinline__ bool dw_bits(double x, float* h, float* l) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const unsigned long long a = b & 0x7fffffffffffffffull;
  const int e = (int)(a >> 52);
  if (a == 0) {
    *h = *l = 0.f;
    return true;
  }
  if (e < 960 || e > 1140) return false;
  const unsigned top = (unsigned)(a >> 29);  // exponent (modulo 2^9) and leading 23 bits
  const unsigned r = (unsigned)((a + 0x0fffffffu + (top & 1u)) >> 29);
  *h = __uint_as_float((r - (unsigned)(896ull << 23)) | sign);
  const int rest = (int)((unsigned)a & 0x1fffffffu) - (int)((r - top) << 29);
  *l = __uint_as_float(
      __float_as_uint(__fmul_rn((float)rest, __uint_as_float((unsigned)(e - 948) << 23))) ^ sign);
  return true;
}
// (double)x, exact (subnormal floats, infinities and NaN through the conversion)
__device__ __forceinline__ double widen_bits(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  if (m != 0 && m - 0x00800000u >= 0x7f000000u) return (double)x;
  const unsigned hi = (b & 0x80000000u) | (m != 0 ? (m >> 3) + (896u << 20) : 0u);
  return __hiloint2double((int)hi, (int)(b << 29));
}

// an expansion's coefficient (FP64 in memory) in a kernel's arithmetic, and back
template <typename T>
__device__ __forceinline__ T coef_in(double x);
template <>
__device__ __forceinline__ double coef_in<double>(double x) { return x; }
template <>
__device__ __forceinline__ float coef_in<float>(double x) {
  float h, l;
  return dw_bits(x, &h, &l) ? h : (float)x;
}
template <>
__device__ __forceinline__ dwf coef_in<dwf>(double x) {
  float h, l;
  return dw_bits(x, &h, &l) ? dwf(h, l) : dwf(x);
}
__device__ __forceinline__ double coef_out(double x) { return x; }
__device__ __forceinline__ double coef_out(float x) { return widen_bits(x); }
__device__ __forceinline__ double coef_out(dwf x) {
  return __dadd_rn(widen_bits(x.h), widen_bits(x.l));
}
