// FP64 logarithm of the 2D near field (leaf.cu), and its table.
//
// Table-driven (P. T. P. Tang, "Table-driven implementation of the logarithm
// function in IEEE floating-point arithmetic", ACM TOMS 16, 1990): x = 2^e m,
// m in [3/4, 3/2), c = k/128 the nearest table point, b an 8-bit 1/c, r = m b - 1
// by one FMA, log x = e log 2 - log b + log1p(r), |r| < 2^-7.2, the last by its
// series to r^7.  At c = 1 the table is exact, so log keeps its relative accuracy
// as x -> 1.
//
// The table and log 2 come in two parts, the leading ones multiples of 2^-42, so
// that their sum is exact; b is short, so that r is exact near 1; and r is added in
// two parts, the leading 20 bits exactly, the rest with the small terms.  At most
// 0.58 ulp, rms 0.289 (a correctly rounded logarithm has 0.5 and 0.289; only past
// |log x| = 32, where r < 2^-22 may not add exactly, up to 0.99); one-part
// constants and a 24-bit 1/c gave 1.6 and 0.41 to 0.48.
//
// The FP64 pipe (two lanes a cycle) bounds the near field, so what lies 2^-32 and
// more below the result is formed in float (the series from r^5, the trailing
// parts of the table and of log 2) and widened through its bits: eleven FP64
// instructions, against about 25 of log().  Planar biharmonic with gradient, 120k
// points: 1,363 us; 1,543 with all of it in FP64 (sixteen), 1,368 with the one-part
// constants (eleven).
#pragma once

#include <cmath>

#include "fmm_internal.cuh"

struct LogTab {
  // b = 1/c (8 bits) and -log b in two parts, k = 96 .. 192
  double inv[kLogTab], hi[kLogTab];
  float lo[kLogTab];
};

// (double)x for x = 0 or a normal float (the conversion without its FP64 work)
__device__ __forceinline__ double widen_normal(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  const unsigned hi = (b & 0x80000000u) | (m != 0 ? (m >> 3) + (896u << 20) : 0u);
  return __hiloint2double((int)hi, (int)(b << 29));
}

__device__ __forceinline__ double log_tab(double x, const LogTab& t) {  // x > 0
  const int hi = __double2hiint(x);
  if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return log(x);  // subnormal, inf
  const int up = (hi & 0x000fffff) >= 0x00080000 ? 1 : 0;          // m >= 3/2: halve it
  const int e = (hi >> 20) - 1023 + up;
  const int mh = (hi & 0x000fffff) | (0x3ff00000 - (up << 20));
  const double m = __hiloint2double(mh, __double2loint(x));
  // nearest k/128: m in [1, 3/2): 1/128 is bit 13 of the high word; in [3/4, 1): bit 14
  const int hm = mh & 0x000fffff;
  const int k = (up ? 64 + ((hm + (1 << 13)) >> 14) : 128 + ((hm + (1 << 12)) >> 13)) - 96;
  const double b = t.inv[k];
  const double r = fma(m, b, -1.0);
  // r^5 (1/5 - r/6 + r^2/7) with the bracket, and its r, in float (m and b cut to floats)
  const unsigned off = 896u << 20;
  const float mf = __uint_as_float((((unsigned)mh - off) << 3) | ((unsigned)__double2loint(x) >> 29));
  const float rf = __fmaf_rn(mf, __uint_as_float(((unsigned)__double2hiint(b) - off) << 3), -1.f);
  const float c = __fmaf_rn(rf, __fmaf_rn(rf, 1.f / 7.f, -1.f / 6.f), 0.2f);
  const unsigned cb = __float_as_uint(c);  // (c > 0)
  double q = fma(r, __hiloint2double((int)((cb >> 3) + off), (int)(cb << 29)), -1.0 / 4.0);
  q = fma(r, q, 1.0 / 3.0);
  q = fma(r, q, -1.0 / 2.0);
  // log 2 rounded to a multiple of 2^-42, and the rest
  const float ef = (float)e;
  const double s = fma(widen_normal(ef), 0x1.62e42fefa38p-1, t.hi[k]);  // exact
  const double p = fma(r * r, q, widen_normal(__fmaf_rn(ef, 0x1.ef3579p-45f, t.lo[k])));
  const double rh = __hiloint2double(__double2hiint(r), 0);
  return (s + rh) + ((r - rh) + p);
}

// -log(c) = hi + lo, hi a multiple of 2^-42, for c of at most 8 bits in (1/2, 2):
// -2 atanh(z), z = (c - 1)/(c + 1), |z| < 1/3, by its series in double-doubles
inline void log_parts(double c, double* hi, double* lo) {
  struct dd {
    double h, l;
  };
  auto norm = [](double h, double l) {
    const double s = h + l;
    return dd{s, l - (s - h)};
  };
  auto mul = [&](dd a, dd b) {
    const double p = a.h * b.h;
    return norm(p, std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
  };
  const double num = c - 1.0, den = c + 1.0;  // exact
  const double z0 = num / den;
  const dd z{z0, std::fma(-z0, den, num) / den};
  const dd z2 = mul(z, z);
  dd s{1.0 / 71.0, 0.0};
  for (int k = 69; k >= 1; k -= 2) {  // 1/k + z^2 s
    const dd t = mul(s, z2);
    const double a = 1.0 / k, al = std::fma(-a, (double)k, 1.0) / k;
    const double h = a + t.h;
    s = norm(h, (t.h - (h - a)) + (al + t.l));
  }
  const dd v = mul(z, s);
  const double big = 1.5 * 1024.0;  // (adding it rounds to multiples of 2^-42)
  const double r = (-2.0 * v.h + big) - big;
  *hi = r;
  *lo = (-2.0 * v.h - r) - 2.0 * v.l;
}

// b and the two parts of -log b, kLogTab doubles each
inline void fill_log_tab(double* t) {
  for (int k = 0; k < kLogTab; ++k) {
    t[k] = std::nearbyint(256.0 * 128.0 / (96 + k)) / 256.0;
    log_parts(t[k], &t[kLogTab + k], &t[2 * kLogTab + k]);
  }
}
