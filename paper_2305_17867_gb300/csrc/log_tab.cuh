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
// that their sum is exact; b is short, so that r is exact near 1; and r is added
// by Fast2Sum, its error going to the small terms.  At most 0.58 ulp, rms 0.289
// (a correctly rounded logarithm has 0.5 and 0.289); one-part constants and a 24-bit
// 1/c gave 1.6 and 0.41 to 0.48.
#pragma once

#include <cmath>

#include "fmm_internal.cuh"

struct LogTab {
  // b = 1/c (8 bits) and -log b in two parts, k = 96 .. 192
  double inv[kLogTab], hi[kLogTab], lo[kLogTab];
};

__device__ __forceinline__ double log_tab(double x, const LogTab& t) {  // x > 0
  const int hi = __double2hiint(x);
  if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return log(x);  // subnormal, inf
  const int up = (hi & 0x000fffff) >= 0x00080000 ? 1 : 0;          // m >= 3/2: halve it
  const int e = (hi >> 20) - 1023 + up;
  const double m = __hiloint2double((hi & 0x000fffff) | (0x3ff00000 - (up << 20)),
                                    __double2loint(x));
  // nearest k/128: m in [1, 3/2): 1/128 is bit 13 of the high word; in [3/4, 1): bit 14
  const int hm = __double2hiint(m) & 0x000fffff;
  const int k = (up ? 64 + ((hm + (1 << 13)) >> 14) : 128 + ((hm + (1 << 12)) >> 13)) - 96;
  const double r = fma(m, t.inv[k], -1.0);
  double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
  q = fma(r, q, 1.0 / 5.0);
  q = fma(r, q, -1.0 / 4.0);
  q = fma(r, q, 1.0 / 3.0);
  q = fma(r, q, -1.0 / 2.0);
  const double ed = __hiloint2double(0x43300000, (int)((unsigned)e ^ 0x80000000u)) -
                    __hiloint2double(0x43300000, (int)0x80000000u);
  // log 2 rounded to a multiple of 2^-42, and the rest
  const double s = fma(ed, 0x1.62e42fefa38p-1, t.hi[k]);  // exact
  const double p = fma(r * r, q, fma(ed, 0x1.ef35793c7673p-45, t.lo[k]));
  const double u = s + r;  // s = 0 or |s| > |r|
  return u + (((s - u) + r) + p);
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

// the table's 3 kLogTab doubles in the order of LogTab
inline void fill_log_tab(double* t) {
  for (int k = 0; k < kLogTab; ++k) {
    t[k] = std::nearbyint(256.0 * 128.0 / (96 + k)) / 256.0;
    log_parts(t[k], &t[kLogTab + k], &t[2 * kLogTab + k]);
  }
}
