// FP64 Box-Muller on one word pair, for a GPU with two FP64 lanes an SM: the
// arguments are 32-bit integers, so the logarithm, the sine and the cosine are
// computed in 64-bit integers, and FP64 does the square root and the products
// (8 instructions a pair instead of the 110 of log, sqrt and sincospi: the
// 512^3 z forward pass 12.9 -> 2.50 ms together with its fixed-point transform).
//
// * ln u, u = (r + 1) 2^-32 = y 2^(-1-z), y in [1, 2) from the 32 bits: the top
//   seven fraction bits select c ~ 1/y (11 bits), t = y c - 1 is exact, ln u =
//   (L - n ln 2) + ln(1 + t), |t| < 2^-7.8, the series to t^7 (next term below
//   2^-57 of t). For y >= 1.414 the entry holds L = -ln(2c) and n = z (else
//   -ln c and z + 1), so that nothing cancels. Units: 2^-61 where n = 0 (then
//   -2 ln u < 0.7), else 2^-57. Near u = 1 (above 1 - 2^-8, where c = 1/2 and
//   L = 0) the series runs in FP64, which keeps its relative accuracy.
// * rho = sqrt(-2 ln u): the FP32 reciprocal root and two Newton steps in FP64
//   with a final correction of the root (Markstein).
// * 2 pi u': the nearest quarter turn and 2^-10 of a turn by integers, then
//   sin and cos of the remainder (below 2^-8.3) by their series and one complex
//   product with the table's entry, in units of 2^-62; within 2^-11 of a turn from
//   an axis the small one of the two by its series in FP64, which keeps its
//   relative accuracy (units of 2^-62 had left it 10 digits at the smallest
//   angles).
// Against extended precision over 128^3 cells: relative L2 8.05e-17 (log and
// sincospi: 8.4e-17).
#pragma once

#include <stdint.h>

#include "gg_fixed.cuh"

namespace gg {
namespace gauss64 {

// The tables are rounded once from sums in two-double arithmetic (error-free
// sums and Dekker's products), evaluated by the compiler.
struct Dd {
  double h, l;
};
__host__ __device__ constexpr Dd two_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return Dd{s, (a - (s - t)) + (b - t)};
}
__host__ __device__ constexpr Dd dd_add(Dd a, Dd b) {
  const Dd s = two_sum(a.h, b.h);
  const double e = s.l + a.l + b.l, h = s.h + e;
  return Dd{h, e - (h - s.h)};
}
__host__ __device__ constexpr Dd two_prod(double a, double b) {
  const double ca = 134217729.0 * a, cb = 134217729.0 * b;  // 2^27 + 1
  const double ah = ca - (ca - a), al = a - ah, bh = cb - (cb - b), bl = b - bh;
  const double p = a * b;
  return Dd{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
__host__ __device__ constexpr Dd dd_mul(Dd a, Dd b) {
  const Dd p = two_prod(a.h, b.h);
  const double e = p.l + a.h * b.l + a.l * b.h, h = p.h + e;
  return Dd{h, e - (h - p.h)};
}
__host__ __device__ constexpr Dd dd_div(Dd a, double b) {
  const double q = a.h / b;
  const Dd p = two_prod(q, b);
  const double r = ((a.h - p.h) - p.l) + a.l, q2 = r / b, h = q + q2;
  return Dd{h, q2 - (h - q)};
}
__host__ __device__ constexpr Dd ln_series(double c) {  // ln c = 2 atanh((c - 1) / (c + 1)), c of 12 bits
  const Dd z = dd_div(Dd{c - 1.0, 0.0}, c + 1.0), z2 = dd_mul(z, z);
  Dd t = z, s = Dd{0.0, 0.0};
  for (int i = 0; i < 34; ++i) {
    s = dd_add(s, dd_div(t, 2.0 * i + 1.0));
    t = dd_mul(t, z2);
  }
  return Dd{2.0 * s.h, 2.0 * s.l};
}
// sum of (-1)^i x^(2i + odd) / (2i + odd)!
__host__ __device__ constexpr Dd circle_series(Dd x, int odd) {
  const Dd x2 = dd_mul(x, x);
  Dd t = odd ? x : Dd{1.0, 0.0}, s = Dd{0.0, 0.0};
  for (int i = 0; i < 14; ++i) {
    s = dd_add(s, t);
    t = dd_div(dd_mul(t, x2), -(2.0 * i + odd + 1.0) * (2.0 * i + odd + 2.0));
  }
  return s;
}

struct Tables {
  int4 ln[128];  // {low and high word of round(-2 L 2^61), 2^11 c, 0}
  int4 cs[257];  // cos, sin of 2 pi (j - 128) / 1024 as twiddles: round(v 2^62) = h 2^32 + l, {h, l, h, l}
};
constexpr int kRoot2 = 53;  // first entry with y >= 1.414
__host__ __device__ constexpr long long rounded(Dd v, double unit) {  // |v unit| < 2^63
  const double h = v.h * unit, l = v.l * unit;  // exact: powers of two
  const long long i = (long long)h;             // h - i exact
  const double f = (h - (double)i) + l;
  return i + (long long)(f < 0 ? f - 0.5 : f + 0.5);
}
__host__ __device__ constexpr Tables make_tables() {
  Tables t = {};
  for (int j = 0; j < 128; ++j) {
    const double y = 1.0 + (j + 0.5) / 128.0;
    const int q = j == 127 ? 1024 : (int)(2048.0 / y + 0.5);
    const double c = q / 2048.0;
    const long long w = j == 127 ? 0 : rounded(ln_series(j >= kRoot2 ? 2.0 * c : c), 0x1p62);  // -2 L
    t.ln[j] = int4{fx::low_half(w), fx::high_half(w) + (fx::low_half(w) < 0 ? -1 : 0), q, 0};
  }
  for (int j = 0; j <= 256; ++j) {
    // 2 pi = 6.283185307179586 + 2.4492935982947064e-16
    const Dd x = dd_mul(Dd{0x1.921fb54442d18p+2, 0x1.1a62633145c07p-52}, Dd{(j - 128) / 1024.0, 0.0});
    const long long c = rounded(circle_series(x, 0), 0x1p62), n = rounded(circle_series(x, 1), 0x1p62);
    t.cs[j] = int4{fx::high_half(c), fx::low_half(c), fx::high_half(n), fx::low_half(n)};
  }
  return t;
}
static __device__ const Tables kTables = make_tables();

__device__ __forceinline__ double neg2_ln_near1(uint32_t r) {  // u > 1 - 2^-8
  const double t = -((double)(~r) * 0x1p-32);                  // u - 1, exact
  double q = fma(t, 1.0 / 7.0, -1.0 / 6.0);
  q = fma(t, q, 0.2);
  q = fma(t, q, -0.25);
  q = fma(t, q, 1.0 / 3.0);
  q = fma(t, q, -0.5);
  return -2.0 * fma(t * t, q, t);
}
__device__ __forceinline__ double neg2_ln(uint32_t r) {  // -2 ln((r + 1) 2^-32)
  if (r >= 0xff000000u) return neg2_ln_near1(r);
  const uint32_t x = r + 1u;
  const int z = __clz((int)x);
  const uint32_t m = x << z;
  const int j = (int)((m >> 24) & 127u);
  const int4 e = __ldg(&kTables.ln[j]);
  const long long w = ((long long)e.y << 32) | (uint32_t)e.x;
  const long long t42 = (long long)((unsigned long long)m * (uint32_t)e.z) - (1ll << 42);  // t 2^42, exact
  const long long t70 = (long long)((unsigned long long)t42 << 28);
  const long long t2 = __mul64hi(t70, t70);                          // t^2 2^76
  const long long t3 = __mul64hi(t70, 6148914691236517205ll);        // t/3 2^70
  // 1/4 - t (1/5 - t (1/6 - t/7)) 2^32, then times t^2 2^47
  const int t31 = (int)(t42 >> 11);
  const int q7 = 715827883 - 2 * __mulhi(t31, 613566757);            // 1/6 - t/7
  const int q6 = 858993459 - 2 * __mulhi(t31, q7);                   // 1/5 - t (...)
  const uint32_t q5 = 1073741824u - 2 * __mulhi(t31, q6);            // 1/4 - t (...)
  const uint32_t r2 = __umulhi((uint32_t)(t2 >> 29), q5);            // 2^47
  const long long q = (1ll << 61) - (t3 >> 8) + ((long long)r2 << 15);  // 1/2 - t/3 + t^2/4 - ... 2^62
  const long long l1 = (long long)((unsigned long long)t42 << 20) - (__mul64hi(t2, q) >> 12);  // ln(1 + t) 2^62
  const int n = z + (j < kRoot2 ? 1 : 0);
  // -2 ln u = 2 n ln 2 - 2 L - 2 ln(1 + t); 2 ln(1 + t) in units of 2^-61 is l1
  if (n == 0) return fx::scaled_double(w - l1, 61);
  return fx::scaled_double((long long)n * 199786072581291495ll + ((w - l1) >> 4), 57);
}
__device__ __forceinline__ double root(double a) {  // sqrt(a), 0 or 2^-31 < a < 64
  const int hi = __double2hiint(a);
  if (hi == 0) return 0.0;
  // FP32 value and its reciprocal root, moved between the formats by their bits
  const float f = __int_as_float((hi - ((1023 - 127) << 20)) << 3);
  const int yb = __float_as_int(rsqrtf(f));
  const double y = __hiloint2double((yb >> 3) + ((1023 - 127) << 20), yb << 29);
  double g = a * y, h = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  const double d = fma(-g, g, a);
  return fma(d, h, g);
}
// sin(2 pi d 2^-32), |d| <= 2^21: x - x^3/6 + x^5/120 (next term below 2^-62 of x),
// within 1.4 units of the last place. One warp in eight gets here.
__device__ __forceinline__ double small_sine(int d) {
  const double x = (double)d * 0x1.921fb54442d18p-30, x2 = x * x;  // 2 pi 2^-32
  return fma(x * x2, fma(x2, 1.0 / 120.0, -1.0 / 6.0), x);
}
// 2 pi 2^38 = kTurnHi 2^32 + kTurnLo + kTurnFrac 2^-31
constexpr int kTurnHi = 402, kTurnLo = 531973186, kTurnFrac = 1757557957;
__device__ __forceinline__ void sincos_turn(uint32_t rb, double &s, double &c) {
  const uint32_t q = (rb + (1u << 29)) >> 30;   // nearest quarter turn (mod 4)
  const int t = (int)(rb - (q << 30));          // remainder, |t| <= 2^29
  const int j = (t + (1 << 21)) >> 22;          // |j| <= 128
  const int d = t - j * (1 << 22);              // |d| <= 2^21
  const int4 e = __ldg(&kTables.cs[j + 128]);
  // x = 2 pi d 2^-32 in units of 2^-70
  const long long x = (long long)((unsigned long long)((long long)d * kTurnHi) << 32) + (long long)d * kTurnLo + (((long long)d * kTurnFrac) >> 31);
  const long long x2 = __mul64hi(x, x);                              // x^2 2^76
  const uint32_t xs = (uint32_t)(x2 >> 28);                          // 2^48, below 2^31.4
  const uint32_t x4 = __umulhi(xs, xs);                              // x^4 2^64, below 2^30.7
  // 1 - sin x / x = x^2/6 - x^4/120 in units of 2^-76; sin x in units of 2^-70
  const long long u = __mul64hi(x2, 3074457345618258603ll) - ((long long)__umulhi(x4, 35791394u) << 12);
  const long long sn = x - (__mul64hi(x, u) >> 12);
  // 1 - cos x = x^2/2 - x^4/24 in units of 2^-76
  const long long cm = (x2 >> 1) - ((long long)__umulhi(x4, 178956971u) << 12);
  const Fx a = fx::mul(Fx{(1ll << 62) - (cm >> 14), sn >> 8}, e.x, e.y, e.z, e.w);
  const long long p = (q & 1) ? a.x : a.y, w = (q & 1) ? a.y : a.x;  // sin, cos by quarter turns
  s = fx::scaled_double((q & 2) ? -p : p, 62);
  c = fx::scaled_double(((q + 1) & 2) ? -w : w, 62);
  if (j == 0) {  // near an axis one of the two is as small as the angle
    const double v = small_sine(d);
    if (q & 1) c = (q & 2) ? v : -v;
    else s = (q & 2) ? -v : v;
  }
}

}  // namespace gauss64
}  // namespace gg
