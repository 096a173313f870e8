// 64-bit fixed-point complex arithmetic for the FP64 transforms.
//
// GB300 has two FP64 lanes an SM (a warp instruction holds the pipe for 16
// cycles), against 64 integer ones: a 512-point FP64 transform needs 28 FP64
// instructions a point, 14 SM cycles, however it is scheduled, and the FP64
// kernels ran at 84% of that bound. The same transform on 64-bit integers takes
// about 120 integer instructions a point, two to three cycles. 512^3 noise ->
// pos + vel 59.1 -> 12.8 ms (z forward 12.9 -> 2.50, y 3.38 -> 0.90, x 11.1 -> 3.04,
// y inverses 11.0 -> 2.63, z inverses 20.7 -> 3.74), bound by the latency of the
// integer chains at 16 warps an SM (12 at 192 to 384, 8 at 768 and 1536).
//
// Each transform of N points (a column of a tile, a line) gets one power of two
// as its scale, from the sum A of the moduli of its inputs, estimated from above by
// the sum of |re| + |im|, above N = 768 more closely (modulus): the largest one for
// which that stays below 2^62.5. Every intermediate and output of the transform is
// bounded by A (all twiddles have modulus one), and the sums re + im that products
// by (1 + i) / sqrt(2) take by sqrt(2) A, so nothing reaches 2^63. (The i m outputs of the
// strided passes 2^62; z forward, whose last step adds two outputs, 2^61, above N =
// 512, where that bit counts, 2^62 and the outputs halved first.)
//
// Rounding the inputs to their unit u changes each output by 0.41 sqrt(N) u rms.
// The unit is A 2^-62.5 to A 2^-61.5 and A <= sqrt(N) L2 (L2: root of the sum of
// squares of the inputs, the rms of the outputs), so a flat spectrum or white
// noise is off by up to 0.41 N 2^-61.5 of its rms, a steep one by less. Products by
// twiddles keep 62 bits; those of the first stages add a third. Emulated for a
// strided column of white noise, rms over the position of the power of two: 1.1e-16
// at N = 1024, 1.8e-16 at 1536 (an FP64 transform there: 2.5e-16, 2.7e-16).
// Six transforms forward and back on white noise, against the identity, fixed
// point and FP64 transforms:
//   N             64    256   384   512   768   1024  1536
//   fixed point   1.5   1.6   2.8   2.2   3.4   3.0   4.4   e-16 relative L2 (largest: 4.7)
//   FP64          4.3   5.4   5.8   5.7   6.2   6.2   6.6
// Every rounding is unbiased: the modes along the axes are off by 1.5e-16 to 4.6e-16
// (FP64: 2.7e-16 to 5.6e-16), the worst cell by 6 to 11 times the rms error.
// Measured against 113-bit arithmetic, the density chain of six transforms is
// off by 1.2e-16 to 2.7e-16 relative L2 (white, steep, spike and single-mode
// fields of 32^3 to 128^3; the FP64 transforms: 3.0e-16 to 5.2e-16).
// Infinities and NaN turn their whole transform into NaN, as the FP64 sums did.
#pragma once

#include <type_traits>

#include "gg_device.cuh"

namespace gg {

template <> struct CxOf<long long> { using T = Fx; };

namespace fx {

constexpr float kRootHalf = 0.70710684f;                // sqrt(1/2), from above
constexpr long long kSqrtHalf = 3260954456333195553ll;  // sqrt(1/2) 2^62
constexpr long long kSin60 = 3993837246235628775ll;     // sqrt(3)/2 2^62

}  // namespace fx

__device__ __forceinline__ Fx cmul(Fx a, TwFx w) { return fx::mul(a, w.x, w.y, w.z, w.w); }
__device__ __forceinline__ Fx cmulc(Fx a, TwFx w) { return fx::mul(a, w.x, w.y, -w.z, -w.w); }

template <bool INV> struct Butterfly<3, INV, Fx> {
  static __device__ __forceinline__ void run(Fx *v) {
    constexpr int h = fx::high_half(fx::kSin60), l = fx::low_half(fx::kSin60);
    const Fx s = cadd(v[1], v[2]), d = csub(v[1], v[2]);
    const Fx t = {v[0].x - fx::half_even(s.x), v[0].y - fx::half_even(s.y)};
    const Fx r = mul_wi<INV>(Fx{fx::mul_real(d.x, h, l), fx::mul_real(d.y, h, l)});
    v[0] = cadd(v[0], s);
    v[1] = cadd(t, r);
    v[2] = csub(t, r);
  }
};
template <bool INV> struct Butterfly<8, INV, Fx> {
  static __device__ __forceinline__ void run(Fx *v) {
    constexpr int h = fx::high_half(fx::kSqrtHalf), l = fx::low_half(fx::kSqrtHalf);
    Fx e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    Butterfly<4, INV, Fx>::run(e);
    Butterfly<4, INV, Fx>::run(o);
    // o_1 w8, o_3 w8^3 from the two sums of their components
    const long long s1 = fx::mul_real(o[1].x + o[1].y, h, l), d1 = fx::mul_real(o[1].x - o[1].y, h, l);
    const long long s3 = fx::mul_real(o[3].x + o[3].y, h, l), d3 = fx::mul_real(o[3].x - o[3].y, h, l);
    const Fx o1 = INV ? Fx{d1, s1} : Fx{s1, -d1};
    const Fx o3 = INV ? Fx{-s3, d3} : Fx{-d3, -s3};
    const Fx o2 = mul_wi<INV>(o[2]);
    v[0] = cadd(e[0], o[0]);
    v[4] = csub(e[0], o[0]);
    v[1] = cadd(e[1], o1);
    v[5] = csub(e[1], o1);
    v[2] = cadd(e[2], o2);
    v[6] = csub(e[2], o2);
    v[3] = cadd(e[3], o3);
    v[7] = csub(e[3], o3);
  }
};

namespace fx {

// ------------------------------------------------------------ scale and conversion
__device__ __forceinline__ uint32_t mag_hi(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }
// |value| / 2^(e - 1023) from its high word (20 mantissa bits; 0 below 2^-126; for
// values up to 2^128 above 2^(e - 1023))
__device__ __forceinline__ float rel(uint32_t h, int e) {
  const int v = (int)h - ((e - 127) << 20);
  return __int_as_float((v > 0 ? v : 0) << 3);
}
__device__ __forceinline__ float pow2(int e) {  // 2^e, 0 below -126, for e <= 0
  return __int_as_float((e > -127 ? e + 127 : 0) << 23);
}

// Scale of a transform: values are integers in units of 2^-s; k: see to_fixed.
struct Scale {
  int k, s, e;
  bool bad;  // an infinity or a NaN among the inputs
};
// e: largest biased exponent; sum: the transform's bound in units of 2^(e - 1023)
__device__ __forceinline__ Scale scale_of(int e, float sum) {
  Scale c;
  // sum 1.0001 covers the truncated mantissas and the FP32 rounding; es below 0
  // would take a lone value out of to_fixed's range
  const int es = (int)(__float_as_uint(fmaxf(sum * 1.0001f, 1.0f)) >> 23) - 127;
  c.s = 1084 - e - es;   // the sum times 2^s is below 2^62
  c.k = 1075 - c.s;
  c.e = e;
  c.bad = e == 2047;
  return c;
}

// A partial sum over some threads: (largest exponent, sum relative to it).
__device__ __forceinline__ void merge(int &e, float &sum, int e2, float s2) {
  const int m = e > e2 ? e : e2;
  sum = sum * pow2(e - m) + s2 * pow2(e2 - m);
  e = m;
}

// v times the weight m (as normalised by Weight) as an integer in units of 2^-s:
// the 53-bit mantissa times m' in [2^10, 2^11), shifted right.
struct Weight {
  uint32_t m;  // 0: the value is dropped
  int c;
  bool neg;
};
__device__ __forceinline__ Weight weight_one() { return Weight{1u << 10, 10, false}; }
__device__ __forceinline__ Weight weight_int(int f) {  // |f| < 2^11
  const uint32_t a = (uint32_t)(f < 0 ? -f : f);
  const int c = a ? __clz(a) - 21 : 0;
  return Weight{a << c, c, f < 0};
}
__device__ __forceinline__ long long to_fixed(double v, const Scale &sc, const Weight &w) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  // a zero or subnormal has no leading bit and the exponent of a field of 1
  const uint32_t field = (hi >> 20) & 0x7ffu, lead = min(field, 1u);
  const uint32_t mh = (hi & 0xfffffu) + (lead << 20);
  const unsigned long long p = (unsigned long long)lo * w.m;
  const unsigned long long m = p + ((unsigned long long)(mh * w.m) << 32);
  // m >= 2^62 (normal values) and the result is below 2^62: r >= 0, except for a value dropped by
  // its weight (m = 0), whose r may be anything. Rounded to nearest: cutting off
  // would shrink every transform by up to 2^-53.
  const uint32_t r = min((uint32_t)(sc.k + w.c - 2) - field + lead, 63u);
  const unsigned long long f = ((m >> r) + 1) >> 1;
  const long long g = (long long)f;
  return ((int)hi < 0) != w.neg ? -g : g;
}

// An integer in units of 2^-s rounded to FP64.
static __device__ __noinline__ double slow_scale(double v, int s) { return scalbn(v, -s); }
__device__ __forceinline__ double to_double(long long f, const Scale &sc) {
  if (sc.s > 960 || sc.s < -960) return slow_scale((double)f, sc.s);
  return scaled_double(f, sc.s);
}
__device__ __forceinline__ double2 to_double2(const Fx &f, const Scale &sc) {
  double2 d = {to_double(f.x, sc), to_double(f.y, sc)};
  if (sc.bad) d.x = d.y = __hiloint2double(0x7ff80000, 0);
  return d;
}

// The scale of a transform whose inputs are spread over the lanes of a CTA.
// maxf(): this thread's largest exponent; sumf(e): its sum relative to e. The
// lanes of a warp that share the transform are those with equal lane / GROUP
// (STRIDE = 1: GROUP neighbours) or equal lane % STRIDE. slots > 1: partial
// results of several warps (or, without WARP, threads) meet in `parts`
// (slots x width). Every thread of the CTA calls it; it ends with (at least)
// a CTA barrier when BAR is set.
template <bool WARP, int FIRST, int LAST, bool BAR, class MaxF, class SumF>
__device__ __forceinline__ Scale transform_scale(int slot, int slots, int col, int width, bool writer,
                                                 int2 *parts, const MaxF &maxf, const SumF &sumf) {
  int e = maxf();
  if constexpr (WARP) {
#pragma unroll
    for (int o = FIRST; o < LAST; o <<= 1) {
      const int x = __shfl_xor_sync(0xffffffffu, e, o);
      e = e > x ? e : x;
    }
  }
  float sum = sumf(e);
  if constexpr (WARP) {
#pragma unroll
    for (int o = FIRST; o < LAST; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  }
  if (slots > 1) {
    if (writer) parts[slot * width + col] = make_int2(e, __float_as_int(sum));
    __syncthreads();
    int2 q = parts[col];
    e = q.x;
    sum = __int_as_float(q.y);
#pragma unroll 4
    for (int i = 1; i < slots; ++i) {
      q = parts[i * width + col];
      merge(e, sum, q.x, __int_as_float(q.y));
    }
  } else if constexpr (BAR) {
    __syncthreads();
  }
  return scale_of(e, sum);
}

__device__ __forceinline__ int max_exp(int e, double2 v) {
  const uint32_t a = mag_hi(v.x), b = mag_hi(v.y);
  const int x = (int)((a > b ? a : b) >> 20);
  return e > x ? e : x;
}
// the grids that need every bit of the block scale (see the head of the file)
__host__ __device__ constexpr bool fine(int n) { return n > 768; }
// modulus of v / 2^(e - 1023), from above: max + (sqrt(2) - 1) min, within 1.083 of it,
// where a quarter bit counts; else |re| + |im| (two instructions a value less: 1% of
// a run at 64^3 and 512^3)
template <int N> __device__ __forceinline__ float modulus(double2 v, int e) {
  const float a = rel(mag_hi(v.x), e), b = rel(mag_hi(v.y), e);
  return fine(N) ? fmaf(fminf(a, b), 0.41421357f, fmaxf(a, b)) : a + b;
}

}  // namespace fx
}  // namespace gg
