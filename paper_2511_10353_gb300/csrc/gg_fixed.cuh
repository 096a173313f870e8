// 64-bit fixed-point complex products: values in units of 2^-s, factors of
// modulus up to one in units of 2^-62, split into 32-bit halves.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gg {

struct Fx {
  long long x, y;
};

// Twiddle w: round(w 2^62) = h 2^32 + l per component, l signed: (re h, re l, im h, im l).
using TwFx = int4;

namespace fx {

__device__ __forceinline__ int lo_of(long long a) { return (int)(uint32_t)a; }  // signed low half
__device__ __forceinline__ int hi_of(long long a) {                             // a = hi 2^32 + lo
  return (int)(a >> 32) + (int)((uint32_t)lo_of(a) >> 31);
}
__device__ __forceinline__ long long wide(int a, int b, long long c) { return (long long)a * b + c; }
// (H 2^64 + C 2^32) / 2^62, C carrying its rounding constant: |H| < 2^60, |C| < 2^63
__device__ __forceinline__ long long join(long long h, long long c) { return (h << 2) + (c >> 30); }
constexpr long long kRound = 1ll << 29;

// The low x low products (below half a unit) are left out.
__device__ __forceinline__ Fx mul(Fx a, int rh, int rl, int ih, int il) {
  const int xl = lo_of(a.x), xh = hi_of(a.x), yl = lo_of(a.y), yh = hi_of(a.y);
  Fx o;
  o.x = join(wide(yh, -ih, (long long)xh * rh),
             wide(yl, -ih, wide(yh, -il, wide(xl, rh, wide(xh, rl, kRound)))));
  o.y = join(wide(yh, rh, (long long)xh * ih),
             wide(yl, rh, wide(yh, rl, wide(xl, ih, wide(xh, il, kRound)))));
  return o;
}
__device__ __forceinline__ long long mul_real(long long a, int h, int l) {
  const int al = lo_of(a), ah = hi_of(a);
  return join((long long)ah * h, wide(al, h, wide(ah, l, kRound)));
}
// An integer rounded to FP64: its halves exactly in the mantissas of 2^84 and
// 2^52 and two additions.
__device__ __forceinline__ double rounded_double(long long f) {
  const double a = __hiloint2double(0x45300000, (int)((uint32_t)(f >> 32) ^ 0x80000000u));
  const double b = __hiloint2double(0x43300000, (int)(uint32_t)f);
  return (a - (0x1p84 + 0x1p63 + 0x1p52)) + b;
}
// halves of a constant of modulus below one in 2^62 units
__host__ __device__ constexpr long long units(double c) {
  return (long long)(c * 4611686018427387904.0);  // exact: a power of two times a double
}
__host__ __device__ constexpr int low_half(long long w) {
  return (int)((w & 0xffffffffll) >= 0x80000000ll ? (w & 0xffffffffll) - 0x100000000ll : (w & 0xffffffffll));
}
__host__ __device__ constexpr int high_half(long long w) { return (int)((w - low_half(w)) / 4294967296ll); }

}  // namespace fx
}  // namespace gg
