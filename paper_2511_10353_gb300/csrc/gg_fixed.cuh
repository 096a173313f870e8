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

// The low x low products are left out: each a unit at most, a third of one rms and
// without a bias.
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
// a / 2, halves to even. Cut off, a quarter of a unit would be lost on average, the
// same everywhere; the transforms along the other axes gather such a constant in
// single modes and cells (1536^3, forward and back: one cell off by 2000 times the
// rms error).
__device__ __forceinline__ long long half_even(long long a) {
  const long long h = a >> 1;
  return h + (long long)((uint32_t)a & (uint32_t)h & 1u);
}
// An integer, times 2^-s, rounded to FP64 without the FP64 pipe: normalised,
// rounded to nearest even and put together by integers (26 instructions; two exact
// halves and two FP64 additions, 32 cycles of that pipe, took 13.9 instead of
// 12.3 ms in the 512^3 FP64 run). |s| <= 960.
__device__ __forceinline__ double scaled_double(long long f, int s) {
  const long long sign = f >> 63;
  const unsigned long long u = (unsigned long long)((f ^ sign) - sign);
  const int z = __clzll((long long)u);
  const unsigned long long n = u << (z & 63);  // bit 63 set
  const uint32_t rest = ((uint32_t)n & 0x7ffu) + (((uint32_t)n >> 11) & 1u);  // ties to even
  const unsigned long long m = (n >> 11) + (rest > 0x400u ? 1ull : 0ull);   // a carry goes on into the exponent
  const uint32_t hi = (uint32_t)(m >> 32) + ((uint32_t)(1085 - z - s) << 20);
  return __hiloint2double(u ? (int)(hi | ((uint32_t)(sign >> 32) & 0x80000000u)) : 0, (int)(uint32_t)m);
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
