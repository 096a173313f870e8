// Sec. 2.1 diagnostics on sm_103a: shell sums of a half spectrum for the
// power-spectrum estimator, and the moments of a real field.
//
// Shell sums: warps stride over the (x, y) lines of the half spectrum; the
// shell index by exact integer arithmetic: b = floor(|m| + 1/2) is the smallest b
// with 4 m^2 < (2b + 1)^2, from an FP32 estimate (m^2 < 2^24) corrected by one.
// An FP64 square root a mode had bound the kernel (two FP64 lanes an SM): 512^3
// 1375 -> 259 us. Adding the eight lines of an orbit (+-m_x, +-m_y) before
// the shared-memory sums took 63 us, but rounds P(k), which callers get in
// FP64, differently by 4e-9; the order of the additions is kept instead. The
// grid's sums (weight, weight |m|) are formed once per plan and shell count.
//
// Moments: per-CTA FP64 sum (first pass) or sum of squared deviations
// (second pass), minimum and maximum, one slot per CTA, added in a fixed
// order (the result does not depend on scheduling); the mean stays on the
// device between the passes. FP32 fields: adding every value in FP64 is
// bound by the FP64 rate (512^3 1537 us a pass, 20 times the read), so a
// thread adds 32 values exactly, as 64-bit integers in units of 2^-55 of
// their largest binary order, and makes one FP64 addition of them. The second
// pass does the same with the squares of d = v - c for the FP32 value c nearest to
// the mean: d is an integer in units of 2^-58 of the group's largest order, squared
// by its halves (three multiply-adds), and
// sum (v - mean)^2 = sum d^2 - (sum d)^2 / count. (Squares in FP32 with their
// rounding errors added beside them were off by up to 3e-15.) Groups that hold an
// infinity or a NaN add in FP64. 512^3: 132 and 186 us (squares in FP32 163).
#include <cfloat>
#include <cstdint>

#include <cuda_runtime.h>

#include "gg_device.cuh"
#include "gg_internal.h"

namespace gg {
namespace {

// Shell of a mode: floor(|m| + 1/2), m2 < 2^24 (exact in FP32).
__device__ __forceinline__ int shell_of(int m2) {
  int b = (int)(sqrtf((float)m2) + 0.5f);
  if ((2 * b + 1) * (2 * b + 1) <= 4 * m2) ++b;
  if (b > 0 && 4 * m2 < (2 * b - 1) * (2 * b - 1)) --b;
  return b;
}

// Power sums: one warp per (x, y) line of the half spectrum at a time, its own
// copy of the shell sums in shared memory (copies = warps of the CTA, or fewer
// when the bins are many), accumulated in the field's precision per CTA (A) and
// in FP64 across CTAs. A line's values are read before the first addition.
template <typename R, typename A>
__global__ void __launch_bounds__(256) k_shell_power(const ShellArgs a, int copies) {
  extern __shared__ __align__(16) unsigned char raw[];
  A *acc = reinterpret_cast<A *>(raw);  // [copies][nbins]
  const int nb = a.nbins;
  for (int i = threadIdx.x; i < copies * nb; i += blockDim.x) acc[i] = (A)0;
  __syncthreads();
  const Cx<R> *spec = reinterpret_cast<const Cx<R> *>(a.spec);
  const int n = a.n, half = n / 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  A *mine = acc + (size_t)(warp % copies) * nb;
  const int lines = n * n, wstep = (int)gridDim.x * (int)(blockDim.x >> 5);
  for (int line = (int)(blockIdx.x * (blockDim.x >> 5)) + warp; line < lines; line += wstep) {
    const int x = line / n, y = line - x * n;
    if (x == half || y == half) continue;  // |m_j| = N/2 left out (k_z = N/2 is not stored)
    const int mx = x < half ? x : x - n, my = y < half ? y : y - n;
    const int p2 = mx * mx + my * my;
    const Cx<R> *row = spec + (int64_t)line * half;
    constexpr int AHEAD = 8;
    for (int k0 = 0; k0 < half; k0 += 32 * AHEAD) {
      if (shell_of(p2 + k0 * k0) >= nb) break;  // the shells grow along the line
      Cx<R> v[AHEAD];
#pragma unroll
      for (int q = 0; q < AHEAD; ++q) {
        const int kz = k0 + 32 * q + lane;
        if (kz < half) v[q] = row[kz];
      }
#pragma unroll
      for (int q = 0; q < AHEAD; ++q) {
        const int kz = k0 + 32 * q + lane;
        const int b = shell_of(p2 + kz * kz);
        if (kz < half && b < nb) atomicAdd(&mine[b], (A)(kz == 0 ? 1 : 2) * (v[q].x * v[q].x + v[q].y * v[q].y));
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    double t = 0.0;
    for (int c = 0; c < copies; ++c) t += (double)acc[(size_t)c * nb + i];
    if (t != 0.0) atomicAdd(&a.sums[i], t);
  }
}

// The grid's own sums (weight, weight |m|: FP64, once per plan and shell
// count): a warp per orbit (+-u, +-v), (+-v, +-u) of lines, which share every
// |m|. `copies` of the sums per CTA, taken by lane, at an odd stride.
__global__ void __launch_bounds__(256) k_shell_grid(const ShellArgs a, int copies) {
  extern __shared__ __align__(16) unsigned char raw[];
  double *acc = reinterpret_cast<double *>(raw);  // [copies][stride], 2 nbins used
  const int nb = a.nbins, stride = (2 * nb) | 1;
  for (int i = threadIdx.x; i < copies * stride; i += blockDim.x) acc[i] = 0.0;
  __syncthreads();
  const int half = a.n / 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double *mine = acc + (lane & (copies - 1)) * stride;
  const int orbits = half * (half + 1) / 2;  // 0 <= v <= u < N/2 (|m_j| = N/2 left out)
  const int wstep = (int)gridDim.x * (int)(blockDim.x >> 5);
  for (int o = (int)(blockIdx.x * (blockDim.x >> 5)) + warp; o < orbits; o += wstep) {
    int u = (int)((sqrtf(8.0f * (float)o + 1.0f) - 1.0f) * 0.5f);
    while (u * (u + 1) / 2 > o) --u;
    while ((u + 1) * (u + 2) / 2 <= o) ++u;
    const int v = o - u * (u + 1) / 2;
    const int lines = (u ? 2 : 1) * (v ? 2 : 1) * (u != v ? 2 : 1);
    for (int kz = lane; kz < half; kz += 32) {
      const int m2 = u * u + v * v + kz * kz;
      const int b = shell_of(m2);
      if (b >= nb) break;  // the shells grow along the line
      const double w = (double)((kz == 0 ? 1 : 2) * lines);
      atomicAdd(&mine[b], w);
      atomicAdd(&mine[nb + b], w * sqrt((double)m2));
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * nb; i += blockDim.x) {
    double t = 0.0;
    for (int c = 0; c < copies; ++c) t += acc[c * stride + i];
    if (t != 0.0) atomicAdd(&a.sums[i], t);
  }
}

// v (24-bit mantissa times 2^(e - 150)) in units of 2^(E - 182), E the group's
// largest biased exponent (0 counts as 1): exact for e > E - 33, else cut off
// below 2^-55 of the group's largest binary order.
__device__ __forceinline__ long long fixed32(float v, int E) {
  const uint32_t b = __float_as_uint(v);
  const int e = (int)((b >> 23) & 255u);
  const uint32_t m = (b & 0x7fffffu) | (e ? 0x800000u : 0u);
  const int sh = E - (e ? e : 1);
  const long long f = (long long)(((unsigned long long)m << 32) >> (sh < 63 ? sh : 63));
  return (int)b < 0 ? -f : f;
}
// v in units of 2^(E - 184), modulo 2^64: v - c below 2^(E - 126) is then the exact
// difference of two such values, below 2^58, however large v and c are themselves
// (a value that the shift takes out of the word is a multiple of 2^64 units). Bits
// below one unit (v below 2^-34 of that bound) are cut off.
__device__ __forceinline__ long long units58(float v, int E) {
  const uint32_t b = __float_as_uint(v);
  const int field = (int)((b >> 23) & 255u), lead = min(field, 1);
  const int m = (int)((b & 0x7fffffu) + ((uint32_t)lead << 23));
  const int sh = field + 1 - lead - E + 34;
  const long long w = ((int)b < 0 ? -m : m) >> min(max(-sh, 0), 31);
  long long f;  // shl.b64 clamps its shift at 64
  asm("shl.b64 %0, %1, %2;" : "=l"(f) : "l"(w), "r"(max(sh, 0)));
  return f;
}
__device__ __forceinline__ double unfixed(long long f, int E) {  // E >= 1
  return (double)f * __hiloint2double((E - 182 + 1023) << 20, 0);
}
__device__ __forceinline__ int exponent_of(uint32_t bits) {
  const int e = (int)((bits >> 23) & 255u);
  return e ? e : 1;
}

constexpr int kMomentVec = 8;  // float4 a thread and group

// The sum of 32 FP32 values; SECOND: of the squares of d = v - c, and in `lin` of d.
template <bool SECOND>
__device__ __forceinline__ double group_sum(const float4 *v, float c, double &lin) {
  float x[4 * kMomentVec];
#pragma unroll
  for (int i = 0; i < kMomentVec; ++i) {
    x[4 * i] = v[i].x;
    x[4 * i + 1] = v[i].y;
    x[4 * i + 2] = v[i].z;
    x[4 * i + 3] = v[i].w;
  }
  uint32_t top = 0;
  if constexpr (!SECOND) {
#pragma unroll
    for (int i = 0; i < 4 * kMomentVec; ++i) top = max(top, __float_as_uint(x[i]) & 0x7fffffffu);
    if (top < 0x7f800000u) {
      const int E = exponent_of(top);
      long long s = 0;
#pragma unroll
      for (int i = 0; i < 4 * kMomentVec; ++i) s += fixed32(x[i], E);
      return unfixed(s, E);
    }
    double s = 0.0;  // an infinity or a NaN
    for (int i = 0; i < 4 * kMomentVec; ++i) s += (double)x[i];
    return s;
  } else {
#pragma unroll
    for (int i = 0; i < 4 * kMomentVec; ++i)
      top = max(top, __float_as_uint(__fsub_rn(x[i], c)) & 0x7fffffffu);
    if (top < 0x7f800000u) {
      // of the largest |d|, below 1 for subnormals
      const int E = top >= 0x800000u ? (int)(top >> 23) : 9 - __clz((int)top);
      const long long fc = units58(c, E);
      // d = dh 2^32 + dl: the sums of d, dh^2, dh dl and (dl / 8)^2, each below 2^63
      long long l = 0, hh = 0, hl = 0, ll = 0;
#pragma unroll
      for (int i = 0; i < 4 * kMomentVec; ++i) {
        const long long d = units58(x[i], E) - fc;
        const int dl = (int)(uint32_t)d, dh = (int)(d >> 32) + (int)((uint32_t)dl >> 31);
        l += d;
        hh += (long long)dh * dh;
        hl += (long long)dh * dl;
        ll += (long long)(dl >> 3) * (dl >> 3);
      }
      lin += (double)l * __hiloint2double((E - 184 + 1023) << 20, 0);
      const long long t = (hh << 5) + (hl >> 26) + (ll >> 53);  // in units of 2^59
      return (double)t * __hiloint2double((2 * E - 309 + 1023) << 20, 0);
    }
    double s = 0.0;
    for (int i = 0; i < 4 * kMomentVec; ++i) {
      const double d = (double)x[i] - (double)c;
      s += d * d;
      lin += d;
    }
    return s;
  }
}

// {sum of s, minimum of lo, maximum of hi} of the CTA; LIN: lo adds up as s does.
template <bool LIN> __device__ __forceinline__ double join_lo(double a, double b) { return LIN ? a + b : fmin(a, b); }
template <bool LIN = false>
__device__ __forceinline__ void block_slots(double s, double lo, double hi, double *slots) {
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    lo = join_lo<LIN>(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  __shared__ double ws[3][8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    ws[0][warp] = s;
    ws[1][warp] = lo;
    ws[2][warp] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double ts = 0.0, tl = LIN ? 0.0 : DBL_MAX, th = -DBL_MAX;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      ts += ws[0][w];
      tl = join_lo<LIN>(tl, ws[1][w]);
      th = fmax(th, ws[2][w]);
    }
    slots[3 * blockIdx.x] = ts;
    slots[3 * blockIdx.x + 1] = tl;
    slots[3 * blockIdx.x + 2] = th;
  }
}

template <typename R, bool SECOND>
__global__ void __launch_bounds__(256) k_moments(const MomentArgs a) {
  double s = 0.0, lo = SECOND ? 0.0 : DBL_MAX, hi = -DBL_MAX;  // SECOND: lo sums the deviations
  const double mean = SECOND ? a.slots[3 * gridDim.x] : 0.0;  // k_moments_mean's
  if constexpr (sizeof(R) == 4) {
    const float4 *f = reinterpret_cast<const float4 *>(a.field);
    // N even: whole quads; a field off the 16-byte grid takes the FP64 loop below
    const int64_t quads = ((uintptr_t)a.field & 15u) ? 0 : a.count / 4;
    const float c = (float)mean;
    float flo = __int_as_float(0x7f800000), fhi = __int_as_float(0xff800000);
    constexpr int GROUP = 256 * kMomentVec;
    const int64_t whole = quads / GROUP;
    for (int64_t g = blockIdx.x; g < whole; g += gridDim.x) {
      float4 v[kMomentVec];
#pragma unroll
      for (int i = 0; i < kMomentVec; ++i) v[i] = __ldg(f + g * GROUP + i * 256 + threadIdx.x);
      s += group_sum<SECOND>(v, c, lo);
      if constexpr (!SECOND) {
#pragma unroll
        for (int i = 0; i < kMomentVec; ++i) {
          flo = fminf(flo, fminf(fminf(v[i].x, v[i].y), fminf(v[i].z, v[i].w)));
          fhi = fmaxf(fhi, fmaxf(fmaxf(v[i].x, v[i].y), fmaxf(v[i].z, v[i].w)));
        }
      }
    }
    const float *fs = reinterpret_cast<const float *>(a.field);
    for (int64_t i = whole * GROUP * 4 + (int64_t)blockIdx.x * 256 + threadIdx.x; i < a.count;
         i += (int64_t)gridDim.x * 256) {  // the rest, in FP64
      const float v = fs[i];
      const double d = SECOND ? (double)v - (double)c : (double)v;
      s += SECOND ? d * d : d;
      if constexpr (SECOND) lo += d;
      flo = fminf(flo, v);
      fhi = fmaxf(fhi, v);
    }
    if constexpr (!SECOND) {
      lo = fmin(lo, (double)flo);
      hi = fmax(hi, (double)fhi);
    }
  } else {
    const R *f = reinterpret_cast<const R *>(a.field);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.count;
         i += (int64_t)gridDim.x * blockDim.x) {
      const double v = (double)f[i];
      const double d = SECOND ? v - mean : v;
      s += SECOND ? d * d : d;
      if constexpr (!SECOND) {
        lo = fmin(lo, v);
        hi = fmax(hi, v);
      }
    }
  }
  block_slots<SECOND>(s, lo, hi, a.slots + (SECOND ? 3 * gridDim.x + 3 : 0));
}

// The first pass's slots added in a fixed order: {mean, min, max} after them.
__global__ void __launch_bounds__(256) k_moments_mean(double *slots, int blocks, int64_t count) {
  double s = 0.0, lo = DBL_MAX, hi = -DBL_MAX;
  for (int b = threadIdx.x; b < blocks; b += 256) {
    s += slots[3 * b];
    lo = fmin(lo, slots[3 * b + 1]);
    hi = fmax(hi, slots[3 * b + 2]);
  }
  double *out = slots + 3 * blocks;
  block_slots(s, lo, hi, out);
  if (threadIdx.x == 0) out[0] = out[0] / (double)count;
}

int grid_for(int64_t work, int per_sm) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (work + 255) / 256;
  const int64_t cap = (int64_t)(sms > 0 ? sms : 1) * per_sm;
  return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

}  // namespace

template <typename K> cudaError_t shell_launch(K kern, const ShellArgs &a, int copies, size_t per_copy, int blocks,
                                               cudaStream_t s) {
  const size_t smem = per_copy * copies;
  const cudaError_t e = raise_smem(reinterpret_cast<const void *>(kern), smem);
  if (e != cudaSuccess) return e;
  kern<<<blocks, 256, smem, s>>>(a, copies);
  return cudaGetLastError();
}

template <typename R> cudaError_t launch_shell_sums(const ShellArgs &a, bool geometry, cudaStream_t s) {
  if (geometry) {
    const size_t per_copy = (size_t)((2 * a.nbins) | 1) * sizeof(double);
    int copies = 8;
    while (copies > 1 && copies * per_copy > 48 * 1024) copies /= 2;
    const int64_t half = a.n / 2;
    return shell_launch(k_shell_grid, a, copies, per_copy, grid_for(half * (half + 1) / 2 * 32, 4), s);
  }
  const size_t per_copy = (size_t)a.nbins * sizeof(R);
  int copies = (int)((192 * 1024) / per_copy);
  copies = copies > 8 ? 8 : (copies < 1 ? 1 : copies);
  return shell_launch(k_shell_power<R, R>, a, copies, per_copy, grid_for((int64_t)a.n * a.n * 32 / 8, 2), s);
}

template <typename R> int moment_blocks(int64_t count) {
  return sizeof(R) == 4 ? grid_for(count / (4 * kMomentVec), 4) : grid_for(count, 8);
}

template <typename R> cudaError_t launch_moments(const MomentArgs &a, int blocks, cudaStream_t s) {
  k_moments<R, false><<<blocks, 256, 0, s>>>(a);
  k_moments_mean<<<1, 256, 0, s>>>(a.slots, blocks, a.count);
  k_moments<R, true><<<blocks, 256, 0, s>>>(a);
  return cudaGetLastError();
}

template cudaError_t launch_shell_sums<float>(const ShellArgs &, bool, cudaStream_t);
template cudaError_t launch_shell_sums<double>(const ShellArgs &, bool, cudaStream_t);
template int moment_blocks<float>(int64_t);
template int moment_blocks<double>(int64_t);
template cudaError_t launch_moments<float>(const MomentArgs &, int, cudaStream_t);
template cudaError_t launch_moments<double>(const MomentArgs &, int, cudaStream_t);

}  // namespace gg
