// Size-specialised FP64 passes on fixed-point transforms (see gg_fx.cuh): the
// data flow of gg_ct_kernels.cuh (persistent CTAs, TMA tiles, the spectrum
// handed from the forward to the inverse transforms in registers), FP64 in
// memory and between the transforms, 64-bit integers inside them. One tile
// shape a size: 16-byte values leave no room for a choice.
#pragma once

#include "gg_ct_kernels.cuh"

namespace gg {
namespace fx {

using I = long long;

// Strided tile: rows of up to 128 bytes; two CTAs of 256 threads an SM where
// three tiles of each fit (two being loaded and transformed, one stored).
template <int N> struct AxisShape {
  static constexpr int K = ct::skey<I>(N);
  static constexpr int E = ct::elems(K), P = N / E;
  static constexpr int pick() {
    int b = 8;
    while (b > 4 && ((N / 2) % b != 0 || P * b > 256 || N * b > 2304)) b /= 2;
    return b;
  }
  static constexpr int B = pick(), THREADS = P * B;
  static constexpr int TILE = N * B;
  static constexpr int TILE_BYTES = (TILE * 16 + 127) / 128 * 128;
  static constexpr bool WARP = THREADS % 32 == 0 && 32 % B == 0;
  static constexpr int SLOTS = WARP ? THREADS / 32 : P;
  static constexpr int PARTS_BYTES = (SLOTS * B * 8 + 127) / 128 * 128;
  static constexpr bool TW_SMEM = N * 16 <= 8192;
  static constexpr int FIXED_BYTES = 128 + PARTS_BYTES + (TW_SMEM ? N * 16 : 0);
  static constexpr int REGS = E <= 8 ? 128 : (E <= 12 ? 168 : 255);
  static constexpr int fit(int tiles) { return (228 * 1024) / (FIXED_BYTES + tiles * TILE_BYTES + 1024); }
  static constexpr int by_regs() { return 65536 / (THREADS * REGS) > 0 ? 65536 / (THREADS * REGS) : 1; }
  // a third tile for the outputs where it costs no CTA
  static constexpr bool STG = fit(3) >= 1 && (fit(3) >= by_regs() || fit(3) == fit(2));
  static constexpr int smem_ctas() { return STG ? fit(3) : fit(2); }
  static constexpr int cap() {
    const int m = smem_ctas() < by_regs() ? smem_ctas() : by_regs();
    return m < 1 ? 1 : (m > 12 ? 12 : m);
  }
  static constexpr int MINB = cap();
  static constexpr int SMEM = FIXED_BYTES + (STG ? 3 : 2) * TILE_BYTES;
  static constexpr int rows_box() {
    int rows = 0;
    for (int d = 1; d <= 256 && d <= N; ++d)
      if (N % d == 0 && (d == N || d * B * 16 % 128 == 0)) rows = d;
    return rows;
  }
  static constexpr int ROWS_BOX = rows_box();
  static_assert((N / 2) % B == 0 && SMEM <= 227 * 1024 && ROWS_BOX > 0, "strided tile");
};

template <int N, int MODE>
__global__ void __launch_bounds__(AxisShape<N>::THREADS, AxisShape<N>::MINB)
    k_axis_fx(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap smap0,
              const __grid_constant__ CUtensorMap smap1, const AxisArgs a) {
  pass_begin();
  using Sh = AxisShape<N>;
  constexpr bool FWD = MODE != kAxisInv, INV = MODE != kAxisFwd;
  constexpr int K = Sh::K, E = Sh::E, P = Sh::P, B = Sh::B, HALF = N / 2, S = ct::nstages(K);
  constexpr int INNER = HALF / B, STRIDE = Sh::TILE_BYTES / 16;
  constexpr int RF = ct::radix_of(K, 0, false), SPANF = N / RF, NBF = E / RF;  // first forward stage
  constexpr int RH = ct::radix_of(K, 0, true), SPAN = N / RH, NB = E / RH;     // hand-off
  constexpr int RL = ct::radix_of(K, S - 1, true), SPANL = N / RL, NBL = E / RL;  // last inverse stage
  static_assert(S > 1, "two stages at least");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem_raw);
  int2 *parts = reinterpret_cast<int2 *>(smem_raw + 128);
  int4 *tw_s = reinterpret_cast<int4 *>(smem_raw + 128 + Sh::PARTS_BYTES);
  unsigned char *tiles = smem_raw + Sh::FIXED_BYTES;
  const int tid = threadIdx.x;
  const int64_t per_real = (int64_t)N * INNER;
  const int64_t ntiles = per_real * (a.nbatch > 0 ? a.nbatch : 1);
  const double *table = reinterpret_cast<const double *>(a.table);
  if constexpr (Sh::TW_SMEM) {
    const int4 *src = reinterpret_cast<const int4 *>(a.tw);
    for (int i = tid; i < N; i += Sh::THREADS) tw_s[i] = src[i];
  }
  const ct::Tw<int4, Sh::TW_SMEM> tw{Sh::TW_SMEM ? tw_s : reinterpret_cast<const int4 *>(a.tw)};
  if (tid == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    fence_mbar_init();
  }
  __syncthreads();
  const bool cin = a.chunked_in != 0, chunk_outer = cin && a.axis == 0;
  auto decode = [&](int64_t t, int64_t &rr, int64_t &outer, int &chunk) {
    rr = t / per_real;
    const int64_t tt = t - rr * per_real;
    if (chunk_outer) {
      chunk = (int)(tt / N);
      outer = tt - (int64_t)chunk * N;
    } else {
      outer = tt / INNER;
      chunk = (int)(tt - outer * INNER);
    }
  };
  auto issue = [&](int64_t t, int sb) {
    int64_t rr, outer;
    int chunk;
    decode(t, rr, outer, chunk);
    unsigned char *dst = tiles + sb * Sh::TILE_BYTES;
    if (a.test_skip_copy) return;  // fault test: the wait for this tile runs out
    mbar_arrive_expect_tx(&bars[sb], (uint32_t)(Sh::TILE * 16));
#pragma unroll
    for (int i = 0; i < N; i += Sh::ROWS_BOX) {
      unsigned char *d = dst + i * B * 16;
      if (cin) {
        if (a.axis == 1) tma_load_5d(d, &map, &bars[sb], 0, i, (int)outer, chunk, (int)rr);
        else tma_load_5d(d, &map, &bars[sb], 0, (int)outer, i, chunk, (int)rr);
      } else if (a.axis == 1) {
        tma_load_4d(d, &map, &bars[sb], chunk * B * 2, i, (int)outer, (int)rr);
      } else {
        tma_load_4d(d, &map, &bars[sb], chunk * B * 2, (int)outer, i, (int)rr);
      }
    }
  };
  int64_t t = blockIdx.x;
  if (tid == 0 && t < ntiles) issue(t, 0);
  for (int it = 0; t < ntiles; t += gridDim.x, ++it) {
    const int sb = it & 1;
    const int64_t tn = t + gridDim.x;
    if (tid == 0 && tn < ntiles) {
      if constexpr (!Sh::STG) bulk_wait_read0();  // the previous tile's outputs left from that buffer
      fence_proxy_async_smem();
      issue(tn, sb ^ 1);
    }
    int c = tid & (B - 1), p = tid / B;
    asm volatile("" : "+r"(c), "+r"(p));
    __builtin_assume(c >= 0 && c < B && p >= 0 && p < P);
    int64_t rr, outer;
    int chunk;
    decode(t, rr, outer, chunk);
    const int kz = chunk * B + c;
    Fx *buf = reinterpret_cast<Fx *>(tiles) + sb * STRIDE;
    double2 *bufd = reinterpret_cast<double2 *>(buf);
    double2 *outd = Sh::STG ? reinterpret_cast<double2 *>(tiles) + 2 * STRIDE : bufd;
    const int m_outer = a.axis == 0 ? ct_freq((int)outer, N) : 0;
    const bool nyq_outer = a.axis == 0 && (int)outer == HALF;
    auto tab_index = [&](int n) {
      const int m = ct_freq(n, N);
      return (n == HALF || nyq_outer) ? -1 : m * m + m_outer * m_outer + kz * kz;
    };
    if (FWD && a.pre) {
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int r = 0; r < RH; ++r) {
          const int q = tab_index(p + P * b + r * SPAN);
          if (q >= 0) prefetch_l1(table + q);
        }
    }
    const bool ok = __syncthreads_and(mbar_wait(&bars[sb], (uint32_t)((it >> 1) & 1), a.err, a.wait_us));
    if (!ok) {
      if (tid == 0) {
        if (tn < ntiles && !a.test_skip_copy)
          mbar_wait(&bars[sb ^ 1], (uint32_t)(((it + 1) >> 1) & 1), nullptr, a.wait_us);
        bulk_wait0();  // the output stores, before the CTA exits
      }
      return;
    }
    auto ld = [&](int n) { return buf[n * B + c]; };
    auto st = [&](int n, Fx v) { buf[n * B + c] = v; };
    auto scale = [&](auto maxf, auto sumf) {
      const int warp = tid >> 5, lane = tid & 31;
      return transform_scale<Sh::WARP, B, 32, true>(Sh::WARP ? warp : p, Sh::SLOTS, c, B,
                                                    !Sh::WARP || lane < B, parts, maxf, sumf);
    };
    auto tma_out = [&](int o) {
      const CUtensorMap *sm = o == 0 ? &smap0 : &smap1;
#pragma unroll
      for (int i = 0; i < N; i += Sh::ROWS_BOX) {
        const double2 *s = outd + i * B;
        if (a.chunked_out) {
          if (a.axis == 1) tma_store_5d(sm, s, 0, i, (int)outer, chunk, (int)rr);
          else tma_store_5d(sm, s, 0, (int)outer, i, chunk, (int)rr);
        } else if (a.axis == 1) {
          tma_store_4d(sm, s, chunk * B * 2, i, (int)outer, (int)rr);
        } else {
          tma_store_4d(sm, s, chunk * B * 2, (int)outer, i, (int)rr);
        }
      }
      bulk_commit();
    };
    double2 X[E];  // the spectrum at p + P b + r SPAN
    if constexpr (FWD) {
      Fx v[E];
      Scale sc;
      {
        double2 d[E];
#pragma unroll
        for (int b = 0; b < NBF; ++b)
#pragma unroll
          for (int r = 0; r < RF; ++r) d[b * RF + r] = bufd[(p + P * b + r * SPANF) * B + c];
        sc = scale(
            [&]() {
              int e = 1;
#pragma unroll
              for (int i = 0; i < E; ++i) e = max_exp(e, d[i]);
              return e;
            },
            [&](int e) {
              float s = 0.0f;
#pragma unroll
              for (int i = 0; i < E; ++i) s += modulus<N>(d[i], e);
              return kRootHalf * s;
            });  // its barrier: every thread has read the tile
        const Weight one = weight_one();
#pragma unroll
        for (int i = 0; i < E; ++i) v[i] = Fx{to_fixed(d[i].x, sc, one), to_fixed(d[i].y, sc, one)};
      }
#pragma unroll
      for (int b = 0; b < NBF; ++b) {
        Butterfly<RF, false, Fx>::run(&v[b * RF]);
#pragma unroll
        for (int r = 0; r < RF; ++r) st((p + P * b) * RF + r, v[b * RF + r]);
      }
      __syncthreads();
      ct::stages<I, N, E, false, 1, S - 1>(p, tw, ld, st);
      ct::last_stage_regs<I, N, E, false>(p, tw, ld, v);
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int r = 0; r < RH; ++r) {
          double2 x = to_double2(v[b * RH + r], sc);
          if (a.pre) {
            const int q = tab_index(p + P * b + r * SPAN);
            const double f = (q >= 0 && q >= a.qmin) ? __ldg(table + q) : 0.0;  // qmin: Eq. 4
            x.x *= f;
            x.y *= f;
          }
          X[b * RH + r] = x;
        }
    } else {
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int r = 0; r < RH; ++r) X[b * RH + r] = bufd[(p + P * b + r * SPAN) * B + c];
    }
    if constexpr (!INV) {  // the spectrum out
      if constexpr (Sh::STG) {
        if (tid == 0) bulk_wait_read0();  // the staging tile is free
      }
      __syncthreads();  // ... and the last stage has read the work tile
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int r = 0; r < RH; ++r) outd[(p + P * b + r * SPAN) * B + c] = X[b * RH + r];
      fence_proxy_async_smem();
      __syncthreads();
      if (tid == 0) tma_out(0);
      continue;
    }
    for (int o = 0; o < a.nout; ++o) {
      asm volatile("" : "+r"(c), "+r"(p));
      __builtin_assume(c >= 0 && c < B && p >= 0 && p < P);
      const bool im = a.mul[o] == kMulIm;
      auto freq = [&](int i) {  // i m, 0 at -N/2
        const int n = p + P * (i / RH) + (i % RH) * SPAN;
        return n == HALF ? 0 : ct_freq(n, N);
      };
      // the previous output has left the work tile (in place), or the staging tile
      if (tid == 0) bulk_wait_read0();
      const Scale sc = scale(
          [&]() {
            int e = 1;
#pragma unroll
            for (int i = 0; i < E; ++i) {
              const int x = max_exp(0, X[i]);
              e = e > x || (im && freq(i) == 0) ? e : x;
            }
            return e;
          },
          [&](int e) {
            float s = 0.0f;
#pragma unroll
            for (int i = 0; i < E; ++i) {
              const float x = modulus<N>(X[i], e);
              // i m: without the half bit, so that a lone weighted value stays in to_fixed's range
              s += im ? (freq(i) == 0 ? 0.0f : x * fabsf((float)freq(i))) : kRootHalf * x;
            }
            return s;
          });  // its barrier: every thread has read the work tile
      Fx v[E];
#pragma unroll
      for (int i = 0; i < E; ++i) {
        if (im) {
          Weight w = weight_int(freq(i));
          const I y = to_fixed(X[i].x, sc, w);
          w.neg = !w.neg;
          v[i] = Fx{to_fixed(X[i].y, sc, w), y};
        } else {
          v[i] = Fx{to_fixed(X[i].x, sc, weight_one()), to_fixed(X[i].y, sc, weight_one())};
        }
      }
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        Butterfly<RH, true, Fx>::run(&v[b * RH]);
#pragma unroll
        for (int r = 0; r < RH; ++r) st((p + P * b) * RH + r, v[b * RH + r]);
      }
      __syncthreads();
      ct::stages<I, N, E, true, 1, S - 1>(p, tw, ld, st);
      ct::last_stage_regs<I, N, E, true>(p, tw, ld, v);
      if constexpr (!Sh::STG) __syncthreads();  // every thread has read the work tile
#pragma unroll
      for (int b = 0; b < NBL; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r) outd[(p + P * b + r * SPANL) * B + c] = to_double2(v[b * RL + r], sc);
      fence_proxy_async_smem();
      __syncthreads();
      if (tid == 0) tma_out(o);
    }
  }
  if (tid == 0) bulk_wait0();  // the output stores, before the CTA exits
}

// ------------------------------------------------------------ z passes
// Lines of M = N/2 complex values, P threads each. Padded by one value in 8:
// a quarter-warp then spreads the strided accesses of the stages over the banks.
template <int N> struct ZShape {
  static constexpr int M = N / 2, K = ct::skey<I>(M);
  static constexpr int E = ct::elems(K), P = M / E;
  static constexpr int LD = M + M / 8 + 1;
  static constexpr int pick() {
    int l = 1;
    while (l < 32 && P * l * 2 <= 128) l *= 2;
    return l;
  }
  static constexpr int L = pick(), THREADS = P * L;
  static constexpr bool WARP = P % 32 == 0 || (32 % P == 0 && THREADS % 32 == 0);
  static constexpr int LAST = P >= 32 ? 32 : P;              // lanes of a warp that share a line
  static constexpr int SLOTS = !WARP ? P : (P > 32 ? P / 32 : 1);  // partial results of a line
  static constexpr int PARTS_BYTES = (SLOTS * L * 8 + 127) / 128 * 128;
  static constexpr int DENSE = L * M;
  static constexpr int DENSE_BYTES = (DENSE * 16 + 127) / 128 * 128;
  static constexpr int WORK_BYTES = (L * LD * 16 + 127) / 128 * 128;
  static constexpr int Q_BYTES = N * 8;
  static constexpr int SMEM_COPY = 128 + PARTS_BYTES + DENSE_BYTES + WORK_BYTES;  // with a dense tile
  static constexpr int SMEM_GEN = 128 + PARTS_BYTES + WORK_BYTES;
  static constexpr int REGS = E <= 8 ? 128 : (E <= 12 ? 168 : 255);
  static constexpr int ctas(int smem) {
    const int s = (228 * 1024) / (smem + 1024), r = 65536 / (THREADS * REGS);
    const int m = s < r ? s : r;
    return m < 1 ? 1 : (m > 12 ? 12 : m);
  }
  static_assert((M / 2) % P == 0 && E % 2 == 0, "conjugate pairs");
};
template <int N> __device__ __forceinline__ int zat(int l, int n) {
  return l * ZShape<N>::LD + n + (int)((unsigned)n >> 3);
}
// the scale of line l from a thread's inputs
template <int N, bool BAR, class MaxF, class SumF>
__device__ __forceinline__ Scale line_scale(int tid, int l, int p, int2 *parts, const MaxF &m, const SumF &s) {
  using Sh = ZShape<N>;
  const int slot = Sh::WARP ? (Sh::P > 32 ? p / 32 : 0) : p;
  return transform_scale<Sh::WARP, 1, Sh::LAST, BAR>(slot, Sh::SLOTS, l, Sh::L,
                                                     !Sh::WARP || (p & 31) == 0, parts, m, s);
}

template <int N, bool NOISE>
__global__ void __launch_bounds__(ZShape<N>::THREADS,
                                  ZShape<N>::ctas(NOISE ? ZShape<N>::SMEM_COPY : ZShape<N>::SMEM_GEN))
    k_zfwd_fx(const ZFwdArgs a) {
  pass_begin();
  using Sh = ZShape<N>;
  constexpr int M = Sh::M, K = Sh::K, E = Sh::E, P = Sh::P, L = Sh::L, S = ct::nstages(K);
  constexpr int RF = ct::radix_of(K, 0, false), SPANF = M / RF, NBF = E / RF;
  constexpr bool HALVE = N > 512;  // see the head of gg_fx.cuh
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw);
  int2 *parts = reinterpret_cast<int2 *>(smem_raw + 128);
  Fx *work = reinterpret_cast<Fx *>(smem_raw + 128 + Sh::PARTS_BYTES);
  double2 *workd = reinterpret_cast<double2 *>(work);
  double2 *dense = reinterpret_cast<double2 *>(smem_raw + 128 + Sh::PARTS_BYTES + Sh::WORK_BYTES);  // NOISE
  const int tid = threadIdx.x;
  const int64_t ntiles = a.nlines / L;
  const ct::Tw<int4, false> tw{reinterpret_cast<const int4 *>(a.tw_half)};
  const int4 *twf = reinterpret_cast<const int4 *>(a.tw_full);
  auto issue = [&](int64_t t) {
    mbar_arrive_expect_tx(bar, (uint32_t)(Sh::DENSE * 16));
    bulk_load(dense, reinterpret_cast<const double2 *>(a.noise) + t * Sh::DENSE, (uint32_t)(Sh::DENSE * 16), bar);
  };
  if constexpr (NOISE) {
    if (tid == 0) {
      mbar_init(bar, 1);
      fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0 && blockIdx.x < ntiles) issue(blockIdx.x);
  }
  uint32_t phase = 0;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    int l = tid / P, p = tid - (tid / P) * P;
    asm volatile("" : "+r"(l), "+r"(p));
    __builtin_assume(l >= 0 && l < L && p >= 0 && p < P);
    const int64_t line = t * L + l;
    if constexpr (NOISE) {
      const bool ok = __syncthreads_and(mbar_wait(bar, phase, a.err));
      if (!ok) return;  // nothing else in flight
      phase ^= 1;
    } else {
      const uint32_t lpr = (uint32_t)(a.lines_per_real > 0 ? a.lines_per_real : a.nlines);
      const uint32_t rr = (uint32_t)line / lpr, local = (uint32_t)line - rr * lpr;
      const uint64_t seed = a.seeds ? a.seeds[rr] : a.seed;
      const uint64_t g0 = (uint64_t)local * (uint64_t)(N / 4);
      static_assert(N % 4 == 0 && P * (E / 2) == M / 2, "lines start on a Philox group");
#pragma unroll 1
      for (int i = 0; i < E / 2; ++i) {
        const int q = p + P * i;
        double w[4];
        gauss4(noise_words(seed, g0 + q), w);
        workd[zat<N>(l, 2 * q)] = double2{w[0], w[1]};
        workd[zat<N>(l, 2 * q + 1)] = double2{w[2], w[3]};
      }
      __syncthreads();
    }
    auto ld = [&](int n) { return work[zat<N>(l, n)]; };
    auto st = [&](int n, Fx v) { work[zat<N>(l, n)] = v; };
    Fx v[E];
    Scale sc;
    {
      double2 d[E];
#pragma unroll
      for (int b = 0; b < NBF; ++b)
#pragma unroll
        for (int r = 0; r < RF; ++r) {
          const int n = p + P * b + r * SPANF;
          d[b * RF + r] = NOISE ? dense[l * M + n] : workd[zat<N>(l, n)];
        }
      sc = line_scale<N, true>(
          tid, l, p, parts,
          [&]() {
            int e = 1;
#pragma unroll
            for (int i = 0; i < E; ++i) e = max_exp(e, d[i]);
            return e;
          },
          [&](int e) {
            float s = 0.0f;
#pragma unroll
            for (int i = 0; i < E; ++i) s += modulus<N>(d[i], e);
            return HALVE ? s : 2.0f * s;
          });  // its barrier: every thread has read its values
      if constexpr (NOISE) {
        if (tid == 0 && t + gridDim.x < ntiles) {
          fence_proxy_async_smem();
          issue(t + gridDim.x);
        }
      }
      const Weight one = weight_one();
#pragma unroll
      for (int i = 0; i < E; ++i) v[i] = Fx{to_fixed(d[i].x, sc, one), to_fixed(d[i].y, sc, one)};
    }
#pragma unroll
    for (int b = 0; b < NBF; ++b) {
      Butterfly<RF, false, Fx>::run(&v[b * RF]);
#pragma unroll
      for (int r = 0; r < RF; ++r) st((p + P * b) * RF + r, v[b * RF + r]);
    }
    __syncthreads();
    ct::stages<I, M, E, false, 1, S>(p, tw, ld, st);
    // the real-input spectrum by conjugate pairs: X_k = S/2 - i (D/2) w_k, X_{M-k} =
    // conj(S/2 + i (D/2) w_k), S and D twice their bound
    double2 *dst = reinterpret_cast<double2 *>(a.out) + line * M;
    auto part = [](I q) { return HALVE ? half_even(q) : q; };
    Scale so = sc;
    if constexpr (!HALVE) ++so.s;
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
      const int k = p + P * i;
      const Fx zk = ld(k);
      if (k == 0) {
        const Fx zh = ld(M / 2);
        dst[0] = to_double2(Fx{zk.x + zk.y, 0}, sc);
        dst[M / 2] = to_double2(Fx{zh.x, -zh.y}, sc);
      } else {
        const Fx zm = ld(M - k);
        const Fx s = {part(zk.x + zm.x), part(zk.y - zm.y)};
        const Fx d = cmul(Fx{part(zk.x - zm.x), part(zk.y + zm.y)}, __ldg(twf + k));
        dst[k] = to_double2(Fx{s.x + d.y, s.y - d.x}, so);
        dst[M - k] = to_double2(Fx{s.x - d.y, -(s.y + d.x)}, so);
      }
    }
    __syncthreads();  // the work tile is rewritten next tile
  }
}

// The inverse z pass and the Eq. 3 epilogue (see zinv_body). A pair of the c2r
// pre-processing, Z_k = S + T and Z_{M-k} = conj(S - T), has |Z_k|^2 + |Z_{M-k}|^2 =
// 4 (|X_k|^2 + |X_{M-k}|^2): the line's sum of moduli grows by at most 2 sqrt(2),
// and each value fits far below it. Lines above 384 (N > 768) form the pairs in a
// finer unit (2^-6 of the transform's where the line leaves room, as a flat spectrum
// does) and round them once, so that the transform's inputs carry one rounding at its
// unit instead of those of four inputs, which alone came to 5e-16 at N = 1536. At N =
// 512 (2.9e-16 for six transforms without it) it would cost 1.5% of the run.
__host__ __device__ constexpr int im_bits(int m) {  // frequencies below m are below 2^im_bits
  int b = 0;
  while ((1 << b) < m) ++b;
  return b;
}
template <int N, bool EXT>
__global__ void __launch_bounds__(ZShape<N>::THREADS, ZShape<N>::ctas(ZShape<N>::SMEM_COPY + ZShape<N>::Q_BYTES))
    k_zinv_fx(const ZInvArgs a) {
  pass_begin();
  using Sh = ZShape<N>;
  using R = double;
  constexpr int M = Sh::M, K = Sh::K, E = Sh::E, P = Sh::P, L = Sh::L, S = ct::nstages(K);
  constexpr int RL = ct::radix_of(K, S - 1, true), SPANL = M / RL, NBL = E / RL;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw);
  int2 *parts = reinterpret_cast<int2 *>(smem_raw + 128);
  Fx *work = reinterpret_cast<Fx *>(smem_raw + 128 + Sh::PARTS_BYTES);
  double2 *dense = reinterpret_cast<double2 *>(smem_raw + 128 + Sh::PARTS_BYTES + Sh::WORK_BYTES);
  double *q_s = reinterpret_cast<double *>(smem_raw + Sh::SMEM_COPY);  // lattice coordinates
  const int tid = threadIdx.x;
  const int64_t ntiles = a.nlines / L;
  const ct::Tw<int4, false> tw{reinterpret_cast<const int4 *>(a.tw_half)};
  const int4 *twf = reinterpret_cast<const int4 *>(a.tw_full);
  const R box = a.box, cell = a.cell, qo = a.q_offset, vfac = a.vfac;
  for (int i = tid; i < N; i += Sh::THREADS) q_s[i] = mul_rn((R)i + qo, cell);
  if (tid == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  auto issue = [&](int64_t t) {
    mbar_arrive_expect_tx(bar, (uint32_t)(Sh::DENSE * 16));
    bulk_load(dense, reinterpret_cast<const double2 *>(a.src) + t * Sh::DENSE, (uint32_t)(Sh::DENSE * 16), bar);
  };
  int64_t t = blockIdx.x;
  if (tid == 0 && t < ntiles) issue(t);
  uint32_t phase = 0;
  for (; t < ntiles; t += gridDim.x, phase ^= 1) {
    int l = tid / P, p = tid - (tid / P) * P;
    asm volatile("" : "+r"(l), "+r"(p));
    __builtin_assume(l >= 0 && l < L && p >= 0 && p < P);
    const bool ok = __syncthreads_and(mbar_wait(bar, phase, a.err));
    if (!ok) return;  // nothing else in flight
    auto ld = [&](int n) { return work[zat<N>(l, n)]; };
    auto st = [&](int n, Fx v) { work[zat<N>(l, n)] = v; };
    const bool im = a.mul_kz != 0;
    Scale sc;
    {
      double2 xk[E / 2], xm[E / 2];  // the pairs (k, M - k), k = p + P i; k = 0: (0, M/2)
#pragma unroll
      for (int i = 0; i < E / 2; ++i) {
        const int k = p + P * i;
        xk[i] = dense[l * M + k];
        xm[i] = dense[l * M + (k ? M - k : M / 2)];
      }
      sc = line_scale<N, true>(
          tid, l, p, parts,
          [&]() {
            int e = 1;
#pragma unroll
            for (int i = 0; i < E / 2; ++i) {
              const int x = max_exp(0, xk[i]);
              e = e > x || (im && p + P * i == 0) ? e : x;
              e = max_exp(e, xm[i]);
            }
            return e;
          },
          [&](int e) {
            float s = 0.0f;
#pragma unroll
            for (int i = 0; i < E / 2; ++i) {
              const int k = p + P * i;
              const float x = modulus<N>(xk[i], e), y = modulus<N>(xm[i], e);
              s += im ? (k ? x * (float)k : 0.0f) + y * (float)(k ? M - k : M / 2) : x + y;
            }
            return 2.0f * s;  // sum of |Z| below 2^62.5
          });  // its barrier: the dense tile has been read
      if (tid == 0 && t + gridDim.x < ntiles) {
        fence_proxy_async_smem();
        issue(t + gridDim.x);
      }
      Scale su = sc;
      int g = 0;
      if constexpr (fine(N)) {  // weighted inputs stay below 2^60 in the finer unit
        const int room = 1082 - sc.s - sc.e - (im ? im_bits(M) : 0);
        g = room < 6 ? 0 : 6;
        su.k -= g;
      }
      const I low = ((1ll << g) - 1) >> 1, tie = g ? 1 : 0;
      auto round = [&](I q) { return (q + low + ((q >> g) & tie)) >> g; };  // halves to even
      auto put = [&](int n, Fx v) { st(n, Fx{round(v.x), round(v.y)}); };
#pragma unroll
      for (int i = 0; i < E / 2; ++i) {
        const int k = p + P * i, km = k ? M - k : M / 2;
        Fx u, w;
        if (im) {  // i m_z on both members
          Weight wk = weight_int(k), wm = weight_int(km);
          u.y = to_fixed(xk[i].x, su, wk);
          w.y = to_fixed(xm[i].x, su, wm);
          wk.neg = wm.neg = true;
          u.x = to_fixed(xk[i].y, su, wk);
          w.x = to_fixed(xm[i].y, su, wm);
        } else {
          const Weight one = weight_one();
          u = Fx{to_fixed(xk[i].x, su, one), to_fixed(xk[i].y, su, one)};
          w = Fx{to_fixed(xm[i].x, su, one), to_fixed(xm[i].y, su, one)};
        }
        if (k == 0) {  // X_{N/2} = 0; the self-paired X_{M/2}: Z = 2 conj X
          // S = X_0, D = X_0, Z = X_0 + i X_0
          put(0, Fx{u.x - u.y, u.x + u.y});
          put(M / 2, Fx{2 * w.x, -2 * w.y});
        } else {
          const Fx s = {u.x + w.x, u.y - w.y}, d = {u.x - w.x, u.y + w.y};
          const Fx q = mul_pi(cmulc(d, __ldg(twf + k)));  // Z_k = S + i D conj w
          put(k, Fx{s.x + q.x, s.y + q.y});
          put(M - k, Fx{s.x - q.x, q.y - s.y});  // conj(S - i D conj w)
        }
      }
    }
    __syncthreads();
    ct::stages<I, M, E, true, 0, S - 1>(p, tw, ld, st);
    Fx v[E];
    ct::last_stage_regs<I, M, E, true>(p, tw, ld, v);
    double2 z[E];
#pragma unroll
    for (int i = 0; i < E; ++i) z[i] = to_double2(v[i], sc);
    const uint32_t line = (uint32_t)(t * L + l);
    const uint32_t lpr = (uint32_t)(a.lines_per_real > 0 ? a.lines_per_real : a.nlines);
    const uint32_t rr = line / lpr, local = line - rr * lpr;
    const uint32_t ix = local / (uint32_t)a.n, iy = local - ix * (uint32_t)a.n;
    const int comp = a.comp;
    const R qline = q_s[comp == 0 ? ix : iy];
    void *psi_b = a.psi_list ? a.psi_list[rr] : a.psi;
    void *pos_b = a.pos_list ? a.pos_list[rr] : a.pos;
    void *vel_b = a.vel_list ? a.vel_list[rr] : a.vel;
    const int64_t off = (int64_t)(a.psi_list || a.pos_list || a.vel_list ? local : line) * M;
    double2 *psi = psi_b ? reinterpret_cast<double2 *>(psi_b) + off : nullptr;
    double2 *pos = pos_b ? reinterpret_cast<double2 *>(pos_b) + off : nullptr;
    double2 *vel = vel_b ? reinterpret_cast<double2 *>(vel_b) + off : nullptr;
    auto each = [&](auto f) {
#pragma unroll
      for (int b = 0; b < NBL; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r) f(p + P * b + r * SPANL, z[b * RL + r]);
    };
    if constexpr (EXT) {  // Sec. 2.4: the interpolated coarse large scales
      const R *large = reinterpret_cast<const R *>(a.large);
      if (large) {
        const CicAxis<R> cx = cic_axis<R>((int)ix, a.n_low, N), cy = cic_axis<R>((int)iy, a.n_low, N);
        each([&](int n, double2 &q) {
          R l0, l1;
          cic_pair<R>(large, a.n_low, N, cx, cy, n, l0, l1);
          q.x += l0;
          q.y += l1;
        });
      }
    }
    if (psi) {
      if (a.accumulate) {
        each([&](int n, double2 q) {
          const double2 o = psi[n];
          psi[n] = double2{o.x + a.alpha * q.x, o.y + a.alpha * q.y};
        });
      } else {
        each([&](int n, double2 q) { psi[n] = q; });
      }
    }
    if (pos) {
      const R sh1 = EXT ? a.shift : 0.0;
      each([&](int n, double2 q) {
        const R q0 = comp == 2 ? q_s[2 * n] : qline, q1 = comp == 2 ? q_s[2 * n + 1] : qline;
        if constexpr (EXT) {  // Sec. 2.2: periodic shift
          pos[n] = double2{wrap_box<R>(q0 + sh1 + q.x, box), wrap_box<R>(q1 + sh1 + q.y, box)};
        } else {
          pos[n] = double2{wrap_box<R>(q0 + q.x, box), wrap_box<R>(q1 + q.y, box)};
        }
      });
      if constexpr (EXT) {  // gas partners
        if (a.pos2) {
          double2 *pos2 = reinterpret_cast<double2 *>(a.pos2) + off;
          const R sh2 = a.shift2;
          each([&](int n, double2 q) {
            const R q0 = comp == 2 ? q_s[2 * n] : qline, q1 = comp == 2 ? q_s[2 * n + 1] : qline;
            pos2[n] = double2{wrap_box<R>(q0 + sh2 + q.x, box), wrap_box<R>(q1 + sh2 + q.y, box)};
          });
        }
      }
    }
    if (vel) each([&](int n, double2 q) { vel[n] = double2{vfac * q.x, vfac * q.y}; });
    __syncthreads();  // the work tile is rewritten next tile
  }
}

// ------------------------------------------------------------ launchers
template <int N, int MODE> cudaError_t launch_axis(const AxisArgs &in, cudaStream_t s) {
  using Sh = AxisShape<N>;
  AxisArgs a = in;
  if ((a.chunked_in || a.chunked_out) && a.cols != Sh::B) return cudaErrorInvalidValue;
  if (a.nout > 2) return cudaErrorInvalidValue;
  a.cols = Sh::B;
  a.inner_chunks = (N / 2) / Sh::B;
  a.rows_box = Sh::ROWS_BOX;
  CUtensorMap map;
  cudaError_t e = make_map<double>(&map, a);
  if (e != cudaSuccess) return e;
  CUtensorMap smap[2] = {map, map};
  for (int o = 0; o < a.nout; ++o) {
    AxisArgs b = a;
    b.src = a.dst[o];
    b.chunked_in = a.chunked_out;
    if ((e = make_map<double>(&smap[o], b)) != cudaSuccess) return e;
  }
  auto kern = k_axis_fx<N, MODE>;
  if ((e = set_smem(kern, Sh::SMEM)) != cudaSuccess) return e;
  const int64_t tiles = (int64_t)N * a.inner_chunks * (a.nbatch > 0 ? a.nbatch : 1);
  return launch_pass(kern, tiles, Sh::THREADS, Sh::SMEM, s, a.overlap, map, smap[0], smap[1], a);
}
template <int N, bool NOISE> cudaError_t launch_zfwd(const ZFwdArgs &a, cudaStream_t s) {
  using Sh = ZShape<N>;
  const int smem = NOISE ? Sh::SMEM_COPY : Sh::SMEM_GEN;
  auto kern = k_zfwd_fx<N, NOISE>;
  cudaError_t e = set_smem(kern, smem);
  if (e != cudaSuccess) return e;
  return launch_pass(kern, a.nlines / Sh::L, Sh::THREADS, smem, s, a.overlap, a);
}
template <int N, bool EXT> cudaError_t launch_zinv(const ZInvArgs &a, cudaStream_t s) {
  using Sh = ZShape<N>;
  const int smem = Sh::SMEM_COPY + Sh::Q_BYTES;
  auto kern = k_zinv_fx<N, EXT>;
  cudaError_t e = set_smem(kern, smem);
  if (e != cudaSuccess) return e;
  return launch_pass(kern, a.nlines / Sh::L, Sh::THREADS, smem, s, a.overlap, a);
}

template <int... NS> struct Table {
  static bool has(int n) { return ((n == NS) || ...); }
  static int cols(int n) {
    int c = 0;
    ((n == NS ? (c = AxisShape<NS>::B, 0) : 0), ...);
    return c;
  }
  template <int N> static cudaError_t axis_n(const AxisArgs &a, cudaStream_t s) {
    if (a.fwd && a.inv) return launch_axis<N, kAxisFwdInv>(a, s);
    if (a.fwd) return launch_axis<N, kAxisFwd>(a, s);
    return a.inv ? launch_axis<N, kAxisInv>(a, s) : cudaErrorInvalidValue;
  }
  template <int N> static cudaError_t zfwd_n(const ZFwdArgs &a, cudaStream_t s) {
    return a.noise ? launch_zfwd<N, true>(a, s) : launch_zfwd<N, false>(a, s);
  }
  template <int N> static cudaError_t zinv_n(const ZInvArgs &a, cudaStream_t s) {
    const bool ext = a.large || a.pos2 || a.shift != 0.0 || a.shift2 != 0.0;
    return ext ? launch_zinv<N, true>(a, s) : launch_zinv<N, false>(a, s);
  }
  static cudaError_t axis(const AxisArgs &a, cudaStream_t s) {
    cudaError_t e = cudaErrorInvalidValue;
    ((a.n == NS ? (e = axis_n<NS>(a, s), 0) : 0), ...);
    return e;
  }
  static cudaError_t zfwd(const ZFwdArgs &a, cudaStream_t s) {
    cudaError_t e = cudaErrorInvalidValue;
    ((a.n == NS ? (e = zfwd_n<NS>(a, s), 0) : 0), ...);
    return e;
  }
  static cudaError_t zinv(const ZInvArgs &a, cudaStream_t s) {
    cudaError_t e = cudaErrorInvalidValue;
    ((a.n == NS ? (e = zinv_n<NS>(a, s), 0) : 0), ...);
    return e;
  }
};

}  // namespace fx
}  // namespace gg
