// Cloud-in-cell density of the Zel'dovich particles (one per Lagrangian
// cell, positions q + psi) and the adjoint of that map with respect to psi:
// the differentiable density used by the adjoint form (gradients of a loss on
// the smoothed density with respect to the white noise).
#include "gg_device.cuh"

namespace gg {

// Walk of both kernels: a warp owns 32 neighbouring z of one x plane and steps
// along y, so that no particle costs a division (the 64-bit divisions of a
// linear index had been most of both kernels' instructions), its loads are
// whole lines, and the nodes above one row are those below the next.
template <typename R> struct Cic {
  int i0[3];  // lower node
  int i1[3];  // upper node (periodic)
  R f[3];
};

// Lower node and fractional offset of coordinate u along one axis.
template <typename R> __device__ __forceinline__ void cic_axis_of(R u, int n, int &i0, int &i1, R &f) {
  const R fl = floor(u);
  f = u - fl;
  i0 = (int)fl;
  if ((unsigned)i0 >= (unsigned)n) {  // across the box edge
    i0 %= n;
    if (i0 < 0) i0 += n;
  }
  i1 = i0 + 1 == n ? 0 : i0 + 1;
}
// The particle of cell (x, y, z): psi its displacement, off = q_offset - 1/2.
template <typename R>
__device__ __forceinline__ Cic<R> cic_of(int x, int y, int z, const R psi[3], R off, R inv_cell, int n) {
  Cic<R> c;
  cic_axis_of<R>((R)x + off + psi[0] * inv_cell, n, c.i0[0], c.i1[0], c.f[0]);
  cic_axis_of<R>((R)y + off + psi[1] * inv_cell, n, c.i0[1], c.i1[1], c.f[1]);
  cic_axis_of<R>((R)z + off + psi[2] * inv_cell, n, c.i0[2], c.i1[2], c.f[2]);
  return c;
}
// Address of node (row, z), row = x n + y (below 2^24): two wide multiply-adds.
template <typename R> __device__ __forceinline__ R *node(R *base, int row, int n, int z) {
  return base + (uint64_t)(uint32_t)row * (uint32_t)n + (uint32_t)z;
}

// The rows of one warp: x, rows y0 .. y0 + ny - 1, cells z0 + lane.
struct CicWalk {
  int x, y0, y1, z;
  bool live;
};
// The displacements of the walk's rows, read two rows ahead of their use: one
// row's three loads a warp do not cover the latency of HBM.
template <typename R> struct CicRows {
  const R *psi[3];
  int64_t p;  // the cell of the row two ahead
  int left, n;
  R next[2][3];
  __device__ __forceinline__ void load(R v[3]) {
#pragma unroll
    for (int j = 0; j < 3; ++j) v[j] = left > 0 ? __ldg(psi[j] + p) : (R)0;
    p += n;
    --left;
  }
  __device__ __forceinline__ CicRows(const CicArgs &a, const CicWalk &k) {
#pragma unroll
    for (int j = 0; j < 3; ++j) psi[j] = reinterpret_cast<const R *>(a.psi[j]);
    n = a.n;
    p = ((int64_t)k.x * n + k.y0) * n + k.z;
    left = k.live ? k.y1 - k.y0 : 0;
    load(next[0]);
    load(next[1]);
  }
  __device__ __forceinline__ void take(R d[3]) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      d[j] = next[0][j];
      next[0][j] = next[1][j];
    }
    load(next[1]);
  }
};

__device__ __forceinline__ CicWalk cic_walk(int n, int rows) {
  const int zc = (n + 31) >> 5, yc = (n + rows - 1) / rows;
  const uint32_t w = (uint32_t)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
  const uint32_t t = w / (uint32_t)zc;
  CicWalk k;
  k.z = (int)(w - t * (uint32_t)zc) * 32 + (int)(threadIdx.x & 31);
  k.x = (int)(t / (uint32_t)yc);
  k.y0 = (int)(t - (uint32_t)k.x * (uint32_t)yc) * rows;
  k.y1 = k.y0 + rows < n ? k.y0 + rows : n;
  k.live = k.z < n;
  return k;
}

template <typename R>
__global__ void k_fill(R *x, int64_t count, R value) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x)
    x[i] = value;
}

// Eight nodes a particle. Displacements vary slowly, so most of them meet in
// registers first: a lane's upper-z values join the lower-z values of the
// next lane where that lane's lower node is this one's upper, and the upper-y
// values wait for the next row. Two atomic additions a particle remain on a
// smooth field, all eight where neighbours scatter. Bound by issue (nodes,
// weights, addresses). 512^3: 1407 -> 917 us.
template <typename R>
__global__ void __launch_bounds__(256) k_cic_deposit(const CicArgs a, int rows) {
  const int n = a.n;
  const CicWalk k = cic_walk(n, rows);
  if (k.x >= n) return;  // the whole warp
  const int lane = (int)(threadIdx.x & 31);
  R *delta = reinterpret_cast<R *>(a.delta);
  CicRows<R> rd(a, k);
  const R off = (R)(a.q_offset - 0.5), inv_cell = (R)(1.0 / a.cell);
  R carry0 = (R)0, carry1 = (R)0;  // waiting for the nodes at cp0, cp1
  R *cp0 = nullptr, *cp1 = nullptr;
  for (int y = k.y0; y < k.y1; ++y) {
    R d[3];
    rd.take(d);
    const Cic<R> c = cic_of<R>(k.x, y, k.z, d, off, inv_cell, n);
    // weights by corner: (1 * wx) * wy * wz
    const R x0 = (R)1 - c.f[0], x1 = c.f[0], y0 = (R)1 - c.f[1], y1 = c.f[1];
    const R z0 = k.live ? (R)1 - c.f[2] : (R)0, z1 = k.live ? c.f[2] : (R)0;
    const R w00 = x0 * y0, w01 = x0 * y1, w10 = x1 * y0, w11 = x1 * y1;
    R lo[4] = {w00 * z0, w01 * z0, w10 * z0, w11 * z0};  // (x, y) = 00, 01, 10, 11
    const R hi[4] = {w00 * z1, w01 * z1, w10 * z1, w11 * z1};
    const int r00 = c.i0[0] * n + c.i0[1], r10 = c.i1[0] * n + c.i0[1];
    // along z: take over the upper values of the lane below
    const int br = __shfl_up_sync(0xffffffffu, r00, 1), bz = __shfl_up_sync(0xffffffffu, c.i1[2], 1);
    const bool takes = lane > 0 && k.live && br == r00 && bz == c.i0[2];
    const unsigned taken = __ballot_sync(0xffffffffu, takes) >> 1;  // bit l: lane l + 1 took
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const R up = __shfl_up_sync(0xffffffffu, hi[q], 1);
      lo[q] += takes ? up : (R)0;
    }
    if (!k.live) continue;
    const int r01 = r00 + c.i1[1] - c.i0[1], r11 = r10 + c.i1[1] - c.i0[1];
    if (!((taken >> lane) & 1u)) {
      atomicAdd(node(delta, r00, n, c.i1[2]), hi[0]);
      atomicAdd(node(delta, r01, n, c.i1[2]), hi[1]);
      atomicAdd(node(delta, r10, n, c.i1[2]), hi[2]);
      atomicAdd(node(delta, r11, n, c.i1[2]), hi[3]);
    }
    // along y: the waiting values are this row's lower nodes, or they leave
    R *p0 = node(delta, r00, n, c.i0[2]), *p1 = node(delta, r10, n, c.i0[2]);
    if (cp0 == p0 && cp1 == p1) {
      lo[0] += carry0;
      lo[2] += carry1;
    } else if (cp0) {
      atomicAdd(cp0, carry0);
      atomicAdd(cp1, carry1);
    }
    atomicAdd(p0, lo[0]);
    atomicAdd(p1, lo[2]);
    carry0 = lo[1];
    carry1 = lo[3];
    cp0 = node(delta, r01, n, c.i0[2]);
    cp1 = node(delta, r11, n, c.i0[2]);
  }
  if (cp0) {
    atomicAdd(cp0, carry0);
    atomicAdd(cp1, carry1);
  }
}

// g_psi_j(p) = sum over the 8 nodes c of g(c) d w_c / d psi_j: the gradient of
// the trilinear interpolant, by differences and interpolations along z, y, x.
// The gathers hit the L1 cache (neighbouring lanes, the previous row).
// 512^3: 1490 -> 742 us (the three reads and writes of the fields: 480).
template <typename R>
__global__ void __launch_bounds__(256) k_cic_adjoint(const CicArgs a, int rows) {
  const int n = a.n;
  const CicWalk k = cic_walk(n, rows);
  if (k.x >= n || !k.live) return;
  const R *g = reinterpret_cast<const R *>(a.g_delta);
  CicRows<R> rd(a, k);
  const R off = (R)(a.q_offset - 0.5), inv_cell = (R)(1.0 / a.cell);
  R *out[3] = {reinterpret_cast<R *>(a.g_psi[0]), reinterpret_cast<R *>(a.g_psi[1]),
               reinterpret_cast<R *>(a.g_psi[2])};
  int64_t p = ((int64_t)k.x * n + k.y0) * n + k.z;
  for (int y = k.y0; y < k.y1; ++y, p += n) {
    R d[3];
    rd.take(d);
    const Cic<R> c = cic_of<R>(k.x, y, k.z, d, off, inv_cell, n);
    const int dy = c.i1[1] - c.i0[1], dz = c.i1[2] - c.i0[2];
    const int r0 = c.i0[0] * n + c.i0[1], r1 = c.i1[0] * n + c.i0[1];
    R v[2][2], s[2][2];  // per (x, y) node line: value at the particle's z, z slope
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const R *l = node(g, ((q >> 1) ? r1 : r0) + ((q & 1) ? dy : 0), n, c.i0[2]);
      const R g0 = __ldg(l), g1 = __ldg(l + dz);
      s[q >> 1][q & 1] = g1 - g0;
      v[q >> 1][q & 1] = ((R)1 - c.f[2]) * g0 + c.f[2] * g1;
    }
    const R y0 = (R)1 - c.f[1], y1 = c.f[1], x0 = (R)1 - c.f[0], x1 = c.f[0];
    const R gx = (y0 * v[1][0] + y1 * v[1][1]) - (y0 * v[0][0] + y1 * v[0][1]);
    const R gy = x0 * (v[0][1] - v[0][0]) + x1 * (v[1][1] - v[1][0]);
    const R gz = x0 * (y0 * s[0][0] + y1 * s[0][1]) + x1 * (y0 * s[1][0] + y1 * s[1][1]);
    if (out[0]) out[0][p] = gx * inv_cell;
    if (out[1]) out[1][p] = gy * inv_cell;
    if (out[2]) out[2][p] = gz * inv_cell;
  }
}

static int grid_blocks(int64_t work, int threads) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t b = (work + threads - 1) / threads;
  const int64_t cap = (int64_t)sms * 16;
  return (int)(b < cap ? (b > 0 ? b : 1) : cap);
}

// Rows a warp walks: sixteen, fewer where that would leave the chip short of
// warps (64 an SM), and the CTAs of eight warps that cover the grid.
static int walk_rows(int n) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t lanes = (int64_t)n * ((n + 31) / 32) * n;  // warps at one row each
  int rows = 16;
  while (rows > 1 && lanes / rows < (int64_t)sms * 64) rows /= 2;
  return rows;
}
static unsigned walk_blocks(int n, int rows) {
  const int64_t warps = (int64_t)n * ((n + rows - 1) / rows) * ((n + 31) / 32);
  return (unsigned)((warps + 7) / 8);
}

template <typename R>
cudaError_t launch_cic_deposit(const CicArgs &a, cudaStream_t s) {
  const int64_t cells = (int64_t)a.n * a.n * a.n;
  k_fill<R><<<grid_blocks(cells, 256), 256, 0, s>>>(reinterpret_cast<R *>(a.delta), cells, (R)-1);
  const int rows = walk_rows(a.n);
  k_cic_deposit<R><<<walk_blocks(a.n, rows), 256, 0, s>>>(a, rows);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_cic_adjoint(const CicArgs &a, cudaStream_t s) {
  const int rows = walk_rows(a.n);
  k_cic_adjoint<R><<<walk_blocks(a.n, rows), 256, 0, s>>>(a, rows);
  return cudaGetLastError();
}

template cudaError_t launch_cic_deposit<float>(const CicArgs &, cudaStream_t);
template cudaError_t launch_cic_deposit<double>(const CicArgs &, cudaStream_t);
template cudaError_t launch_cic_adjoint<float>(const CicArgs &, cudaStream_t);
template cudaError_t launch_cic_adjoint<double>(const CicArgs &, cudaStream_t);

}  // namespace gg
