// F32 size-specialised kernels, strided passes, of the grids 2^a 3^b with at
// least three factors of two from 32 to 1152 that have no tile variants: the
// run-time kernels spend most of their instructions on index arithmetic.
// noise -> pos + vel: 1024^3 44.3 -> 23.2 ms; density 96^3 76 -> 35 us (see
// gg_ct.cuh for the shapes). Other sizes keep the run-time kernels: rows of
// N / 2 not a multiple of 4 make 16-byte TMA rows, and above 1152 a tile of
// 64-byte rows no longer leaves room for two.
#include "gg_ct_kernels.cuh"

namespace gg {

using MoreF32 = CtTable<float, GG_MORE_F32>;
bool spec_more_has_f32(int n) { return MoreF32::has(n); }
int spec_more_cols_f32(int n, int v) { return MoreF32::cols(n, v); }
cudaError_t spec_more_axis_filter_f32(const AxisArgs &a, cudaStream_t s) { return MoreF32::axis_filter(a, s); }
cudaError_t spec_more_axis_f32(const AxisArgs &a, cudaStream_t s) { return MoreF32::axis(a, s); }

}  // namespace gg
