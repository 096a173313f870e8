// FP64 size-specialised strided passes (fixed-point transforms, gg_fx_kernels.cuh):
// the grids 2^a 3^b with three or more factors of two up to 384, and 512, 768,
// 1024, 1536.
#include "gg_fx_kernels.cuh"

namespace gg {

using TableF64 = fx::Table<GG_FX_SIZES>;
template <> bool spec_has<double>(int n) { return TableF64::has(n); }
template <> bool spec_tuned<double>(int) { return false; }
template <> cudaError_t spec_axis<double>(const AxisArgs &a, cudaStream_t s) { return TableF64::axis(a, s); }
template <> int spec_axis_cols<double>(int n, int) { return TableF64::cols(n); }

}  // namespace gg
