// F32 size-specialised strided-pass kernels of the sizes with tile variants
// (the z-pass kernels of the same sizes are in gg_ct_z_f32.cu, the sizes with
// one tile shape in gg_ct_more*_f32.cu: translation units that compile in
// parallel).
#include "gg_ct_kernels.cuh"

namespace gg {

using TableF32 = CtTable<float, 64, 128, 192, 256, 384, 512, 1536>;
template <> bool spec_has<float>(int n) { return TableF32::has(n) || spec_more_has_f32(n); }
template <> bool spec_tuned<float>(int n) { return TableF32::has(n); }
template <> bool spec_three_ctas<float>(int n) { return TableF32::three(n); }
template <> cudaError_t spec_axis<float>(const AxisArgs &a, cudaStream_t s) {
  return TableF32::has(a.n) ? TableF32::axis(a, s) : spec_more_axis_f32(a, s);
}
cudaError_t spec_axis_filter_f32(const AxisArgs &a, cudaStream_t s) {
  return TableF32::has(a.n) ? TableF32::axis_filter(a, s) : spec_more_axis_filter_f32(a, s);
}
template <> int spec_axis_cols<float>(int n, int v) {
  return TableF32::has(n) ? TableF32::cols(n, v) : spec_more_cols_f32(n, v);
}

}  // namespace gg
