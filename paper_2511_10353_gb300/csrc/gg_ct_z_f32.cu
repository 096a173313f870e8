// F32 size-specialised z-pass and two-input strided kernels of the sizes with
// tile variants.
#include "gg_ct_kernels.cuh"

namespace gg {

using TableF32 = CtTable<float, 64, 128, 192, 256, 384, 512, 1536>;
template <> cudaError_t spec_zinv<float>(const ZInvArgs &a, cudaStream_t s) {
  return TableF32::has(a.n) ? TableF32::zinv(a, s) : spec_more_zinv_f32(a, s);
}
template <> cudaError_t spec_axis_dual<float>(const AxisArgs &a, cudaStream_t s) {
  return TableF32::has(a.n) ? TableF32::dual(a, s) : spec_more_dual_f32(a, s);
}
cudaError_t spec_zfilter_f32(const ZFilterArgs &a, cudaStream_t s) {
  return TableF32::has(a.n) ? TableF32::zfilter(a, s) : spec_more_zfilter_f32(a, s);
}
template <> cudaError_t spec_zfwd<float>(const ZFwdArgs &a, cudaStream_t s) {
  return TableF32::has(a.n) ? TableF32::zfwd(a, s) : spec_more_zfwd_f32(a, s);
}

}  // namespace gg
