// F32 size-specialised kernels, z passes and two-input strided passes, of the sizes in gg_ct_more_f32.cu.
#include "gg_ct_kernels.cuh"

namespace gg {

using MoreF32 = CtTable<float, GG_MORE_F32>;
cudaError_t spec_more_zinv_f32(const ZInvArgs &a, cudaStream_t s) { return MoreF32::zinv(a, s); }
cudaError_t spec_more_dual_f32(const AxisArgs &a, cudaStream_t s) { return MoreF32::dual(a, s); }
cudaError_t spec_more_zfilter_f32(const ZFilterArgs &a, cudaStream_t s) { return MoreF32::zfilter(a, s); }
cudaError_t spec_more_zfwd_f32(const ZFwdArgs &a, cudaStream_t s) { return MoreF32::zfwd(a, s); }

}  // namespace gg
