// FP64 size-specialised z passes (fixed-point transforms) of the sizes in
// gg_fx_axis.cu.
#include "gg_fx_kernels.cuh"

namespace gg {

using TableF64 = fx::Table<GG_FX_SIZES>;
template <> cudaError_t spec_zinv<double>(const ZInvArgs &a, cudaStream_t s) { return TableF64::zinv(a, s); }
template <> cudaError_t spec_zfwd<double>(const ZFwdArgs &a, cudaStream_t s) { return TableF64::zfwd(a, s); }

}  // namespace gg
