// Fused FP32 kernel for the stencil G1..G6.
#include "rlbm_fused.cuh"
#include "rlbm_persist.cuh"
#include "rlbm_fused_launch.h"

namespace rlbm {
template <>
cudaError_t launch_fused<StencilG16>(const FusedParams& p, const void* fin, void* fout, int mode, cudaStream_t s) {
  return launch_fused_impl<StencilG16>(p, fin, fout, mode, s);
}
template <>
cudaError_t launch_f32_io<StencilG16>(bool init, const FusedParams& fp, const StepParams<double>& p, FieldPtrs fd,
                                    void* cur, void* other, MomentOut mo, cudaStream_t s) {
  return launch_f32_io_impl<StencilG16>(init, fp, p, fd, cur, other, mo, s);
}
template <>
const void* fused_kernel_fn<StencilG16>(int mode) {
  return fused_kernel_fn_impl<StencilG16>(mode);
}
template <>
const void* persist_kernel_fn<StencilG16>(int mode) {
  return persist_kernel_fn_impl<StencilG16>(mode);
}
}  // namespace rlbm
