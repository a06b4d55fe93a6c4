// fused_bands.cu - the persistent batched kernel for small batches, whose panels
// are cut into row bands so that every CTA has work (band_shape in
// fused_kernel.cu chooses them).
#include "fused_device.cuh"

namespace roibin {

FusedKernel fused_band_kernel(uint32_t kG) { return kG > 1 ? k_fused<kMaxG, 2, true> : k_fused<1, 2, true>; }

}  // namespace roibin
