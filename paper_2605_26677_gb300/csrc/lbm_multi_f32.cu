// lbm_multi_f32.cu -- the many-steps kernels for f32 storage.
#include "lbm_multi_kernels.cuh"

namespace tlv {

const void *multi_kernel_f32(int law) { return multi_kernel<float>(law); }

} // namespace tlv
