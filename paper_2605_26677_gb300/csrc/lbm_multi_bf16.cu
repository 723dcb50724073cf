// lbm_multi_bf16.cu -- the many-steps kernels for bf16 storage.
#include "lbm_multi_kernels.cuh"

namespace tlv {

const void *multi_kernel_bf16(int law) { return multi_kernel<__nv_bfloat16>(law); }

} // namespace tlv
