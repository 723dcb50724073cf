// lbm_multi_f16.cu -- the many-steps kernels for f16 storage.
#include "lbm_multi_kernels.cuh"

namespace tlv {

const void *multi_kernel_f16(int law) { return multi_kernel<__half>(law); }

} // namespace tlv
