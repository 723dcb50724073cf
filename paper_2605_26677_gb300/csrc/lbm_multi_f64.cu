// lbm_multi_f64.cu -- the many-steps kernels for f64 storage.
#include "lbm_multi_kernels.cuh"

namespace tlv {

const void *multi_kernel_f64(int law) { return multi_kernel<double>(law); }

} // namespace tlv
