// lbm_pair_f32.cu -- the two-step kernel for FP32 storage.
#include "lbm_pair_kernels.cuh"

namespace tlv {

cudaError_t launch_pair_f32(int law, const void *args, int grid, cudaStream_t st)
{
    return launch_pair<float, PAIR_VEC>(law, args, grid, st);
}

cudaError_t launch_wide_f32(void *f, const Layout &L, cudaStream_t st)
{
    const int n = 24 * (L.ny + 2);
    k_wide<float><<<(n + 127) / 128, 128, 0, st>>>(static_cast<float *>(f), L);
    return cudaGetLastError();
}

int pair_blocks_f32(int law) { return pair_blocks<float, PAIR_VEC>(law); }

} // namespace tlv
