// lbm_multi_plan.h -- how the many-steps kernel (k_multi) shares out a
// lattice: its blocks, and which nodes a task takes. Plain C++: the library,
// the kernel and a test on the CPU compile the same functions.
#pragma once
#include <algorithm>

#ifdef __CUDACC__
#define TLV_HD __host__ __device__ __forceinline__
#else
#define TLV_HD inline
#endif

namespace tlv {

constexpr int MULTI_WARPS = 8;  // warps per block at most (4: more blocks meet at the barrier,
                                // 512^2 FP32 8.7 against 8.0 us a step; 16: 7.7, but FP64 512^2 138
                                // against 113)

struct MultiGrid {
    int warps, blocks;  // warps per block
};

// `tasks` over the SMs, at most per_sm blocks of MULTI_WARPS warps on each: as
// few rounds as these allow, and the blocks small enough that the SMs get
// equally many (FP64 39 x 798, traction sides, 1596 tasks: 200 blocks of eight
// warps took 74 us a step, 266 of six 40).
inline MultiGrid multi_grid(long long tasks, int sms, int per_sm)
{
    const long long k = std::min<long long>(per_sm, std::max<long long>(1, (tasks + MULTI_WARPS * sms - 1) / (MULTI_WARPS * sms)));
    MultiGrid g;
    g.warps = (int)std::min<long long>(MULTI_WARPS, std::max<long long>(1, (tasks + k * sms - 1) / (k * sms)));
    g.blocks = (int)std::min<long long>((tasks + g.warps - 1) / g.warps, k * sms);
    return g;
}

// Row and 32-node segment of a task: the bottom and top rows first and the
// segments rotated by the row (as task_coords), and with `twist` once more every
// nseg rows. Where the warps are a multiple of nseg^2 (multi_twist), the rows'
// rotation alone gives a warp the same segment in every round, and the side
// edges' Newton solves to few warps (traction sides, MR, us a step, so / in
// single launches / twisted: FP32 225 x 4533 88, 64, 48, 254 x 1021 21, 18, 11;
// FP64 249 x 250 115, 74, 91). Elsewhere it would only make other lattices meet.
TLV_HD bool multi_twist(int nseg, int warps)
{
    // (nor where the second rotation comes round with the first)
    return nseg > 2 && warps % (nseg * nseg) == 0 && warps / (nseg * nseg) % nseg != 0;
}

TLV_HD void multi_coords(int task, int nseg, int ny, bool twist, int &y, int &seg)
{
    const int r = task / nseg;
    y = (r == 0 || ny < 2) ? r : (r == 1 ? ny - 1 : r - 1);
    seg = (task - r * nseg + y + (twist ? r / nseg : 0)) % nseg;
}

} // namespace tlv
