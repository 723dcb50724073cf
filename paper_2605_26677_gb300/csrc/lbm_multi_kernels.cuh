// lbm_multi_kernels.cuh -- many steps of a small lattice in one cooperative
// launch.
#pragma once
#include "lbm_grid_barrier.cuh"
#include "lbm_internal.h"
#include "lbm_step_core.cuh"

namespace tlv {

// Loads past the L1 cache, for values that other SMs stored in this launch
__device__ __forceinline__ double ld_l2(const double *p) { return __ldcg(p); }
__device__ __forceinline__ float ld_l2(const float *p) { return __ldcg(p); }
template <typename H>
__device__ __forceinline__ H ld_l2(const H *p)  // the 16-bit types
{
    static_assert(sizeof(H) == 2, "a 16-bit type");
    const unsigned short b = __ldcg(reinterpret_cast<const unsigned short *>(p));
    H r;
    memcpy(&r, &b, 2);
    return r;
}

// One node per lane: the same arithmetic as step_task, arranged for latency.
// Each lane loads its 24 populations and u* at once (no shuffles: the
// neighbouring columns' lines are the same), and a boundary node's ghost
// cells are formed from the registers instead of from a re-read of what was
// stored.
template <typename S, int LAW>
__device__ __forceinline__ void node_step(const StepArgs<typename Prec<S>::R> &a,
                                          const StepTimes<typename Prec<S>::R> &tab, int s, const void *from, void *to,
                                          int x, int y, unsigned &flags)
{
    using T = typename Prec<S>::R;
    const long long plane = a.L.plane;
    const int pitch = a.L.pitch;
    const long long cell = (long long)(y + 1) * pitch + a.L.xoff + x;
    const S *__restrict__ fin = static_cast<const S *>(from);
    S *__restrict__ fout = static_cast<S *>(to);
    double *us = a.ustar + (long long)y * a.L.upitch + x;
    S in[4][6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        in[0][k] = ld_l2(fin + (0 * 6 + k) * plane + cell - 1);
        in[2][k] = ld_l2(fin + (2 * 6 + k) * plane + cell + 1);
        in[1][k] = ld_l2(fin + (1 * 6 + k) * plane + cell - pitch);
        in[3][k] = ld_l2(fin + (3 * 6 + k) * plane + cell + pitch);
    }
    const double u1 = us[0], u2 = us[a.L.uplane];
    T f[4][6], v1, v2;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 6; ++k) f[q][k] = ld_r(in[q][k]);
    const LawP<T> m{a.lam, a.mu, a.p2, a.p3};
    collide_node<LAW, T>(f, a, m, true, flags, v1, v2);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const S o = to_store<S>(f[q][k]);
            fout[(q * 6 + k) * plane + cell] = o;
            f[q][k] = ld_r(o);
        }
    us[0] = u1 + a.dt * (double)v1;
    us[a.L.uplane] = u2 + a.dt * (double)v2;
    if (x == 0 || y == 0 || x == a.L.nx - 1 || y == a.L.ny - 1) {
        auto ev = [&](int e, int p) {
            return a.profile[e] ? edge_val<T>(a.value[e], tab.g[s][e] * a.profile[e][p], a.c) : tab.val[s][e];
        };
        node_ghosts<LAW, S, T>(f, x, y, a, ev, m, fout, flags);
    }
}

// Steps 0 .. nsteps - 1 of one lattice, a grid barrier between them. A step
// of such a lattice is all latency: launched on its own with four nodes per
// lane it takes 5 us (64^2 FP32) to 12 us (256 x 128 with traction edges).
// Here one node per lane spreads the lattice over every SM and shortens each
// warp's chain, and a barrier (1.2 us over 152 blocks) replaces the launch:
// us per step, launches of their own / this kernel,
//   64^2 FP32 periodic 4.8 / 2.4, 131 x 37 FP32 with traction edges 11.0 /
//   3.7, 256 x 128 FP32 the same 11.7 / 4.0, 512^2 FP32 11.7 / 8.0,
//   1000 x 517 FP32 24.8 / 17.4, 64^2 FP64 11.3 / 5.5.
// What is left at 64^2 is the barrier, one L2 round trip and the chain of one
// node's arithmetic (FP64: 64 cycles per warp instruction). Four nodes per
// lane in this kernel gave no gain (64^2 FP32 4.8, 131 x 37 10.4). The same
// warp takes the same tasks in every step, so u* stays with its thread; the
// populations, which other SMs wrote, are read past the L1 cache.
template <typename S, int LAW>
__global__ void __launch_bounds__(32 * MULTI_WARPS) k_multi(const __grid_constant__ StepArgs<typename Prec<S>::R> a,
                                               const __grid_constant__ StepTimes<typename Prec<S>::R> tab, int nsteps, unsigned *count)
{
    const int lane = threadIdx.x & 31;
    // consecutive tasks to different blocks: a last round that is not full
    // still loads every SM alike (FP64, bound by its pipe)
    const int gw = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const int nw = gridDim.x * (blockDim.x >> 5);
    const int nseg = (a.L.nx + 31) / 32, ntask = a.L.ny * nseg;
    const bool twist = multi_twist(nseg, nw);
    unsigned flags = 0;
    void *const f0 = const_cast<void *>(a.fin);
    for (int s = 0; s < nsteps; ++s) {
        const void *from = (s & 1) ? a.fout : f0;
        void *to = (s & 1) ? f0 : a.fout;
        for (int task = gw; task < ntask; task += nw) {
            int y, seg;
            multi_coords(task, nseg, a.L.ny, twist, y, seg);
            const int x = seg * 32 + lane;
            if (x < a.L.nx) node_step<S, LAW>(a, tab, s, from, to, x, y, flags);
        }
        if (s + 1 < nsteps && !grid_barrier(count, gridDim.x * (unsigned)(s + 1))) {
            flags |= ST_STALL;
            break;
        }
    }
    flags = __reduce_or_sync(FULL_MASK, flags);
    if (flags && lane == 0) atomicOr(a.status, (int)flags);
}

template <typename S>
const void *multi_kernel(int law)
{
    switch (law) {
    case LAW_SVK: return (const void *)k_multi<S, LAW_SVK>;
    case LAW_NH: return (const void *)k_multi<S, LAW_NH>;
    case LAW_LOGNH: return (const void *)k_multi<S, LAW_LOGNH>;
    case LAW_MR: return (const void *)k_multi<S, LAW_MR>;
    case LAW_YEOH: return (const void *)k_multi<S, LAW_YEOH>;
    case LAW_GENT: return (const void *)k_multi<S, LAW_GENT>;
    default: return nullptr;
    }
}

} // namespace tlv
