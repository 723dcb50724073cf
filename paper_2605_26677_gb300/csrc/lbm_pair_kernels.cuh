// lbm_pair_kernels.cuh -- two steps of a large lattice in one pass over its
// populations.
#pragma once
#include "lbm_bulk.cuh"
#include "lbm_internal.h"
#include "lbm_launch.cuh"
#include "lbm_pair_plan.h"
#include "lbm_step_core.cuh"
#include "lbm_step_kernels.cuh"
#include <type_traits>


namespace tlv {

// Nodes per lane and blocks per SM: eight warps of four nodes each and a
// staged row per warp fill the shared memory (113 KB a block). 8192^2, us per
// step: 1406; two nodes per lane with 12 warps 1490, with 16 warps 1570.
constexpr int PAIR_BLOCKS = 2;

// 16 bytes from global to shared memory without waiting
__device__ __forceinline__ void copy_async(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(cta_smem(dst)), "l"(src) : "memory");
}

template <typename S, int VEC>
__device__ __forceinline__ Pack<S, VEC> pack_of(const S (&v)[VEC])
{
    Pack<S, VEC> o;
#pragma unroll
    for (int e = 0; e < VEC; ++e) o.v[e] = v[e];
    return o;
}

// u += dt v. The FP64 pipe takes a warp's conversion as long as its FMA (64
// cycles), so normal floats are widened on the integer pipe.
template <int VEC>
__device__ __forceinline__ void add_scaled(double (&u)[VEC], double dt, const float (&v)[VEC])
{
    bool normal = true;
#pragma unroll
    for (int e = 0; e < VEC; ++e) normal = normal && ((__float_as_uint(v[e]) >> 23) & 255u) - 1u < 254u;
    if (normal) {
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            const unsigned b = __float_as_uint(v[e]);
            const unsigned hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u);
            u[e] += dt * __hiloint2double((int)hi, (int)(b << 29));
        }
    } else {
#pragma unroll
        for (int e = 0; e < VEC; ++e) u[e] += dt * (double)v[e];
    }
}

// Shared memory of one warp: what the second step takes over from earlier
// rows of the first, as packed vectors per lane ...
template <typename S, int VEC>
struct PairSmem {
    Pack<S, VEC> s0[6][32], s2[6][32];  // f*^{n+1}_0 and _2 of the previous row
    Pack<S, VEC> s1[2][6][32];          // f*^{n+1}_1 of the last two rows, by row parity
    Pack<float, VEC> v[2][32];          // v^n of the previous row
    Pack<S, VEC> in[4][6][32];          // f*^n of the next row and u* of the one before it, on their way
    Pack<double, VEC> u[2][32];
    float side[2][PAIR_SIDE_ROWS][6];   // and the side-edge ghosts of f*^{n+1}, by row
};

// Ghost value of f*^{n+1} at a node of a bottom or top edge row (out of line:
// it runs once per task)
template <int LAW, typename T>
__device__ __noinline__ void pair_row_ghost(const PairArgs<T> &p, int e, int x, const T (*f)[6], T out[6],
                                            unsigned &flags)
{
    const StepArgs<T> &a = p.a;
    T U[6];
    state_from_fstar(f[0], f[1], f[2], f[3], a.hdtb1, a.hdtb2, U);
    const LawP<T> m{a.lam, a.mu, a.p2, a.p3};
    const EdgeVal<T> val = a.profile[e] ? edge_val<T>(a.value[e], p.g1[e] * a.profile[e][x], a.c) : p.v1[e];
    if (e == EDGE_BOTTOM)
        edge_ghost<LAW, T>(EDGE_BOTTOM, a.kind[EDGE_BOTTOM], f[edge_dout(EDGE_BOTTOM)], U, val, m, out, flags);
    else
        edge_ghost<LAW, T>(EDGE_TOP, a.kind[EDGE_TOP], f[edge_dout(EDGE_TOP)], U, val, m, out, flags);
}

// Ghosts of f*^{n+1} at PAIR_SIDE_ROWS / 2 rows of each side edge (the first
// lanes left, the next as many right), from row base on within [ya, yb): the edge node's first
// step and its edge rule, one row per lane, into the warp's table.
template <typename S, int LAW, int VEC>
__device__ __noinline__ void pair_side_ghosts(const PairArgs<S> &p, PairSmem<S, VEC> *sm, int base,
                                              int ya, int yb, bool left, bool right, int lane, unsigned &flags)
{
    using T = S;
    const StepArgs<T> &a = p.a;
    const int nx = a.L.nx, ny = a.L.ny;
    constexpr int H = PAIR_SIDE_ROWS / 2;
    const int sd = lane / H, y = base + (lane & (H - 1));
    if ((sd == 0 ? left : sd == 1 && right) && y >= ya && y < yb) {
        const bool yper = a.kind[EDGE_BOTTOM] == BC_PERIODIC;
        const int x = sd == 0 ? 0 : nx - 1;
        const int yd = (yper && y == 0) ? ny - 1 : y - 1, yu = (yper && y == ny - 1) ? 0 : y + 1;
        const S *fin = static_cast<const S *>(a.fin) + a.L.xoff + x;
        T f[4][6], v1, v2;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            f[0][k] = fin[(0 * 6 + k) * a.L.plane + (long long)(y + 1) * a.L.pitch - 1];
            f[2][k] = fin[(2 * 6 + k) * a.L.plane + (long long)(y + 1) * a.L.pitch + 1];
            f[1][k] = fin[(1 * 6 + k) * a.L.plane + (long long)(yd + 1) * a.L.pitch];
            f[3][k] = fin[(3 * 6 + k) * a.L.plane + (long long)(yu + 1) * a.L.pitch];
        }
        const LawP<T> m{a.lam, a.mu, a.p2, a.p3};
        unsigned none = 0;
        collide_node<LAW, T>(f, a, m, false, none, v1, v2);
        T U[6], out[6];
        state_from_fstar(f[0], f[1], f[2], f[3], a.hdtb1, a.hdtb2, U);
        const int e = sd == 0 ? EDGE_LEFT : EDGE_RIGHT;
        const EdgeVal<T> val = a.profile[e] ? edge_val<T>(a.value[e], p.g1[e] * a.profile[e][y], a.c) : p.v1[e];
        if (sd == 0)
            edge_ghost<LAW, T>(EDGE_LEFT, a.kind[EDGE_LEFT], f[edge_dout(EDGE_LEFT)], U, val, m, out, flags);
        else
            edge_ghost<LAW, T>(EDGE_RIGHT, a.kind[EDGE_RIGHT], f[edge_dout(EDGE_RIGHT)], U, val, m, out, flags);
#pragma unroll
        for (int k = 0; k < 6; ++k) sm->side[sd][y & (PAIR_SIDE_ROWS - 1)][k] = out[k];
    }
    __syncwarp();
}

// Columns -2, -1 and nx, nx + 1 of one row (r: its column 0), from those of
// nx - 2, nx - 1 and 0, 1 that lie in [x0, x1)
template <typename S>
__device__ __forceinline__ void wide_columns(S *r, int nx, int x0, int x1)
{
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (i >= x0 && i < x1) r[nx + i] = r[i];
        if (nx - 2 + i >= x0 && nx - 2 + i < x1) r[i - 2] = r[nx - 2 + i];
    }
}

// What the next launch pulls from beyond the side edges, for rows [ya, yb) of
// the strip of columns [x0, x1), one row per lane from the stored values: the
// edge rules' ghosts, or with periodic x two columns of every plane (ghost
// rows included).
template <typename S, int LAW>
__device__ __noinline__ void pair_side_columns(const PairArgs<S> &p, int ya, int yb, int x0, int x1,
                                               int lane, unsigned &flags)
{
    const StepArgs<S> &a = p.a;
    const int nx = a.L.nx, ny = a.L.ny;
    if (x0 > 1 && x1 < nx - 1) return;
    __syncwarp();  // the other lanes' stores
    S *fout = static_cast<S *>(a.fout);
    if (a.kind[EDGE_LEFT] == BC_PERIODIC) {
        const bool yper = a.kind[EDGE_BOTTOM] == BC_PERIODIC;
        const int r0 = (ya == 0 && !yper) ? -1 : ya, r1 = (yb == ny && !yper) ? ny + 1 : yb;
        for (int y = r0 + lane; y < r1; y += 32) {
            S *r = fout + (long long)(y + 1) * a.L.pitch + a.L.xoff;
#pragma unroll 6
            for (int pl = 0; pl < 24; ++pl) wide_columns(r + pl * a.L.plane, nx, x0, x1);
        }
    } else {
        const StepIO io{a.fin, a.fout, nullptr};
        for (int y = ya + lane; y < yb; y += 32) {
            if (y == 0 || y == ny - 1) continue;
            if (x0 == 0) xedge_node<LAW, S>(a, io, 0, y, flags);
            if (nx - 1 >= x0 && nx - 1 < x1 && !(x0 == 0 && nx == 1)) xedge_node<LAW, S>(a, io, nx - 1, y, flags);
        }
    }
    __syncwarp();
}

// One task: rows [ya, yb) of one strip. Lane l holds columns c .. c + VEC - 1,
// c = 30 VEC strip + VEC (l - 1); lanes 1 to 30 write, lanes 0 and 31 are the
// strip's halo (their outermost columns go stale by one column per step).
template <typename S, int LAW, int VEC>
__device__ __forceinline__ void pair_task(const PairArgs<S> &p, int chunk, int strip, int lane,
                                          PairSmem<S, VEC> *sm, unsigned &flags)
{
    using T = S;
    using PK = Pack<S, VEC>;
    using PD = Pack<double, VEC>;
    const StepArgs<T> &a = p.a;
    const int nx = a.L.nx, ny = a.L.ny, pitch = a.L.pitch;
    const long long plane = a.L.plane;
    const S *__restrict__ fin = static_cast<const S *>(a.fin);
    S *__restrict__ fout = static_cast<S *>(a.fout);
    int ya, yb;
    pair_rows(p.plan, ny, chunk, ya, yb);
    const int c = (30 * strip + lane - 1) * VEC;
    const bool xper = a.kind[EDGE_LEFT] == BC_PERIODIC, yper = a.kind[EDGE_BOTTOM] == BC_PERIODIC;
    const bool ld = c <= (xper ? nx + 1 : nx);  // the lane's vector holds a column that some output needs
    const bool out = lane >= 1 && lane <= 30 && c < nx;
    const bool left = !xper && strip == 0;
    const bool right = !xper && 30 * VEC * strip < nx && nx - 1 < 30 * VEC * (strip + 1);
    const int rfirst = (ya == 0 && !yper) ? 0 : ya - 1;

    // row r of f*^n into the warp's staging rows, each lane its own vectors,
    // in the background of the row before
    auto fetch = [&](int r) {
        if (r > yb) return;
        if (out && r > ya) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const double *us = a.ustar + i * a.L.uplane + (long long)(r - 1) * a.L.upitch + c;
#pragma unroll
                for (int h = 0; h < VEC / 2; ++h) copy_async(&sm->u[i][lane].v[2 * h], us + 2 * h);
            }
        }
        if ((!yper && r == ny) || !ld) return;
        const int y = yper ? (r < 0 ? r + ny : r >= ny ? r - ny : r) : r;
        const int yd = (yper && y == 0) ? ny - 1 : y - 1, yu = (yper && y == ny - 1) ? 0 : y + 1;
        const S *b = fin + a.L.xoff + c;
        const S *b0 = b + (long long)(y + 1) * pitch, *b1 = b + (long long)(yd + 1) * pitch + 6 * plane,
                *b3 = b + (long long)(yu + 1) * pitch + 18 * plane;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            copy_async(&sm->in[0][k][lane], b0 + k * plane);
            copy_async(&sm->in[2][k][lane], b0 + (12 + k) * plane);
            copy_async(&sm->in[1][k][lane], b1 + k * plane);
            copy_async(&sm->in[3][k][lane], b3 + k * plane);
        }
    };
    fetch(rfirst);
    for (int r = rfirst; r <= yb; ++r) {
        if ((left || right) && ((r - rfirst) & (PAIR_SIDE_ROWS / 2 - 1)) == 0) pair_side_ghosts<S, LAW, VEC>(p, sm, r, ya, yb, left, right, lane, flags);
        const int yo = r - 1;  // the row whose second step this pass finishes
        T f[4][6][VEC], vel[2][VEC];
        asm volatile("cp.async.wait_all;" ::: "memory");
        // Eq. (22), the first step's share; the second's follows below
        PD us[2];
        if (yo >= ya && out) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                us[i] = sm->u[i][lane];
                add_scaled(us[i].v, a.dt, sm->v[i][lane].v);
            }
        }
#pragma unroll 1
        for (int ph = 0; ph < 2; ++ph) {
            bool real;
            if (ph == 0) {
                // first step at row r: pull f*^n
                if (!yper && r == ny) {
                    // past the top edge: only the ghosts of f*^{n+1}_3, left
                    // in the ghost row of fout by the row before
                    if (out)
#pragma unroll
                        for (int k = 0; k < 6; ++k) {
                            const PK t = *reinterpret_cast<const PK *>(fout + (3 * 6 + k) * plane + (long long)(ny + 1) * pitch + a.L.xoff + c);
#pragma unroll
                            for (int e = 0; e < VEC; ++e) f[3][k][e] = t.v[e];
                        }
                    continue;
                }
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    const PK c0 = sm->in[0][k][lane], c1 = sm->in[1][k][lane], c2 = sm->in[2][k][lane],
                             c3 = sm->in[3][k][lane];
                    const T lf = __shfl_up_sync(FULL_MASK, c0.v[VEC - 1], 1);
                    const T rt = __shfl_down_sync(FULL_MASK, c2.v[0], 1);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        f[0][k][e] = e == 0 ? lf : c0.v[e - 1];
                        f[2][k][e] = e == VEC - 1 ? rt : c2.v[e + 1];
                        f[1][k][e] = c1.v[e];
                        f[3][k][e] = c3.v[e];
                    }
                }
                __syncwarp();
                fetch(r + 1);
                real = out && r >= ya && r < yb;
            } else {
                // second step at row yo: take over what the rows before left
                // and leave this row's
                PK q1[6];
                const bool first = yper || r < ny;
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    const PK t0 = sm->s0[k][lane], t2 = sm->s2[k][lane];
                    q1[k] = sm->s1[r & 1][k][lane];
                    if (first) {
                        sm->s0[k][lane] = pack_of<S, VEC>(f[0][k]);
                        sm->s2[k][lane] = pack_of<S, VEC>(f[2][k]);
                        sm->s1[r & 1][k][lane] = pack_of<S, VEC>(f[1][k]);
                    }
                    T lf = __shfl_up_sync(FULL_MASK, t0.v[VEC - 1], 1);
                    T rt = __shfl_down_sync(FULL_MASK, t2.v[0], 1);
                    if (left && lane == 1) lf = sm->side[0][yo & (PAIR_SIDE_ROWS - 1)][k];
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        f[0][k][e] = e == 0 ? lf : t0.v[e - 1];
                        f[2][k][e] = e == VEC - 1 ? rt : t2.v[e + 1];
                        f[1][k][e] = q1[k].v[e];
                    }
                    if (right)
#pragma unroll
                        for (int e = 0; e < VEC; ++e)
                            if (c + e == nx - 1) f[2][k][e] = sm->side[1][yo & (PAIR_SIDE_ROWS - 1)][k];
                }
                if (yo < ya) break;
                real = out;
            }
            const LawP<T> m{a.lam, a.mu, a.p2, a.p3};
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                T fq[4][6];
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int k = 0; k < 6; ++k) fq[q][k] = f[q][k][e];
                collide_node<LAW, T>(fq, a, m, real && c + e < nx, flags, vel[0][e], vel[1][e]);
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int k = 0; k < 6; ++k) f[q][k][e] = fq[q][k];
            }
            if (ph == 0) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    Pack<float, VEC> t;
#pragma unroll
                    for (int e = 0; e < VEC; ++e) t.v[e] = vel[i][e];
                    sm->v[i][lane] = t;
                }
                // ghosts of f*^{n+1} along a bottom or top edge
                if (!yper && out && ((r == 0 && ya == 0) || (r == ny - 1 && yb == ny))) {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        if (c + e >= nx) continue;
                        T fq[4][6], g[6];
#pragma unroll
                        for (int q = 0; q < 4; ++q)
#pragma unroll
                            for (int k = 0; k < 6; ++k) fq[q][k] = f[q][k][e];
                        if (r == 0) {
                            pair_row_ghost<LAW, T>(p, EDGE_BOTTOM, c + e, fq, g, flags);
#pragma unroll
                            for (int k = 0; k < 6; ++k) sm->s1[1][k][lane].v[e] = g[k];
                        } else {
                            // read back by the pass that follows the last row
                            pair_row_ghost<LAW, T>(p, EDGE_TOP, c + e, fq, g, flags);
#pragma unroll
                            for (int k = 0; k < 6; ++k)
                                fout[(3 * 6 + k) * plane + (long long)(ny + 1) * pitch + a.L.xoff + c + e] = g[k];
                        }
                    }
                }
            }
        }
        if (yo < ya || !out) continue;
        const long long row = (long long)(yo + 1) * pitch + a.L.xoff + c;
        const bool full = c + VEC <= nx;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                S *dst = fout + (q * 6 + k) * plane + row;
                const PK o = pack_of<S, VEC>(f[q][k]);
                if (full) {
                    *reinterpret_cast<PK *>(dst) = o;
                } else {
#pragma unroll
                    for (int e = 0; e < VEC; ++e)
                        if (c + e < nx) dst[e] = o.v[e];
                }
            }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            add_scaled(us[i].v, a.dt, vel[i]);
            *reinterpret_cast<PD *>(a.ustar + i * a.L.uplane + (long long)yo * a.L.upitch + c) = us[i];
        }
        if (yo == 0 || yo == ny - 1) lane_ghosts<LAW, S, VEC>(a, nullptr, fout, row, c, yo, flags);
    }
    pair_side_columns<S, LAW>(p, ya, yb, 30 * VEC * strip, 30 * VEC * (strip + 1), lane, flags);
}

// Two steps in one pass: f*^n is read, f*^{n+1} lives in registers and shared
// memory only, f*^{n+2} is written, and u* moves once for both steps: 112
// instead of 224 bytes per node and step, 122 measured (4096^2). A warp goes
// down a strip of columns row by row (pair_task); the strips overlap by a lane
// on either side and the row chunks by a row, 7% and 4 to 12% of reads done
// twice. The warps need nothing of one another. Its next row is copied to
// shared memory in the background of the current one (without that copy 1591
// instead of 1406 us a step on 8192^2, with u* read when it is needed and its
// velocities widened on the FP64 pipe 1580). Barriers that keep the warps of
// a block on the same row made it slower (1756). The same bits as two
// launches of k_step; us per step, k_step / k_pair: 8192^2 periodic 2145 /
// 1366, 4096 x 2048 clamped 284 / 187, 2048^2 periodic 149 / 106. What binds it now
// is the latency of a warp's own chain at eight warps per SM (33% of issue
// slots) and HBM at 5.5 TB/s; with the collisions taken out it moves its
// data at 5.7 TB/s.
template <typename S, int LAW, int VEC>
__global__ void __launch_bounds__(128, PAIR_BLOCKS) k_pair(const __grid_constant__ PairArgs<S> p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    pdl_enter();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    PairSmem<S, VEC> *sm = reinterpret_cast<PairSmem<S, VEC> *>(smem) + wid;
    unsigned flags = 0;
    // one counter: the tasks are few, and only a common order puts the long
    // ones before the short ones (over four stripes 8192^2 took 1425 instead
    // of 1386 us a step, 4096 x 2048 clamped 200 instead of 194). The counter
    // sets alternate as in dyn_tasks.
    if (blockIdx.x == 0 && threadIdx.x < DYN_STRIPES) p.a.ctr_next[threadIdx.x * DYN_CTR_STRIDE] = 0u;
    pair_tasks(
        4 * gridDim.x, (unsigned)(p.plan.nstrip * p.plan.nchunk), [&] { return lane == 0 ? atomicAdd(p.a.ctr, 1u) : 0u; },
        [&](unsigned next) { return __shfl_sync(FULL_MASK, next, 0); },
        [&](int task) {
            __syncwarp();
            const int i = task / p.plan.nstrip;
            pair_task<S, LAW, VEC>(p, pair_chunk(p.plan, i), task - i * p.plan.nstrip, lane, sm, flags);
        });
    flags = __reduce_or_sync(FULL_MASK, flags);
    if (flags && lane == 0) atomicOr(p.a.status, (int)flags);
}

// Periodic x: columns -2, -1 and nx, nx + 1 of every plane and row (ghost rows
// included) before the first pair of a call
template <typename S>
__global__ void __launch_bounds__(128) k_wide(S *f, Layout L)
{
    const int rows = L.ny + 2;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 24 * rows; i += gridDim.x * blockDim.x) {
        S *r = f + (long long)(i / rows) * L.plane + (long long)(i % rows) * L.pitch + L.xoff;
        wide_columns(r, L.nx, 0, L.nx);
    }
}

// The kernel of a law with its shared-memory limit raised (once per device)
template <typename S, int LAW, int VEC>
static cudaError_t pair_prepare()
{
    static unsigned long long done = 0;  // one bit per device ordinal < 64
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (__atomic_load_n(&done, __ATOMIC_ACQUIRE) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(k_pair<S, LAW, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             4 * (int)sizeof(PairSmem<S, VEC>));
    if (e == cudaSuccess) __atomic_fetch_or(&done, bit, __ATOMIC_ACQ_REL);
    return e;
}

template <typename Fn>
static auto with_law(int law, Fn fn)
{
    switch (law) {
    case LAW_SVK: return fn(std::integral_constant<int, LAW_SVK>());
    case LAW_NH: return fn(std::integral_constant<int, LAW_NH>());
    case LAW_LOGNH: return fn(std::integral_constant<int, LAW_LOGNH>());
    case LAW_MR: return fn(std::integral_constant<int, LAW_MR>());
    case LAW_YEOH: return fn(std::integral_constant<int, LAW_YEOH>());
    default: return fn(std::integral_constant<int, LAW_GENT>());
    }
}

template <typename S, int VEC>
static cudaError_t launch_pair(int law, const void *args, int grid, cudaStream_t st)
{
    PairArgs<S> p = *static_cast<const PairArgs<S> *>(args);
    return with_law(law, [&](auto L) {
        constexpr int LAW = decltype(L)::value;
        const cudaError_t e = pair_prepare<S, LAW, VEC>();
        if (e != cudaSuccess) return e;
        // the counter set that the previous dynamic launch zeroed
        p.a.ctr = p.a.ctr2 + *p.a.ctr_par * DYN_SET_WORDS;
        p.a.ctr_next = p.a.ctr2 + (*p.a.ctr_par ^ 1) * DYN_SET_WORDS;
        *p.a.ctr_par ^= 1;
        return launch_pdl(k_pair<S, LAW, VEC>, grid, 128, 4 * sizeof(PairSmem<S, VEC>), st, p);
    });
}

// resident blocks per SM, 0 if it cannot run
template <typename S, int VEC>
static int pair_blocks(int law)
{
    return with_law(law, [](auto L) {
        constexpr int LAW = decltype(L)::value;
        int n = 0;
        if (pair_prepare<S, LAW, VEC>() != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_pair<S, LAW, VEC>, 128, 4 * sizeof(PairSmem<S, VEC>)) !=
                cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        return n;
    });
}

} // namespace tlv
