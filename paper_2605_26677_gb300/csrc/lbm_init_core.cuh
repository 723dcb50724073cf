// lbm_init_core.cuh -- per-node pieces of the second-order initialization
// (Sec. 3.4, Eqs. 16-21) shared by the init kernel and the adjoint's init
// step, in a compute type R: FP64 for FP64 storage and for the adjoint, FP32
// for FP32 and 16-bit storage (whose populations are rounded to FP32 or
// less anyway, and whose every step computes in FP32).
#pragma once
#include "lbm_device.cuh"
#include "lbm_edges.cuh"
#include "lbm_internal.h"
#include <type_traits>

namespace tlv {

__device__ __forceinline__ long long pidx(const Layout &L, int q, int k, int x, int y)
{
    return (long long)(q * 6 + k) * L.plane + (long long)(y + 1) * L.pitch + L.xoff + x;
}


// coordinates of node n (32-bit division where it suffices)
__device__ __forceinline__ void node_xy(long long n, int nx, int &x, int &y)
{
    if (n >> 31) {
        y = (int)(n / nx);
    } else {
        y = (int)((unsigned)n / (unsigned)nx);
    }
    x = (int)(n - (long long)y * nx);
}

// Second-order difference of a compact field along x (dir 0) or y (dir 1)
// without its factor h = 1 / (2 dx): central inside, wrap-around when
// periodic, one-sided three-point stencil at a non-periodic end (Sec. 3.4).
__device__ __forceinline__ double fd(const double *a, int nx, int ny, int x, int y, int dir, int per)
{
    const int n = dir == 0 ? nx : ny;
    const int i = dir == 0 ? x : y;
    auto at = [&](int j) { return dir == 0 ? a[(long long)y * nx + j] : a[(long long)j * nx + x]; };
    if (per) return at(i + 1 == n ? 0 : i + 1) - at(i == 0 ? n - 1 : i - 1);
    if (i == 0) return -3.0 * at(0) + 4.0 * at(1) - at(2);
    if (i == n - 1) return 3.0 * at(n - 1) - 4.0 * at(n - 2) + at(n - 3);
    return at(i + 1) - at(i - 1);
}

// f^eq_q(U) - f^eq_q(U_rest) of Eq. (12): U_ofs = U - U_rest (v, F - I), P the
// stress; f^eq is linear in U and in P, and P(I) = 0.
template <typename R>
__device__ __forceinline__ void feq_ofs(const R U[6], const R P[4], R r2c, R feq[4][6])
{
    const R PhiX[6] = {-P[0], -P[2], -U[0], R(0), -U[1], R(0)};
    const R PhiY[6] = {-P[1], -P[3], R(0), -U[0], R(0), -U[1]};
    const int ci[4] = {1, 0, -1, 0}, cj[4] = {0, 1, 0, -1};
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 6; ++k) feq[q][k] = R(0.25) * (U[k] + r2c * (ci[q] * PhiX[k] + cj[q] * PhiY[k]));
}

// dP_i = C : dF_i for three directions at one F in FP64, the law chosen once
// so that they share its reciprocal and cofactors
__device__ __forceinline__ void tangent_jvp3(int law, const double G[4], const double d[3][4], const LawP<double> &m,
                                             double dP[3][4])
{
    auto three = [&](auto L) {
#pragma unroll
        for (int i = 0; i < 3; ++i) jvp_ofs<decltype(L)::value, double>(G, d[i], m, dP[i]);
    };
    switch (law) {
    case LAW_SVK: three(std::integral_constant<int, LAW_SVK>()); break;
    case LAW_NH: three(std::integral_constant<int, LAW_NH>()); break;
    case LAW_LOGNH: three(std::integral_constant<int, LAW_LOGNH>()); break;
    case LAW_MR: three(std::integral_constant<int, LAW_MR>()); break;
    case LAW_YEOH: three(std::integral_constant<int, LAW_YEOH>()); break;
    default: three(std::integral_constant<int, LAW_GENT>()); break;
    }
}

// f^0 - f_rest at node (x, y) in compute type R (f_rest = U_rest / 4: 1/4 in
// the F11 and F22 components, 0 elsewhere): f^eq(U0) and, for order 2, the
// correction -(dt/2) D_q f^eq of Eqs. (16)-(21), with the node's parameters.
// Returns false if det F0 <= 0.
template <typename R>
__device__ inline bool init_node_ofs(const InitArgs &a, const InitConst<R> &K, int x, int y, const LawP<R> &m,
                                     R f[4][6])
{
    const int nx = a.L.nx, ny = a.L.ny;
    const long long N = (long long)nx * ny, n = (long long)y * nx + x;
    const int ci[4] = {1, 0, -1, 0}, cj[4] = {0, 1, 0, -1};
    const R c = (R)a.c, dt = (R)a.dt;
    const R r2c = R(2) / c;
    R U[6];  // U0 - U_rest
#pragma unroll
    for (int k = 0; k < 6; ++k) U[k] = (R)(a.U0[k * N + n] - ((k == 2 || k == 5) ? 1.0 : 0.0));
    const R G[4] = {U[2], U[3], U[4], U[5]};
    const R F[4] = {R(1) + U[2], U[3], U[4], R(1) + U[5]};
    R P[4], dJ;
    piola_any_t<R>(a.m.law, G, m, P, dJ);
    feq_ofs<R>(U, P, r2c, f);
    if (a.order == 2) {
        R gX[6], gY[6], dPX[4], dPY[4];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            gX[k] = (R)(fd(a.U0 + k * N, nx, ny, x, y, 0, a.xper) * K.h);
            gY[k] = (R)(fd(a.U0 + k * N, nx, ny, x, y, 1, a.yper) * K.h);
        }
        // d_alpha P = C : d_alpha F (text after Eq. 18), as Jacobian actions (Eq. 8)
        tangent_jvp_t<R>(a.m.law, F, gX + 2, m, dPX);
        tangent_jvp_t<R>(a.m.law, F, gY + 2, m, dPY);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const R i = (R)ci[q], j = (R)cj[q];
            R Z[6], dP[4];
            // Eq. (18): Z_q = D_q U0 with d_t U0 taken from the continuum system
            Z[0] = (R)a.b1 + dPX[0] + dPY[1] + c * i * gX[0] + c * j * gY[0];
            Z[1] = (R)a.b2 + dPX[2] + dPY[3] + c * i * gX[1] + c * j * gY[1];
            Z[2] = gX[0] + c * i * gX[2] + c * j * gY[2];
            Z[3] = gY[0] + c * i * gX[3] + c * j * gY[3];
            Z[4] = gX[1] + c * i * gX[4] + c * j * gY[4];
            Z[5] = gY[1] + c * i * gX[5] + c * j * gY[5];
            tangent_jvp_t<R>(a.m.law, F, Z + 2, m, dP); // Eq. (20)
            // Eq. (21): D_q f^eq = (f^eq)'(U0) Z_q, then Eq. (16)
            const R Dq[6] = {R(0.25) * (Z[0] - r2c * (i * dP[0] + j * dP[1])),
                             R(0.25) * (Z[1] - r2c * (i * dP[2] + j * dP[3])),
                             R(0.25) * (Z[2] - (r2c * i) * Z[0]),
                             R(0.25) * (Z[3] - (r2c * j) * Z[0]),
                             R(0.25) * (Z[4] - (r2c * i) * Z[1]),
                             R(0.25) * (Z[5] - (r2c * j) * Z[1])};
#pragma unroll
            for (int k = 0; k < 6; ++k) f[q][k] -= R(0.5) * dt * Dq[k];
        }
    }
    return dJ > R(-1);
}

// f^0 - f_rest at node (x, y) in FP64 with the node's parameters, its terms
// added to fz (without P) and fm (with P), which may be one array: the terms
// of init_node_ofs without the products with the directions' zeros. SPLIT: fm
// starts from zero. For SVK, NH and log-NH with lambda = r mu the stress and its
// tangent are linear in mu, and f^0 is fz + mu fm with fm that of mu = 1.
// Returns false if det F0 <= 0.
template <bool SPLIT>
__device__ __forceinline__ bool init_node_parts(const InitArgs &a, const InitConst<double> &K, int x, int y,
                                                const LawP<double> &m, double fz[4][6], double fm[4][6])
{
    const int nx = a.L.nx, ny = a.L.ny;
    const long long N = (long long)nx * ny, n = (long long)y * nx + x;
    const double c = a.c;
    double U[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) U[k] = a.U0[k * N + n] - ((k == 2 || k == 5) ? 1.0 : 0.0);
    const double G[4] = {U[2], U[3], U[4], U[5]};
    double P[4], dJ;
    piola_any(a.m.law, G, m, P, dJ);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const double s = (q < 2 ? 0.25 : -0.25) * K.r2c;  // of Phi_X (even q) or Phi_Y
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            fz[q][k] = 0.25 * U[k];
            if (SPLIT) fm[q][k] = 0.0;
        }
        const int o = q & 1;
        fz[q][2 + o] -= s * U[0];
        fz[q][4 + o] -= s * U[1];
        fm[q][0] -= s * P[o];
        fm[q][1] -= s * P[2 + o];
    }
    const bool ok = dJ > -1.0;
    if (a.order != 2) return ok;
    double gX[6], gY[6], dP[3][4];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        gX[k] = fd(a.U0 + k * N, nx, ny, x, y, 0, a.xper) * K.h;
        gY[k] = fd(a.U0 + k * N, nx, ny, x, y, 1, a.yper) * K.h;
    }
    const double d[3][4] = {{gX[2], gX[3], gX[4], gX[5]}, {gY[2], gY[3], gY[4], gY[5]}, {gX[0], gY[0], gX[1], gY[1]}};
    tangent_jvp3(a.m.law, G, d, m, dP);
    const double zb0 = dP[0][0] + dP[1][1], zb1 = dP[0][2] + dP[1][3];
    const double dt8 = 0.125 * a.dt;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int o = q & 1;
        const double sg = q < 2 ? 1.0 : -1.0, ci = sg * c, r = sg * K.r2c;
        const double *g = o ? gY : gX;  // the difference along the direction
        const double za0 = a.b1 + ci * g[0], za1 = a.b2 + ci * g[1];
        const double Z[4] = {gX[0] + ci * g[2], gY[0] + ci * g[3], gX[1] + ci * g[4], gY[1] + ci * g[5]};
        fz[q][0] -= dt8 * za0;
        fz[q][1] -= dt8 * za1;
#pragma unroll
        for (int k = 0; k < 4; ++k) fz[q][2 + k] -= dt8 * Z[k];
        fz[q][2 + o] += dt8 * (r * za0);
        fz[q][4 + o] += dt8 * (r * za1);
        const double e0 = dP[2][o] + ci * dP[o][o], e1 = dP[2][2 + o] + ci * dP[o][2 + o];  // Eq. (20)
        fm[q][0] -= dt8 * (zb0 - r * e0);
        fm[q][1] -= dt8 * (zb1 - r * e1);
        fm[q][2 + o] += dt8 * (r * zb0);
        fm[q][4 + o] += dt8 * (r * zb1);
    }
    return ok;
}

} // namespace tlv
