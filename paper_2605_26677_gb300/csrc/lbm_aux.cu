// lbm_aux.cu -- initialization, read-out and diagnostics kernels of the TL
// vectorial D2Q4x6 LBM. Read-out and diagnostics compute in FP64 whatever the
// storage; the initialization computes in FP64 for FP64 storage and in FP32
// otherwise (u* always in FP64).
#include <cfloat>

#include "lbm_init_core.cuh"
#include <type_traits>

namespace tlv {

// Initial populations (Sec. 3.4) followed by the collision of step 0, so the
// stored state is f*^0; u* receives u0 - (dt/2) v0 + dt v^0 (Eq. 22).
// FP32 and 16-bit storage: bound by latency at the 12 warps per SM that its
// registers leave (4096 x 2048: 2.02 -> 1.81 ms with the constants from the
// host, 1.78 in blocks of two warps; 1.17 ms at six blocks per SM, but with fewer registers the compiler
// contracts its products differently and the start's last bits change). FP64
// storage: bound by the FP64 pipe (11.9 -> 9.4 ms with one reciprocal for the
// three tangent actions and Eq. (20) formed from them, 7.2 without the
// products with the directions' zeros).
template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? 2 : 3)
    k_init(const InitArgs a, const InitConst<typename std::conditional<sizeof(T) == 8, double, float>::type> K)
{
    using R = typename std::conditional<sizeof(T) == 8, double, float>::type;  // compute type
    const int nx = a.L.nx, ny = a.L.ny;
    const long long N = (long long)nx * ny;
    T *fout = static_cast<T *>(a.fout);
    const double dt = a.dt;
    const R c = (R)a.c, w = (R)a.omega;
    const long long n1 = (long long)a.y1 * nx;
    for (long long n = (long long)a.y0 * nx + (long long)blockIdx.x * blockDim.x + threadIdx.x; n < n1;
         n += (long long)gridDim.x * blockDim.x) {
        int x, y;
        node_xy(n, nx, x, y);
        R f[4][6];  // f^0 - f_rest
        const LawP<R> m = law_cast<R>(law_at(a.m, n));
        bool valid;
        if constexpr (sizeof(R) == 8)
            valid = init_node_parts<false>(a, K, x, y, m, f, f);
        else
            valid = init_node_ofs<R>(a, K, x, y, m, f);
        if (!valid) atomicOr(a.status, ST_BAD_J);
        // step-0 collision (Eqs. 10, 12, 14) on the offsets from the rest
        // state, which the collision leaves fixed
        R Un[6], dJ;
#pragma unroll
        for (int k = 0; k < 6; ++k) Un[k] = (f[0][k] + f[2][k]) + (f[1][k] + f[3][k]);
        Un[0] += K.hb1;
        Un[1] += K.hb2;
        const R Gn[4] = {Un[2], Un[3], Un[4], Un[5]};
        R Pn[4], feq[4][6];
        piola_any_t<R>(a.m.law, Gn, m, Pn, dJ);
        if constexpr (sizeof(R) == 8) {
            // feq_ofs without the products with the directions' zeros
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int o = q & 1;
                const R s = (q < 2 ? R(0.25) : R(-0.25)) * K.r2c;
#pragma unroll
                for (int k = 0; k < 6; ++k) feq[q][k] = R(0.25) * Un[k];
                feq[q][0] -= s * Pn[o];
                feq[q][1] -= s * Pn[2 + o];
                feq[q][2 + o] -= s * Un[0];
                feq[q][4 + o] -= s * Un[1];
            }
        } else {
            feq_ofs<R>(Un, Pn, R(2) / c, feq);
        }
        const R src[2] = {K.src1, K.src2};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                R fs = f[q][k] + w * (feq[q][k] - f[q][k]);
                if (k < 2) fs += src[k];
                fout[pidx(a.L, q, k, x, y)] = to_store<T>(fs);
            }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const double u0 = a.u0 ? a.u0[k * N + n] : 0.0;
            bool ok = true;
            double v;
            if constexpr (sizeof(R) == 8) {
                v = Un[k];
            } else {
                v = widen_int(Un[k], ok);
                if (!ok) v = (double)Un[k];
            }
            a.ustar[k * a.L.uplane + (long long)y * a.L.upitch + x] = (u0 - 0.5 * dt * a.U0[k * N + n]) + dt * v;
        }
    }
}

template <typename R>
__global__ void k_mu_plane(const double *mu, R *plane, Layout L)
{
    const long long N = (long long)L.nx * L.ny;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(n % L.nx), y = (int)(n / L.nx);
        plane[(long long)y * L.upitch + x] = (R)mu[n];
    }
}

// Components [K0, K1) of sum_q f*_q at the node of b (its plane K0), in FP64
// (offset form). A call of its own: as a branch the compiler would execute
// its conversions beside the integer ones.
template <typename T, int K0, int K1>
__device__ __noinline__ void node_sums_cvt(const T *b, long long plane, double *S)
{
    for (int k = 0; k < K1 - K0; ++k) {
        double s = 0.0;
        for (int q = 0; q < 4; ++q) s += (double)ld_r(b[(q * 6 + k) * plane]);
        S[k] = s;
    }
}

// The same with the values widened on the integer pipe where they are normal
template <typename T, int K0, int K1>
__device__ __forceinline__ void node_sums(const T *f, const Layout &L, int x, int y, double *S)
{
    constexpr int n = K1 - K0;
    const T *b = f + pidx(L, 0, K0, x, y);
    T v[4][n];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < n; ++k) v[q][k] = b[(q * 6 + k) * L.plane];
    double d[4][n];
    bool ok = true;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < n; ++k) {
            if constexpr (sizeof(T) == 8)
                d[q][k] = v[q][k];
            else
                d[q][k] = widen_int(ld_r(v[q][k]), ok);
        }
#pragma unroll
    for (int k = 0; k < n; ++k) S[k] = ((d[0][k] + d[1][k]) + d[2][k]) + d[3][k];
    if constexpr (sizeof(T) < 8)
        if (!ok) node_sums_cvt<T, K0, K1>(b, L.plane, S);
}

// U^n = sum_q f*_q - (dt/2) B, P(F^n), sigma = J^{-1} P F^T, u^n = u* - (dt/2) v^n
// (the stored u* already holds u*^{n+1} = u*^n + dt v^n). Bound by the FP64
// pipe: with the conversions off it, 18 sums and about 40 operations of the
// stress per node are left (4096 x 2048 FP32: U and P 1.36 -> 0.88 ms,
// u 0.33 -> 0.17 ms).
// ST: U, P or sigma wanted, DISP: u.
template <typename T, bool ST, bool DISP>
__global__ void __launch_bounds__(128) k_read(const ReadArgs a)
{
    const int nx = a.L.nx, ny = a.L.ny;
    const long long N = (long long)nx * ny;
    const T *f = static_cast<const T *>(a.f);
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        int x, y;
        node_xy(n, nx, x, y);
        double S[6];
        if (DISP || a.U) node_sums<T, 0, 2>(f, a.L, x, y, S);
        if (ST) node_sums<T, 2, 6>(f, a.L, x, y, S + 2);
        const double v1 = S[0] - a.hb1, v2 = S[1] - a.hb2;
        const double G[4] = {S[2], S[3], S[4], S[5]};
        if (ST && a.U) {
            a.U[0 * N + n] = v1;
            a.U[1 * N + n] = v2;
            a.U[2 * N + n] = 1.0 + G[0];
            a.U[3 * N + n] = G[1];
            a.U[4 * N + n] = G[2];
            a.U[5 * N + n] = 1.0 + G[3];
        }
        if (ST && (a.P || a.sigma)) {
            double P[4], dJ;
            piola_any(a.m.law, G, law_at(a.m, n), P, dJ);
            if (a.P)
                for (int m = 0; m < 4; ++m) a.P[m * N + n] = P[m];
            if (a.sigma) {
                const double F[4] = {1.0 + G[0], G[1], G[2], 1.0 + G[3]};
                const double J = 1.0 + dJ;
                a.sigma[0 * N + n] = (P[0] * F[0] + P[1] * F[1]) / J;
                a.sigma[1 * N + n] = (P[0] * F[2] + P[1] * F[3]) / J;
                a.sigma[2 * N + n] = (P[2] * F[0] + P[3] * F[1]) / J;
                a.sigma[3 * N + n] = (P[2] * F[2] + P[3] * F[3]) / J;
            }
        }
        if (DISP) {
            const long long ui = (long long)y * a.L.upitch + x;
            a.u[0 * N + n] = a.ustar[ui] - a.hdt * v1;
            a.u[1 * N + n] = a.ustar[a.L.uplane + ui] - a.hdt * v2;
        }
    }
}

// ---------------------------------------------------------------- diagnostics
// Ten reduced values: 7 sums (v1, v2, G11, G12, G21, G22, energy density),
// min J, max J, max |F - I|_F. Per-block partials, then one block combines them
// in a fixed order, so the result does not depend on scheduling.
constexpr int DIAG_THREADS = 256;
constexpr int DIAG_MAX_BLOCKS = 1024;

struct Red {
    double s[7];
    double jmin, jmax, gmax;
};

static __device__ __forceinline__ void red_combine(Red &r, const Red &o)
{
    for (int i = 0; i < 7; ++i) r.s[i] += o.s[i];
    r.jmin = fmin(r.jmin, o.jmin);
    r.jmax = fmax(r.jmax, o.jmax);
    r.gmax = fmax(r.gmax, o.gmax);
}

static __device__ Red block_reduce(Red r)
{
    __shared__ double sh[DIAG_THREADS / 32][10];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int off = 16; off > 0; off >>= 1) {
        Red o;
        for (int i = 0; i < 7; ++i) o.s[i] = __shfl_down_sync(0xffffffffu, r.s[i], off);
        o.jmin = __shfl_down_sync(0xffffffffu, r.jmin, off);
        o.jmax = __shfl_down_sync(0xffffffffu, r.jmax, off);
        o.gmax = __shfl_down_sync(0xffffffffu, r.gmax, off);
        red_combine(r, o);
    }
    if (lane == 0) {
        for (int i = 0; i < 7; ++i) sh[w][i] = r.s[i];
        sh[w][7] = r.jmin;
        sh[w][8] = r.jmax;
        sh[w][9] = r.gmax;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int ww = 1; ww < DIAG_THREADS / 32; ++ww) {
            Red o;
            for (int i = 0; i < 7; ++i) o.s[i] = sh[ww][i];
            o.jmin = sh[ww][7];
            o.jmax = sh[ww][8];
            o.gmax = sh[ww][9];
            red_combine(r, o);
        }
    }
    return r;
}

template <typename T>
__global__ void __launch_bounds__(DIAG_THREADS) k_diag_partial(const DiagArgs a)
{
    const int nx = a.L.nx, ny = a.L.ny;
    const long long N = (long long)nx * ny;
    const T *f = static_cast<const T *>(a.f);
    Red r;
    for (int i = 0; i < 7; ++i) r.s[i] = 0.0;
    r.jmin = DBL_MAX;
    r.jmax = -DBL_MAX;
    r.gmax = 0.0;
    for (long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        int x, y;
        node_xy(n, nx, x, y);
        double S[6];
        node_sums<T, 0, 6>(f, a.L, x, y, S);
        const double v1 = S[0] - a.hb1, v2 = S[1] - a.hb2;
        const double dJ = S[2] + S[5] + (S[2] * S[5] - S[3] * S[4]);
        r.s[0] += v1;
        r.s[1] += v2;
        for (int m = 0; m < 4; ++m) r.s[2 + m] += S[2 + m];
        r.s[6] += 0.5 * (v1 * v1 + v2 * v2) + energy_ofs(a.m.law, S[2], S[3], S[4], S[5], law_at(a.m, n));
        const double J = 1.0 + dJ;
        r.jmin = fmin(r.jmin, J);
        r.jmax = fmax(r.jmax, J);
        r.gmax = fmax(r.gmax, S[2] * S[2] + S[3] * S[3] + S[4] * S[4] + S[5] * S[5]);
    }
    r.gmax = sqrt(r.gmax);  // the root of the largest square: the rounded root is monotone
    r = block_reduce(r);
    if (threadIdx.x == 0) {
        double *p = a.partial + (long long)blockIdx.x * 10;
        for (int i = 0; i < 7; ++i) p[i] = r.s[i];
        p[7] = r.jmin;
        p[8] = r.jmax;
        p[9] = r.gmax;
    }
}

__global__ void __launch_bounds__(DIAG_THREADS) k_diag_final(const DiagArgs a, int nblocks)
{
    Red r;
    for (int i = 0; i < 7; ++i) r.s[i] = 0.0;
    r.jmin = DBL_MAX;
    r.jmax = -DBL_MAX;
    r.gmax = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
        const double *p = a.partial + (long long)b * 10;
        Red o;
        for (int i = 0; i < 7; ++i) o.s[i] = p[i];
        o.jmin = p[7];
        o.jmax = p[8];
        o.gmax = p[9];
        red_combine(r, o);
    }
    r = block_reduce(r);
    if (threadIdx.x == 0) {
        const double N = (double)a.L.nx * (double)a.L.ny;
        a.out[0] = r.s[0];
        a.out[1] = r.s[1];
        a.out[2] = 1.0 + r.s[2] / N;
        a.out[3] = r.s[3] / N;
        a.out[4] = r.s[4] / N;
        a.out[5] = 1.0 + r.s[5] / N;
        a.out[6] = a.dx * a.dx * r.s[6];
        a.out[7] = r.jmin;
        a.out[8] = r.jmax;
        a.out[9] = r.gmax;
    }
}

// ---------------------------------------------------------------- launchers
static int grid_for(long long n, int threads)
{
    long long g = (n + threads - 1) / threads;
    if (g > 65535LL * 16) g = 65535LL * 16;
    return (int)(g < 1 ? 1 : g);
}

cudaError_t launch_init(int storage, const InitArgs &a, cudaStream_t st)
{
    // the kernel writes rows [y0, y1) and reads U0 around them: a range
    // outside the lattice is an error, an empty one a no-op
    if (a.y0 < 0 || a.y1 > a.L.ny || a.y1 < a.y0) return cudaErrorInvalidValue;
    if (a.y1 == a.y0) return cudaSuccess;
    // two warps to a block: 14 instead of 12 fit an SM's registers (FP32)
    const int g = grid_for((long long)a.L.nx * (a.y1 - a.y0), 64);
    return with_storage(storage, [&](auto tag) {
        using R = typename std::conditional<sizeof(tag) == 8, double, float>::type;
        k_init<decltype(tag)><<<g, 64, 0, st>>>(a, init_const<R>(a));
        return cudaGetLastError();
    });
}

cudaError_t launch_read(int storage, const ReadArgs &a, cudaStream_t st)
{
    const int g = grid_for((long long)a.L.nx * a.L.ny, 128);
    return with_storage(storage, [&](auto tag) {
        using T = decltype(tag);
        const bool state = a.U || a.P || a.sigma;
        if (state && a.u)
            k_read<T, true, true><<<g, 128, 0, st>>>(a);
        else if (state)
            k_read<T, true, false><<<g, 128, 0, st>>>(a);
        else
            k_read<T, false, true><<<g, 128, 0, st>>>(a);
        return cudaGetLastError();
    });
}

int diag_blocks(const Layout &L)
{
    const long long n = (long long)L.nx * L.ny;
    long long b = (n + DIAG_THREADS - 1) / DIAG_THREADS;
    if (b > DIAG_MAX_BLOCKS) b = DIAG_MAX_BLOCKS;
    return (int)(b < 1 ? 1 : b);
}

cudaError_t launch_diag(int storage, const DiagArgs &a, cudaStream_t st)
{
    const int nb = diag_blocks(a.L);
    with_storage(storage, [&](auto tag) {
        k_diag_partial<decltype(tag)><<<nb, DIAG_THREADS, 0, st>>>(a);
        return 0;
    });
    k_diag_final<<<1, DIAG_THREADS, 0, st>>>(a, nb);
    return cudaGetLastError();
}

cudaError_t launch_mu_plane(int storage, const double *mu, void *plane, const Layout &L, cudaStream_t st)
{
    const long long N = (long long)L.nx * L.ny;
    const int grid = (int)((N + 255) / 256 < 4096 ? (N + 255) / 256 : 4096);
    if (storage == STORE_F64)
        k_mu_plane<double><<<grid, 256, 0, st>>>(mu, static_cast<double *>(plane), L);
    else
        k_mu_plane<float><<<grid, 256, 0, st>>>(mu, static_cast<float *>(plane), L);
    return cudaGetLastError();
}

constexpr int STATS_BLOCKS = 256;

__global__ void __launch_bounds__(256) k_field_stats(const double *v, long long n, double *partial)
{
    __shared__ double smin[256], smax[256], sbad[256];
    double lo = DBL_MAX, hi = -DBL_MAX, bad = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double x = v[i];
        if (!isfinite(x)) {
            bad += 1.0;
        } else {
            lo = fmin(lo, x);
            hi = fmax(hi, x);
        }
    }
    smin[threadIdx.x] = lo;
    smax[threadIdx.x] = hi;
    sbad[threadIdx.x] = bad;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            smin[threadIdx.x] = fmin(smin[threadIdx.x], smin[threadIdx.x + s]);
            smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[threadIdx.x + s]);
            sbad[threadIdx.x] += sbad[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partial[3 * blockIdx.x] = smin[0];
        partial[3 * blockIdx.x + 1] = smax[0];
        partial[3 * blockIdx.x + 2] = sbad[0];
    }
}

cudaError_t launch_field_stats(const double *v, long long n, double out[3], cudaStream_t st)
{
    double *partial = nullptr;
    cudaError_t e = cudaMallocAsync((void **)&partial, 3 * STATS_BLOCKS * sizeof(double), st);
    if (e != cudaSuccess) return e;
    k_field_stats<<<STATS_BLOCKS, 256, 0, st>>>(v, n, partial);
    double h[3 * STATS_BLOCKS];
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, partial, sizeof h, cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(partial, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    out[0] = DBL_MAX;
    out[1] = -DBL_MAX;
    out[2] = 0.0;
    for (int b = 0; b < STATS_BLOCKS; ++b) {
        out[0] = fmin(out[0], h[3 * b]);
        out[1] = fmax(out[1], h[3 * b + 1]);
        out[2] += h[3 * b + 2];
    }
    return cudaSuccess;
}

} // namespace tlv
