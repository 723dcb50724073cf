// lbm_pair_plan.h -- which lattices the two-step kernel (k_pair) takes, how it
// cuts them into tasks, and which warp takes which. Plain C++: the library, the
// kernel and a test on the CPU compile the same functions.
#pragma once
#include <algorithm>

#ifdef __CUDACC__
#define TLV_HD __host__ __device__ __forceinline__
#else
#define TLV_HD inline
#endif

namespace tlv {

constexpr int PAIR_VEC = 4, PAIR_COLUMNS = 30 * PAIR_VEC;  // nodes per lane, columns per strip

// Tasks: strips of PAIR_COLUMNS columns, each cut into nlong chunks of hlong
// rows and then chunks of hend rows
struct PairPlan {
    int nstrip, nchunk;
    int nlong, hlong, hend;
};

// rows [ya, yb) of a chunk
TLV_HD void pair_rows(const PairPlan &p, int ny, int chunk, int &ya, int &yb)
{
    const int over = chunk > p.nlong ? chunk - p.nlong : 0;  // short chunks before this one
    ya = (chunk - over) * p.hlong + over * p.hend;
    yb = ya + (chunk < p.nlong ? p.hlong : p.hend);
    if (yb > ny) yb = ny;
}

// the i-th chunk to be taken: those of the bottom and top rows, whose edge
// rules take longest, first
TLV_HD int pair_chunk(const PairPlan &p, int i) { return i == 0 ? 0 : i == 1 ? p.nchunk - 1 : i - 1; }

// Tasks of one of `warps` warps, from the launch's counter (claim() adds one and
// returns the old value; the lanes get it by wait()): claimed one task ahead, so
// that the counter's latency passes during the task, but not where there is a
// warp for every task. The blocks of a launch that no other launch waits for
// start one after another: the early warps would claim two tasks each and half
// the warps none (2048^2, lbm_step(2): 334 us a pass, now 241; in the middle of
// a long call, where all blocks are placed when the tasks begin, 217).
template <typename Claim, typename Wait, typename Run>
TLV_HD void pair_tasks(unsigned warps, unsigned ntask, Claim claim, Wait wait, Run run)
{
    unsigned t = wait(claim());
    while (t < ntask) {
        const unsigned next = ntask > warps ? claim() : ntask;
        run((int)t);
        t = wait(next);
    }
}

// What plan and choice depend on
struct PairLattice {
    int nx, ny;
    bool log_law, heavy_law;  // log-NH; a law of the isochoric invariants (MR, Yeoh, Gent)
    bool xper, yper;          // periodic in x, y
    bool ytraction;           // a traction edge at the bottom or top
    int warps;                // resident warps of the kernel
};

// Rows per task. us per step, FP32, NH unless named.
// Where tasks of 16 rows come in more than three rounds of one per warp: 16,
// or 24 from 16 rounds on, and 6 for about the last two rounds, which leave
// the warps idle for less at the launch's end (16 rows throughout / this:
// 4096 x 2048 clamped 194.5 / 187, 4096^2 377 / 370, 8192^2 1386 / 1366).
// Smaller lattices: one task per warp (2049^2 with a traction top 114, with 4
// rows 132; 250 x 6000 with traction edges 60, 70). Only where the tasks of a
// traction bottom or top, which take longest, can be shared out among many
// strips, and x is not periodic (whose wrapped columns each task at the sides
// copies): 4 rows, 6 from 20 rows a warp on, 12 from 30 on with the heavy laws
// (traction edges, one task per warp / this: 8197 x 257 64.8 / 59.9, Gent 93.4 /
// 78.7; 4899 x 613 86.2 / 82.1, MR 121 / 101; 2449^2 158 / 150, Gent 208 / 193).
inline PairPlan pair_plan(const PairLattice &l)
{
    PairPlan p{};
    p.nstrip = (l.nx + PAIR_COLUMNS - 1) / PAIR_COLUMNS;
    auto tasks = [&](int h) { return (long long)p.nstrip * ((l.ny + h - 1) / h); };
    if (tasks(16) > 3LL * l.warps) {
        p.hlong = tasks(16) > 16LL * l.warps ? 24 : 16;
        p.hend = 6;
        const int tail = std::min(l.ny, (int)((p.hlong == 16 ? 2.0 : 1.5) * l.warps / p.nstrip * p.hend));
        p.nlong = (l.ny - tail) / p.hlong;
        p.nchunk = p.nlong + (l.ny - p.nlong * p.hlong + p.hend - 1) / p.hend;
        return p;
    }
    int h = std::max(4, (int)((long long)l.ny * p.nstrip / l.warps));
    while (tasks(h) > l.warps && h < l.ny) ++h;
    if (l.ytraction && !l.xper && p.nstrip >= 8 && h >= 11) h = h < 20 ? 4 : l.heavy_law && h >= 30 ? 12 : 6;
    p.hlong = h;
    p.nlong = p.nchunk = (l.ny + h - 1) / h;
    return p;
}

// Whether k_pair beats the step kernel on a lattice: no, yes, or a guess that
// the context's first call of enough steps replaces by a comparison
enum PairAdvice { PAIR_NO, PAIR_GUESS_NO, PAIR_GUESS_YES, PAIR_YES };

// Both kernels were timed on 2500 lattices of 1 to 12 M nodes, 24 to 750000
// nodes wide, with twelve kinds of edges and every law, from a wave field and
// from rest (step kernel / k_pair, the better task order of the former):
// - periodic x below 130 columns loses (122 x 36000 0.81, 60 x 73000 0.85),
//   as do fewer than 24 rows between edges (500000 x 12 0.89);
// - SVK, NH and log-NH win (1.05 to 1.59), but for traction bottoms and tops
//   below 1.5 M nodes (5825 x 182 with periodic x 0.93, 254 x 5821 0.94, 2913 x
//   364 with traction all round 1.08) and strips of rows (200000 x 30 0.94);
// - MR, Yeoh and Gent, whose collisions bound k_pair, win from 8 M nodes on
//   (1.1 to 1.4) and mostly below (0.9 to 1.25), but for a traction bottom or
//   top below 3 M nodes (0.74 to 1.1), narrow lattices and strips of rows (0.6
//   to 1.05); the same lattice varied by up to 0.2 between processes.
inline PairAdvice pair_advice(const PairLattice &l)
{
    const double m = (double)l.nx * l.ny / (1 << 20);
    const bool odd = l.nx < 160 || l.ny < 64;
    if (l.nx < 8 || l.ny < 8 || (l.xper && l.nx < 130) || (!l.yper && l.ny < 24)) return PAIR_NO;
    if (l.heavy_law) {
        if (m >= 8.0 && !odd) return PAIR_YES;
        return odd || (l.ytraction && m < 3.0) ? PAIR_GUESS_NO : PAIR_GUESS_YES;
    }
    if (l.ytraction && (odd || m < 1.5)) return odd || l.xper || l.log_law ? PAIR_GUESS_NO : PAIR_GUESS_YES;
    return odd ? PAIR_GUESS_YES : PAIR_YES;
}

} // namespace tlv
