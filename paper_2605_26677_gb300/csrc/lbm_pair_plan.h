// lbm_pair_plan.h -- which warp of the two-step kernel (k_pair) takes which
// task. Plain C++: the kernel and a test on the CPU compile the same function.
#pragma once

#ifdef __CUDACC__
#define TLV_HD __host__ __device__ __forceinline__
#else
#define TLV_HD inline
#endif

namespace tlv {

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

} // namespace tlv
