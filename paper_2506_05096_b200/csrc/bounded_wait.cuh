// Warp-uniform election and the bounded mbarrier wait shared by the tcgen05 kernels.
#pragma once

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace astraea {

constexpr uint64_t kWaitLimitNs = 1000000000ull; // bounded waits: one second

__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile("{\n\t.reg .pred px;\n\telect.sync _|px, 0xffffffff;\n\tselp.u32 %0, 1, 0, px;\n\t}" : "=r"(pred));
    return pred != 0;
}

// Bounded mbarrier wait.  Gives up after the limit, or at once when another wait of this CTA
// already gave up; the caller carries on (its results are void, the error word says so).
// CLUSTER: for arrivals from other CTAs, relaxed at cluster scope (see mbar_try_wait_cluster).
template <bool CLUSTER = false>
__device__ __forceinline__ void wait_bar(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *err_word,
                                         uint64_t limit_ns = kWaitLimitNs) {
    auto arrived = [&] { return CLUSTER ? ptx::mbar_try_wait_cluster(bar, parity) : ptx::mbar_try_wait(bar, parity); };
    if (arrived()) return;
    if (*abort_flag) return;
    const uint64_t t0 = ptx::globaltimer_ns();
    uint32_t spins = 0;
    while (!arrived()) {
        if ((++spins & 255u) == 0) {
            if (*abort_flag) return;
            if (ptx::globaltimer_ns() - t0 > limit_ns) {
                *abort_flag = 1;
                atomicExch(err_word, kErrTimeout);
                return;
            }
        }
    }
}

// Bounded wait for copies (or MMAs) of this CTA that are under way, before its memory is given up: it does not mind that
// the CTA has given up, and returns after the limit all the same.
__device__ __forceinline__ void drain_bar(uint32_t bar, uint32_t parity, uint64_t limit_ns = kWaitLimitNs) {
    if (ptx::mbar_try_wait(bar, parity)) return;
    const uint64_t t0 = ptx::globaltimer_ns();
    while (!ptx::mbar_try_wait(bar, parity) && ptx::globaltimer_ns() - t0 <= limit_ns) {}
}

}  // namespace astraea
