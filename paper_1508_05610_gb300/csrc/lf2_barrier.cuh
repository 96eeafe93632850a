#pragma once
// lf2_barrier.cuh -- the grid barrier of the cooperative multi-step kernels.
//
// One 64-bit word in the field's scratch, zeroed before each launch: the low 63 bits count arrivals
// and are never reset, the top bit says that a block gave up.  Barrier number b (from 0) is complete
// when the count has reached (b + 1) * blocks, so the last arrival releases the waiters by itself, and
// one load tells a waiter both the count and the flag.  (A counter that the last block reset before it
// advanced a generation, a fence on each side and a second load for the error flag made a barrier
// 1.2 us longer.)  Every access is to the whole 64-bit word: the memory model orders a release and an
// acquire only when the two accesses overlap completely.
//
// Waits are bounded: a cooperative launch keeps every block resident, so real waits take
// microseconds; after kBarrierPolls polls of about half a microsecond (about a second) the waiter sets the
// flag, every block stops and the host reports it (lf2_field_check).  The flag goes with the launch's
// word; a status word beside it, which launches leave alone, keeps the event until it is reported.
#include <cuda_runtime.h>

namespace lf2 {
namespace {

constexpr unsigned kBarrierPolls = 1u << 21;
constexpr unsigned long long kBarrierGaveUp = 1ull << 63;

// All of the block's earlier writes are visible to every block that has waited for this barrier.
__device__ __forceinline__ void grid_arrive(unsigned long long *bar) {
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(bar) : "memory");
}

// False when the wait ran out after polls_max polls, here or in another block.
__device__ __forceinline__ bool grid_wait(unsigned long long *bar, unsigned long long *status, unsigned long long target,
                                          unsigned polls_max) {
    __shared__ int s_ok;
    if (threadIdx.x == 0) {
        int ok = 1;
        unsigned polls = 0;
        while (true) {
            unsigned long long v;
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(bar) : "memory");
            if (v & kBarrierGaveUp) {
                ok = 0;
                break;
            }
            if (v >= target && polls_max) break;
            if (++polls > polls_max) {
                asm volatile("red.relaxed.gpu.global.or.b64 [%0], %1;" ::"l"(bar), "l"(kBarrierGaveUp) : "memory");
                asm volatile("red.relaxed.gpu.global.or.b64 [%0], 1;" ::"l"(status) : "memory");
                ok = 0;
                break;
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

}  // namespace
}  // namespace lf2
