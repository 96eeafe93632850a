#pragma once
// lf2_barrier.cuh -- the grid barrier of the cooperative multi-step kernels.
//
// One 64-bit word in the field's scratch, zeroed before each launch: the low half counts arrivals
// and is never reset, the high half is an error flag.  Barrier number b (from 0) is complete when
// the count has reached (b + 1) * blocks, so the last arrival releases the waiters by itself, and one
// load tells a waiter both the count and the error.  (A counter that the last block reset before it
// advanced a generation, a fence on each side and a second load for the error flag made a barrier
// 1.2 us longer.)  The count wraps modulo 2^32; a waiter is never more than one barrier behind.
//
// Waits are bounded: a cooperative launch keeps every block resident, so real waits take
// microseconds; after kBarrierPolls polls of about half a microsecond (about a second) the waiter sets the
// flag, every block stops and the host reports it (lf2_field_check).
#include <cuda_runtime.h>

namespace lf2 {
namespace {

constexpr unsigned kBarrierPolls = 1u << 21;

// All of the block's earlier writes are visible to every block that has waited for this barrier.
__device__ __forceinline__ void grid_arrive(unsigned *bar) {
    __syncthreads();
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}

// False when the wait ran out after polls_max polls, here or in another block.
__device__ __forceinline__ bool grid_wait(unsigned *bar, unsigned target, unsigned polls_max) {
    __shared__ int s_ok;
    if (threadIdx.x == 0) {
        int ok = 1;
        unsigned polls = 0;
        while (true) {
            unsigned long long v;
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(bar) : "memory");
            if ((unsigned)(v >> 32) != 0u) {
                ok = 0;
                break;
            }
            if ((int)((unsigned)v - target) >= 0 && polls_max) break;
            if (++polls > polls_max) {
                atomicExch(bar + 1, 1u);
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
