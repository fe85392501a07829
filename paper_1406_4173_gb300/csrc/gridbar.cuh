// Barrier between the phases of a cooperative launch.
#pragma once
#include "common.cuh"

namespace bcpp {

// words at the start of a kernel's control block (zeroed before the launch)
constexpr int CTL_BAR = 0, CTL_GEN = 1, CTL_ABORT = 2, CTL_WORDS = 8;
constexpr unsigned GRID_SPIN_MAX = 1u << 28;   // polls before the barrier gives up

// Barrier over all blocks of the cooperative launch.  false: gave up (never with co-resident blocks).
__device__ __forceinline__ bool grid_barrier(uint32_t* ctl, uint32_t* flags) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile uint32_t* gen = ctl + CTL_GEN;
        volatile uint32_t* ab = ctl + CTL_ABORT;
        const uint32_t g = *gen;
        __threadfence();
        if (atomicAdd(ctl + CTL_BAR, 1u) == gridDim.x - 1) {
            ctl[CTL_BAR] = 0u;
            __threadfence();
            atomicAdd(ctl + CTL_GEN, 1u);
        } else {
            unsigned polls = 0;
            while (*gen == g && *ab == 0u) {
                __nanosleep(20);
                if (++polls == GRID_SPIN_MAX) {
                    atomicOr(&flags[FLAG_TIMEOUT], 1u);
                    atomicExch(ctl + CTL_ABORT, 1u);
                }
            }
        }
        s_ok = *ab == 0u;
        __threadfence();
    }
    __syncthreads();
    return s_ok != 0;
}

}  // namespace bcpp
