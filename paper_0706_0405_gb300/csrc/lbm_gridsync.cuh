// lbm_gridsync.cuh -- the bounded grid-wide barrier of the persistent batch
// kernels (each translation unit has its own copy of the bound).
#pragma once

#include "lbm_device.cuh"
#include "lbm_ptx.cuh"

namespace lbm {
namespace {

constexpr long long kBarrierCycles = 4000000000LL;  // ~2 s at 2 GHz, then give up
// SM cycles an inter-CTA wait (grid barrier, neighbour wait) lasts before it
// gives up (batch_set_wait_cycles)
__device__ long long g_wait_cycles = kBarrierCycles;

// Bounded grid-wide barrier for a cooperative launch.  Returns false (and
// sets ST_TIMEOUT) if the barrier did not complete in time or another CTA
// has given up (ST_TIMEOUT already set); the decision is the CTA's, taken
// by one thread and passed on by the CTA barrier, so all its threads leave
// together.  The stores of
// the step are ordered before the async-proxy reads (tensor copies) of the
// next step on both sides: every thread fences after its stores, and the
// thread that issues the copies fences after the barrier.
__device__ bool grid_barrier(unsigned* count, volatile unsigned* gen, unsigned* status) {
    __shared__ int ok;
    fence_proxy_async_global();
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        const unsigned g = *gen;
        __threadfence();
        const unsigned arrived = atomicAdd(count, 1u);
        if (arrived == gridDim.x - 1) {
            *count = 0u;
            __threadfence();
            atomicAdd(const_cast<unsigned*>(gen), 1u);
        } else {
            const long long t0 = clock64();
            while (*gen == g) {
                if (clock64() - t0 > g_wait_cycles || (*(volatile unsigned*)status & ST_TIMEOUT)) {
                    atomicOr(status, ST_TIMEOUT);
                    ok = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
        fence_proxy_async_global();
    }
    __syncthreads();
    return ok != 0;
}

}  // namespace
}  // namespace lbm
