// Grid-wide meeting points inside one cooperative kernel (every block
// resident), with bounded waits.
#pragma once

#include "device.cuh"

namespace packsell {

struct Meet {
    unsigned *arrived, *left;  // 0 between launches
    int *timeout;              // set when a wait ran out: later launches return at once
};

constexpr unsigned kMeetPolls = 1u << 22;

// Wait (bounded) until all blocks have arrived `round` times in this launch;
// false when the wait ran out. What every thread of every block wrote before
// it is visible to every thread after it (through loads that are not marked
// read-only: no __ldg, no const __restrict__ on memory that the kernel writes).
__device__ __forceinline__ bool meet(const Meet &m, unsigned round) {
    __shared__ bool ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(m.arrived, 1u);
        const unsigned all = gridDim.x * round;
        unsigned polls = 0;
        while (*(volatile unsigned *)m.arrived < all && ++polls < kMeetPolls) {
        }
        ok = polls < kMeetPolls;
        if (!ok) *m.timeout = PACKSELL_ERR_TIMEOUT;
        __threadfence();
    }
    __syncthreads();
    return ok;
}

// Called by every block after its last meet(): the last one puts the counters back.
__device__ __forceinline__ void meet_done(const Meet &m) {
    if (threadIdx.x == 0 && atomicAdd(m.left, 1u) == gridDim.x - 1u) {
        *m.arrived = 0u;
        *m.left = 0u;
    }
}

// A cooperative launch: fails instead of running when not every block fits.
template <typename... KArgs, typename... Args>
cudaError_t launch_coop(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem,
                        cudaStream_t s, Args &&...args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace packsell
