// Protocols on the reduction cells of a handle (DeviceState): who may publish a call's sums and clear its cells.
#pragma once
#include "eoq_device.cuh"
#include "eoq_internal.h"

namespace eoq {

// Every thread of every block calls this after the block's last use of the handle's reduction cells (no early
// returns before it).  True in thread 0 of the block that arrives last: by then every block has read what it
// needed and added what it had to add, so that thread may publish the sums and must put the cells back to zero.
__device__ __forceinline__ bool last_block_done(DeviceState *dev)
{
    __shared__ unsigned last_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned t = atomicAdd(&dev->ticket, 1u);
        last_s = (t == gridDim.x - 1) ? 1u : 0u;
        if (last_s) {
            __threadfence();
            dev->ticket = 0;
        }
    }
    __syncthreads();
    return last_s != 0 && threadIdx.x == 0;
}

// For kernels that only read what the launch shares (maxima, a step counter): one thread of every block calls this once
// its values have arrived (they went through shared memory and a barrier).  True in the block that comes last, whose
// thread may then change them.  The counter wraps to zero by itself; taken early, its latency hides behind the block's
// work.
__device__ __forceinline__ bool last_reader(DeviceState *dev)
{
    const unsigned blocks = gridDim.x * gridDim.y;
    return atomicInc(&dev->ticket, blocks - 1) == blocks - 1;
}

}  // namespace eoq
