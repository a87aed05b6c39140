// Kernel of the batched form (plds_set_*).
#include "plds_device.cuh"
#include "plds_kernels.h"

namespace pl {

__global__ void __launch_bounds__(kSetThreads, 2)
    k_batch_set(const SetItem *__restrict__ items, int32_t count, int32_t *next) {
    extern __shared__ int32_t sh[];
    __shared__ GraphCtx gsh;
    __shared__ int32_t idx;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) idx = atomicAdd(next, 1);
        __syncthreads();
        const int i = idx;
        if (i >= count) return;
        for (int h = 0; h < 2; ++h) {
            __syncthreads();
            const int32_t *src = reinterpret_cast<const int32_t *>(&items[i].half[h]);
            int32_t *dst = reinterpret_cast<int32_t *>(&gsh);
            for (int k = threadIdx.x; k < (int)(sizeof(GraphCtx) / 4); k += blockDim.x) dst[k] = src[k];
            __syncthreads();
            // the host reads both halves' control blocks: clear them even for an empty half
            int32_t *cw = reinterpret_cast<int32_t *>(gsh.ctl);
            for (int k = threadIdx.x; k < (int)(sizeof(Ctl) / 4); k += blockDim.x) cw[k] = 0;
            if (gsh.B == 0) continue;  // an empty half changes nothing
            for (int64_t k = threadIdx.x; k < gsh.hcap; k += blockDim.x) gsh.hset[k] = kEmptyKey;
            if (gsh.op == kOpInsert)
                for (int k = threadIdx.x; k <= gsh.K; k += blockDim.x) gsh.bins[k] = 0;
            __syncthreads();
            BlockTeam T{gsh.ctl};
            run_batch(T, gsh, BatchIn{gsh.edges, gsh.B, gsh.op, gsh.stamp_base}, sh, kSetStageShift);
            __syncthreads();
            if (ld_volatile(&gsh.ctl->err) != 0) break;  // the host resolves it and reruns this graph
        }
    }
}

}  // namespace pl
