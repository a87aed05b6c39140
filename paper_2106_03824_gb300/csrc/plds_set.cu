// Kernel of the batched form (plds_set_*): the graphs that one block each takes.
#include "plds_set.cuh"

namespace pl {

// Starts next to the cluster kernel (programmatic dependent launch: once every
// cluster is resident) and ends after it.
__global__ void __launch_bounds__(kSetThreads, 2) k_batch_set(const SetItem *__restrict__ items, SetQueue *q) {
    extern __shared__ int32_t sh[];
    __shared__ GraphCtx gsh;
    __shared__ int32_t idx;
    const int32_t count = q->count;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) idx = q->large + atomicAdd(&q->next[1], 1);
        __syncthreads();
        const int i = idx;
        if (i >= count) break;
        BlockTeam T{nullptr};
        set_graph(T, gsh, items[i], sh, [] { __syncthreads(); });
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace pl
