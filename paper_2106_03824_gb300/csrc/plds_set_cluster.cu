// Kernel of the batched form (plds_set_*): the graphs that a cluster of blocks takes.
#include "plds_set.cuh"

namespace pl {

__global__ void __launch_bounds__(kSetThreads, 2)
    k_batch_set_cluster(const SetItem *__restrict__ items, SetQueue *q) {
    extern __shared__ int32_t sh[];
    __shared__ GraphCtx gsh;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int32_t rank, cid;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%clusterid.x;" : "=r"(cid));
    const int32_t large = q->large;
    for (;;) {
        ClusterTeam::barrier();  // the slot's last readers are done
        if (rank == 0 && threadIdx.x == 0) q->slot[cid] = atomicAdd(&q->next[0], 1);
        ClusterTeam::barrier();
        const int i = ld_volatile(&q->slot[cid]);
        if (i >= large) break;
        ClusterTeam T{nullptr, rank, kSetCluster};
        set_graph(T, gsh, items[i], sh, [] { ClusterTeam::barrier(); });
    }
}

}  // namespace pl
