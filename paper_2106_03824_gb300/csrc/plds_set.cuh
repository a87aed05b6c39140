// One graph's round of the batched form, by a block or a cluster of blocks.
#pragma once
#include "plds_device.cuh"
#include "plds_kernels.h"

namespace pl {

// The insertion half, then the deletion half, of item; gsh: the block's shared copy of
// the half's context; barrier: the team's plain barrier.
template <class Team, class Bar>
__device__ __forceinline__ void set_graph(Team &T, GraphCtx &gsh, const SetItem &item, int32_t *sh, Bar barrier) {
    for (int h = 0; h < 2; ++h) {
        barrier();
        const int32_t *src = reinterpret_cast<const int32_t *>(&item.half[h]);
        int32_t *dst = reinterpret_cast<int32_t *>(&gsh);
        for (int k = threadIdx.x; k < (int)(sizeof(GraphCtx) / 4); k += blockDim.x) dst[k] = src[k];
        __syncthreads();
        // the host reads both halves' control blocks: clear them even for an empty half
        int32_t *cw = reinterpret_cast<int32_t *>(gsh.ctl);
        for (int k = T.tid(); k < (int)(sizeof(Ctl) / 4); k += T.nthreads()) cw[k] = 0;
        if (gsh.B == 0) continue;  // an empty half changes nothing
        for (int64_t k = T.tid(); k < gsh.hcap; k += T.nthreads()) gsh.hset[k] = kEmptyKey;
        if (gsh.op == kOpInsert)
            for (int k = T.tid(); k <= gsh.K; k += T.nthreads()) gsh.bins[k] = 0;
        barrier();
        T.ctl = gsh.ctl;
        run_batch(T, gsh, BatchIn{gsh.edges, gsh.B, gsh.op, gsh.stamp_base, gsh.hcap}, sh, kSetStageShift);
        barrier();
        const int32_t err = ld_volatile(&gsh.ctl->err);
        barrier();
        if (err != 0) break;  // the host resolves it and reruns this graph
    }
}

}  // namespace pl
