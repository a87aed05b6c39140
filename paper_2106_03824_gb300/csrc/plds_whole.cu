// Kernels of small batches: the steps before the level rounds and the rounds in one
// cooperative launch, grid barriers between the steps.
#include "plds_device.cuh"
#include "plds_kernels.h"

namespace pl {

template <int kWhat>
__device__ __forceinline__ void whole_batch(const GraphCtx &g) {
    extern __shared__ int32_t sh[];
    GridTeam T{g.ctl, g.wait_limit_ns, g.barrier_sleep_ns};
    run_batch<GridTeam, false, kWhat>(T, g, BatchIn{g.edges, g.B, g.op, g.stamp_base, g.hcap}, sh, 0);
}

__global__ void __launch_bounds__(512) k_whole_insert(const __grid_constant__ GraphCtx g) {
    whole_batch<kInsertRounds>(g);
}

// (The second launch bound as for the rounds kernel.)
__global__ void __launch_bounds__(512, 1) k_whole_jump(const __grid_constant__ GraphCtx g) {
    whole_batch<kJumpRounds>(g);
}

__global__ void __launch_bounds__(512) k_whole_delete(const __grid_constant__ GraphCtx g) {
    whole_batch<kDeleteRounds>(g);
}

}  // namespace pl
