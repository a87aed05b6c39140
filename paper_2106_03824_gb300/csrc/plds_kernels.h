// The persistent kernels of the batched and the serving form, each compiled in a
// translation unit of its own, and the records they share with the host runtime.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "plds_types.h"

namespace pl {

// A small batch in one launch (insertion, insertion by the jump variant, deletion).
__global__ void k_whole_insert(const __grid_constant__ GraphCtx g);
__global__ void k_whole_jump(const __grid_constant__ GraphCtx g);
__global__ void k_whole_delete(const __grid_constant__ GraphCtx g);

// Batched form: one graph's work of a round.
struct SetItem {
    GraphCtx half[2];  // 0: insertion half, 1: deletion half
};
constexpr int kSetThreads = 256;
constexpr int kSetStageShift = 1;
// Blocks per large graph.  Rounds of 16 / 64 / 128 / 512 graphs of 1e3-1e5 vertices, level reads
// included, with 4: 4.4 / 7.7 / 9.2 / 23.6 ms, with 8: 3.3 / 5.4 / 7.0 / 25.6, with 16: 2.7 / 6.3 /
// 11.2 / 32.7 (one block per graph: 10.7 / 19.7 / 23.6 / 42.8).
constexpr int kSetCluster = 8;

// A round's work: graphs items[0..large) for the clusters, items[large..count) for
// single blocks; next[0] and next[1] are the two queues' heads, slot[c] the graph that
// cluster c works on.
struct SetQueue {
    int32_t next[2];
    int32_t large, count;
    int32_t slot[1024];
};

__global__ void k_batch_set(const SetItem *items, SetQueue *q);
__global__ void k_batch_set_cluster(const SetItem *items, SetQueue *q);

// Serving form.
enum : int32_t { kSlotFree = 0, kSlotReady = 1, kSlotDone = 2 };
enum : int32_t { kReqInsert = 0, kReqDelete = 1, kReqCoreness = 2 };
enum : int32_t { kExitNone = 0, kExitIdle = 1, kExitNeedPool = 2, kExitError = 3, kExitLeaving = 4 };
constexpr int kMaxSeg = 64;  // requests merged into one batch at most

struct alignas(64) ReqSlot {
    int32_t state;  // kSlot*
    int32_t op;     // kReq*
    int64_t B;
    const int32_t *edges;  // device-accessible
    double *out;           // device-accessible (coreness queries)
    int64_t ticket;
    int64_t merge_cap;  // edges one merged batch may hold (0: never merge)
    // written by the device
    int32_t status;   // device error bits
    int32_t batch_n;  // requests in the batch this one was applied in
    int64_t batch_first;  // ticket of that batch's first request
    uint64_t t_begin, t_end;  // device globaltimer
    unsigned long long pool_top;  // adjacency slots handed out after the request
    unsigned long long st[kStCount];
    unsigned long long valid;
};

struct ServeCtl {  // device memory
    int32_t exit_reason;
    int32_t cmd;
    int64_t head;        // next slot sequence number
    int32_t stamp_next;  // stamps of the next request start here
    int32_t nseg;        // requests in the current batch (0: a query or an unmerged request)
    unsigned long long grow_total;
    int64_t seg_total;   // edges gathered (after rejected requests are dropped)
    ReqSlot cur;         // the head request (copied from the ring)
    const int2 *seg_ptr[kMaxSeg];
    int64_t seg_off[kMaxSeg + 1];
    int32_t seg_bad[kMaxSeg];
};

// Why and where the loop stopped, written into pinned host memory as it leaves
// (reason kExitNone: not written, an error stopped it).  An idle loop first writes
// kExitLeaving and looks at its slot once more: either it sees a request marked ready
// meanwhile, takes the mark back and serves it, or the host, which reads the reason after
// marking its slot, sees that the loop is leaving.
struct ServeExit {
    int32_t reason;
    int32_t stamp_next;
    int64_t head;
    unsigned long long grow_total;
};

struct ServeArgs {
    ReqSlot *ring;  // device pointer of the pinned ring
    int32_t slots;
    int64_t idle_ns;
    ServeCtl *sc;
    const double *powtab;
    int2 *ebuf;  // gathered edges of a merged batch [max_batch]
    ServeExit *exit;
};

__global__ void k_serve(const __grid_constant__ GraphCtx base, const ServeArgs a);

}  // namespace pl
