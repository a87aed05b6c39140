// Kernel of the serving form (plds_server_*): the device-resident request loop.
#include <cstddef>

#include "plds_device.cuh"
#include "plds_kernels.h"

namespace pl {

// Word-by-word copy that reads through volatile loads (the source may be host memory
// the host is writing, or device memory written by another block).
__device__ __forceinline__ void copy_slot(ReqSlot *dst, const ReqSlot *src) {
    const volatile int32_t *sv = reinterpret_cast<const volatile int32_t *>(src);
    int32_t *dv = reinterpret_cast<int32_t *>(dst);
    for (int k = 0; k < (int)(sizeof(ReqSlot) / 4); ++k) dv[k] = sv[k];
}

// Leader: extend the batch that starts with the head request by the waiting
// requests that follow it (same kind, total edges within the cap).
__device__ void serve_select(const ServeArgs &a, ServeCtl *sc) {
    const ReqSlot &c = sc->cur;
    sc->nseg = 0;
    if (c.op == kReqCoreness || c.merge_cap <= 0 || c.B > c.merge_cap) return;
    int64_t total = c.B;
    sc->seg_ptr[0] = reinterpret_cast<const int2 *>(c.edges);
    sc->seg_off[0] = 0;
    sc->seg_bad[0] = 0;
    int ns = 1;
    for (int j = 1; j < a.slots && ns < kMaxSeg; ++j) {
        const ReqSlot *r = a.ring + ((sc->head + j) % a.slots);
        if (*(volatile const int32_t *)&r->state != kSlotReady) break;
        __threadfence_system();
        const int32_t op = *(volatile const int32_t *)&r->op;
        const int64_t B = *(volatile const int64_t *)&r->B;
        if (op != c.op || total + B > c.merge_cap) break;
        sc->seg_ptr[ns] = reinterpret_cast<const int2 *>(*(const int32_t *volatile *)&r->edges);
        sc->seg_off[ns] = total;
        sc->seg_bad[ns] = 0;
        total += B;
        ++ns;
    }
    sc->seg_off[ns] = total;
    sc->seg_total = total;
    sc->nseg = ns > 1 ? ns : 0;  // a request alone is read in place
}

// Grid: copy the batch's requests into one contiguous edge array; with `check`,
// flag each request holding an id outside [0, n).  Segment offsets are in shared
// memory (s_off[0..ns]).
__device__ void serve_gather(GridTeam &T, const ServeCtl *sc, int ns, const int64_t *s_off, int2 *ebuf, int32_t n,
                             bool check, int32_t *bad) {
    const int64_t total = s_off[ns];
    for (int64_t i = T.tid(); i < total; i += T.nthreads()) {
        int lo = 0, hi = ns - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_off[mid] <= i) lo = mid;
            else hi = mid - 1;
        }
        const int2 uv = sc->seg_ptr[lo][i - s_off[lo]];
        if (check && (uv.x < 0 || uv.x >= n || uv.y < 0 || uv.y >= n)) *(volatile int32_t *)&bad[lo] = 1;
        ebuf[i] = uv;
    }
}

// Key-set entries the current batch uses: a power of two of at least four times its edges,
// as far as the buffer has them (it is sized for max_batch).
__device__ __forceinline__ int64_t serve_hcap(const GraphCtx &base, const ServeCtl *sc) {
    const int64_t B = max((long long)1024, (long long)(*(volatile const int32_t *)&sc->nseg > 0
                                                           ? *(volatile const int64_t *)&sc->seg_total
                                                           : *(volatile const int64_t *)&sc->cur.B));
    return min((long long)base.hcap, 4ll << (64 - __clzll(B - 1)));
}

// Leader: the loop is about to leave.
__device__ __forceinline__ void serve_leave(const ServeArgs &a, const ServeCtl *sc, int32_t reason) {
    volatile ServeExit *x = a.exit;
    x->stamp_next = sc->stamp_next;
    x->head = sc->head;
    x->grow_total = sc->grow_total;
    __threadfence_system();
    x->reason = reason;
}

__global__ void __launch_bounds__(512) k_serve(const __grid_constant__ GraphCtx base, const ServeArgs a) {
    extern __shared__ int32_t sh[];
    __shared__ int64_t s_off[kMaxSeg + 1];
    GridTeam T{base.ctl, base.wait_limit_ns, base.barrier_sleep_ns};
    ServeCtl *sc = a.sc;
    for (;;) {
        // the leader waits for the next slot (bounded by the idle limit)
        if (T.leader()) {
            ReqSlot *r = a.ring + (sc->head % a.slots);
            const uint64_t t0 = global_ns();
            int32_t st;
            while ((st = *(volatile int32_t *)&r->state) != kSlotReady && global_ns() - t0 < (uint64_t)a.idle_ns)
                __nanosleep(256);
            if (st != kSlotReady) {
                *(volatile int32_t *)&a.exit->reason = kExitLeaving;
                __threadfence_system();
                st = *(volatile int32_t *)&r->state;
                if (st == kSlotReady) *(volatile int32_t *)&a.exit->reason = kExitNone;
            }
            if (st == kSlotReady) {
                __threadfence_system();
                copy_slot(&sc->cur, r);
                serve_select(a, sc);
                sc->cmd = 1;
            } else {
                sc->cmd = 0;
                sc->exit_reason = kExitIdle;
                serve_leave(a, sc, kExitIdle);
            }
            __threadfence();
        }
        if (!T.sync()) return;
        if (ld_volatile(&sc->cmd) == 0) return;
        const int64_t hcap = serve_hcap(base, sc);  // (before rejected requests are dropped)
        // a fresh control block and key set for this request (the barrier words stay)
        {
            int32_t *cw = reinterpret_cast<int32_t *>(base.ctl);
            const int first = (int)(offsetof(Ctl, err) / 4);
            for (int k = T.tid() + first; k < (int)(sizeof(Ctl) / 4); k += T.nthreads()) cw[k] = 0;
            for (int64_t k = T.tid(); k < hcap; k += T.nthreads()) base.hset[k] = kEmptyKey;
            for (int k = T.tid(); k <= base.K; k += T.nthreads()) base.bins[k] = 0;
            if (sc->stamp_next + 2 * base.K + 8 >= 0x7fffffff) {  // stamps wrap: clear them
                for (int k = T.tid(); k < base.n; k += T.nthreads()) base.stamp[k] = 0;
            }
        }
        ReqSlot req;
        copy_slot(&req, &sc->cur);
        const int ns = ld_volatile(&sc->nseg);
        if (ns > 0) {  // gather the batch's requests, rejecting those with a bad id
            for (int k = threadIdx.x; k <= ns; k += blockDim.x) s_off[k] = sc->seg_off[k];
            __syncthreads();
            serve_gather(T, sc, ns, s_off, a.ebuf, base.n, true, sc->seg_bad);
            if (!T.sync()) return;
            bool anybad = false;
            for (int k = 0; k < ns; ++k) anybad |= ld_volatile(&sc->seg_bad[k]) != 0;
            if (anybad) {  // gather again without the rejected requests (they keep length 0)
                __syncthreads();
                if (threadIdx.x == 0) {
                    int64_t t = 0;
                    for (int k = 0; k < ns; ++k) {
                        s_off[k] = t;
                        if (!ld_volatile(&sc->seg_bad[k])) t += sc->seg_off[k + 1] - sc->seg_off[k];
                    }
                    s_off[ns] = t;
                }
                __syncthreads();
                if (T.leader()) sc->seg_total = s_off[ns];
                // a zero-length segment is never selected by the search below (offsets
                // equal), so the remaining requests' edges land contiguously
                serve_gather(T, sc, ns, s_off, a.ebuf, base.n, false, sc->seg_bad);
            }
        }
        if (!T.sync()) return;
        int32_t sbase = sc->stamp_next;
        if (sbase + 2 * base.K + 8 >= 0x7fffffff) sbase = 1;
        const uint64_t t_begin = global_ns();
        if (req.op == kReqCoreness) {
            for (int64_t v = T.tid(); v < base.n; v += T.nthreads()) {
                int32_t g = -1;
                if (base.deg[v] > 0) g = max((base.level[v] + 1) / base.Lg - 1, 0);
                req.out[v] = g < 0 ? 0.0 : a.powtab[g];
            }
        } else {
            const BatchIn in{ns > 0 ? reinterpret_cast<const int32_t *>(a.ebuf) : req.edges,
                             ns > 0 ? *(volatile const int64_t *)&sc->seg_total : req.B,
                             req.op == kReqInsert ? kOpInsert : kOpDelete, sbase, hcap};
            run_batch(T, base, in, sh, 0);
        }
        const bool ok = T.sync();
        if (T.leader()) {
            const int32_t err = ld_volatile(&base.ctl->err);
            if (err == kErrNeedPool) {  // leave the slots ready; the host grows the pool and relaunches
                sc->exit_reason = kExitNeedPool;
                sc->grow_total = base.ctl->grow_total;
                sc->stamp_next = sbase + base.K + 2;
                serve_leave(a, sc, kExitNeedPool);
            } else {
                const int nr = ns > 0 ? ns : 1;
                const uint64_t t_end = global_ns();
                const unsigned long long top = *(volatile unsigned long long *)base.pool_top;
                for (int j = 0; j < nr; ++j) {
                    ReqSlot *r = a.ring + ((sc->head + j) % a.slots);
                    r->status = (ns > 0 && ld_volatile(&sc->seg_bad[j])) ? kErrInvalidId : err;
                    r->batch_n = nr;
                    r->batch_first = req.ticket;
                    r->t_begin = t_begin;
                    r->t_end = t_end;
                    r->pool_top = top;
                    for (int k = 0; k < kStCount; ++k) r->st[k] = base.ctl->st[k];
                    r->valid = base.ctl->vcount;
                }
                __threadfence_system();
                for (int j = 0; j < nr; ++j)
                    *(volatile int32_t *)&a.ring[(sc->head + j) % a.slots].state = kSlotDone;
                sc->head += nr;
                sc->stamp_next = sbase + base.K + 2;
                if (err) sc->exit_reason = kExitError;
            }
            __threadfence();
        }
        if (!ok) return;
        if (!T.sync()) return;
    }
}

}  // namespace pl
