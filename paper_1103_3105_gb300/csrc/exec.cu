// exec.cu -- the three bulk execution strategies (Section 5).
//
//   K-SET (Section 5.3)  the k-sets run in order with no conflict control
//       inside a level (Property 1).  Three launch shapes:
//         wide level     one full-grid launch per level (kernel boundary =
//                        the level barrier);
//         narrow levels  one thread-block cluster (or one CTA) walks a run of
//                        consecutive narrow levels, separated by cluster (or
//                        CTA) barriers, loading the next level's signatures
//                        and prefetching its rows into L2 before each barrier;
//         persistent     a grid claims level-ordered chunks of one CTA; a
//                        chunk of level k starts once every transaction of
//                        level k-1 has finished (per-level counters).  Chunks
//                        are claimed in increasing order, so every chunk a
//                        waiting CTA depends on is held by a running CTA.
//   PART (Section 5.2)   one thread per non-empty partition runs its
//       transactions serially in timestamp order.
//   (K-SET under the read/write model and PART of debit-credit-only bulks:
//   exec_dc.cu; K-SET of blind increments and SCAN: analysis.cu; K-SET of
//   order-entry-only bulks: exec_oe.cu.)
//   TPL (Section 5.1)    ordered counter locks: an operation whose group has
//       `ticket` earlier operations before its run waits until that many have
//       released the item's counter, then the transaction runs and every
//       operation releases (+1).  Transactions are handed out in timestamp
//       order, so the earliest unfinished one never waits: no deadlock.
// Every wait is bounded by the configured limit; on expiry the kernel sets
// ERR_TIMEOUT in the bulk's error word and returns.
#include <algorithm>
#include <vector>
#include <cooperative_groups.h>

#include "engine.h"
#include "procs.cuh"
#include "ranges.cuh"

namespace cg = cooperative_groups;

namespace gtx {

namespace {

struct LevelArgs {
    DevDB db;
    DevBulk b;
    const BulkCtl *ctl;
    const uint32_t *level_off;
    const uint32_t *type_cut; // per level, where the new-orders and payments start (or null)
    uint32_t k0, k1;          // levels [k0, k1)
    bool orders;              // new-orders are registered (launch_orders follows)
    bool atomic_add;
};

struct KsetArgs {
    DevDB db;
    DevBulk b;
    BulkCtl *ctl;
    const uint32_t *level_off, *chunk_off, *chunk_level;
    const uint32_t *type_cut;   // per level, where the new-orders and payments start (or null)
    uint32_t *done;
    uint64_t spin_limit_ns;
    bool orders;                // new-orders are registered (launch_orders follows)
    bool atomic_add;
};

// waits until *p >= need; false on timeout.  The sleep between polls grows
// with the number of releases still missing (each costs at least one
// hand-off), so a waiter far back in a long chain polls rarely instead of
// flooding L2 with acquire loads.
// per_gap_ns = 0 keeps a short fixed poll (level counters, whose missing
// releases arrive together).
__device__ __forceinline__ bool wait_at_least(const uint32_t *p, uint32_t need, uint64_t limit_ns,
                                              uint32_t per_gap_ns = 0)
{
    uint32_t v = ld_acquire(p);
    if (v >= need) return true;
    const uint64_t t0 = globaltimer();
    uint32_t spins = 0;
    while (v < need) {
        const uint32_t gap = need - v;
        if (per_gap_ns && gap > 1) __nanosleep(gap > 64 ? 64 * per_gap_ns : per_gap_ns * gap);
        else if (++spins > 64) __nanosleep(32);
        if (globaltimer() - t0 > limit_ns) return false;
        v = ld_acquire(p);
    }
    return true;
}

// a bulk known to hold no two conflicting transactions (a 0-set): every
// transaction at once, straight from the bulk's signatures (timestamp order)
__global__ void __launch_bounds__(256) independent_kernel(DevDB db, DevBulk b, const BulkCtl *ctl, bool atomic_add)
{
    if (ctl->err) return;
    const int64_t hb = ctl->base.hist;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < b.n; t += (int64_t)gridDim.x * blockDim.x)
        exec_txn(db, b, view_of(b, (uint32_t)t, hb), atomic_add);
}

// The lanes of one level.  Records are sorted by (level, type) (Appendix
// D's grouping by type), so a level is a run of each type in turn.  With
// type cuts, order-entry's new-orders take 16 lanes each (their line-parallel
// procedure), their run starting on a half warp; every other transaction takes
// one lane.  Lane x maps to the record at `pos`; gl = its index in a group, or
// -1 for a one-lane transaction.
struct LevelLanes {
    uint32_t lo, c8, c9, a1, b1, v;
    __device__ __forceinline__ void make(uint32_t lo_, uint32_t hi, const uint32_t *cut)
    {
        lo = lo_;
        if (!cut) {
            c8 = c9 = hi;
            a1 = b1 = v = hi - lo;
            return;
        }
        c8 = __ldg(&cut[0]);
        c9 = __ldg(&cut[1]);
        a1 = (c8 - lo + kGroup - 1) & ~(uint32_t)(kGroup - 1);   // new-order groups start here
        b1 = a1 + kGroup * (c9 - c8);                            // the types after them
        v = b1 + (hi - c9);
    }
    // false for an idle lane (alignment padding before the groups)
    __device__ __forceinline__ bool at(uint32_t x, uint32_t &pos, int &gl) const
    {
        gl = -1;
        if (x < c8 - lo) { pos = lo + x; return true; }
        if (x < a1) return false;
        if (x < b1) { pos = c8 + (x - a1) / kGroup; gl = (int)((x - a1) % kGroup); return true; }
        pos = c9 + (x - b1);
        return true;
    }
};

// One lane of a level.  Order-entry's procedures run in their first parts
// (launch_orders runs the second ones after the last level).
__device__ __forceinline__ void exec_lane(const DevDB &db, const DevBulk &b, const TxnView &v, int gl, bool first,
                                          bool atomic_add)
{
    if (first && gl < 0 && v.type == GPUTX_T_OE_NEW_ORDER) {
        new_order_first_lane(db, b, v);
    } else if (gl >= 0) {
        int64_t p2, p3;
        const int64_t line = new_order_params(b, v, (uint32_t)gl, p2, p3);
        new_order_first(db, b, v, (uint32_t)gl, p2, p3, line, b.slot_ord[v.t], b.slot_ol[v.t]);
    } else if (first && v.type == GPUTX_T_OE_ORDER_STATUS) {
        order_status_first(db, b, v, __ldg(&v.p[2]));
    } else {
        exec_txn(db, b, v, atomic_add);
    }
}

// The second parts of a bulk's new-orders (orders = true: order rows, lines,
// index entries, outputs), then of its order-statuses, 16 lanes a transaction
// in timestamp order, so slots and outputs are written side by side.  Only
// transactions whose first part ran have a second one: an order that never ran
// has an insert slot all the same, which may lie past the area.  `decided`: every
// new-order with status 0 ran (order_status_kernel set it).
__global__ void __launch_bounds__(256) orders_kernel(DevDB db, DevBulk b, const BulkCtl *ctl, bool orders, bool decided)
{
    if (ctl->err & ~(uint32_t)ERR_CAPACITY) return;
    const int64_t n = b.n_live ? (int64_t)*b.n_live : b.n;
    const uint32_t gl = threadIdx.x & (kGroup - 1);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x / kGroup;
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kGroup; t < n; t += stride) {
        const int32_t type = __ldg(&b.type[t]);
        if (type != (orders ? GPUTX_T_OE_NEW_ORDER : GPUTX_T_OE_ORDER_STATUS) || b.status[t] != 0) continue;
        if (!decided && b.out[t * b.R + (orders ? 2 : 1)] == 0) continue;
        const TxnView v = view_of(b, (uint32_t)t, 0);
        if (orders) {
            NewOrderPart o;
            int64_t p2, p3;
            o.line = new_order_params(b, v, gl, p2, p3);
            o.o_id = b.out[t * b.R];
            o.w = v.p0;
            o.d = v.p0 * OE_DIST + v.p1;
            o.c = o.d * OE_CUST + p2;
            o.oslot = b.base->ord + b.slot_ord[t];
            o.lslot = b.base->ol + b.slot_ol[t];
            o.cnt = (int)p3;
            o.run = true;
            new_order_finish(db, b, v, gl, o);
        } else {
            order_status_finish(db, b, v, gl);
        }
    }
}

// one wide level [level_off[k0], level_off[k0+1]) over the whole grid
__global__ void __launch_bounds__(256) kset_level_kernel(LevelArgs a)
{
    if (a.ctl->err) return;
    const int64_t hb = a.ctl->base.hist;
    const uint32_t lo = __ldg(&a.level_off[a.k0]), hi = __ldg(&a.level_off[a.k0 + 1]);
    LevelLanes L;
    L.make(lo, hi, a.type_cut ? a.type_cut + 2 * (int64_t)a.k0 : nullptr);
    for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < L.v; x += gridDim.x * blockDim.x) {
        uint32_t pos;
        int gl;
        if (L.at(x, pos, gl)) exec_lane(a.db, a.b, view_at(a.b, pos, hb), gl, a.orders, a.atomic_add);
    }
}

// one lane's record of a level, in registers before the level runs
struct LaneRecord {
    TxnView v;
    int64_t p2, p3, line;    // order-entry: parameters 2, 3 and 4 + gl
    uint32_t os, ls;         // insert slots of a new-order
    int gl;                  // index in the lane group, or -1
    bool has;
};

// the record of lane `rank` of a level into L1
__device__ __forceinline__ void lane_prefetch(const DevBulk &b, const LevelLanes &L, uint32_t rank)
{
    uint32_t pos = 0;
    int gl;
    if (!(rank < L.v && L.at(rank, pos, gl))) return;
    if (kDebug && pos >= b.n) return;
    prefetch_record_l1(b, pos);
    if (gl > 0 && 4 + gl < b.P)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(b.rec_params + (int64_t)pos * b.P + 4 + gl));
}

// the loads of lane `rank` of a level; none depends on another
__device__ __forceinline__ LaneRecord lane_record(const DevBulk &b, const LevelLanes &L, uint32_t rank)
{
    LaneRecord r{};
    uint32_t pos = 0;
    r.gl = -1;
    r.has = rank < L.v && L.at(rank, pos, r.gl);
    if (!r.has) return r;
    r.v = record_at(b, pos);
    if (b.P > 3) {
        r.p2 = __ldg(&r.v.p[2]);
        r.p3 = __ldg(&r.v.p[3]);
    } else if (b.P > 2) {
        r.p2 = __ldg(&r.v.p[2]);
    }
    if (r.gl >= 0 && 4 + r.gl < b.P) r.line = __ldg(&r.v.p[4 + r.gl]);
    return r;
}

// a run of narrow levels [k0, k1) on one thread-block cluster (CLUSTER) or
// one CTA.
//
// What bounds it is the latency of a level, so whatever need not lie between
// two barriers does not.  A level's bounds are loaded four levels ahead, its
// records come into L1 three and into registers two levels ahead, its rows into
// L2 and its insert slots into registers one level ahead; order rows, lines,
// index entries and the order-statuses' sums are left to launch_orders, and the
// payments' totals follow the barrier's arrival.  200,003 order-entry
// transactions (which run item by item unless other schemas' share the database),
// 317 a level: 3.5 us a level; 7.3 when the records were
// loaded during the level before and the procedures ran whole (of it 3.0
// without any procedure, 1.2 the index entry's compare-and-swap).
template <bool CLUSTER, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) kset_narrow_kernel(LevelArgs a)
{
    if (a.ctl->err) return;   // set by an earlier launch only: uniform here
    const int64_t hb = a.ctl->base.hist;
    uint32_t nthreads = blockDim.x, rank = threadIdx.x;
    if (CLUSTER) {
        cg::cluster_group cl = cg::this_cluster();
        nthreads = cl.num_threads();
        rank = cl.thread_rank();
    }
    const uint32_t *cut = a.type_cut;
    const bool first = a.orders;
    // the bounds of level j; levels from k1 on are empty
    auto lanes_of = [&](uint32_t j) {
        LevelLanes L;
        if (j < a.k1) L.make(__ldg(&a.level_off[j]), __ldg(&a.level_off[j + 1]), cut ? cut + 2 * (int64_t)j : nullptr);
        else L.make(0, 0, nullptr);
        return L;
    };
    // what hangs on a record's contents: its insert slots, its rows in L2
    auto slots = [&](LaneRecord &r) {
        if (!r.has) return;
        if (r.gl >= 0) {
            r.os = __ldg(&a.b.slot_ord[r.v.t]);
            r.ls = __ldg(&a.b.slot_ol[r.v.t]);
            prefetch_new_order(a.db, r.v, (uint32_t)r.gl, r.p2, r.p3, r.line);
        } else {
            prefetch_txn(a.db, r.v);
        }
        if (a.b.slot_hist) r.v.hist_slot = __ldg(&a.b.slot_hist[r.v.t]);
    };
    LevelLanes L0 = lanes_of(a.k0), L1 = lanes_of(a.k0 + 1), L2 = lanes_of(a.k0 + 2), L3 = lanes_of(a.k0 + 3);
    LaneRecord r0 = lane_record(a.b, L0, rank), r1 = lane_record(a.b, L1, rank);
    slots(r0);
    lane_prefetch(a.b, L2, rank);
    for (uint32_t k = a.k0; k < a.k1; k++) {
        const LevelLanes L4 = lanes_of(k + 4);
        slots(r1);
        LaneRecord r2 = lane_record(a.b, L2, rank);
        lane_prefetch(a.b, L3, rank);
        const bool pay = r0.has && first && r0.v.type == GPUTX_T_OE_PAYMENT;
        r0.v.hist_slot += hb;
        if (r0.has) {
            if (r0.gl >= 0)
                new_order_first(a.db, a.b, r0.v, (uint32_t)r0.gl, r0.p2, r0.p3, r0.line, r0.os, r0.ls);
            else if (pay) payment_first(a.db, a.b, r0.v, r0.p2, r0.p3);
            else exec_lane(a.db, a.b, r0.v, -1, first, a.atomic_add);
        }
        for (uint32_t x = rank + nthreads; x < L0.v; x += nthreads) {
            uint32_t p2;
            int g2;
            if (L0.at(x, p2, g2)) exec_lane(a.db, a.b, view_at(a.b, p2, hb), g2, first, a.atomic_add);
        }
        __syncwarp();
        if (CLUSTER) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        if (pay) payment_totals(a.db, r0.v, r0.p3);
        __syncwarp();
        if (CLUSTER) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        else __syncthreads();
        L0 = L1;
        L1 = L2;
        L2 = L3;
        L3 = L4;
        r0 = r1;
        r1 = r2;
    }
}

__global__ void kset_kernel(KsetArgs a)
{
    __shared__ uint32_t s_k, s_start, s_cnt, s_stop;
    const int64_t levels = (int64_t)a.ctl->last_level + 1;   // from the analysis, on the device
    const uint32_t nchunks = a.chunk_off[levels];
    const int64_t hb = a.ctl->base.hist;
    const uint32_t *cut = a.type_cut;
    while (true) {
        if (threadIdx.x == 0) {
            uint32_t stop = *(volatile uint32_t *)&a.ctl->err ? 1u : 0u;
            const uint32_t c = stop ? nchunks : atomicAdd(&a.ctl->claim, 1u);
            if (c < nchunks) {
                // a chunk is a run of blockDim lanes of one level
                const uint32_t k = a.chunk_level[c];
                const uint32_t w = level_lane_count(a.level_off[k], a.level_off[k + 1], cut ? cut + 2 * (int64_t)k : nullptr);
                const uint32_t start = (c - a.chunk_off[k]) * blockDim.x;
                const uint32_t cnt = (w - start) < blockDim.x ? (w - start) : blockDim.x;
                s_k = k;
                s_start = start;
                s_cnt = cnt;
            } else {
                stop = 1;
            }
            s_stop = stop;
        }
        __syncthreads();
        if (s_stop) break;
        LevelLanes L;
        L.make(a.level_off[s_k], a.level_off[s_k + 1], cut ? cut + 2 * (int64_t)s_k : nullptr);
        // signatures are immutable: load them and prefetch the rows while the
        // previous level may still be running
        TxnView v{};
        uint32_t pos;
        int gl = -1;
        const bool mine = threadIdx.x < s_cnt && L.at(s_start + threadIdx.x, pos, gl);
        if (mine) {
            v = view_at(a.b, pos, hb);
            if (gl < 0) {
                prefetch_txn(a.db, v);
            } else {
                int64_t p2, p3;
                const int64_t line = new_order_params(a.b, v, (uint32_t)gl, p2, p3);
                prefetch_new_order(a.db, v, (uint32_t)gl, p2, p3, line);
            }
        }
        if (threadIdx.x == 0 && s_k > 0) {
            const uint32_t k = s_k;
            const uint32_t prev = level_lane_count(a.level_off[k - 1], a.level_off[k], cut ? cut + 2 * (int64_t)(k - 1) : nullptr);
            if (!wait_at_least(&a.done[k - 1], prev, a.spin_limit_ns)) {
                set_err(&a.ctl->err, ERR_TIMEOUT);
                s_stop = 1;
            }
        }
        __syncthreads();
        if (s_stop) break;
        if (mine) {
            exec_lane(a.db, a.b, v, gl, a.orders, a.atomic_add);
            __threadfence();
        }
        __syncthreads();
        if (threadIdx.x == 0) red_release_add(&a.done[s_k], s_cnt);
    }
}

// K-SET for bulks whose transactions have one operation each (subscriber types,
// mixed with debit-credit): the graph is one path of runs per item, and a
// transaction of the k-th k-set depends on the k-th run of its own item only, so
// no barrier across items is needed and no level table either.  A CTA runs the
// groups that begin in its slice of the operations sorted by item, a window of
// kRoundWindow positions at a time: a segmented scan gives every transaction its
// run within the window, round r runs the r-th run of every group in it (a run
// of reads at once), dealt to the threads by type so that a warp runs one
// procedure, and a CTA barrier ends the round.  The rows and index slots of the
// whole window are prefetched before its first round.
//
// What bounds it is random access to rows and indexes (wide rounds) and a
// procedure's chain of round trips (a hot item's rounds).  1M subscribers, 2^20
// transactions: 260 us, where the levels took 221 (one launch per wide
// level, a cluster for the rest) after 95 us of regrouping, tables, gathering
// and two host round trips.
constexpr int kRoundThreads = 256, kRoundWindow = 512, kRoundPer = kRoundWindow / kRoundThreads;
constexpr int kRoundSlots = kRoundWindow + 32 * GPUTX_NUM_TYPES;

struct RoundArgs {
    DevDB db;
    DevBulk b;
    BulkCtl *ctl;
    const uint32_t *sk, *sv;
    bool stats;                 // record d and w0
    bool atomic_add;
};

__global__ void __launch_bounds__(kRoundThreads, 3) kset_rounds_kernel(RoundArgs a)
{
    __shared__ uint32_t s_min, s_stop, s_rounds, s_first, s_last;
    __shared__ uint32_t s_txn[kRoundWindow];
    __shared__ uint16_t s_list[kRoundSlots];
    __shared__ uint32_t s_cnt[GPUTX_NUM_TYPES], s_at[GPUTX_NUM_TYPES + 1];
    __shared__ uint64_t s_warp[kRoundThreads / 32];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = (uint32_t)a.b.n;
    if (tid == 0) s_stop = *(volatile uint32_t *)&a.ctl->err;
    __syncthreads();
    uint32_t lo, hi;
    if (s_stop || !group_range<kRoundThreads>(a.sk, n, kRoundWindow, &s_min, lo, hi)) return;   // uniform
    const int64_t hb = a.ctl->base.hist;
    uint32_t carry = 0;                      // rank of the position before the window within its group
    uint32_t dmax = 0, zero = 0;
    for (uint32_t base = lo; base < hi; base += kRoundWindow) {
        // thread t owns positions kRoundPer t .. of the window
        uint32_t rank[kRoundPer];            // (set below: the round)
        int32_t type[kRoundPer];
        bool own[kRoundPer];                 // the position's group begins in the window
        uint64_t acc = 0;                    // segmented: head flag << 32 | runs since
        if (tid == 0) s_rounds = 0;
#pragma unroll
        for (int u = 0; u < kRoundPer; u++) {
            const uint32_t e = tid * kRoundPer + u, pos = base + e;
            type[u] = -1;
            uint32_t head = 0, runhead = 0;
            if (pos < hi) {
                const uint32_t k = __ldg(&a.sk[pos]), v = __ldg(&a.sv[pos]), t = v >> 7;
                head = pos == lo || __ldg(&a.sk[pos - 1]) != k;
                if (!head) {
                    const uint32_t c = v & 3u, pc = __ldg(&a.sv[pos - 1]) & 3u;
                    runhead = !(c == pc && cls_shares(c));
                }
                s_txn[e] = t;
                const TxnView w = view_of(a.b, t, hb);
                type[u] = w.type;
                prefetch_txn(a.db, w);
            }
            const uint64_t x = head ? 1ull << 32 : (uint64_t)runhead;
            acc = x >> 32 ? x : acc + x;
            rank[u] = (uint32_t)acc;
            own[u] = (acc >> 32) != 0;
        }
        // the scan over the threads' positions
        uint64_t x = acc;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint64_t o = __shfl_up_sync(kFull, x, off);
            if (lane >= (uint32_t)off && !(x >> 32)) x += o;
        }
        uint64_t excl = __shfl_up_sync(kFull, x, 1);
        if (lane == 0) excl = 0;
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        uint64_t before = 0;
        for (uint32_t w = 0; w < warp; w++) before = s_warp[w] >> 32 ? s_warp[w] : before + s_warp[w];
        const uint64_t pre = excl >> 32 ? excl : before + excl;
        uint32_t rmax = 0;
#pragma unroll
        for (int u = 0; u < kRoundPer; u++) {
            if (!own[u]) {
                rank[u] += (uint32_t)pre;
                own[u] = (pre >> 32) != 0;
            }
            const uint32_t e = tid * kRoundPer + u, pos = base + e;
            if (pos >= hi) continue;
            const uint32_t r = own[u] ? rank[u] : rank[u] + carry;   // the k-set of the transaction
            dmax = r > dmax ? r : dmax;
            zero += r == 0;
            // the group open since the last window goes on with round 0
            if (e == 0) s_first = own[u] ? 0u : rank[u];
            if (pos + 1 == hi || e + 1 == kRoundWindow) s_last = r;
        }
        __syncthreads();
        const uint32_t first = s_first;
        carry = s_last;
#pragma unroll
        for (int u = 0; u < kRoundPer; u++) {
            if (base + tid * kRoundPer + u >= hi) continue;
            if (!own[u]) rank[u] -= first;
            rmax = rank[u] > rmax ? rank[u] : rmax;
        }
        rmax = __reduce_max_sync(kFull, rmax);
        if (lane == 0 && rmax) atomicMax(&s_rounds, rmax);
        if (tid < GPUTX_NUM_TYPES) s_cnt[tid] = 0;
        __syncthreads();
        const uint32_t rounds = s_rounds;
        for (uint32_t r = 0; r <= rounds; r++) {
            // this round's transactions by type, each type from a multiple of 32
            uint32_t at[kRoundPer];
#pragma unroll
            for (int u = 0; u < kRoundPer; u++)
                if (type[u] >= 0 && rank[u] == r) at[u] = atomicAdd(&s_cnt[type[u]], 1u);
            __syncthreads();
            if (warp == 0) {
                const uint32_t c = lane < GPUTX_NUM_TYPES ? (s_cnt[lane] + 31u) & ~31u : 0u;
                uint32_t y = c;
#pragma unroll
                for (int off = 1; off < 16; off <<= 1) {
                    const uint32_t o = __shfl_up_sync(kFull, y, off);
                    if (lane >= (uint32_t)off) y += o;
                }
                if (lane < GPUTX_NUM_TYPES) s_at[lane] = y - c;
                if (lane == GPUTX_NUM_TYPES - 1) s_at[GPUTX_NUM_TYPES] = y;
            }
            __syncthreads();
            const uint32_t total = s_at[GPUTX_NUM_TYPES];
            for (uint32_t i = tid; i < total; i += kRoundThreads) s_list[i] = 0xffffu;
            __syncthreads();
            if (tid < GPUTX_NUM_TYPES) s_cnt[tid] = 0;
#pragma unroll
            for (int u = 0; u < kRoundPer; u++)
                if (type[u] >= 0 && rank[u] == r) s_list[s_at[type[u]] + at[u]] = (uint16_t)(tid * kRoundPer + u);
            __syncthreads();
            for (uint32_t i = tid; i < total; i += kRoundThreads) {
                const uint32_t e = s_list[i];
                if (e != 0xffffu) exec_txn(a.db, a.b, view_of(a.b, s_txn[e], hb), a.atomic_add);
            }
            __syncthreads();                 // the round's writes before the next one's reads
        }
    }
    if (a.stats) {
        dmax = __reduce_max_sync(kFull, dmax);
        zero = __reduce_add_sync(kFull, zero);
        if (lane == 0) {
            if (dmax) atomicMax(&a.ctl->depth, dmax);
            if (zero) atomicAdd(&a.ctl->w0, zero);
        }
    }
}

__global__ void part_kernel(DevDB db, DevBulk b, const BulkCtl *ctl, const uint32_t *pkeys,
                            const uint32_t *part_start)
{
    extern __shared__ unsigned long long part_smem[];
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    // the partition's cells stay with this thread for the whole launch: a
    // write-through cache in shared memory serves its repeated reads
    CachedCells cells;
    cells.tag = part_smem + threadIdx.x * CachedCells::kSlots;
    cells.val = (int64_t *)(part_smem + (blockDim.x + threadIdx.x) * CachedCells::kSlots);
    for (int i = 0; i < CachedCells::kSlots; i++) cells.tag[i] = 0;
    if (p >= ctl->npart || ctl->err) return;
    const int64_t hb = ctl->base.hist;
    const uint32_t n = (uint32_t)b.n;
    uint32_t i = part_start[p];
    if (!dbg_in(i, n, b.err)) return;
    const uint32_t key = __ldg(&pkeys[i]);
    // a two-deep pipeline along the partition's timestamp order: while
    // transaction i executes, i+1's rows are already in L2 and i+2's record
    // is loading; the partition's own order is the only dependency
    TxnView v = view_at(b, i, hb);
    prefetch_txn(db, v);
    bool has1 = i + 1 < n && __ldg(&pkeys[i + 1]) == key;
    TxnView v1{};
    if (has1) {
        v1 = view_at(b, i + 1, hb);
        prefetch_txn(db, v1);
    }
    while (true) {
        const bool has2 = has1 && i + 2 < n && __ldg(&pkeys[i + 2]) == key;
        TxnView v2{};
        if (has2) v2 = view_at(b, i + 2, hb);
        exec_txn(db, b, v, false, cells);
        if (!has1) break;
        if (has2) prefetch_txn(db, v2);
        v = v1;
        v1 = v2;
        has1 = has2;
        i++;
    }
}

// sum of `x` over the lanes of `m` (this lane's group) and its inclusive
// prefix up to this lane, in lane order; every lane of the warp calls it
__device__ __forceinline__ void group_sum(uint32_t m, int64_t x, int64_t &pre, int64_t &tot)
{
    pre = lanes_prefix(m, x);
    tot = __shfl_sync(kFull, pre, 31 - __clz(m));
}

// one addition per distinct cell among the lanes with `on`, by the lowest
// lane of each: `key` selects the cell; every lane of the warp calls it
__device__ __forceinline__ void warp_add(bool on, uint32_t key, unsigned long long *cell, int64_t x)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t m = __match_any_sync(kFull, on ? key : (0xFFFFFFE0u | lane));
    if (__any_sync(kFull, on && __popc(m) > 1)) {
        int64_t pre, tot;
        group_sum(m, x, pre, tot);
        x = tot;
    }
    if (on && lane == (uint32_t)(__ffs(m) - 1)) atomicAdd(cell, (unsigned long long)x);
}

struct TplArgs {
    DevDB db;
    DevBulk b;
    BulkCtl *ctl;
    const uint32_t *lock_key, *lock_ticket, *op_off;
    uint32_t *done;
    int uniform_k;
    uint64_t spin_limit_ns;
    bool atomic_add;
    bool graph;          // fixed-capacity bulk: K slots per transaction, only the
                         // first op_count are real; padding transactions skipped
    bool orders;         // new-orders are registered: launch_orders completes them and the order-statuses
    LockSlots slot;      // item -> its counter in `done`
    const uint32_t *sk, *sv;   // debit-credit: the operations sorted by lock
    int steps;           // tpl_dc_kernel in lock order: times 32 positions a warp takes
};

// releases of the lanes with `rel` (every lane of the warp calls it): lanes
// releasing the same counter are grouped by __match_any_sync and their
// lowest lane adds the group's size (warp-aggregated atomics)
__device__ __forceinline__ void warp_release(const TplArgs &a, bool rel, int64_t off, int cnt)
{
    const uint32_t lane = threadIdx.x & 31;
    const int jmax = __reduce_max_sync(kFull, rel ? (uint32_t)cnt : 0u);
    for (int j = 0; j < jmax; j++) {
        const bool r = rel && j < cnt;
        const uint32_t key = r ? a.slot(__ldg(&a.lock_key[off + j])) : (0xFFFFFFE0u | lane);
        const uint32_t m = __match_any_sync(kFull, key);
        if (r && lane == (uint32_t)(__ffs(m) - 1)) red_release_add(&a.done[key], (uint32_t)__popc(m));
    }
}

// TPL for any registered types.  Each transaction holds one ordered counter
// lock per basic operation (Section 5.1, Appendix C's counter lock with
// ticket semantics): an operation whose group has `ticket` operations before
// its run may proceed once that many have released the item's counter.
// Tickets follow the timestamp order of the group, so the earliest unfinished
// transaction never waits and no deadlock can form.
//
// A warp runs its 32 transactions in lockstep rounds.  A waiting lane polls
// all its locks not yet granted at once (relaxed loads in flight together:
// one round trip, not one per lock; a granted lock stays granted, since no
// later operation releases before this one), then only the lock furthest
// behind, again after about 500 ns per release that lock still misses.
// Every lane whose locks are all granted takes one acquire fence and runs
// its procedure: first the short ones, then the new-orders (up to four of
// them on a half warp each, one lane per order line), each phase followed by
// its releases.  Order-entry's procedures hold their locks for their first
// parts only (launch_orders runs the second ones after this kernel; 200,003
// transactions: 12.9 ms, 14.5 with the procedures whole under the locks).  Releases are warp-aggregated: lanes releasing the same
// counter in a phase are grouped by __match_any_sync and their lowest lane
// adds the group's size.  A round in which nothing is granted sleeps until
// the first lane is due to poll, so a lane about to be granted never sleeps
// behind one far back in its chain.
__global__ void __launch_bounds__(512) tpl_kernel(TplArgs a)
{
    __shared__ uint32_t s_c, s_stop;
    const int64_t n = a.b.n;
    const int64_t hb = a.ctl->base.hist;
    const uint32_t lane = threadIdx.x & 31;
    while (true) {
        if (threadIdx.x == 0) {
            s_stop = *(volatile uint32_t *)&a.ctl->err ? 1u : 0u;
            s_c = atomicAdd(&a.ctl->claim, 1u);
        }
        __syncthreads();
        const int64_t start = (int64_t)s_c * blockDim.x;
        if (s_stop || start >= n) break;
        const int64_t t = start + threadIdx.x;
        const bool live = t < n && !(a.b.n_live && t >= (int64_t)*a.b.n_live);
        int64_t off = 0;
        int cnt = 0;
        TxnView v{};
        if (live) {
            off = a.op_off ? (int64_t)a.op_off[t] : t * a.uniform_k;
            cnt = a.op_off ? (int)(a.op_off[t + 1] - a.op_off[t])
                           : (a.graph ? op_count(a.db, a.b.type[t], a.b.params + t * a.b.P) : a.uniform_k);
            v = view_of(a.b, (uint32_t)t, hb);
            prefetch_txn(a.db, v);
        }
        uint32_t granted = 0;                                  // bit j: lock j granted
        const uint32_t all = cnt >= 32 ? kFull : ((1u << cnt) - 1u);
        int blk = -1;              // the lock holding this lane back (-1: poll every lock)
        uint64_t t_next = 0;       // when this lane polls next
        bool pending = live;
        uint64_t t_prog = globaltimer();
        uint32_t idle = 0;
        while (__any_sync(kFull, pending)) {
            const uint64_t now = globaltimer();
            if (pending && granted != all && now >= t_next) {
                uint32_t gap = 0;
                if (blk >= 0) {        // only the lock that held it back last time
                    const uint32_t tk = __ldg(&a.lock_ticket[off + blk]);
                    const uint32_t c = ld_relaxed_gpu(&a.done[a.slot(__ldg(&a.lock_key[off + blk]))]);
                    if (c >= tk) {
                        granted |= 1u << blk;
                        blk = -1;
                    } else {
                        gap = tk - c;
                    }
                }
                if (blk < 0 && granted != all) {
                    uint32_t c[MAX_OPS], tk[MAX_OPS];
#pragma unroll
                    for (int j = 0; j < MAX_OPS; j++) {         // the polls, all in flight
                        tk[j] = 0;
                        c[j] = 0;
                        if (j < cnt && !((granted >> j) & 1u)) {
                            tk[j] = __ldg(&a.lock_ticket[off + j]);
                            if (tk[j]) c[j] = ld_relaxed_gpu(&a.done[a.slot(__ldg(&a.lock_key[off + j]))]);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < MAX_OPS; j++) {
                        if (j < cnt && !((granted >> j) & 1u)) {
                            if (c[j] >= tk[j]) {
                                granted |= 1u << j;
                            } else if (tk[j] - c[j] > gap) {   // the furthest behind
                                gap = tk[j] - c[j];
                                blk = j;
                            }
                        }
                    }
                }
                // a lock missing `gap` releases needs at least that many
                // hand-offs: poll again after about that long
                if (granted != all) t_next = now + (gap > 1 ? (uint64_t)(gap > 64 ? 64 : gap) * 500 : 0);
            }
            bool ready = pending && granted == all;
            bool failed = false;
            if (!__any_sync(kFull, ready)) {
                if (now - t_prog > a.spin_limit_ns) {
                    // nothing granted within the limit: give up, but release,
                    // so no later waiter hangs on these counters
                    failed = ready = pending;
                    if (failed) set_err(&a.ctl->err, ERR_TIMEOUT);
                } else {
                    // sleep until the first lane is due to poll
                    const uint32_t due = (pending && t_next > now) ? (uint32_t)min(t_next - now, (uint64_t)32000)
                                                                    : (pending ? 0u : kFull);
                    const uint32_t d = __reduce_min_sync(kFull, due);
                    if (d > 0 && d != kFull) __nanosleep(d);
                    else if (++idle > 64) __nanosleep(32);
                    continue;
                }
            }
            if (ready && !failed) fence_acquire_gpu();   // with the polls: acquire of every granted lock
            // The round runs in two phases, each ending with its releases, so
            // a short transaction's hand-off never waits for a new-order of
            // the same warp.  Phase 1: every other granted transaction, one
            // lane each (and the releases of timed-out ones).
            const bool no = ready && !failed && v.type == GPUTX_T_OE_NEW_ORDER;
            const bool r1 = ready && !no, pay = r1 && !failed && v.type == GPUTX_T_OE_PAYMENT;
            if (pay) payment_first(a.db, a.b, v, __ldg(&v.p[2]), __ldg(&v.p[3]));
            else if (r1 && !failed && v.type == GPUTX_T_OE_ORDER_STATUS && a.orders)
                order_status_first(a.db, a.b, v, __ldg(&v.p[2]));
            else if (r1 && !failed) exec_txn(a.db, a.b, v, a.atomic_add);
            __syncwarp();   // every lane's writes precede the releases of its phase
            warp_release(a, r1, off, cnt);
            // no transaction of the bulk reads the totals and additions commute
            if (pay) payment_totals(a.db, v, __ldg(&v.p[3]));
            // Phase 2: the granted new-orders.  Up to four run on a half warp
            // each, two at a time (the line-parallel procedure: one lane per
            // order line, as in the K-SET runners); more run one lane each.
            uint32_t m2 = __ballot_sync(kFull, no);
            if (m2 && __popc(m2) <= 4) {
                while (m2) {
                    const int l0 = __ffs(m2) - 1;
                    m2 &= m2 - 1;
                    const int l1 = m2 ? __ffs(m2) - 1 : -1;
                    if (l1 >= 0) m2 &= m2 - 1;
                    const int src = (lane < 16 || l1 < 0) ? l0 : l1;
                    TxnView g;
                    g.p = (const int64_t *)__shfl_sync(kFull, (unsigned long long)v.p, src);
                    g.p0 = __shfl_sync(kFull, v.p0, src);
                    g.p1 = __shfl_sync(kFull, v.p1, src);
                    g.ts = __shfl_sync(kFull, v.ts, src);
                    g.hist_slot = __shfl_sync(kFull, v.hist_slot, src);
                    g.t = __shfl_sync(kFull, v.t, src);
                    g.type = __shfl_sync(kFull, v.type, src);
                    if (lane < 16 || l1 >= 0) {
                        int64_t p2, p3;
                        const int64_t line = new_order_params(a.b, g, lane & 15u, p2, p3);
                        new_order_first(a.db, a.b, g, lane & 15u, p2, p3, line, a.b.slot_ord[g.t], a.b.slot_ol[g.t]);
                    }
                }
            } else if (no) {
                new_order_first_lane(a.db, a.b, v);
            }
            __syncwarp();
            warp_release(a, no, off, cnt);
            pending = pending && !ready;
            t_prog = globaltimer();
            idle = 0;
        }
        __syncthreads();
    }
}

// TPL for debit-credit-only bulks.  A transaction's one lock is its root
// key's counter (the branch under R/W, the account under ADD).  Once it is
// granted, the account takes a fetch-and-add at L2 (its old value gives the
// output) and the lock is released; the teller and branch additions, the
// history row and the outputs follow the release.  No transaction of the
// bulk reads a teller or branch balance or the history, and integer
// additions commute, so the next holder may run before those land: the
// hand-off waits for one atomic round trip instead of a load, the stores and
// their acknowledgement.
//
// A warp works on 32 transactions and resolves the conflicts among them
// itself.  They are consecutive in timestamp order, or, once the ticket scan has
// found a chain of more than kTplHot operations, consecutive in the operations
// sorted by lock: a lock's queue then changes hands once per 32 transactions
// instead of once per transaction.  Where the longest chain is a small part of the
// bulk (kTplMany), a warp takes a run of 32s side by side, so many that the grid
// holds the whole bulk and all chains move at once: with 32 a warp, 2^20
// transactions had 148 of 1,000 chains at work.  The end of a chain that began in
// an earlier run comes last in its warp's, as nothing waits for it.  A chain that
// is a large part of the bulk is better off with 32 a warp: the next warp is ready
// while the last one writes its rows (Zipf 0.99, one chain of a 16th of 200,003: 680
// against 800 us a bulk).  Always a transaction waits for ones handed out before
// it, or earlier in its warp's run, only.  What bounds a long chain is its hand-offs, about
// 2 us each through L2; in lock order the signatures and outputs are scattered,
// which costs about 50 us per 2^20, hence the line.  1,000 branches, 2^20
// transactions (chains of 1,050): 145 us, 360 with 32 a warp, 1,900 in timestamp
// order; Zipf 0.99 accounts, 200,003: 490 us, 5,500 with CTA-wide groups in
// timestamp order.
//
// __match_any_sync groups the lanes that need the same counter.  Every
// operation here is a write and no other transaction's operation on that item
// lies between two lanes of a group (the warp holds consecutive timestamps, or
// consecutive tickets): their tickets are consecutive, and the whole group runs,
// in lane (timestamp) order, as soon as its first lane's ticket is granted.
// Only that lane polls the counter, and one addition of the group's size
// releases it.  Within a group, lanes on the same account combine their deltas
// (warp-aggregated atomics): one fetch-and-add of the sum, each lane's new
// balance = the old value plus the inclusive prefix of the deltas in lane order
// -- the serial result bit for bit.  Teller and branch additions are aggregated
// the same way.  The warp polls in lockstep rounds: each group polls again after
// about 500 ns per release it still misses, and the warp sleeps until the first
// group is due, so a group whose counter is about to be released never sleeps
// behind one far back in its chain.  A warp in which no two lanes share a
// counter needs none of this: there each lane waits on its own counter and runs
// as soon as it is granted.
__global__ void __launch_bounds__(1024) tpl_dc_kernel(TplArgs a)
{
    __shared__ uint32_t s_c, s_stop;
    const int64_t n = a.b.n;
    const int64_t hb = a.ctl->base.hist;
    const uint32_t lane = threadIdx.x & 31;
    const bool by_lock = a.ctl->hot != 0, many = by_lock && (int64_t)a.ctl->hot * kTplMany <= n;
    while (true) {
        if (threadIdx.x == 0) {
            s_stop = *(volatile uint32_t *)&a.ctl->err ? 1u : 0u;
            s_c = atomicAdd(&a.ctl->claim, 1u);
        }
        __syncthreads();
        // in lock order a warp takes `steps` times 32 positions side by side
        const int steps = many ? a.steps : 1;
        const int64_t start = (int64_t)s_c * blockDim.x * steps;
        if (s_stop || start >= n) break;
        // the warp's positions [lo, hi); those before `head` end a queue that began
        // in an earlier warp's: they come last, as nothing waits for them and what
        // follows them waits for no other warp
        const int64_t lo = min(n, start + (int64_t)(threadIdx.x & ~31u) * steps);
        const int64_t hi = min(n, lo + 32 * (int64_t)steps);
        int64_t head = lo;
        if (steps > 1) {
            head = hi;
            for (int64_t p = lo; p < hi; p += 32) {
                const int64_t q = p + lane;
                const uint32_t m = __ballot_sync(kFull, q < hi && (q == 0 || __ldg(&a.sk[q]) != __ldg(&a.sk[q - 1])));
                if (m) {
                    head = p + __ffs(m) - 1;
                    break;
                }
            }
            if (head == hi) head = lo;
        }
        const int after = (int)((hi - head + 31) / 32), total = after + (int)((head - lo + 31) / 32);
        auto place = [&](int step) { return (step < after ? head + 32 * step : lo + 32 * (step - after)) + lane; };
        auto there = [&](int step) { return step < total && place(step) < (step < after ? hi : head); };
        // a step's record, loaded while the step before runs
        DcRecord ahead{};
        uint32_t ahead_key = 0, ahead_tk = 0;
        auto txn_at = [&](int step) {
            return !there(step) ? 0u : by_lock ? __ldg(&a.sv[place(step)]) >> 7 : (uint32_t)place(step);
        };
        auto load = [&](int step, uint32_t t) {
            if (!there(step)) return;
            ahead.a = (uint32_t)__ldg(&a.b.params[(int64_t)t * a.b.P]);
            ahead.delta = __ldg(&a.b.params[(int64_t)t * a.b.P + 1]);
            ahead.ts = __ldg(&a.b.ts[t]);
            ahead.t = t;
            ahead_key = by_lock ? __ldg(&a.sk[place(step)]) : a.lock_key[t];
            ahead_tk = a.lock_ticket[t];
        };
        uint32_t t1 = txn_at(1);
        load(0, txn_at(0));
        for (int step = 0; step < total; step++) {
            const bool live = there(step);
            DcRecord r = ahead;
            const int64_t t = live ? (int64_t)r.t : 0;
            uint32_t key = 0xFFFFFFE0u | lane, tk = 0;   // a key of its own for an idle lane
            bool rows_ok = true;   // a debug build's check of the record's rows
            if (live) {
                r.tl = a.db.div_tel.div(r.a);
                r.br = a.db.div_br.div(r.a);
                rows_ok = dbg_dc_rows(a.db, a.b, r.a, r.tl, r.br, r.t);
                if (rows_ok) prefetch_l2(&a.db.acc_bal[r.a]);
                key = a.slot(ahead_key);
                tk = ahead_tk;
            }
            load(step + 1, t1);
            t1 = txn_at(step + 2);
            const uint32_t grp = __match_any_sync(kFull, key);
            if (!__any_sync(kFull, live && __popc(grp) > 1)) {
                // no two lanes of the warp share a counter: each waits on its own,
                // without the warp's lockstep rounds
                if (live) {
                    const bool ok = !tk || wait_at_least(&a.done[key], tk, a.spin_limit_ns, 500);
                    if (!ok) set_err(&a.ctl->err, ERR_TIMEOUT);
                    DcOut o;
                    const bool pend = ok && dc_account_rmw(a.db, a.b, r, hb + t, o);
                    red_release_add(&a.done[key], 1u);
                    if (pend) dc_finish_rmw(a.db, a.b, o);
                }
            } else {
                const uint32_t leader = __ffs(grp) - 1;
                const uint32_t need = __shfl_sync(kFull, tk, leader);   // the group's first ticket
                bool pending = live;
                uint64_t t_prog = globaltimer(), t_next = 0;   // t_next: when the group polls next
                uint32_t idle = 0, seen = 0;
                while (__any_sync(kFull, pending)) {
                    const uint64_t now = globaltimer();
                    uint32_t v = need ? seen : need;
                    if (pending && lane == leader && need && now >= t_next) {
                        v = seen = ld_acquire(&a.done[key]);
                        // missing `gap` releases take at least that many hand-offs
                        // (in lock order: a hand-off releases a warp's 32)
                        const uint32_t gap = v >= need ? 0 : by_lock ? (need - v + 31) / 32 : need - v;
                        t_next = now + (gap > 1 ? (uint64_t)(gap > 64 ? 64 : gap) * 500 : 0);
                    }
                    v = __shfl_sync(kFull, v, leader);
                    bool ready = pending && v >= need;
                    bool failed = false;
                    if (!__any_sync(kFull, ready)) {
                        if (now - t_prog > a.spin_limit_ns) {
                            // no group made progress within the limit: give up, but
                            // release, so no later waiter hangs on these counters
                            failed = ready = pending;
                            if (failed && lane == leader) set_err(&a.ctl->err, ERR_TIMEOUT);
                        } else {
                            // sleep until the first group is due to poll
                            const uint32_t due = (pending && lane == leader)
                                                     ? (t_next > now ? (uint32_t)min(t_next - now, (uint64_t)32000) : 0u)
                                                     : kFull;
                            const uint32_t d = __reduce_min_sync(kFull, due);
                            if (d > 0 && d != kFull) __nanosleep(d);
                            else if (++idle > 64) __nanosleep(32);
                            continue;
                        }
                    }
                    // the lanes of `ready` groups run now; the leader's acquire
                    // orders the members' accesses after the previous holder's
                    __syncwarp();
                    const int64_t slot = hb + t;
                    const bool run = ready && !failed && rows_ok && slot < a.db.hist_cap;
                    if (ready && !failed && rows_ok && !run) {      // history full: not executed
                        set_err(a.b.err, ERR_CAPACITY);
                        a.b.status[r.t] = 3;
                    }
                    // the account: one fetch-and-add per distinct account
                    const uint32_t am = __match_any_sync(kFull, run ? r.a : (0xFFFFFFE0u | lane));
                    int64_t pre = r.delta, tot = r.delta;
                    if (__any_sync(kFull, run && __popc(am) > 1)) group_sum(am, r.delta, pre, tot);
                    const uint32_t al = __ffs(am) - 1;
                    int64_t old = 0;
                    if (run && lane == al)
                        old = (int64_t)atomicAdd((unsigned long long *)&a.db.acc_bal[r.a], (unsigned long long)tot);
                    old = __shfl_sync(kFull, old, al);
                    __syncwarp();
                    // one release per group: every member's update precedes it
                    if (ready && lane == leader) red_release_add(&a.done[key], (uint32_t)__popc(grp));
                    warp_add(run, r.tl, (unsigned long long *)&a.db.tel_bal[r.tl], r.delta);
                    warp_add(run, r.br, (unsigned long long *)&a.db.br_bal[r.br], r.delta);
                    if (run) {
                        DcOut o;
                        o.slot = slot;
                        o.ts = r.ts;
                        o.delta = r.delta;
                        o.na = wrap_add(old, pre);
                        o.a = r.a;
                        o.tl = r.tl;
                        o.br = r.br;
                        o.t = r.t;
                        dc_finish(a.db, a.b, o);
                    }
                    pending = pending && !ready;
                    t_prog = globaltimer();
                    idle = 0;
                }
            }
            if (there(step + 1)) prefetch_l2(&a.db.acc_bal[ahead.a]);
        }
        __syncthreads();
    }
}

}  // namespace

// size class of the launch shape a level of width w needs.  Class 0: one
// CTA of up to 64 threads (a CTA barrier).  Class 1: a cluster of up to
// 16 x 64 threads, whose level costs about what one CTA's does.  Classes 2,
// 3, 4: 16 CTAs of 128, 256, 512 threads, each class markedly dearer per
// level than the one below.
static int width_class(uint32_t w)
{
    if (w <= 64) return 0;
    int c = 1;
    while (c < 16 && (1024u << (c - 1)) < w) c++;
    return c;
}

// The end of the segment of narrow levels that starts at k within the run
// [k, run_end).  One launch executes a segment in the shape its widest level
// needs, so a long tail of narrow levels (a skewed bulk's hot chain) must not
// share a launch with a few wide ones: the segment is cut where the width
// class rises, or where a stretch of at least kMinSegment levels of a smaller
// class begins.  Shorter stretches stay in the segment, so every launch but a
// run's last covers at least kMinSegment levels and the launch overhead stays
// small against the levels' own latency.
static int64_t narrow_segment_end(const uint32_t *width, int64_t k, int64_t run_end)
{
    constexpr int64_t kMinSegment = 64;
    auto cls = [&](int64_t j) { return width_class(width[j]); };
    int cmax = cls(k);
    int64_t j = k + 1;
    while (j < run_end) {
        const int c = cls(j);
        if (c > cmax) {
            if (j - k >= kMinSegment) break;
            cmax = c;
            j++;
        } else if (c < cmax) {
            int64_t r = j;
            while (r < run_end && r - j < kMinSegment && cls(r) < cmax) r++;
            if (r - j >= kMinSegment) break;
            j = r;
        } else {
            j++;
        }
    }
    return j;
}

// clusters of this size that fit the device at once (0 = none)
int max_cluster_ok(int csize)
{
    static int cache[17] = {0};
    static bool done[17] = {false};
    if (csize < 1 || csize > 16) return 0;
    if (done[csize]) return cache[csize];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(csize, 1, 1);
    cfg.blockDim = dim3(1024, 1, 1);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = csize;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kset_narrow_kernel<true, 1024>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    cache[csize] = n;
    done[csize] = true;
    return n;
}

int exec_blocks_per_sm(int kind, int block)
{
    int nb = 1;
    if (kind == 0) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kset_kernel, block, 0);
    else if (kind == 2) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, tpl_dc_kernel, block, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, tpl_kernel, block, 0);
    return nb < 1 ? 1 : nb;
}

cudaError_t launch_kset(gputx_bulk *b, int64_t nchunks, int block, bool atomic_add)
{
    gputx_db *db = b->db;
    if (b->n == 0 || nchunks == 0) return cudaSuccess;
    KsetArgs a{};
    a.db = db->dev;
    a.b = make_dev_bulk(b, atomic_add ? GPUTX_CONFLICT_ADD : GPUTX_CONFLICT_PAPER);
    a.ctl = b->ctl;
    a.level_off = b->sc.level_off;
    a.chunk_off = b->sc.chunk_off;
    a.chunk_level = b->sc.chunk_level;
    a.type_cut = b->sc.type_cut;
    a.done = b->sc.done;
    a.orders = db->dev.registered >> GPUTX_T_OE_NEW_ORDER & 1u;
    a.spin_limit_ns = (uint64_t)db->cfg.spin_limit_ns;
    a.atomic_add = atomic_add;
    cudaError_t e = cudaMemsetAsync(b->sc.done, 0, (size_t)(b->n + 1) * sizeof(uint32_t), b->stream);
    if (e) return e;
    e = cudaMemsetAsync(&b->ctl->claim, 0, sizeof(uint32_t), b->stream);
    if (e) return e;
    int64_t grid = (int64_t)db->num_sms * exec_blocks_per_sm(0, block);
    if (grid > nchunks) grid = nchunks;
    kset_kernel<<<(unsigned)grid, block, 0, b->stream>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_kset_levels(gputx_bulk *b, const uint32_t *level_off_host, int64_t depth, int narrow_max,
                               bool atomic_add, const uint32_t *type_cut_host)
{
    gputx_db *db = b->db;
    if (b->n == 0) return cudaSuccess;
    LevelArgs a{};
    a.db = db->dev;
    a.b = make_dev_bulk(b, atomic_add ? GPUTX_CONFLICT_ADD : GPUTX_CONFLICT_PAPER);
    a.ctl = b->ctl;
    a.level_off = b->sc.level_off;
    a.type_cut = type_cut_host ? b->sc.type_cut : nullptr;
    a.orders = db->dev.registered >> GPUTX_T_OE_NEW_ORDER & 1u;
    a.atomic_add = atomic_add;
    const int64_t levels = depth + 1;
    // lanes per level: the launch shapes follow them
    std::vector<uint32_t> width((size_t)levels);
    for (int64_t j = 0; j < levels; j++)
        width[j] = level_lane_count(level_off_host[j], level_off_host[j + 1], a.type_cut ? type_cut_host + 2 * j : nullptr);
    static bool attr_set = false;
    if (!attr_set) {
        cudaFuncSetAttribute(kset_narrow_kernel<true, 256>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaFuncSetAttribute(kset_narrow_kernel<true, 512>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaFuncSetAttribute(kset_narrow_kernel<true, 1024>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        attr_set = true;
    }
    int64_t k = 0, run_end = 0;
    while (k < levels) {
        const uint32_t w = width[k];
        if ((int64_t)w > narrow_max) {
            a.k0 = (uint32_t)k;
            a.k1 = (uint32_t)k + 1;
            int64_t grid = ((int64_t)w + 255) / 256;
            const int64_t cap = (int64_t)db->num_sms * 8;
            if (grid > cap) grid = cap;
            kset_level_kernel<<<(unsigned)grid, 256, 0, b->stream>>>(a);
            count_launches(1);
            k++;
            continue;
        }
        // a run of narrow levels (found once), cut where a long stretch of
        // levels needs a launch shape of another size class (see
        // narrow_segment_end)
        if (run_end <= k) {
            run_end = k;
            while (run_end < levels && (int64_t)width[run_end] <= narrow_max) run_end++;
        }
        const int64_t e = narrow_segment_end(width.data(), k, run_end);
        uint32_t wmax = 0;
        for (int64_t j = k; j < e; j++) wmax = width[j] > wmax ? width[j] : wmax;
        a.k0 = (uint32_t)k;
        a.k1 = (uint32_t)e;
        // spread a level over up to 16 SMs, about 64 transactions each, so
        // no single SM's load/store pipeline carries a whole level
        int csize = (int)((wmax + 63) / 64);
        csize = csize < 1 ? 1 : (csize > 16 ? 16 : csize);
        while (csize > 1 && max_cluster_ok(csize) == 0) csize >>= 1;
        int threads = (int)((wmax + csize - 1) / csize);
        threads = ((threads + 31) / 32) * 32;
        threads = threads < 32 ? 32 : (threads > 1024 ? 1024 : threads);
        if (csize <= 1) {
            if (threads <= 256) kset_narrow_kernel<false, 256><<<1, threads, 0, b->stream>>>(a);
            else kset_narrow_kernel<false, 1024><<<1, threads, 0, b->stream>>>(a);
        } else {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(csize, 1, 1);
            cfg.blockDim = dim3(threads, 1, 1);
            cfg.stream = b->stream;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = csize;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            // up to 256 threads a CTA: more registers per thread for the
            // loads in flight
            cudaError_t e2 = threads <= 256   ? cudaLaunchKernelEx(&cfg, kset_narrow_kernel<true, 256>, a)
                             : threads <= 512 ? cudaLaunchKernelEx(&cfg, kset_narrow_kernel<true, 512>, a)
                                              : cudaLaunchKernelEx(&cfg, kset_narrow_kernel<true, 1024>, a);
            if (e2) return e2;
        }
        count_launches(1);
        cudaError_t e3 = cudaGetLastError();
        if (e3) return e3;
        k = e;
    }
    return cudaGetLastError();
}

cudaError_t launch_part(gputx_bulk *b, const uint32_t *pkeys, int block, int64_t max_parts)
{
    gputx_db *db = b->db;
    if (b->n == 0) return cudaSuccess;
    const DevBulk d = make_dev_bulk(b, GPUTX_CONFLICT_PAPER);
    // few partitions per SM: their scattered stores share one load/store
    // pipeline, so spread the possible partitions over every SM
    const int64_t parts = std::max<int64_t>(1, std::min<int64_t>(b->n, max_parts));
    int threads = (int)((parts + db->num_sms - 1) / db->num_sms);
    threads = ((threads + 7) / 8) * 8;
    threads = threads < 8 ? 8 : (threads > block ? block : threads);
    const int64_t grid = (parts + threads - 1) / threads;   // npart <= parts, read on the device
    const size_t smem = (size_t)threads * 2 * CachedCells::kSlots * sizeof(unsigned long long);
    part_kernel<<<(unsigned)grid, threads, smem, b->stream>>>(db->dev, d, b->ctl, pkeys, b->sc.part_start);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_kset_rounds(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, bool stats, bool atomic_add)
{
    if (b->n == 0) return cudaSuccess;
    RoundArgs a;
    a.db = b->db->dev;
    a.b = make_dev_bulk(b, atomic_add ? GPUTX_CONFLICT_ADD : GPUTX_CONFLICT_PAPER);
    a.ctl = b->ctl;
    a.sk = sk;
    a.sv = sv;
    a.stats = stats;
    a.atomic_add = atomic_add;
    const int64_t grid = (b->n + kRoundWindow - 1) / kRoundWindow;
    kset_rounds_kernel<<<(unsigned)grid, kRoundThreads, 0, b->stream>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_orders(gputx_bulk *b, bool decided)
{
    gputx_db *db = b->db;
    // without new-orders registered the levels and TPL run order-statuses whole;
    // the items never do
    const bool made = db->dev.registered >> GPUTX_T_OE_NEW_ORDER & 1u;
    const bool read = (made || decided) && (db->dev.registered >> GPUTX_T_OE_ORDER_STATUS & 1u);
    if (b->n == 0 || !(made || read)) return cudaSuccess;
    const DevBulk d = make_dev_bulk(b, GPUTX_CONFLICT_PAPER);
    const unsigned grid = (unsigned)std::min<int64_t>((b->n * kGroup + 255) / 256, (int64_t)db->num_sms * 8);
    if (made) {
        orders_kernel<<<grid, 256, 0, b->stream>>>(db->dev, d, b->ctl, true, decided);
        count_launches(1);
    }
    if (read) {
        orders_kernel<<<grid, 256, 0, b->stream>>>(db->dev, d, b->ctl, false, decided);
        count_launches(1);
    }
    return cudaGetLastError();
}

cudaError_t launch_independent(gputx_bulk *b, bool atomic_add)
{
    gputx_db *db = b->db;
    if (b->n == 0) return cudaSuccess;
    int64_t grid = (b->n + 255) / 256;
    if (grid > (int64_t)db->num_sms * 8) grid = (int64_t)db->num_sms * 8;
    independent_kernel<<<(unsigned)grid, 256, 0, b->stream>>>(
        db->dev, make_dev_bulk(b, atomic_add ? GPUTX_CONFLICT_ADD : GPUTX_CONFLICT_PAPER), b->ctl, atomic_add);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_tpl(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int block, bool atomic_add)
{
    gputx_db *db = b->db;
    if (b->n == 0) return cudaSuccess;
    TplArgs a{};
    a.db = db->dev;
    a.b = make_dev_bulk(b, atomic_add ? GPUTX_CONFLICT_ADD : GPUTX_CONFLICT_PAPER);
    a.ctl = b->ctl;
    a.lock_key = b->sc.lock_key;
    a.lock_ticket = b->sc.lock_ticket;
    a.op_off = (db->uniform_k || b->graph) ? nullptr : b->sc.op_off;
    a.done = db->d_done;
    a.uniform_k = b->graph ? db->kmax : db->uniform_k;
    a.graph = b->graph;
    a.spin_limit_ns = (uint64_t)db->cfg.spin_limit_ns;
    a.atomic_add = atomic_add;
    cudaError_t e = cudaMemsetAsync(&b->ctl->claim, 0, sizeof(uint32_t), b->stream);
    if (e) return e;
    a.slot = db->lock_slots;
    a.orders = db->dev.registered >> GPUTX_T_OE_NEW_ORDER & 1u;
    // debit-credit-only bulks of single-lock transactions
    const bool dc = db->dev.registered == (1u << GPUTX_T_DC_DEBIT_CREDIT) && !b->graph && db->uniform_k == 1;
    // the general kernel's registers allow CTAs of up to 512 threads; the
    // CTA size changes only how many transactions a CTA claims at once
    if (!dc && block > 512) block = 512;
    int64_t grid = (int64_t)db->num_sms * exec_blocks_per_sm(dc ? 2 : 1, block);
    const int64_t chunks = (b->n + block - 1) / block;
    if (grid > chunks) grid = chunks;
    a.sk = sk;
    a.sv = sv;
    // lock order: as many positions a warp as let the grid hold the whole bulk
    a.steps = (int)((b->n + grid * block - 1) / (grid * block));
    if (dc) tpl_dc_kernel<<<(unsigned)grid, block, 0, b->stream>>>(a);
    else tpl_kernel<<<(unsigned)grid, block, 0, b->stream>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace gtx
