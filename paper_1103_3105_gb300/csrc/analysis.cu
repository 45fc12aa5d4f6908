// analysis.cu -- bulk generation on the device (Section 4.2, Section 5.2 step
// 1-2, Appendix D): basic-operation extraction, grouping by data item with a
// radix sort, per-group ranks, transaction depths (k-set levels), regrouping
// by (level, type), insert slots, partition ids.
#include <algorithm>
#include <atomic>
#include <cooperative_groups.h>
#include <cstdio>

#include "engine.h"
#include "procs.cuh"
#include "scan.cuh"

namespace gtx {

namespace {

constexpr int TB = 256;  // threads per block of the simple map kernels

// what stops the rank scan and the depth pass: errors of the analysis.  The
// others are the executor's, which may run beside them (launch_depths_aside).
constexpr uint32_t kAnalysisErr = ~(uint32_t)(ERR_CAPACITY | ERR_BOUNDS);
__device__ __forceinline__ uint32_t analysis_errors(const BulkCtl *ctl)
{
    return (ctl->err & kAnalysisErr) | ctl->depth_err;
}

inline unsigned grid_for(int64_t n, int block = TB)
{
    int64_t g = (n + block - 1) / block;
    return (unsigned)(g < 1 ? 1 : g);
}

// ---------------------------------------------------------------------------
// bulk begin / finish: insert bases from the device cursors
// ---------------------------------------------------------------------------
// hist_rows < 0: the history rows were counted by the insert-slot scan
__global__ void begin_kernel(const InsertBase *cursor, BulkCtl *ctl, int64_t hist_rows, bool live_rows)
{
    ctl->base = *cursor;
    if (hist_rows >= 0) ctl->total.hist = live_rows ? (int64_t)ctl->n_live : hist_rows;
}

__global__ void finish_kernel(InsertBase *cursor, const BulkCtl *ctl)
{
    if (ctl->err) return;
    cursor->hist += ctl->total.hist;
    cursor->cf += ctl->total.cf;
    cursor->ord += ctl->total.ord;
    cursor->ol += ctl->total.ol;
}

// ---------------------------------------------------------------------------
// a2: basic-operation extraction (map), with validation and partition ids
// ---------------------------------------------------------------------------
struct ExtractArgs {
    DevDB db;
    DevBulk b;
    BulkCtl *ctl;
    uint32_t *keys, *vals;         // op keys / payloads
    const uint32_t *op_off;        // exclusive op offsets or null (uniform)
    int uniform_k;
    int mode;
    int part_size;
    uint32_t *pid_key, *pid_val;   // PART: partition id and txn per transaction (or null)
    bool write_ops;
    bool sentinel_fill;            // fill unused slots with padding operations
    uint32_t sentinel_key;         // object id above every real one
    const uint32_t *bulk_of;       // segmented graph bulks: the bulk under the object id (or null)
    int seg_shift;                 // bits of the bulk under the object id
    uint32_t pad_pid;              // PART: partition id of a padding transaction (after every real one)
};

__device__ __forceinline__ bool txn_padding(const DevBulk &b, int64_t t)
{
    return b.n_live && t >= (int64_t)*b.n_live;
}

__device__ __forceinline__ bool txn_valid(const DevDB &db, const DevBulk &b, int64_t t)
{
    const int64_t *p = b.params + t * b.P;
    if (!valid_txn(db, b.type[t], p, b.P)) return false;
    if (t > 0 && !(b.ts[t] > b.ts[t - 1])) return false;   // ids strictly increase
    return true;
}

__global__ void count_ops_kernel(DevDB db, DevBulk b, BulkCtl *ctl, uint32_t *cnt)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= b.n) return;
    int c = 0;
    if (txn_valid(db, b, t)) c = op_count(db, b.type[t], b.params + t * b.P);
    else set_err(&ctl->err, ERR_INVAL);
    cnt[t] = (uint32_t)c;
}

__global__ void extract_kernel(ExtractArgs a)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    bool cross = false;
    if (t < a.b.n) {
        const int64_t *p = a.b.params + t * a.b.P;
        const int64_t off = a.op_off ? (int64_t)a.op_off[t] : t * a.uniform_k;   // used when writing
        const bool pad = txn_padding(a.b, t);
        const bool ok = pad || txn_valid(a.db, a.b, t);
        uint32_t obj[MAX_OPS], root[MAX_OPS];
        uint8_t cls[MAX_OPS];
        int k = 0;
        if (ok && !pad) {
            k = access_set(a.db, a.b.type[t], p, a.mode, obj, cls, root);
        } else if (!ok) {
            set_err(&a.ctl->err, ERR_INVAL);
        }
        if (a.write_ops && a.sentinel_fill) {
            // padding operations after the real ones: they sort past every
            // real group and every consumer skips their payload
            for (int j = k; j < a.uniform_k; j++) {
                a.keys[off + j] = a.sentinel_key;
                a.vals[off + j] = OP_SENTINEL;
            }
        } else if (a.write_ops && a.op_off == nullptr) {
            // uniform layout: always fill K slots (dummy reads on object 0 for
            // an invalid transaction; the bulk will not execute)
            for (int j = k; j < a.uniform_k; j++) { obj[j] = 0; cls[j] = CLS_R; root[j] = 0; }
            k = a.uniform_k;
        }
        const uint32_t pid = pad ? a.pad_pid : (k ? root[0] / (uint32_t)a.part_size : 0);
        const uint32_t seg = (a.bulk_of && !pad) ? a.bulk_of[t] : 0u;
        for (int j = 0; j < k; j++) {
            if (a.write_ops) {
                a.keys[off + j] = (obj[j] << a.seg_shift) | seg;
                a.vals[off + j] = ((uint32_t)t << 7) | ((uint32_t)j << 2) | cls[j];
            }
            cross |= (root[j] / (uint32_t)a.part_size) != pid;
        }
        if (a.pid_key) {
            a.pid_key[t] = pid;
            a.pid_val[t] = (uint32_t)t;
        }
    }
    const uint32_t cross_mask = __ballot_sync(0xffffffffu, cross);
    if ((threadIdx.x & 31) == 0 && cross_mask) atomicAdd(&a.ctl->cross, (uint32_t)__popc(cross_mask));
}

// Extraction of a bulk whose registered types have one operation each, with
// the digit counts of the sort that follows (`hist`, RB-bit digits; null: that
// sort counts for itself).  Without the general kernel's per-transaction
// arrays it streams: 2^22 debit-credit transactions take 40 us, extraction and
// counting in two kernels took 67.
struct ExtractOneArgs {
    DevDB db;
    DevBulk b;
    BulkCtl *ctl;
    uint32_t *keys, *vals, *hist;
    int64_t *deltas;               // debit-credit-only bulks: each transaction's delta side by side (or null)
    int mode, part_size, passes;
    bool by_part;                  // key = partition, payload = transaction (else the item and launch_extract's payload)
};

template <int RB> __global__ void __launch_bounds__(256) extract_one_kernel(ExtractOneArgs a)
{
    constexpr int D = 1 << RB, MAXP = (32 + RB - 1) / RB;
    __shared__ uint32_t sh[MAXP * D];
    if (a.hist) {
        for (int i = threadIdx.x; i < a.passes * D; i += blockDim.x) sh[i] = 0;
        __syncthreads();
    }
    // kTxns transactions of a thread at once, their loads in flight together
    constexpr int kTxns = 4;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t0 < a.b.n; t0 += kTxns * step) {
        int32_t type[kTxns];
        int64_t p0[kTxns], ts[kTxns], before[kTxns];
#pragma unroll
        for (int u = 0; u < kTxns; u++) {
            const int64_t t = t0 + u * step;
            if (t >= a.b.n) continue;
            type[u] = __ldg(&a.b.type[t]);
            p0[u] = __ldg(&a.b.params[t * a.b.P]);
            ts[u] = __ldg(&a.b.ts[t]);
            before[u] = t ? __ldg(&a.b.ts[t - 1]) : 0;
        }
#pragma unroll
        for (int u = 0; u < kTxns; u++) {
            const int64_t t = t0 + u * step;
            if (t >= a.b.n) continue;
            // an invalid transaction (the bulk will not execute) reads item 0
            uint32_t obj = 0, cls = CLS_R, root = 0;
            if (valid_txn(a.db, type[u], a.b.params + t * a.b.P, a.b.P) && (t == 0 || ts[u] > before[u]))
                single_op(a.db, type[u], p0[u], a.mode, obj, cls, root);
            else
                set_err(&a.ctl->err, ERR_INVAL);
            const uint32_t key = a.by_part ? root / (uint32_t)a.part_size : obj;
            a.keys[t] = key;
            a.vals[t] = a.by_part ? (uint32_t)t : ((uint32_t)t << 7) | cls;
            if (a.deltas) a.deltas[t] = a.b.P > 1 ? __ldg(&a.b.params[t * a.b.P + 1]) : 0;
            if (a.hist)
                for (int q = 0; q < a.passes; q++) atomicAdd(&sh[q * D + ((key >> (RB * q)) & (D - 1))], 1u);
        }
    }
    if (a.hist) {
        __syncthreads();
        for (int i = threadIdx.x; i < a.passes * D; i += blockDim.x)
            if (sh[i]) atomicAdd(&a.hist[i], sh[i]);
    }
}

// exclusive op offsets from per-transaction counts
struct OffsetMode {
    const uint32_t *cnt;
    uint32_t *off;
    int64_t n;
    __device__ uint64_t element(int64_t i) const { return DualSeg::make(0, 0, 0, cnt[i]); }
    __device__ void output(int64_t i, uint64_t s) const
    {
        off[i + 1] = DualSeg::v2(s);
        if (i == 0) off[0] = 0;
    }
};

// ---------------------------------------------------------------------------
// a4/a5: ranks in each group and transaction depth (Section 4.2 steps 2-5)
// ---------------------------------------------------------------------------
// Within a group (one data item, operations in timestamp order) an operation
// starts a new run unless it and its predecessor are both reads or both ADDs.
// rank = run index within the group; depth(t) = max rank over t's operations.
struct RankMode {
    const uint32_t *sk, *sv;
    uint32_t *level;
    uint32_t *rid;   // optional: place within the run, bit 31 = first run of its group
    __device__ uint64_t element(int64_t i) const
    {
        const uint32_t k = sk[i], v = sv[i];
        const bool head = (i == 0) || sk[i - 1] != k;
        uint32_t runhead = 1;
        if (!head) {
            const uint32_t c = v & 3u, pc = sv[i - 1] & 3u;
            runhead = !(c == pc && cls_shares(c));
        }
        return DualSeg::make(head, head ? 0u : runhead, runhead, 1);
    }
    __device__ void output(int64_t i, uint64_t s) const
    {
        if (sv[i] == OP_SENTINEL) return;
        const uint32_t rank = DualSeg::v1(s);
        const uint32_t txn = sv[i] >> 7;
        atomicMax(&level[txn], rank);
        if (rid) rid[i] = (DualSeg::v2(s) - 1u) | (rank == 0 ? 0x80000000u : 0u);
    }
};

// TPL tickets: number of operations of the group before this operation's run
// (Section 5.1 key values, read with ticket semantics).  `hot` becomes the
// largest last ticket of a group if that is at least `hot_ticket`: the longest
// chain, which picks how the debit-credit executor hands transactions out.
struct TicketMode {
    const uint32_t *sk, *sv;
    uint32_t *lock_key, *lock_ticket;
    const uint32_t *op_off;
    int uniform_k;
    uint32_t *hot;
    uint32_t hot_ticket;
    uint32_t n_objects;   // a debug build checks every lock key against it
    uint32_t *err;
    int64_t m;
    __device__ uint64_t element(int64_t i) const
    {
        const uint32_t k = sk[i], v = sv[i];
        const bool head = (i == 0) || sk[i - 1] != k;
        uint32_t runhead = 1;
        if (!head) {
            const uint32_t c = v & 3u, pc = sv[i - 1] & 3u;
            runhead = !(c == pc && cls_shares(c));
        }
        return DualSeg::make(head, 1, runhead, 1);
    }
    __device__ void output(int64_t i, uint64_t s) const
    {
        const uint32_t v = sv[i];
        if (v == OP_SENTINEL) return;
        const uint32_t txn = v >> 7, j = (v >> 2) & 31u;
        const int64_t slot = (op_off ? (int64_t)op_off[txn] : (int64_t)txn * uniform_k) + j;
        const uint32_t tk = DualSeg::v1(s) - DualSeg::v2(s);
        if (!dbg_in(sk[i], n_objects, err)) return;
        lock_key[slot] = sk[i];
        lock_ticket[slot] = tk;
        if (tk >= hot_ticket && (i + 1 >= m || sk[i + 1] != sk[i]) && tk > *(volatile uint32_t *)hot) atomicMax(hot, tk);
    }
};

// Exact depths by dataflow (one pass, no rounds).
//
// Within a group (one item, operations in timestamp order) the runs follow
// one another: every operation of run q conflicts with every operation of run
// q-1, and transitively with all earlier runs.  So a transaction's depth is
// the largest, over its operations outside their group's first run, of one
// more than the deepest transaction of the run before -- the longest path of
// the conflict graph, the depth the Jacobi refinement converges to.  Here each
// transaction computes it once the transactions of the runs before its
// operations have theirs.
//
// Two numbers come out of the same pass: the depth (d and w0 are taken from
// it) and the level the transaction executes in, which leaves out the edges
// between two blind increments of the read/write model (CLS_BW): K-SET applies
// those by atomic additions, so they order nothing.  Order-entry's payments
// then run beside each other although all of a warehouse's write its total.
// A finished transaction publishes both in one 64-bit word with its chunk's lap
// (below), so a waiter needs no fence and no second read.
//
// What bounds the pass is the longest path, so its hops are made short.  One
// cluster runs it: a CTA holds 1,024 consecutive transactions, its neighbours the
// chunks before and after, and a CTA's next chunk is the one kFlowCluster
// further.  A finished transaction stores its word into the shared memory of
// every CTA of the cluster, where the words of the last kFlowCluster chunks lie in
// a ring, so waiting is polling one shared-memory word a lane and nothing goes
// through L2 but what is older.  Warps run by themselves, without barriers: a
// warp whose transactions are finished costs nothing.  Before that, while the
// chunks before still run, a transaction that waits for one other, p, knows its
// depth as max(m, depth(p) + l), and if p does too, it takes over p's p (pointer
// jumping), so a chain through a chunk -- the payments of a warehouse -- is one
// hop behind the chunk before.  A CTA waits for earlier transactions only, and
// all CTAs of a cluster run at the same time: the chain of waits always ends.
// Order-entry, 200,003 transactions under R/W (d = 1,442, 610 levels): 500 us, 0.8
// a level; in rounds of a whole chunk with two CTA barriers each and polls in L2,
// on every SM: 1,050; polls in L2 by each lane alone: 2,950.  A warp works off
// what its lanes find one pass at a time, so a pass is kept short (lanes that each
// went on as far as they could: 820) and what a lane waits for is in timestamp
// order (in operation order: 670).  Chunks of 512: 535, of 256: 723; words for the
// next 2 chunks only, the others' in L2: 888 (670 in the same order with 7); a
// cluster of 16: no faster.

// per operation: the last operation of the run before its own
// (kPredNone: none).  Several transactions in that run: kPredRun | the sorted
// position of the last.  One: its index, and kPredBlind if both are blind
// increments.
constexpr uint32_t kPredNone = 0xffffffffu, kPredRun = 1u << 30, kPredVal = kPredRun - 1u;
constexpr uint32_t kPredBlind = 1u << 31, kPredTxn = (1u << 25) - 1u;
// levels from the predecessor to the transaction (0: it does not order the execution)
__device__ __forceinline__ uint32_t pred_step(uint32_t p) { return !(p & kPredRun) && (p & kPredBlind) ? 0u : 1u; }

__global__ void depth_prep_kernel(const uint32_t *sv, const uint32_t *rid, int64_t m, const uint32_t *op_off,
                                  int kslots, uint32_t *pred, BulkCtl *ctl)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= m || analysis_errors(ctl)) return;
    const uint32_t v = sv[i];
    if (v == OP_SENTINEL) return;
    const uint32_t r = rid[i];
    const uint32_t txn = v >> 7, j = (v >> 2) & 31u;
    const int64_t slot = (op_off ? (int64_t)op_off[txn] : (int64_t)txn * kslots) + j;
    uint32_t p = kPredNone;
    if (!(r & 0x80000000u)) {
        const int64_t q = i - r - 1;                       // the run before ends here
        if (!dbg_in(q, m, &ctl->err)) return;
        const uint32_t w = sv[q];
        p = (rid[q] & 0x7fffffffu) ? (kPredRun | (uint32_t)q) : (w >> 7);
        if (!(p & kPredRun) && (v & 3u) == CLS_BW && (w & 3u) == CLS_BW) p |= kPredBlind;
    }
    pred[slot] = p;
}

constexpr int kFlowThreads = 1024, kFlowCluster = 8;
constexpr int kFlowPush = 7;                // the chunks after a chunk that get its words in shared memory
constexpr unsigned long long kNotYet = ~0ull;

// A word: lap << 50 | depth << 25 | level (a bulk has at most 2^25 transactions).
// A place in the ring takes the words of one CTA, whose chunks lie kFlowCluster
// apart, so the lap (from 1, at most 2^12 + 1) says which chunk's word it holds:
// nothing keeps the CTAs of the cluster in step, and one may be any number of laps
// ahead of another.
constexpr uint32_t kFlowBits = 25, kFlowMask = (1u << kFlowBits) - 1u;
__device__ __forceinline__ uint32_t flow_lap(uint32_t chunk) { return chunk / kFlowCluster + 1; }
constexpr int32_t kLapStep = 1 << (2 * kFlowBits - 32);   // a lap in a word's upper half

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

struct FlowArgs {
    const uint32_t *pred, *op_off, *sv, *rid;
    int kslots;
    unsigned long long *depths;              // per transaction: its word, kNotYet before
    uint32_t *level;
    BulkCtl *ctl;
    uint32_t *err;
    int64_t n;
    bool graph;                              // transactions from n_live on are padding
    uint64_t limit_ns;
};

// what a transaction that waits for one other, p, knows: its depth is
// max(dep, depth(p) + dlen), its level max(lev, level(p) + llen), or lev if llen
// is 0; p = kPredNone while it waits for several
struct FlowNode {
    uint32_t p, len, dep, lev;               // len: dlen << 16 | llen, at most kFlowThreads each
};

__global__ void __launch_bounds__(kFlowThreads, 1) depth_flow_kernel(FlowArgs a)
{
    // [MAX_OPS][kFlowThreads] predecessors, the nodes, the ring of words
    extern __shared__ __align__(16) uint32_t s_pred[];
    FlowNode *s_node = reinterpret_cast<FlowNode *>(s_pred + MAX_OPS * kFlowThreads);
    unsigned long long *s_ring = reinterpret_cast<unsigned long long *>(s_node + kFlowThreads);
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    BulkCtl *ctl = a.ctl;
    const uint32_t tid = threadIdx.x, lane = tid & 31, rank = cl.block_rank();
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(s_ring);
    for (int k = 0; k <= kFlowPush; k++) s_ring[k * kFlowThreads + tid] = 0;
    if (rank == 0 && tid == 0) ctl->rounds = 1;
    __shared__ uint32_t s_stop;
    if (tid == 0) s_stop = analysis_errors(ctl);
    const uint32_t n = (uint32_t)(a.graph ? (int64_t)ctl->n_live : a.n);
    cl.sync();
    const bool stop = *cl.map_shared_rank(&s_stop, 0) != 0;    // the same in every CTA
    cl.sync();
    if (stop) return;
    uint32_t dmax = 0, lmax = 0, zero = 0;
    for (uint32_t c = rank; (uint64_t)c * kFlowThreads < n; c += kFlowCluster) {
        const uint32_t start = c * kFlowThreads, t = start + tid;
        uint32_t dep = 0, lev = 0;
        auto take = [&](unsigned long long w, uint32_t dl, uint32_t ll) {
            const uint32_t d = ((uint32_t)(w >> kFlowBits) & kFlowMask) + dl, l = ((uint32_t)w & kFlowMask) + ll;
            dep = d > dep ? d : dep;
            if (ll) lev = l > lev ? l : lev;
        };
        // where transaction x's word comes to in this CTA's ring
        auto near_word = [&](uint32_t x) { return c - x / kFlowThreads <= (uint32_t)kFlowPush; };
        auto ring_word = [&](uint32_t x) {
            return ring + 8u * ((c - x / kFlowThreads) * kFlowThreads + x % kFlowThreads);
        };
        // the runs before its operations that are not known complete: `left` of
        // one transaction, in timestamp order (the last one's word is the last to
        // come, and then no other look lies between it and this one's), from the
        // column's start; `runs` of several, from its end
        uint32_t left = 0, runs = 0;
        if (t < n) {
            const int64_t s0 = a.op_off ? (int64_t)a.op_off[t] : (int64_t)t * a.kslots;
            const int k = a.op_off ? (int)(a.op_off[t + 1] - a.op_off[t]) : a.kslots;
            for (int j0 = 0; j0 < k; j0 += 6) {
                uint32_t p[6];
                unsigned long long w[6];
#pragma unroll
                for (int u = 0; u < 6; u++) p[u] = j0 + u < k ? __ldg(&a.pred[s0 + j0 + u]) : kPredNone;
#pragma unroll
                for (int u = 0; u < 6; u++)
                    w[u] = p[u] == kPredNone || (p[u] & kPredRun) ? kNotYet : ld_relaxed_u64(&a.depths[p[u] & kPredTxn]);
#pragma unroll
                for (int u = 0; u < 6; u++) {
                    if (p[u] == kPredNone) continue;
                    if (w[u] != kNotYet) {
                        take(w[u], 1, pred_step(p[u]));
                        continue;
                    }
                    if (p[u] & kPredRun) {
                        s_pred[(MAX_OPS - ++runs) * kFlowThreads + tid] = p[u];
                        continue;
                    }
                    uint32_t i = left++;
                    for (; i > 0; i--) {
                        const uint32_t o = s_pred[(i - 1) * kFlowThreads + tid];
                        if ((o & kPredTxn) <= (p[u] & kPredTxn)) break;
                        s_pred[i * kFlowThreads + tid] = o;
                    }
                    s_pred[i * kFlowThreads + tid] = p[u];
                }
            }
        }
        FlowNode me{kPredNone, 0, 0, 0};
        if (left == 1 && !runs) {
            const uint32_t p = s_pred[tid];
            me = FlowNode{p & kPredTxn, 0x10000u | pred_step(p), dep, lev};
        }
        s_node[tid] = me;
        __syncthreads();
        while (true) {
            FlowNode o{kPredNone, 0, 0, 0};
            if (me.p != kPredNone && me.p >= start) o = s_node[me.p - start];
            const bool jump = o.p != kPredNone;
            if (!__syncthreads_or(jump)) break;
            if (jump) {
                const uint32_t dl = me.len >> 16, ll = me.len & 0xffffu, ol = o.len & 0xffffu;
                me.dep = o.dep + dl > me.dep ? o.dep + dl : me.dep;
                if (ll) me.lev = o.lev + ll > me.lev ? o.lev + ll : me.lev;
                me.len = ((dl + (o.len >> 16)) << 16) | (ll && ol ? ll + ol : 0u);
                me.p = o.p;
                s_node[tid] = me;
            }
            __syncthreads();
        }
        // what the lane waits for: x, dl and ll edges from it; then `more` earlier
        // operations of a run, which ends at `end`
        uint32_t x = start, dl = 1, ll = 1, more = 0, end = 0, at_left = tid;
        bool done = t >= n;
        auto next = [&]() -> bool {            // false: nothing left
            if (more | runs) {
                if (more) {
                    more--;
                    end--;
                } else {
                    end = s_pred[(MAX_OPS - runs--) * kFlowThreads + tid] & kPredVal;
                    more = __ldg(&a.rid[end]) & 0x7fffffffu;
                }
                x = __ldg(&a.sv[end]) >> 7;
                return true;
            }
            if (!left) return false;
            const uint32_t p = s_pred[at_left];
            at_left += kFlowThreads;
            left--;
            x = p & kPredTxn;
            ll = pred_step(p);
            return true;
        };
        auto publish = [&]() {
            const unsigned long long w =
                (unsigned long long)flow_lap(c) << (2 * kFlowBits) | (unsigned long long)dep << kFlowBits | lev;
            asm volatile("st.relaxed.cluster.shared::cta.u64 [%0], %1;" ::"r"(ring + 8u * tid), "l"(w) : "memory");
#pragma unroll
            for (uint32_t r = 1; r <= (uint32_t)kFlowPush; r++) {
                uint32_t dst;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                             : "=r"(dst)
                             : "r"(ring + 8u * (r * kFlowThreads + tid)), "r"((rank + r) % kFlowCluster));
                asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(dst), "l"(w) : "memory");
            }
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(&a.depths[t]), "l"(w) : "memory");
            done = true;
        };
        if (me.p != kPredNone) {
            left = 0;
            x = me.p;
            dl = me.len >> 16;
            ll = me.len & 0xffffu;
            dep = me.dep;
            lev = me.lev;
        } else if (!done && !next()) {
            publish();
        }
        // one look a lane and pass; a lane that finds its word goes on to what it
        // waits for next in the next pass, so the lanes stay together
        uint64_t t_prog = 0;
        uint32_t seen = 0;
        // where it looks, and the least upper half of a word there that ends the wait
        // (none for a lane that is done or whose word is in L2 only)
        bool l2;
        uint32_t at;
        int32_t want;
        auto aim = [&]() {
            const bool near = near_word(x) && !done;
            l2 = !near && !done;
            at = near ? ring_word(x) : ring;
            want = near ? (int32_t)flow_lap(x / kFlowThreads) * kLapStep : INT32_MAX;
        };
        aim();
        for (uint32_t spin = 1;; spin++) {
            unsigned long long w;
            asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(w) : "r"(at) : "memory");
            const int32_t ahead = (int32_t)(w >> 32) - want;
            bool hit = ahead >= 0;
            // older than the ring, or overwritten by a later chunk's (that CTA has finished its chunk)
            if (ahead >= kLapStep || (l2 && (spin & 7u) == 0)) {
                w = ld_relaxed_u64(&a.depths[x]);
                hit = w != kNotYet;
            }
            if (__any_sync(kFull, hit)) {
                if (hit) {
                    take(w, dl, ll);
                    if (!next()) publish();
                    aim();
                }
                continue;
            }
            if (__all_sync(kFull, done)) break;
            if ((spin & 1023u) == 0) {         // no chunk finished for the limit: give up, but publish
                const uint32_t f = ld_relaxed_gpu(&ctl->front);
                const uint64_t now = globaltimer();
                if (t_prog == 0 || f != seen) t_prog = now;
                seen = f;
                const bool late = now - t_prog > a.limit_ns || (*(volatile uint32_t *)a.err & ERR_TIMEOUT);
                if (__any_sync(kFull, late)) {
                    if (lane == 0) set_err(a.err, ERR_TIMEOUT);
                    if (!done) publish();
                    aim();
                }
            }
        }
        if (t < n) {
            a.level[t] = lev;
            dmax = dep > dmax ? dep : dmax;
            lmax = lev > lmax ? lev : lmax;
            zero += dep == 0;
        }
        __syncthreads();                       // nobody here waits for this chunk any more
        if (tid == 0) atomicAdd(&ctl->front, 1u);
    }
    dmax = __reduce_max_sync(kFull, dmax);
    lmax = __reduce_max_sync(kFull, lmax);
    zero = __reduce_add_sync(kFull, zero);
    if (lane == 0) {
        if (dmax) atomicMax(&ctl->depth, dmax);
        if (lmax) atomicMax(&ctl->last_level, lmax);
        if (zero) atomicAdd(&ctl->w0, zero);
    }
    cl.sync();                                 // stores into this CTA's ring may still be on their way
}

// d and w0 (Appendix D structural parameters)
__global__ void level_stats_kernel(const uint32_t *level, int64_t n, BulkCtl *ctl)
{
    __shared__ uint32_t s_max, s_zero;
    if (threadIdx.x == 0) { s_max = 0; s_zero = 0; }
    __syncthreads();
    uint32_t mx = 0, zero = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t l = level[i];
        mx = l > mx ? l : mx;
        zero += (l == 0);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    zero = __reduce_add_sync(0xffffffffu, zero);
    if ((threadIdx.x & 31) == 0) { atomicMax(&s_max, mx); atomicAdd(&s_zero, zero); }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&ctl->depth, s_max);
        atomicMax(&ctl->last_level, s_max);
        atomicAdd(&ctl->w0, s_zero);
    }
}

// ---------------------------------------------------------------------------
// a6: regroup by (level, type) -- Appendix D's grouping by type, per level
// ---------------------------------------------------------------------------
__global__ void regroup_keys_kernel(const uint32_t *level, const int32_t *type, int64_t n, int tbits,
                                    uint32_t *keys, uint32_t *vals, const uint32_t *n_live,
                                    const uint32_t *bulk_of, const uint32_t *seg_base)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n) return;
    if (n_live && t >= (int64_t)*n_live) {
        keys[t] = (uint32_t)n << tbits;   // padding: past every real level
    } else {
        const int32_t ty = type[t];
        // a segment's levels run bulk after bulk: global level = the bulk's
        // first global level + the level within the bulk
        const uint32_t lv = level[t] + (bulk_of ? seg_base[bulk_of[t]] : 0u);
        keys[t] = (lv << tbits) | (tbits && ty > 0 ? (uint32_t)ty : 0u);
    }
    vals[t] = (uint32_t)t;
}

// the bulk of each live transaction of a segment (seg_off: first
// transaction of each of its n_seg bulks, ascending from 0)
__global__ void seg_index_kernel(const uint32_t *seg_off, const BulkCtl *ctl, uint32_t *bulk_of, int64_t cap)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= cap) return;
    const uint32_t nseg = ctl->n_seg < 1 ? 1u : (ctl->n_seg > (uint32_t)kSegMax ? (uint32_t)kSegMax : ctl->n_seg);
    uint32_t lo = 0, hi = nseg - 1;   // last bulk whose start is <= t
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (seg_off[mid] <= (uint32_t)t) lo = mid;
        else hi = mid - 1;
    }
    bulk_of[t] = lo;
}

__global__ void seg_depth_kernel(const uint32_t *level, const uint32_t *bulk_of, const BulkCtl *ctl,
                                 uint32_t *seg_depth, int64_t cap)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= cap || t >= (int64_t)ctl->n_live) return;
    atomicMax(&seg_depth[bulk_of[t]], level[t]);
}

// first global level of each bulk; the segment's depth becomes the last
// global level
__global__ void seg_base_kernel(const uint32_t *seg_depth, BulkCtl *ctl, uint32_t *seg_base)
{
    if (threadIdx.x != 0) return;
    const uint32_t nseg = ctl->n_seg < 1 ? 1u : (ctl->n_seg > (uint32_t)kSegMax ? (uint32_t)kSegMax : ctl->n_seg);
    uint32_t acc = 0;
    for (uint32_t i = 0; i < nseg; i++) {
        seg_base[i] = acc;
        acc += seg_depth[i] + 1;
    }
    seg_base[nseg] = acc;
    ctl->depth = ctl->last_level = acc - 1;
}

__global__ void part_fallback_kernel(BulkCtl *ctl)
{
    if (ctl->cross) ctl->err |= ERR_FALLBACK;
}

// Level boundaries from the keys sorted by (level << tbits | type); with
// type_cut, also where each level's new-orders and payments start (type_cut[2 k
// + j] = first position of level k whose type is >= 8 + j), so the executors
// can give the new-orders their lane groups.  A cut (k, type) lands on the first
// key at or above k << tbits | type; levels are contiguous, so between two
// adjacent keys at most two levels' cuts fall.
// a debug build's check of the level table the executors index by: the
// bounds of levels 0..depth rise and stay within the bulk (an executor whose
// bulk carries an error returns before its first gather)
__global__ void check_level_off_kernel(const uint32_t *level_off, int64_t n, BulkCtl *ctl)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (ctl->err || k > (int64_t)ctl->last_level || k >= n) return;
    const uint32_t lo = level_off[k], hi = level_off[k + 1];
    if (lo > hi || !dbg_in(hi, n + 1, &ctl->err)) set_err(&ctl->err, ERR_BOUNDS);
}

__global__ void level_off_kernel(const uint32_t *skeys, int64_t n, int tbits, uint32_t *level_off,
                                 uint32_t *type_cut, const BulkCtl *ctl, const uint32_t *err)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n || *err) return;
    // real levels are 0..depth; a graph bulk's padding sorts after them as
    // level n, whose boundary is the only one needed past depth
    const uint32_t top = ctl->last_level + 1;
    const uint32_t key = skeys[i];
    const uint32_t lv = key >> tbits;
    const uint32_t lvc = lv < top ? lv : top;
    const uint32_t prev = i ? (skeys[i - 1] >> tbits) : 0u;
    if (i == 0) {
        for (uint32_t k = 0; k <= lvc; k++) level_off[k] = 0;
    } else if (lv != prev) {
        for (uint32_t k = prev + 1; k <= lvc; k++) level_off[k] = (uint32_t)i;
    }
    if (i == n - 1 && lv < top) level_off[lv + 1] = (uint32_t)n;
    if (type_cut && (i == 0 || skeys[i - 1] != key)) {
        const uint64_t below = i ? (uint64_t)skeys[i - 1] + 1 : 0;   // cuts in (key[i-1], key[i]]
        const uint32_t kmax = lv < top ? lv : top - 1;
        for (uint32_t k = i ? prev : 0; k <= kmax; k++)
            for (uint32_t j = 0; j < 2; j++) {
                const uint64_t cut = ((uint64_t)k << tbits) | (GPUTX_T_OE_NEW_ORDER + j);
                if (cut >= below && cut <= key) type_cut[2 * k + j] = (uint32_t)i;
            }
    }
    if (type_cut && i == n - 1 && lv < top)
        for (uint32_t j = 0; j < 2; j++) {
            const uint64_t cut = ((uint64_t)lv << tbits) | (GPUTX_T_OE_NEW_ORDER + j);
            if (cut > key) type_cut[2 * lv + j] = (uint32_t)n;
        }
}

struct ChunkMode {
    const uint32_t *level_off;
    uint32_t *chunk_off;
    uint32_t block;
    const BulkCtl *ctl;   // levels = last_level + 1, read on the device
    const uint32_t *type_cut;   // chunks count lanes (order-entry groups) when set
    __device__ uint64_t element(int64_t k) const
    {
        if (k > (int64_t)ctl->last_level) return 0;
        const uint32_t w = level_lane_count(level_off[k], level_off[k + 1], type_cut ? type_cut + 2 * k : nullptr);
        return DualSeg::make(0, 0, 0, (w + block - 1) / block);
    }
    __device__ void output(int64_t k, uint64_t s) const
    {
        chunk_off[k + 1] = DualSeg::v2(s);
        if (k == 0) chunk_off[0] = 0;
    }
};

__global__ void chunk_level_kernel(const uint32_t *chunk_off, const BulkCtl *ctl, uint32_t *chunk_level,
                                   int64_t cap, const uint32_t *err)
{
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (*err) return;
    const int64_t levels = (int64_t)ctl->last_level + 1;
    const uint32_t nchunks = chunk_off[levels];
    if (c >= cap || c >= nchunks) return;
    // largest k with chunk_off[k] <= c
    int64_t lo = 0, hi = levels - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (chunk_off[mid] <= (uint32_t)c) lo = mid;
        else hi = mid - 1;
    }
    chunk_level[c] = (uint32_t)lo;
}

// ---------------------------------------------------------------------------
// a7: deterministic insert slots: exclusive counts in timestamp order
// ---------------------------------------------------------------------------
struct SlotMode {
    const int32_t *type;
    const int64_t *params;
    int P;
    int64_t n;
    uint32_t *slot_a, *slot_b;
    BulkCtl *ctl;
    int which;   // 0: (call-forwarding inserts, orders) 1: (-, order lines)
    __device__ uint32_t a(int64_t t) const
    {
        return which == 0 ? (type[t] == GPUTX_T_SUB_INSERT_CF) : 0u;
    }
    __device__ uint32_t bv(int64_t t) const
    {
        if (type[t] != GPUTX_T_OE_NEW_ORDER) return 0u;
        if (which == 0) return 1u;
        const int64_t c = params[t * P + 3];
        return (c >= 1 && c <= OE_MAX_LINES) ? (uint32_t)c : 0u;
    }
    __device__ uint64_t element(int64_t t) const { return DualSeg::make(0, a(t), 0, bv(t)); }
    __device__ void output(int64_t t, uint64_t s) const
    {
        const uint32_t ia = DualSeg::v1(s), ib = DualSeg::v2(s);
        if (which == 0) {
            slot_a[t] = ia - a(t);
            slot_b[t] = ib - bv(t);
            if (t == n - 1) { ctl->total.cf = ia; ctl->total.ord = ib; }
        } else {
            slot_b[t] = ib - bv(t);
            if (t == n - 1) ctl->total.ol = ib;
        }
    }
};

// ---------------------------------------------------------------------------
// PART: partition starts; TPL: counter reset
// ---------------------------------------------------------------------------
// partition heads in sorted order: part_start[p] = first position of the
// p-th partition, part_start[npart] = n (a compaction by prefix count)
struct HeadMode {
    const uint32_t *skeys;
    uint32_t *part_start;
    BulkCtl *ctl;
    int64_t n;
    const uint32_t *n_live;   // graph bulks: padding (sorted last) forms no partition
    __device__ int64_t live() const { return n_live ? (int64_t)*n_live : n; }
    __device__ bool head(int64_t i) const { return i < live() && (i == 0 || skeys[i] != skeys[i - 1]); }
    __device__ uint64_t element(int64_t i) const { return DualSeg::make(0, 0, 0, head(i) ? 1u : 0u); }
    __device__ void output(int64_t i, uint64_t s) const
    {
        const uint32_t c = DualSeg::v2(s);
        if (head(i)) part_start[c - 1] = (uint32_t)i;
        if (i == live() - 1) {
            part_start[c] = (uint32_t)live();
            ctl->npart = c;
        }
    }
};

__global__ void tpl_reset_kernel(const uint32_t *skeys, int64_t m, uint32_t *done, uint32_t n_objects,
                                 LockSlots slot)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= m) return;
    const uint32_t k = skeys[i];
    if ((i == 0 || skeys[i - 1] != k) && k < n_objects) done[slot(k)] = 0;
}

// scratch of a scan of `tiles` tiles, cleared: one of the areas that the bulk's
// submission cleared, or the first one again
cudaError_t scan_scratch(gputx_bulk *b, int64_t tiles, uint64_t *&z)
{
    z = b->sc.scan_zero;
    if (tiles > b->sc.scan_tiles) return cudaErrorInvalidValue;
    if (b->scans < kScanAreas) {
        z += b->scans++ * (1 + b->sc.scan_tiles);
        return cudaSuccess;
    }
    return cudaMemsetAsync(z, 0, (1 + tiles) * sizeof(uint64_t), b->stream);
}

// where the rank scan and the depth pass note that a wait ran out
uint32_t *analysis_err(gputx_bulk *b, bool aside) { return aside ? &b->ctl->depth_err : &b->ctl->err; }

template <class Mode>
cudaError_t run_scan(gputx_bulk *b, const Mode &mode, int64_t count, uint32_t stop = ~0u, bool aside = false)
{
    if (count <= 0) return cudaSuccess;
    const int64_t tiles = (count + SCAN_TILE - 1) / SCAN_TILE;
    cudaStream_t s = b->stream;
    uint64_t *z = nullptr;
    const cudaError_t e = scan_scratch(b, tiles, z);
    if (e) return e;
    dualseg_scan_kernel<Mode><<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(
        mode, count, z + 1, (uint32_t *)z, analysis_err(b, aside), &b->ctl->err, stop,
        (uint64_t)b->db->cfg.spin_limit_ns);
    count_launches(1);
    return cudaGetLastError();
}

inline DevBulk dev_bulk(gputx_bulk *b, int mode)
{
    DevBulk d{};
    d.n = b->n;
    d.P = b->P;
    d.R = b->R;
    d.ts = b->ts;
    d.type = b->type;
    d.params = b->params;
    d.status = b->status;
    d.out = b->out;
    d.err = &b->ctl->err;
    d.base = &b->ctl->base;
    d.slot_cf = b->sc.slot_cf;
    d.slot_ord = b->sc.slot_ord;
    d.slot_ol = b->sc.slot_ol;
    d.slot_hist = b->sc.slot_hist;
    d.rec_params = b->sc.rec_params;
    d.rec_ts = b->sc.rec_ts;
    d.rec_type = b->sc.rec_type;
    d.rec_t = b->sc.rec_t;
    d.n_live = b->graph ? &b->ctl->n_live : nullptr;
    d.conflict_mode = mode;
    return d;
}

// the bulk's signatures permuted into execution order: executors then read
// them sequentially instead of chasing order[] into random rows
__global__ void gather_kernel(DevBulk b, const uint32_t *order, int64_t *r_params, int64_t *r_ts,
                              int32_t *r_type, uint32_t *r_t, const uint32_t *err)
{
    const int64_t pos = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (pos >= b.n || *err) return;
    const uint32_t t = order[pos];
    if (!dbg_in(t, b.n, b.err)) return;
    r_t[pos] = t;
    r_ts[pos] = b.ts[t];
    r_type[pos] = b.type[t];
    const int64_t *src = b.params + (int64_t)t * b.P;
    int64_t *dst = r_params + pos * b.P;
    for (int j = 0; j < b.P; j++) dst[j] = src[j];
}

// ---------------------------------------------------------------------------
// relaxed timestamps (Appendix G): validation and counter-based grouping
// ---------------------------------------------------------------------------
__global__ void validate_kernel(DevDB db, DevBulk b, BulkCtl *ctl)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < b.n && !txn_valid(db, b, t)) set_err(&ctl->err, ERR_INVAL);
}

// each transaction takes the next counter value of its partition as its
// position in the partition (the order of the atomics is the relaxation).
// With few partitions a block first counts in shared memory, then takes one
// global range per partition it saw (kPartCountItems transactions a thread),
// so 4 M transactions over 1,000 counters do not serialise on the counters.
constexpr int kPartCountThreads = 1024, kPartCountItems = 8, kPartLocalMax = 4096;

__device__ __forceinline__ bool part_of(const DevDB &db, const DevBulk &b, int64_t t, int mode, int part_size,
                                        uint32_t &pid, bool &cross)
{
    if (!txn_valid(db, b, t)) return false;
    uint32_t obj[MAX_OPS], root[MAX_OPS];
    uint8_t cls[MAX_OPS];
    const int k = access_set(db, b.type[t], b.params + t * b.P, mode, obj, cls, root);
    pid = k ? root[0] / (uint32_t)part_size : 0;
    for (int j = 1; j < k; j++) cross |= (root[j] / (uint32_t)part_size) != pid;
    return true;
}

template <bool LOCAL>
__global__ void __launch_bounds__(kPartCountThreads) part_count_kernel(DevDB db, DevBulk b, BulkCtl *ctl, int mode,
                                                                       int part_size, uint32_t *cnt, int64_t parts,
                                                                       uint32_t *pid_of, uint32_t *key_of)
{
    __shared__ uint32_t scnt[LOCAL ? kPartLocalMax : 1], sbase[LOCAL ? kPartLocalMax : 1];
    if (LOCAL) {
        for (int64_t p = threadIdx.x; p < parts; p += blockDim.x) scnt[p] = 0;
        __syncthreads();
    }
    const int64_t base = (int64_t)blockIdx.x * kPartCountThreads * kPartCountItems + threadIdx.x;
    uint32_t pid[kPartCountItems], local[kPartCountItems];
    bool ok[kPartCountItems];
    bool cross = false;
#pragma unroll
    for (int j = 0; j < kPartCountItems; j++) {
        const int64_t t = base + (int64_t)j * kPartCountThreads;
        pid[j] = 0;
        local[j] = 0;
        ok[j] = false;
        if (t < b.n) {
            ok[j] = part_of(db, b, t, mode, part_size, pid[j], cross);
            if (!ok[j]) set_err(&ctl->err, ERR_INVAL);
            else local[j] = LOCAL ? atomicAdd(&scnt[pid[j]], 1u) : atomicAdd(&cnt[pid[j]], 1u);
        }
    }
    if (LOCAL) {
        __syncthreads();
        // the block's first transaction of each partition takes the range
#pragma unroll
        for (int j = 0; j < kPartCountItems; j++)
            if (ok[j] && local[j] == 0) sbase[pid[j]] = atomicAdd(&cnt[pid[j]], scnt[pid[j]]);
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < kPartCountItems; j++) {
        const int64_t t = base + (int64_t)j * kPartCountThreads;
        if (t < b.n) {
            pid_of[t] = pid[j];
            key_of[t] = ok[j] ? (LOCAL ? sbase[pid[j]] + local[j] : local[j]) : 0;
        }
    }
    const uint32_t cross_mask = __ballot_sync(0xffffffffu, cross);
    if ((threadIdx.x & 31) == 0 && cross_mask) atomicAdd(&ctl->cross, (uint32_t)__popc(cross_mask));
}

// position = start of the partition (prefix sum of the counters) + counter value
__global__ void part_scatter_kernel(int64_t n, const uint32_t *off, const uint32_t *pid_of, const uint32_t *key_of,
                                    uint32_t *pkeys, uint32_t *order, const uint32_t *err)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= n || *err) return;
    const uint32_t pid = pid_of[t];
    const uint32_t pos = off[pid] + key_of[t];
    pkeys[pos] = pid;
    order[pos] = (uint32_t)t;
}

// ---------------------------------------------------------------------------
// SCAN executor for bulks of debit-credit transactions (blind increments,
// the ADD refinement taken to its end).  Under Definition 1 the output of
// transaction t is its account's balance before the bulk plus the deltas of
// the bulk's transactions on that account up to and including t, in
// timestamp order: a segmented prefix sum over the operations grouped by
// account (the stable grouping sort keeps timestamp order inside a group).
// Teller and branch balances only receive sums, and wrapping addition is
// associative and commutative, so atomic adds give the serial result.
// ---------------------------------------------------------------------------
struct AcctScanArgs {
    const uint32_t *sk, *sv;     // operations grouped by account object id
    const int64_t *deltas;       // by transaction, side by side
    int64_t *acc_bal, *out;
    uint32_t m;
    int R;
    uint32_t o_acc;
    BulkCtl *stats;              // K-SET: accounts are the graph's paths, d and w0 are recorded (or null)
    const InsertBase *cursor;
    int64_t hist_cap;
    Seg64Status st;
    uint32_t *tile_ctr, *err;
    uint64_t spin_limit_ns;
};

// element i of a tile in shared memory: a thread's SCAN_ITEMS consecutive
// elements lie 9 words of 8 bytes apart, so a warp's reads spread over the banks
__device__ __forceinline__ uint32_t tile_at(uint32_t i) { return i + i / SCAN_ITEMS; }

// A tile's keys, transactions, deltas and balances are loaded, and its results
// stored, element by element across the CTA (thread t takes elements t, t + 256,
// ...); the scan itself wants consecutive elements per thread, so the values
// change places through shared memory.  What bounds it is the sectors touched
// one by one: per element the signature's, the account's (read at a group's
// head, written at its end) and the output's; with consecutive elements per
// thread in global memory too, every load of keys and payloads (six an element)
// touched 32 sectors a warp as well: 2^22 uniform accounts 125 us against 201.
__global__ void __launch_bounds__(SCAN_THREADS, 6) acct_scan_kernel(AcctScanArgs a)
{
    __shared__ uint32_t s_tile, s_abort;
    __shared__ Seg64 s_warp[SCAN_THREADS / 32];
    __shared__ Seg64 s_prefix;
    __shared__ uint64_t s_v[SCAN_TILE + SCAN_TILE / SCAN_ITEMS];
    __shared__ uint32_t s_fc[SCAN_TILE + SCAN_TILE / SCAN_ITEMS];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        s_abort = *(volatile uint32_t *)a.err || !rows_fit(a.cursor, a.m, a.hist_cap, a.err);
        if (!s_abort) s_tile = atomicAdd(a.tile_ctr, 1u);
    }
    __syncthreads();
    if (s_abort) return;
    const uint32_t tile = s_tile, base = tile * SCAN_TILE;
    uint32_t t[SCAN_ITEMS];
    uint32_t heads = 0, lasts = 0;         // bit j: element j begins, ends its account's group
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        const uint32_t i = base + j * SCAN_THREADS + tid;
        t[j] = 0;
        if (i < a.m) {
            const uint32_t k = __ldcs(&a.sk[i]);
            t[j] = __ldcs(&a.sv[i]) >> 7;
            if (i == 0 || __ldg(&a.sk[i - 1]) != k) heads |= 1u << j;
            if (i == a.m - 1 || __ldg(&a.sk[i + 1]) != k) lasts |= 1u << j;
        }
    }
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        const uint32_t i = j * SCAN_THREADS + tid;
        uint64_t v = 0;
        uint32_t fc = 0;
        if (base + i < a.m) {
            v = (uint64_t)__ldg(&a.deltas[t[j]]);
            // the balance before the bulk joins at the account's first operation
            if (heads >> j & 1u) v += (uint64_t)__ldcs(&a.acc_bal[__ldg(&a.sk[base + i]) - a.o_acc]);
            fc = 2u | (heads >> j & 1u);
        }
        s_v[tile_at(i)] = v;
        s_fc[tile_at(i)] = fc;
    }
    __syncthreads();
    Seg64 acc = Seg64::identity();
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        const uint32_t i = tile_at(tid * SCAN_ITEMS + j);
        acc = Seg64::combine(acc, Seg64{s_fc[i], s_v[i]});
    }
    Seg64 x = acc;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const Seg64 o = shfl_up_seg(x, off);
        if (lane >= (uint32_t)off) x = Seg64::combine(o, x);
    }
    if (lane == 31) s_warp[warp] = x;
    Seg64 thread_excl = shfl_up_seg(x, 1);
    if (lane == 0) thread_excl = Seg64::identity();
    __syncthreads();
    if (warp == 0) {
        Seg64 w = (lane < SCAN_THREADS / 32) ? s_warp[lane] : Seg64::identity();
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const Seg64 o = shfl_up_seg(w, off);
            if (lane >= (uint32_t)off) w = Seg64::combine(o, w);
        }
        const Seg64 tile_agg = shfl_seg(w, SCAN_THREADS / 32 - 1);
        Seg64 wexcl = shfl_up_seg(w, 1);
        if (lane == 0) wexcl = Seg64::identity();
        if (lane < SCAN_THREADS / 32) s_warp[lane] = wexcl;
        const Seg64 pre = lookback_seg64(a.st, tile, tile_agg, a.err, a.spin_limit_ns);
        if (lane == 0) s_prefix = pre;
    }
    __syncthreads();
    acc = Seg64::combine(Seg64::combine(s_prefix, s_warp[warp]), thread_excl);
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        const uint32_t i = tile_at(tid * SCAN_ITEMS + j);
        acc = Seg64::combine(acc, Seg64{s_fc[i], s_v[i]});
        s_v[i] = acc.v;
        s_fc[i] = acc.fc;
    }
    __syncthreads();
    uint32_t longest = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        const uint32_t i = j * SCAN_THREADS + tid;
        if (base + i < a.m) {
            const int64_t v = (int64_t)s_v[tile_at(i)];
            a.out[(int64_t)t[j] * a.R] = v;
            // the account's balance after the bulk (every tile reading it
            // published its aggregate before this tile finished its look-back)
            if (lasts >> j & 1u) {
                __stcs(&a.acc_bal[__ldg(&a.sk[base + i]) - a.o_acc], v);
                const uint32_t len = s_fc[tile_at(i)] >> 1;   // the path's length
                longest = len > longest ? len : longest;
            }
        }
    }
    if (a.stats) {
        longest = __reduce_max_sync(0xffffffffu, longest);
        const uint32_t paths = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(lasts));
        if (lane == 0) {
            if (longest > 1) atomicMax(&a.stats->depth, longest - 1);
            if (paths) atomicAdd(&a.stats->w0, paths);
        }
    }
}

// adds x to cell `key` of the lanes with `on`, one atomic per distinct cell and
// warp; every lane of the warp calls it
__device__ __forceinline__ void warp_add_cell(bool on, uint32_t key, unsigned long long *cell, uint64_t x)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t live = __ballot_sync(kFull, on);
    const uint32_t peers = on ? __match_any_sync(live, key) : 1u << lane;
    const int64_t sum = lanes_prefix(peers, (int64_t)x);
    if (on && lane == 31u - (uint32_t)__clz(peers)) atomicAdd(cell, (unsigned long long)sum);
}

// history rows in timestamp order (slot = the cursor + t) and the teller and
// branch sums; reads the signatures sequentially, at the copy rate (2^22: 300 MB
// in 51 us).  With `local` the sums gather in shared memory first (one slot per
// teller and branch) and each block adds its non-zero sums once: the
// same-address atomics on the few branch rows would otherwise serialise in L2.
// With `few` cells (64 branches at most) even the shared-memory atomics collide,
// and a warp adds up what its lanes have for one cell first.  That guards against
// 64-bit additions in shared memory as compare-and-swap loops, which the compiler
// makes of them where it can tell the address space: 4 branches, 4,096
// transactions 42 us, 2^20 258, all of one account 308 (with the warps' sums 5.2,
// 16, 16).  In the code below the address is generic and the additions are single
// instructions, and the warps' sums are not worth their shuffles on either side of
// the line: 4 branches at 2^20 16.0 us against 12.9 without, 64 20.9 against 13.2,
// 128 21.8 against 13.0.
struct DcRowsArgs {
    DevDB db;
    DevBulk b;
    BulkCtl *ctl;
    InsertBase *cursor;
    bool local, few;
};

__global__ void __launch_bounds__(1024) dc_rows_kernel(DcRowsArgs a)
{
    extern __shared__ unsigned long long sums[];   // [n_tel] tellers, then [n_br] branches
    __shared__ uint32_t s_stop;
    const DevDB &db = a.db;
    const DevBulk &b = a.b;
    const int64_t n = b.n_live ? (int64_t)*b.n_live : b.n;
    if (threadIdx.x == 0)
        s_stop = *(volatile uint32_t *)&a.ctl->err || !rows_fit(a.cursor, n, db.hist_cap, &a.ctl->err);
    const uint32_t n_tel = (uint32_t)db.n_tel, n_br = (uint32_t)db.n_br;
    if (a.local)
        for (uint32_t i = threadIdx.x; i < n_tel + n_br; i += blockDim.x) sums[i] = 0;
    __syncthreads();
    if (s_stop) return;                            // uniform
    const int64_t hb = *(volatile int64_t *)&a.cursor->hist;
    // whole warps step together
    for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31u); t0 < n;
         t0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = t0 + (threadIdx.x & 31u);
        const bool on = t < n;
        uint32_t tl = 0, br = 0;
        int64_t d = 0;
        if (on) {
            const uint32_t acct = (uint32_t)b.params[t * b.P];
            d = b.params[t * b.P + 1];
            tl = db.div_tel.div(acct);
            br = db.div_br.div(acct);
            const int64_t slot = hb + t;
            db.h_ts[slot] = b.ts[t];
            db.h_acc[slot] = acct;
            db.h_tel[slot] = tl;
            db.h_br[slot] = br;
            db.h_delta[slot] = d;
            b.status[t] = 0;   // here, in timestamp order, rather than scattered by the account updates
        }
        unsigned long long *tel = a.local ? &sums[tl] : (unsigned long long *)&db.tel_bal[tl];
        unsigned long long *bra = a.local ? &sums[n_tel + br] : (unsigned long long *)&db.br_bal[br];
        if (a.few) {
            warp_add_cell(on, tl, tel, (uint64_t)d);
            warp_add_cell(on, br, bra, (uint64_t)d);
        } else if (on) {
            atomicAdd(tel, (unsigned long long)d);
            atomicAdd(bra, (unsigned long long)d);
        }
    }
    __syncthreads();
    if (a.local)
        for (uint32_t i = threadIdx.x; i < n_tel + n_br; i += blockDim.x) {
            const unsigned long long v = sums[i];
            if (!v) continue;
            unsigned long long *dst = i < n_tel ? (unsigned long long *)&db.tel_bal[i]
                                                : (unsigned long long *)&db.br_bal[i - n_tel];
            atomicAdd(dst, v);
        }
    // the last block moves the cursor on: every block has read it by then
    if (threadIdx.x == 0 && atomicAdd(&a.ctl->rows_done, 1u) == gridDim.x - 1 && !*(volatile uint32_t *)&a.ctl->err)
        a.cursor->hist = hb + n;
}

}  // namespace

DevBulk make_dev_bulk(gputx_bulk *b, int mode) { return dev_bulk(b, mode); }

// The values of a debit-credit-only bulk are cleared just before its executor
// scatters them, 8 bytes at a time: the cleared sectors are still in L2 and the
// scatter need not fetch them (with streaming hints on what passes through
// once, acct_scan_kernel at 2^22: 122 us instead of 156).
cudaError_t clear_outputs(gputx_bulk *b)
{
    return b->n > 0 ? cudaMemsetAsync(b->out, 0, (size_t)b->n * b->R * sizeof(int64_t), b->stream) : cudaSuccess;
}

bool dc_only(const gputx_db *db) { return db->dev.registered == (1u << GPUTX_T_DC_DEBIT_CREDIT); }

cudaError_t launch_scan_exec(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m, bool stats)
{
    if (m == 0) return cudaSuccess;
    gputx_db *db = b->db;
    cudaStream_t s = b->stream;
    const int64_t tiles = (m + SCAN_TILE - 1) / SCAN_TILE;
    uint64_t *z = nullptr;
    cudaError_t e = scan_scratch(b, tiles, z);
    if (!e) e = clear_outputs(b);
    if (e) return e;
    AcctScanArgs a;
    a.sk = sk;
    a.sv = sv;
    a.deltas = b->sc.rec_ts;
    a.acc_bal = db->dev.acc_bal;
    a.out = b->out;
    a.m = (uint32_t)m;
    a.R = b->R;
    a.o_acc = db->dev.o_acc;
    a.stats = stats ? b->ctl : nullptr;
    a.cursor = db->d_cursor;
    a.hist_cap = db->dev.hist_cap;
    a.st.word = (uint32_t *)(z + 1);
    a.st.agg = b->sc.scan_vals;
    a.st.inc = b->sc.scan_vals + tiles;
    a.tile_ctr = (uint32_t *)z;
    a.err = &b->ctl->err;
    a.spin_limit_ns = (uint64_t)db->cfg.spin_limit_ns;
    acct_scan_kernel<<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_dc_rows(gputx_bulk *b)
{
    if (b->n == 0) return cudaSuccess;
    gputx_db *db = b->db;
    // teller and branch sums in shared memory when they fit and there are
    // several transactions per cell (clearing and adding the cells costs each
    // block more than 1,000 transactions' own atomics: 7 us against 3), one
    // block per SM
    const int64_t cells = db->dev.n_tel + db->dev.n_br;
    const size_t smem = (size_t)cells * sizeof(unsigned long long);
    constexpr unsigned kMaxCells = 200u << 10;
    const bool local = smem <= kMaxCells && b->n >= 4 * cells;
    const int threads = 1024;
    int64_t grid = (b->n + threads - 1) / threads;
    if (grid > (int64_t)db->num_sms) grid = db->num_sms;
    if (local && smem > (48u << 10)) {
        // always the same limit: another thread's database may need more than this one
        const cudaError_t e = cudaFuncSetAttribute(dc_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)kMaxCells);
        if (e) return e;
    }
    DcRowsArgs a;
    a.db = db->dev;
    a.b = dev_bulk(b, GPUTX_CONFLICT_ADD);
    a.ctl = b->ctl;
    a.cursor = db->d_cursor;
    a.local = local;
    a.few = db->dev.n_br <= 64;
    dc_rows_kernel<<<(unsigned)grid, threads, local ? smem : 0, b->stream>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_gather(gputx_bulk *b, const uint32_t *order)
{
    if (b->n == 0) return cudaSuccess;
    const DevBulk d = dev_bulk(b, 0);
    gather_kernel<<<grid_for(b->n), TB, 0, b->stream>>>(d, order, b->sc.rec_params, b->sc.rec_ts,
                                                             b->sc.rec_type, b->sc.rec_t, &b->ctl->err);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_validate(gputx_bulk *b)
{
    if (b->n == 0) return cudaSuccess;
    validate_kernel<<<grid_for(b->n), TB, 0, b->stream>>>(b->db->dev, dev_bulk(b, 0), b->ctl);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_part_count(gputx_bulk *b, int mode, int part_size, uint32_t *cnt, int64_t parts,
                              uint32_t *pid_of, uint32_t *key_of)
{
    if (b->n == 0) return cudaSuccess;
    const int64_t per_block = (int64_t)kPartCountThreads * kPartCountItems;
    const unsigned grid = (unsigned)((b->n + per_block - 1) / per_block);
    const int ps = part_size < 1 ? 1 : part_size;
    if (parts <= kPartLocalMax)
        part_count_kernel<true><<<grid, kPartCountThreads, 0, b->stream>>>(b->db->dev, dev_bulk(b, mode), b->ctl,
                                                                          mode, ps, cnt, parts, pid_of, key_of);
    else
        part_count_kernel<false><<<grid, kPartCountThreads, 0, b->stream>>>(b->db->dev, dev_bulk(b, mode), b->ctl,
                                                                           mode, ps, cnt, parts, pid_of, key_of);
    count_launches(1);
    return cudaGetLastError();
}

// exclusive offsets of `parts` counters: off[p] = start of partition p,
// off[parts] = total (scan scratch supplied by the caller)
cudaError_t launch_part_offsets(gputx_bulk *b, const uint32_t *cnt, uint32_t *off, int64_t parts, uint64_t *status,
                                uint32_t *tile_ctr)
{
    if (parts <= 0) return cudaSuccess;
    OffsetMode om{cnt, off, parts};
    const int64_t tiles = (parts + SCAN_TILE - 1) / SCAN_TILE;
    cudaError_t e = cudaMemsetAsync(status, 0, tiles * sizeof(uint64_t), b->stream);
    if (!e) e = cudaMemsetAsync(tile_ctr, 0, sizeof(uint32_t), b->stream);
    if (e) return e;
    dualseg_scan_kernel<OffsetMode><<<(unsigned)tiles, SCAN_THREADS, 0, b->stream>>>(
        om, parts, status, tile_ctr, &b->ctl->err, &b->ctl->err, ~0u, (uint64_t)b->db->cfg.spin_limit_ns);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_part_scatter(gputx_bulk *b, const uint32_t *off, const uint32_t *pid_of, const uint32_t *key_of,
                                uint32_t *pkeys, uint32_t *order)
{
    if (b->n == 0) return cudaSuccess;
    part_scatter_kernel<<<grid_for(b->n), TB, 0, b->stream>>>(b->n, off, pid_of, key_of, pkeys, order,
                                                                &b->ctl->err);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_begin(gputx_bulk *b)
{
    const bool dc = (b->db->dev.registered & 1u) != 0;
    const int64_t rows = b->sc.slot_hist ? -1 : (dc ? b->n : 0);
    begin_kernel<<<1, 1, 0, b->stream>>>(b->db->d_cursor, b->ctl, rows, dc && b->graph);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_finish(gputx_bulk *b)
{
    finish_kernel<<<1, 1, 0, b->stream>>>(b->db->d_cursor, b->ctl);
    count_launches(1);
    return cudaGetLastError();
}

int seg_bits(const gputx_db *db)
{
    // segment bulk ids sit under the object id in a 32-bit key: a group is one
    // bulk's, and an item's groups lie side by side, bulk after bulk
    const int room = 32 - db->obj_bits;
    return room < 1 ? 0 : (room > 6 ? 6 : room);
}

cudaError_t launch_seg_index(gputx_bulk *b)
{
    if (b->n == 0 || !b->sc.bulk_of) return cudaSuccess;
    seg_index_kernel<<<grid_for(b->n), TB, 0, b->stream>>>(b->sc.seg_off, b->ctl, b->sc.bulk_of, b->n);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_seg_levels(gputx_bulk *b)
{
    if (b->n == 0 || !b->sc.bulk_of) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(b->sc.seg_depth, 0, kSegMax * sizeof(uint32_t), b->stream);
    if (e) return e;
    seg_depth_kernel<<<grid_for(b->n), TB, 0, b->stream>>>(b->sc.level, b->sc.bulk_of, b->ctl, b->sc.seg_depth, b->n);
    seg_base_kernel<<<1, 32, 0, b->stream>>>(b->sc.seg_depth, b->ctl, b->sc.seg_base);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_part_fallback_check(gputx_bulk *b)
{
    part_fallback_kernel<<<1, 1, 0, b->stream>>>(b->ctl);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_extract(gputx_bulk *b, int mode, int part_size, uint32_t *pid_key, uint32_t *pid_val,
                           bool write_ops, bool segmented)
{
    gputx_db *db = b->db;
    cudaStream_t s = b->stream;
    if (b->n == 0) return cudaSuccess;
    ExtractArgs a{};
    a.db = db->dev;
    a.b = dev_bulk(b, mode);
    a.ctl = b->ctl;
    a.keys = b->sc.keys_a;
    a.vals = b->sc.vals_a;
    a.uniform_k = db->uniform_k;
    a.mode = mode;
    a.part_size = part_size < 1 ? 1 : part_size;
    a.pid_key = pid_key;
    a.pid_val = pid_val;
    a.write_ops = write_ops;
    a.sentinel_fill = b->graph;
    a.sentinel_key = db->dev.n_objects;
    if (b->graph) a.uniform_k = db->kmax;
    if (segmented && b->graph && b->sc.bulk_of && seg_bits(db) > 0) {
        a.bulk_of = b->sc.bulk_of;
        a.seg_shift = seg_bits(db);
        a.sentinel_key = db->dev.n_objects << a.seg_shift;
    }
    {
        const int64_t roots = std::max<int64_t>({db->dev.n_br, db->dev.n_sub, db->dev.n_wh, 1});
        a.pad_pid = (uint32_t)((roots + a.part_size - 1) / a.part_size);
    }
    if (!db->uniform_k && write_ops && !b->graph) {
        // counts into level[] (free until the rank scan), then offsets
        count_ops_kernel<<<grid_for(b->n), TB, 0, s>>>(db->dev, a.b, b->ctl, b->sc.level);
        count_launches(1);
        cudaError_t e = cudaGetLastError();
        if (e) return e;
        OffsetMode om{b->sc.level, b->sc.op_off, b->n};
        e = run_scan(b, om, b->n);
        if (e) return e;
        a.op_off = b->sc.op_off;
    }
    extract_kernel<<<grid_for(b->n), TB, 0, s>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

// A sort's scratch: a tile counter per pass (8 words), the digit counts, each
// pass's look-back words -- for any number of key bits and up to `count` pairs.
int64_t sort_scratch_words(int64_t count)
{
    int64_t words = 0;
    for (int bits : {10, 32})   // at most three passes of 10-bit digits, four of 8-bit ones
        for (int64_t c : {std::min(count, SORT_WIDE_FROM), count}) {
            const SortShape s = sort_shape(c, bits);
            const int passes = s.digit_bits == 10 ? 3 : 4;
            words = std::max(words, 8 + passes * (int64_t)s.digits() * (1 + s.tiles));
        }
    return words;
}

// where a sort's counters live in its scratch
struct SortScratch {
    uint32_t *ctr, *hist, *status;
    size_t bytes;
    // cleared for the next sort (the first one finds it cleared)
    cudaError_t clear(gputx_bulk *b) const
    {
        const bool done = b->sort_clear;
        b->sort_clear = false;
        return done ? cudaSuccess : cudaMemsetAsync(ctr, 0, bytes, b->stream);
    }
};
static SortScratch sort_scratch(gputx_bulk *b, const SortShape &sh)
{
    SortScratch z;
    z.ctr = b->sc.sort_zero;
    z.hist = z.ctr + 8;
    z.status = z.hist + sh.passes * sh.digits();
    z.bytes = sizeof(uint32_t) * (8 + sh.passes * (size_t)sh.digits() * (1 + sh.tiles));
    return z;
}

template <int RB, int ITEMS>
static cudaError_t launch_radix_passes(gputx_bulk *b, uint32_t *&keys, uint32_t *&vals, uint32_t *&keys_alt,
                                       uint32_t *&vals_alt, uint32_t count, const SortShape &sh, bool counted)
{
    constexpr int D = 1 << RB;
    cudaStream_t s = b->stream;
    const SortScratch z = sort_scratch(b, sh);
    static std::atomic<uint64_t> attr_set{0};   // a bit per device
    const uint64_t dev = 1ull << (b->db->device & 63);
    if (!(attr_set.load(std::memory_order_relaxed) & dev)) {
        const cudaError_t e = cudaFuncSetAttribute(radix_pass_kernel<RB, ITEMS>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)radix_smem<RB, ITEMS>());
        if (e) return e;
        attr_set.fetch_or(dev, std::memory_order_relaxed);
    }
    if (!counted) {
        int hist_blocks = b->db->num_sms * 4;
        const int64_t need = ((int64_t)count + 255) / 256;
        if (hist_blocks > need) hist_blocks = (int)need;
        radix_hist_kernel<RB><<<hist_blocks, 256, 0, s>>>(keys, count, sh.passes, z.hist, &b->ctl->err);
        count_launches(1);
    }
    for (int p = 0; p < sh.passes; p++) {
        radix_pass_kernel<RB, ITEMS><<<(unsigned)sh.tiles, SORT_THREADS, radix_smem<RB, ITEMS>(), s>>>(
            keys, vals, keys_alt, vals_alt, count, RB * p, z.hist + p * D, z.status + (size_t)p * sh.tiles * D,
            z.ctr + p, &b->ctl->err, (uint64_t)b->db->cfg.spin_limit_ns);
        count_launches(1);
        std::swap(keys, keys_alt);
        std::swap(vals, vals_alt);
    }
    return cudaGetLastError();
}

// the sort proper; `counted`: its scratch is cleared and holds the digit counts
static cudaError_t launch_sort_passes(gputx_bulk *b, uint32_t *&keys, uint32_t *&vals, uint32_t *&keys_alt,
                                      uint32_t *&vals_alt, int64_t count, int bits, bool counted)
{
    if (count <= 1 || bits <= 0) return cudaSuccess;
    cudaStream_t s = b->stream;
    if (count <= SMALL_SORT) {
        if (count <= 256 * SMALL_SORT_ITEMS)
            radix_small_kernel<256><<<1, 256, 0, s>>>(keys, vals, keys_alt, vals_alt, (uint32_t)count, bits,
                                                      &b->ctl->err);
        else
            radix_small_kernel<1024><<<1, 1024, 0, s>>>(keys, vals, keys_alt, vals_alt, (uint32_t)count, bits,
                                                        &b->ctl->err);
        count_launches(1);
        std::swap(keys, keys_alt);
        std::swap(vals, vals_alt);
        return cudaGetLastError();
    }
    const SortShape sh = sort_shape(count, bits);
    const SortScratch z = sort_scratch(b, sh);
    if (z.bytes > b->sc.sort_words * sizeof(uint32_t) || bits > 32 || count >= (1ll << 30))
        return cudaErrorInvalidValue;
    if (!counted) {
        const cudaError_t e = z.clear(b);
        if (e) return e;
    }
    const uint32_t n = (uint32_t)count;
    if (sh.digit_bits == 10)
        return sh.items == 4 ? launch_radix_passes<10, 4>(b, keys, vals, keys_alt, vals_alt, n, sh, counted)
                             : launch_radix_passes<10, 16>(b, keys, vals, keys_alt, vals_alt, n, sh, counted);
    return sh.items == 4 ? launch_radix_passes<8, 4>(b, keys, vals, keys_alt, vals_alt, n, sh, counted)
                         : launch_radix_passes<8, 16>(b, keys, vals, keys_alt, vals_alt, n, sh, counted);
}

cudaError_t launch_sort(gputx_bulk *b, uint32_t *&keys, uint32_t *&vals, uint32_t *&keys_alt, uint32_t *&vals_alt,
                        int64_t count, int bits)
{
    return launch_sort_passes(b, keys, vals, keys_alt, vals_alt, count, bits, false);
}

cudaError_t launch_group(gputx_bulk *b, int mode, int part_size, bool by_part, uint32_t *&keys, uint32_t *&vals,
                         uint32_t *&keys_alt, uint32_t *&vals_alt, int bits, int64_t *deltas)
{
    const int64_t n = b->n;
    if (n == 0) return cudaSuccess;
    ExtractOneArgs a;
    a.db = b->db->dev;
    a.b = dev_bulk(b, mode);
    a.ctl = b->ctl;
    a.keys = keys;
    a.vals = vals;
    a.hist = nullptr;
    a.deltas = deltas;
    a.mode = mode;
    a.part_size = part_size < 1 ? 1 : part_size;
    a.passes = 0;
    a.by_part = by_part;
    const SortShape sh = sort_shape(n, bits);
    if (n > SMALL_SORT && bits > 0) {
        const SortScratch z = sort_scratch(b, sh);
        if (z.bytes > b->sc.sort_words * sizeof(uint32_t) || bits > 32) return cudaErrorInvalidValue;
        const cudaError_t e = z.clear(b);
        if (e) return e;
        a.hist = z.hist;
        a.passes = sh.passes;
    }
    // the counts are added up per block: few blocks that stride
    const unsigned grid = (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)b->db->num_sms * 8);
    if (sh.digit_bits == 10) extract_one_kernel<10><<<grid, 256, 0, b->stream>>>(a);
    else extract_one_kernel<8><<<grid, 256, 0, b->stream>>>(a);
    count_launches(1);
    const cudaError_t e = cudaGetLastError();
    if (e) return e;
    return launch_sort_passes(b, keys, vals, keys_alt, vals_alt, n, bits, a.hist != nullptr);
}

cudaError_t launch_rank_scan(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m, bool want_rid,
                             bool aside)
{
    cudaError_t e = cudaMemsetAsync(b->sc.level, 0, b->n * sizeof(uint32_t), b->stream);
    if (e) return e;
    RankMode rm{sk, sv, b->sc.level, want_rid ? b->sc.rid : nullptr};
    return run_scan(b, rm, m, kAnalysisErr, aside);
}

cudaError_t launch_ticket_scan(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m)
{
    const bool fixed = b->db->uniform_k || b->graph;
    TicketMode tm{sk, sv, b->sc.lock_key, b->sc.lock_ticket, fixed ? nullptr : b->sc.op_off,
                  b->graph ? b->db->kmax : b->db->uniform_k, &b->ctl->hot,
                  kTplHot, b->db->dev.n_objects, &b->ctl->err, m};
    cudaError_t e = cudaMemsetAsync(&b->ctl->hot, 0, sizeof(uint32_t), b->stream);
    if (e) return e;
    return run_scan(b, tm, m);
}

// exact depths after the one-pass ranks (A1): the dataflow pass
cudaError_t launch_exact_depth(gputx_bulk *b, const uint32_t *sv, int64_t m, bool aside)
{
    if (b->n == 0) return cudaSuccess;
    if (m >= (int64_t)kPredVal) return cudaErrorInvalidValue;
    cudaStream_t s = b->stream;
    const bool fixed = b->db->uniform_k || b->graph;
    FlowArgs a;
    a.op_off = fixed ? nullptr : b->sc.op_off;
    a.kslots = b->graph ? b->db->kmax : b->db->uniform_k;
    // the per-slot predecessors reuse a TPL buffer (free during the analysis)
    uint32_t *pred = b->sc.lock_key;
    a.pred = pred;
    a.sv = sv;
    a.rid = b->sc.rid;
    a.depths = b->sc.depths;
    a.level = b->sc.level;
    a.ctl = b->ctl;
    a.err = analysis_err(b, aside);
    a.n = b->n;
    a.graph = b->graph;
    a.limit_ns = (uint64_t)b->db->cfg.spin_limit_ns;
    cudaError_t e;
    if (m > 0 && (e = cudaMemsetAsync(pred, 0xff, (size_t)m * sizeof(uint32_t), s))) return e;
    if ((e = cudaMemsetAsync(a.depths, 0xff, (size_t)b->n * sizeof(unsigned long long), s))) return e;
    if ((e = cudaMemsetAsync(&b->ctl->front, 0, sizeof(uint32_t), s))) return e;
    if (m > 0) {
        depth_prep_kernel<<<grid_for(m), TB, 0, s>>>(sv, b->sc.rid, m, a.op_off, a.kslots, pred, b->ctl);
        count_launches(1);
    }
    const size_t smem = (sizeof(uint32_t) * MAX_OPS + sizeof(FlowNode) +
                         sizeof(unsigned long long) * (kFlowPush + 1)) * kFlowThreads;
    if ((e = cudaFuncSetAttribute(depth_flow_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kFlowCluster, 1, 1);
    cfg.blockDim = dim3(kFlowThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kFlowCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if ((e = cudaLaunchKernelEx(&cfg, depth_flow_kernel, a))) return e;
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_depths_aside(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m)
{
    gputx_db *db = b->db;
    const cudaStream_t s = b->stream;
    cudaStream_t side = nullptr;
    for (int i = 0; i < gputx_db::kPool; i++)
        if (db->pool[i] == s) side = db->side[i];
    cudaError_t e = cudaSuccess;
    if (side) {
        e = cudaEventRecord(b->ev_in, s);
        if (!e) e = cudaStreamWaitEvent(side, b->ev_in, 0);
        if (e) return e;
        b->stream = side;
    }
    e = launch_rank_scan(b, sk, sv, m, true, true);
    if (!e) e = launch_exact_depth(b, sv, m, true);
    b->stream = s;
    if (side) {
        const cudaError_t e2 = cudaEventRecord(b->ev_in, side);
        b->aside = true;
        if (!e) e = e2;
    }
    return e;
}

cudaError_t join_depths(gputx_bulk *b)
{
    if (!b->aside) return cudaSuccess;
    b->aside = false;
    return cudaStreamWaitEvent(b->stream, b->ev_in, 0);
}

cudaError_t launch_level_stats(gputx_bulk *b)
{
    if (b->n == 0) return cudaSuccess;
    int blocks = b->db->num_sms * 2;
    const int64_t need = (b->n + 255) / 256;
    if (blocks > need) blocks = (int)need;
    level_stats_kernel<<<blocks, 256, 0, b->stream>>>(b->sc.level, b->n, b->ctl);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_regroup_keys(gputx_bulk *b, uint32_t *keys, uint32_t *vals)
{
    if (b->n == 0) return cudaSuccess;
    const bool seg = b->graph && b->sc.bulk_of;
    regroup_keys_kernel<<<grid_for(b->n), TB, 0, b->stream>>>(b->sc.level, b->type, b->n, b->db->tbits,
                                                               keys, vals, b->graph ? &b->ctl->n_live : nullptr,
                                                               seg ? b->sc.bulk_of : nullptr,
                                                               seg ? b->sc.seg_base : nullptr);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_level_tables(gputx_bulk *b, const uint32_t *skeys, int64_t depth, int block, bool chunks)
{
    cudaStream_t s = b->stream;
    if (b->n == 0) return cudaSuccess;
    level_off_kernel<<<grid_for(b->n), TB, 0, s>>>(skeys, b->n, b->db->tbits, b->sc.level_off, b->sc.type_cut,
                                                   b->ctl, &b->ctl->err);
    count_launches(1);
    if (kDebug) {
        check_level_off_kernel<<<grid_for(b->n + 1), TB, 0, s>>>(b->sc.level_off, b->n, b->ctl);
        count_launches(1);
    }
    if (!chunks) return cudaGetLastError();
    // graph bulks do not know their depth on the host: scan every possible level
    const int64_t levels = b->graph ? b->n : depth + 1;
    ChunkMode cm{b->sc.level_off, b->sc.chunk_off, (uint32_t)block, b->ctl, b->sc.type_cut};
    cudaError_t e = run_scan(b, cm, levels);
    if (e) return e;
    chunk_level_kernel<<<grid_for(b->sc.chunk_cap), TB, 0, s>>>(b->sc.chunk_off, b->ctl, b->sc.chunk_level,
                                                                b->sc.chunk_cap, &b->ctl->err);
    count_launches(1);
    return cudaGetLastError();
}

// history rows of a mixed bulk: exclusive count of debit-credit transactions
// in timestamp order
struct HistSlotMode {
    const int32_t *type;
    int64_t n;
    uint32_t *slot;
    BulkCtl *ctl;
    __device__ uint32_t a(int64_t t) const { return type[t] == GPUTX_T_DC_DEBIT_CREDIT ? 1u : 0u; }
    __device__ uint64_t element(int64_t t) const { return DualSeg::make(0, 0, 0, a(t)); }
    __device__ void output(int64_t t, uint64_t s) const
    {
        const uint32_t v = DualSeg::v2(s);
        slot[t] = v - a(t);
        if (t == n - 1) ctl->total.hist = v;
    }
};

cudaError_t launch_insert_slots(gputx_bulk *b)
{
    if (b->n == 0) return cudaSuccess;
    if (b->sc.slot_hist) {
        HistSlotMode hm{b->type, b->n, b->sc.slot_hist, b->ctl};
        cudaError_t e = run_scan(b, hm, b->n);
        if (e) return e;
    }
    const uint32_t reg = b->db->dev.registered;
    const bool sub_ins = (reg >> GPUTX_T_SUB_INSERT_CF) & 1u;
    const bool oe_no = (reg >> GPUTX_T_OE_NEW_ORDER) & 1u;
    if (!sub_ins && !oe_no) return cudaSuccess;
    SlotMode m0{b->type, b->params, b->P, b->n, b->sc.slot_cf, b->sc.slot_ord, b->ctl, 0};
    cudaError_t e = run_scan(b, m0, b->n);
    if (e || !oe_no) return e;
    SlotMode m1{b->type, b->params, b->P, b->n, nullptr, b->sc.slot_ol, b->ctl, 1};
    return run_scan(b, m1, b->n);
}

cudaError_t launch_part_heads(gputx_bulk *b, const uint32_t *skeys, int64_t n)
{
    if (n <= 0) return cudaSuccess;
    HeadMode hm;
    hm.skeys = skeys;
    hm.part_start = b->sc.part_start;
    hm.ctl = b->ctl;
    hm.n = n;
    hm.n_live = b->graph ? &b->ctl->n_live : nullptr;
    return run_scan(b, hm, n);
}

cudaError_t launch_tpl_reset(gputx_bulk *b, const uint32_t *skeys, int64_t m)
{
    if (m == 0) return cudaSuccess;
    tpl_reset_kernel<<<grid_for(m), TB, 0, b->stream>>>(skeys, m, b->db->d_done, b->db->dev.n_objects,
                                                        b->db->lock_slots);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace gtx
