// exec_dc.cu -- execution of a debit-credit bulk whose transactions are
// grouped by branch (or by a partition of branches), in timestamp order
// inside each group: K-SET under the read/write model (Section 5.3), PART
// (Section 5.2) and relaxed PART (Appendix G).
//
// Under the read/write model every transaction has one basic operation, the
// write of its branch (access_set), so the T-dependency graph is one path per
// branch and the k-th k-set holds the k-th transaction of every path.  No
// edge joins two paths: a transaction of the k-th k-set depends on its own
// path's (k-1)-th transaction and on nothing else of that k-set, so the
// barrier between k-sets is only needed along a path.  Each path therefore
// runs through its own part of the k-sets by itself.  A partition of PART is
// the same thing without the k-set numbers.
#include "dc.cuh"
#include "engine.h"
#include "ranges.cuh"

namespace gtx {

namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kTab = 512;                    // hash slots, at most kThreads used
constexpr uint32_t kFree = 0xffffffffu;      // an unused slot's account

// accounts of one window: the balance after it, for the window that follows
struct Window {
    uint32_t acct[kTab];
    uint32_t warps[kTab];                    // warps that have the account
    int64_t bal[kTab];
};

struct RangeArgs {
    DevDB db;
    DevBulk b;
    BulkCtl *ctl;
    const InsertBase *cursor;
    const uint32_t *keys, *vals;             // sorted by group; transaction = vals >> vshift
    int vshift;
    uint32_t slice;                          // positions per CTA before it follows its last group
    bool stats;                              // record d and w0
    bool pair;                               // a signature's first two parameters are one 16-byte load
};

__device__ __forceinline__ uint32_t acct_hash(uint32_t a) { return (a * 2654435761u) >> 23; }
static_assert(kTab == 512, "acct_hash yields 9 bits");

// A CTA runs the groups that begin in its slice of the sorted positions, from
// the first group's head to the last group's end, 256 positions (a window) at
// a time.  Groups share no account, so windows need not respect their bounds.
// In a window, the transactions on one account form a chain: a transaction's
// new balance is the balance before the window plus the deltas of the chain
// up to it, in position (timestamp) order -- the serial result bit for bit.
// Lanes of a warp that share an account combine by __match_any_sync; their
// lowest lane enters the account and the warp's sum into a shared-memory hash
// table; after a barrier each lane adds the sums of the warps before it, and
// the chain's last warp stores the new balance.
//
// What bounds it is the latency of a window times the windows of the longest
// group, so what a window reads is on its way before it: transaction indices
// four windows ahead, signatures three, balances two (into L2) and one.  A
// balance loaded one window ahead misses that window's own additions; those
// are found in its table.  An otherwise idle SM does a window in 1.2 us (the
// hot branch of Zipf 0.99 accounts), so 256 k-sets of a path cost what the
// barrier of one cost across a cluster (1.3 us; the level runner this replaced).
// Measured on 1,000 branches and 10M accounts under R/W, this kernel against
// the level runner: 2^22 transactions 190 us against 5,600; 200,000 with Zipf
// 0.99 accounts 57 against 6,300; 4 branches, 4,096 transactions 12 against 750.
__global__ void __launch_bounds__(kThreads, 4) dc_range_kernel(RangeArgs a)
{
    __shared__ Window s_win[2];
    __shared__ int64_t s_sum[kTab][kWarps - 1];   // per account and warp but the last: the warp's deltas
    __shared__ uint32_t s_head[kWarps], s_min, s_stop;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const DevBulk &b = a.b;
    const uint32_t n = b.n_live ? *b.n_live : (uint32_t)b.n;
    if (tid == 0) s_stop = *(volatile uint32_t *)&a.ctl->err || !rows_fit(a.cursor, n, a.db.hist_cap, &a.ctl->err);
    __syncthreads();
    uint32_t lo, hi;
    if (s_stop || !group_range<kThreads>(a.keys, n, a.slice, &s_min, lo, hi)) return;   // uniform
    for (uint32_t i = tid; i < kTab; i += kThreads)
        for (int w = 0; w < 2; w++) {
            s_win[w].acct[i] = kFree;
            s_win[w].warps[i] = 0;
        }

    auto txn_at = [&](uint32_t p) { return p < hi ? __ldcs(&a.vals[p]) >> a.vshift : 0u; };
    // the account and delta of position p (kFree: none there)
    auto row_of = [&](uint32_t p, uint32_t t, uint32_t &acct, int64_t &delta) {
        acct = kFree;
        delta = 0;
        if (p >= hi || !dbg_in(t, b.n, b.err)) return;
        const int64_t *row = b.params + (int64_t)t * b.P;
        if (a.pair) {
            const longlong2 r = __ldg(reinterpret_cast<const longlong2 *>(row));
            acct = (uint32_t)r.x;
            delta = r.y;
        } else {
            acct = (uint32_t)__ldg(row);
            delta = __ldg(row + 1);
        }
        if (!dbg_in(acct, a.db.n_acc, b.err)) acct = kFree;
    };
    // this window's transaction, the next two windows' and the index of the third
    uint32_t pos = lo + tid;
    uint32_t t0 = txn_at(pos), t1 = txn_at(pos + kThreads), t2 = txn_at(pos + 2 * kThreads);
    uint32_t t3 = txn_at(pos + 3 * kThreads);
    uint32_t acc0, acc1, acc2;
    int64_t d0, d1, d2;
    row_of(pos, t0, acc0, d0);
    row_of(pos + kThreads, t1, acc1, d1);
    row_of(pos + 2 * kThreads, t2, acc2, d2);
    int64_t bal0 = acc0 != kFree ? __ldcg(&a.db.acc_bal[acc0]) : 0;
    uint32_t key0 = 0, prev0 = 0;
    if (a.stats && pos < hi) {
        key0 = __ldg(&a.keys[pos]);
        prev0 = pos ? __ldg(&a.keys[pos - 1]) : ~key0;
    }
    uint32_t heads = 0, longest = 0, start = lo;   // d, w0: groups seen, the longest, the open one's head
    int cur = 0;
    __syncthreads();
    for (uint32_t base = lo; base < hi; base += kThreads, pos += kThreads) {
        Window &now = s_win[cur], &before = s_win[cur ^ 1];
        const bool act = acc0 != kFree;
        // the balance was loaded before the window before this one stored its own
        int64_t bal = bal0;
        if (act)
            for (uint32_t e = acct_hash(acc0);; e = (e + 1) & (kTab - 1)) {
                const uint32_t k = before.acct[e];
                if (k == acc0) bal = before.bal[e];
                if (k == acc0 || k == kFree) break;
            }
        // in flight during this window: balances of the next (and of the one
        // after it into L2), signatures of the third, indices of the fourth
        const int64_t bal1 = acc1 != kFree ? __ldcg(&a.db.acc_bal[acc1]) : 0;
        if (acc2 != kFree) prefetch_l2(&a.db.acc_bal[acc2]);
        uint32_t acc3;
        int64_t d3;
        row_of(pos + 3 * kThreads, t3, acc3, d3);
        const uint32_t t4 = txn_at(pos + 4 * kThreads);
        uint32_t key1 = 0, prev1 = 0;
        if (a.stats && pos + kThreads < hi) {
            key1 = __ldg(&a.keys[pos + kThreads]);
            prev1 = __ldg(&a.keys[pos + kThreads - 1]);
        }
        // this warp's part of each account's chain
        const uint32_t live = __ballot_sync(kFull, act);
        const uint32_t peers = __match_any_sync(kFull, acc0) & live;
        int64_t pre = d0, tot = d0;
        if (__any_sync(kFull, act && (peers & (peers - 1)))) {
            pre = lanes_prefix(act ? peers : 1u << lane, d0);
            tot = __shfl_sync(kFull, pre, act ? 31 - __clz(peers) : lane);
        }
        const uint32_t first = act ? (uint32_t)__ffs(peers) - 1 : lane;
        uint32_t e = 0;
        if (act && lane == first) {
            e = acct_hash(acc0);
            while (true) {
                const uint32_t k = atomicCAS(&now.acct[e], kFree, acc0);
                if (k == kFree || k == acc0) break;
                e = (e + 1) & (kTab - 1);
            }
            atomicOr(&now.warps[e], 1u << warp);
            if (warp < kWarps - 1) s_sum[e][warp] = tot;
        }
        e = __shfl_sync(kFull, e, first);
        const bool is_head = a.stats && pos < hi && key0 != prev0;
        const uint32_t hm = __ballot_sync(kFull, is_head);
        if (a.stats && lane == 0) s_head[warp] = hm ? base + warp * 32 + 31 - __clz(hm) : kFull;
        __syncthreads();
        if (act) {
            const uint32_t ws = now.warps[e];
            int64_t sum = bal;
#pragma unroll
            for (int w = 0; w < kWarps - 1; w++)
                if (w < (int)warp && (ws >> w & 1u)) sum = wrap_add(sum, s_sum[e][w]);
            if (lane == first && (ws >> warp) == 1u) {   // the chain's last warp
                const int64_t after = wrap_add(sum, tot);
                now.bal[e] = after;
                __stcg(&a.db.acc_bal[acc0], after);
            }
            b.out[(int64_t)t0 * b.R] = wrap_add(sum, pre);
        }
        if (a.stats) {
            heads += is_head;
            // a head closes the group before it, which began at the last head
            // below: in this warp, in a warp before, or in an earlier window
            const uint32_t h = lane < kWarps ? s_head[lane] : kFull;
            const uint32_t with = __ballot_sync(kFull, h != kFull);
            const uint32_t low = with & ((1u << warp) - 1u);
            const uint32_t from_low = __shfl_sync(kFull, h, low ? 31 - __clz(low) : 0);
            const uint32_t last = __shfl_sync(kFull, h, with ? 31 - __clz(with) : 0);
            if (is_head && pos > lo) {
                const uint32_t below = hm & ((1u << lane) - 1u);
                const uint32_t from = below ? base + warp * 32 + 31 - __clz(below) : low ? from_low : start;
                longest = pos - from > longest ? pos - from : longest;
            }
            if (with) start = last;            // the open group of the next window
        }
        // the table before this one is done with: it takes the next window
        for (uint32_t i = tid; i < kTab; i += kThreads) {
            before.acct[i] = kFree;
            before.warps[i] = 0;
        }
        cur ^= 1;
        t0 = t1;
        t1 = t2;
        t2 = t3;
        t3 = t4;
        acc0 = acc1;
        d0 = d1;
        acc1 = acc2;
        d1 = d2;
        acc2 = acc3;
        d2 = d3;
        bal0 = bal1;
        key0 = key1;
        prev0 = prev1;
        __syncthreads();
    }
    if (a.stats) {
        longest = hi - start > longest ? hi - start : longest;   // the last group
        longest = __reduce_max_sync(kFull, longest);
        heads = __reduce_add_sync(kFull, heads);
        if (lane == 0) {
            if (longest > 1) atomicMax(&a.ctl->depth, longest - 1);
            if (heads) atomicAdd(&a.ctl->w0, heads);
        }
    }
}

}  // namespace

cudaError_t launch_dc_ranges(gputx_bulk *b, const uint32_t *keys, const uint32_t *vals, int vshift, bool stats)
{
    if (b->n == 0) return cudaSuccess;
    RangeArgs a;
    a.db = b->db->dev;
    a.b = make_dev_bulk(b, GPUTX_CONFLICT_PAPER);
    a.ctl = b->ctl;
    a.cursor = b->db->d_cursor;
    a.keys = keys;
    a.vals = vals;
    a.vshift = vshift;
    a.stats = stats;
    a.pair = b->P % 2 == 0 && reinterpret_cast<uintptr_t>(b->params) % 16 == 0;
    // small slices spread short groups over the chip; a slice inside a long
    // group costs an empty CTA.  1,000 branches, slices of 256 against 1,024, us:
    // 2^17 12.8 / 18.8, 2^18 22.1 / 21.3, 2^20 62.4 / 59.6, 2^22 217 / 193; with
    // Zipf 0.8 accounts 13.5 / 17.6, 21.7 / 25.1, 72.3 / 69.7, 323 / 303
    a.slice = b->n <= (1 << 20) ? kThreads : 4 * kThreads;
    const int64_t grid = (b->n + a.slice - 1) / a.slice;
    const cudaError_t e = clear_outputs(b);
    if (e) return e;
    dc_range_kernel<<<(unsigned)grid, kThreads, 0, b->stream>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace gtx
