// exec_oe.cu -- K-SET of bulks that hold order-entry transactions only, item by
// item instead of level by level.
//
// No procedure of order-entry carries a value from one item it writes to
// another: the stock rows an order updates, the customer's cells of a payment
// and the district's counter each depend on their own earlier value and on the
// parameters alone, whether an order aborts (an unknown item, no room for its
// rows) is known from its parameters and insert slots, and only the customer's
// last order takes the id that the district's counter gave.  So the k-th run of
// an item needs the runs before it on the same item, as Property 1 has it, but no
// barrier across items: every item's operations are run in timestamp order, all
// items side by side, the customers' last orders after the counters.  The
// results are those of the levels bit for bit (integers, and each item sees the
// same updates in the same order).
#include <algorithm>

#include "engine.h"
#include "procs.cuh"

namespace gtx {

namespace {

constexpr int kItemThreads = 256;

struct ItemArgs {
    DevDB db;
    DevBulk b;
    BulkCtl *ctl;
    const uint32_t *sk, *sv;   // operations sorted by item (key >> shift), then timestamp
    uint32_t m;
    int shift;
};

__device__ __forceinline__ bool items_stop(const BulkCtl *ctl) { return ctl->err & ~(uint32_t)ERR_CAPACITY; }

// Which new-orders run: status 0, 1 (an unknown item) or 3 (no room), 16 lanes
// an order so that its lines are read side by side.
__global__ void __launch_bounds__(kItemThreads) order_status_kernel(DevDB db, DevBulk b, const BulkCtl *ctl)
{
    if (items_stop(ctl)) return;
    const int64_t n = b.n_live ? (int64_t)*b.n_live : b.n;
    const uint32_t gl = threadIdx.x & (kGroup - 1), gm = group_mask();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x / kGroup;
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kGroup; t < n; t += stride) {
        if (__ldg(&b.type[t]) != GPUTX_T_OE_NEW_ORDER) continue;
        const int64_t *p = b.params + t * b.P;
        const int64_t cnt = __ldg(&p[3]);
        const bool bad = (int64_t)gl < cnt && 4 + (int)gl < b.P && (__ldg(&p[4 + gl]) & 0xFFFFFF) >= db.n_items;
        const bool any = __any_sync(gm, bad);
        if (gl == 0) {
            int st = any ? 1 : 0;
            if (!any && (b.base->ord + b.slot_ord[t] >= db.ord_cap || b.base->ol + b.slot_ol[t] + cnt > db.ol_cap)) {
                set_err(b.err, ERR_CAPACITY);
                st = 3;
            }
            b.status[t] = st;
        }
    }
}

enum ItemKind { kItemNone, kItemHouse, kItemDistrict, kItemCustomer, kItemLast, kItemStock };

// an operation on its lane: the item, the transaction, and what it brings
struct ItemOp {
    uint32_t k, v;
    int64_t x;       // a payment's amount, a line's quantity, an order's id
    uint32_t y;      // a payment's district, an order's slot
    bool live;       // it updates the item
};

struct ItemState {   // an item's cells
    int64_t a, b, c;
    uint32_t q;
};

__device__ __forceinline__ ItemKind item_kind(const DevDB &db, uint32_t k)
{
    if (k >= db.n_objects || k < db.o_wytd) return kItemNone;
    if (k >= db.o_stock) return kItemStock;
    if (k >= db.o_clast) return kItemLast;
    if (k >= db.o_cpay) return kItemCustomer;
    return k >= db.o_dnext ? kItemDistrict : kItemHouse;
}

__device__ __forceinline__ ItemOp item_op(const ItemArgs &a, uint64_t i)
{
    ItemOp o{~0u, OP_SENTINEL, 0, 0, false};
    if (i < a.m) {
        o.k = __ldg(&a.sk[i]) >> a.shift;
        o.v = __ldg(&a.sv[i]);
    }
    return o;
}

// what the operation brings: loads that depend on no other item
__device__ __forceinline__ void item_load(const ItemArgs &a, ItemOp &o, ItemKind kind)
{
    const uint32_t t = o.v >> 7;
    if (kind == kItemNone || !dbg_in(t, a.b.n, a.b.err)) return;
    const int64_t *p = a.b.params + (int64_t)t * a.b.P;
    switch (kind) {
    case kItemHouse:
        o.x = __ldg(&p[3]);
        o.y = (uint32_t)__ldg(&p[1]);
        o.live = true;
        break;
    case kItemCustomer:
        o.live = (o.v & 3u) != CLS_R;
        if (o.live) o.x = __ldg(&p[3]);
        break;
    case kItemDistrict: o.live = a.b.status[t] == 0; break;
    case kItemStock:   // operation 2 + l is line l (an order with an unknown item does not run)
        o.live = a.b.status[t] == 0;
        o.x = (__ldg(&p[2 + ((o.v >> 2) & 31u)]) >> 40) & 0xFF;
        break;
    case kItemLast:
        if ((o.v & 3u) == CLS_R) break;
        o.live = a.b.status[t] == 0;
        o.x = a.b.out[(int64_t)t * a.b.R];
        o.y = (uint32_t)(a.b.base->ord + a.b.slot_ord[t]);
        break;
    default: break;
    }
}

// the sum over the lanes [lo, lane] of each lane's segment
__device__ __forceinline__ int64_t lanes_sum(int64_t x, uint32_t lo, uint32_t lane)
{
#pragma unroll
    for (uint32_t d = 1; d < 32; d <<= 1) {
        const int64_t y = __shfl_up_sync(kFull, x, d);
        if (lane >= lo + d) x += y;
    }
    return x;
}

__device__ __forceinline__ uint32_t stock_after(uint32_t q, uint32_t qty)
{
    return (int32_t)q >= (int32_t)(qty + 10) ? q - qty : q - qty + 91;
}

// A warp runs the items whose operations begin in its 32 positions, to the end
// of the last of them: sums and counts by segmented scans, a stock row's
// quantity (whose rule is no sum) step by step in registers.  LAST: the
// customers' last orders, after the counters; else the others.
//
// What bounds it is random access: an operation reads its transaction's
// parameters and status and writes cells or outputs, one 32-byte sector each.
// 200,003 transactions, 1.3 M operations: 73 us (and 11 for the last orders);
// their 610 levels on a cluster took 2,110, after 190 of regrouping, level tables
// and gathering.
// A long run is a chain of windows on one warp, so the next window's operations
// and parameters are on their way while one is worked on.
template <bool LAST> __global__ void __launch_bounds__(kItemThreads) items_kernel(ItemArgs a)
{
    if (items_stop(a.ctl)) return;
    const uint32_t lane = threadIdx.x & 31;
    uint64_t base = ((uint64_t)blockIdx.x * kItemThreads + threadIdx.x) & ~31ull;
    if (base >= a.m) return;
    const DevDB &db = a.db;
    const DevBulk &b = a.b;
    auto kind_of = [&](uint32_t k) {
        const ItemKind kind = item_kind(db, k);
        return (kind == kItemLast) == LAST ? kind : kItemNone;
    };
    ItemOp cur = item_op(a, base + lane), next = item_op(a, base + 32 + lane);
    ItemKind kind = kind_of(cur.k);
    uint32_t prev = base ? __ldg(&a.sk[base - 1]) >> a.shift : ~0u;     // the item before the window
    bool carried = false;
    ItemState carry{};
    if (!__any_sync(kFull, kind != kItemNone)) return;
    item_load(a, cur, kind);
    while (true) {
        const uint32_t before = __shfl_up_sync(kFull, cur.k, 1), nk = __shfl_sync(kFull, next.k, 0);
        const uint32_t heads = __ballot_sync(kFull, cur.k != (lane ? before : prev));
        uint32_t after = __shfl_down_sync(kFull, cur.k, 1);
        if (lane == 31) after = nk;
        const uint32_t below = heads & (0xffffffffu >> (31 - lane));
        const bool first = below == 0;                                  // the item began in an earlier window
        const uint32_t lo = first ? 0 : 31 - __clz(below);
        const bool house = kind == kItemHouse;
        // (a warehouse's total is summed window by window, whoever began it)
        const bool act = kind != kItemNone && (house ? !carried : carried == first);
        const bool ends = after != cur.k;
        const bool more = __shfl_sync(kFull, act && !house && !ends, 31);
        ItemOp ahead{~0u, OP_SENTINEL, 0, 0, false};
        const ItemKind next_kind = more ? kind_of(next.k) : kItemNone;
        if (more) {
            item_load(a, next, next_kind);
            ahead = item_op(a, base + 64 + lane);
        }
        ItemState s = carry;
        if (act && !first) {
            switch (kind) {
            case kItemDistrict: s.a = __ldcg(&db.d_next_o_id[cur.k - db.o_dnext]); break;
            case kItemCustomer: {
                const uint32_t c = cur.k - db.o_cpay;
                s.a = __ldcg(&db.c_balance[c]);
                s.b = __ldcg(&db.c_ytd[c]);
                s.c = __ldcg(&db.c_payment_cnt[c]);
                break;
            }
            case kItemStock: {
                const uint32_t r = cur.k - db.o_stock;
                s.q = (uint32_t)ldg_cg(&db.s_quantity[r]);
                s.b = __ldcg(&db.s_ytd[r]);
                s.c = ldg_cg(&db.s_order_cnt[r]);
                break;
            }
            case kItemLast: {
                const uint32_t c = cur.k - db.o_clast;
                s.a = __ldcg(&db.c_last_o_id[c]);
                s.q = __ldcg(&db.c_last_slot[c]);
                break;
            }
            default: break;
            }
        }
        const bool live = act && cur.live;
        const uint32_t alive = __ballot_sync(kFull, live) & (0xffffffffu >> (31 - lane)) & (0xffffffffu << lo);
        const uint32_t t = cur.v >> 7;
        int64_t *out = b.out + (int64_t)t * b.R;
        if (LAST) {
            // the customer's last order at this operation: the nearest before it
            const int src = alive ? 31 - __clz(alive) : 0;
            const int64_t o = __shfl_sync(kFull, cur.x, src);
            const uint32_t slot = __shfl_sync(kFull, cur.y, src);
            if (alive) {
                s.a = o;
                s.q = slot;
            }
            if (act && (cur.v & 3u) == CLS_R) {
                out[1] = s.a;
                out[2] = s.a == 0 ? 0 : (int64_t)s.q;
                b.status[t] = s.a == 0 ? 1 : 0;
            }
            if (act && ends) {
                const uint32_t c = cur.k - db.o_clast;
                __stcg(&db.c_last_o_id[c], s.a);
                stg_cg(&db.c_last_slot[c], s.q);
            }
        } else {
            const int64_t sum = lanes_sum(live ? cur.x : 0, lo, lane);
            const int cnt = __popc(alive);
            // stock quantities: place by place within the runs of the window
            const bool stock = act && kind == kItemStock;
            const uint32_t qty = (uint32_t)cur.x;
            if (__any_sync(kFull, stock)) {
                if (__all_sync(kFull, stock) && lo == 0 && !(heads & ~1u)) {
                    // one row's: every lane goes through all of them
                    const uint32_t d = live ? qty : 0xffffu;
#pragma unroll
                    for (int i = 0; i < 32; i++) {
                        const uint32_t di = __shfl_sync(kFull, d, i);
                        if (di != 0xffffu) s.q = stock_after(s.q, di);
                    }
                } else {
                    const uint32_t place = lane - lo, steps = __reduce_max_sync(kFull, stock ? place : 0);
                    if (live && place == 0) s.q = stock_after(s.q, qty);
                    for (uint32_t i = 1; i <= steps; i++) {
                        const uint32_t q = __shfl_up_sync(kFull, s.q, 1);
                        if (place == i) s.q = live ? stock_after(q, qty) : q;
                    }
                }
            }
            switch (act ? kind : kItemNone) {
            case kItemHouse: {
                const uint32_t w = cur.k - db.o_wytd;
                if (ends || lane == 31) atomicAdd((unsigned long long *)&db.w_ytd[w], (unsigned long long)sum);
                if (dbg_in(cur.y, OE_DIST, b.err))
                    atomicAdd((unsigned long long *)&db.d_ytd[(int64_t)w * OE_DIST + cur.y], (unsigned long long)cur.x);
                break;
            }
            case kItemDistrict:
                s.a += cnt;
                if (live) out[0] = s.a - 1;
                if (ends) __stcg(&db.d_next_o_id[cur.k - db.o_dnext], s.a);
                break;
            case kItemCustomer: {
                s.a = wrap_add(s.a, -sum);
                s.b = wrap_add(s.b, sum);
                s.c += cnt;
                out[0] = s.a;
                if (live) b.status[t] = 0;
                if (ends) {
                    const uint32_t c = cur.k - db.o_cpay;
                    __stcg(&db.c_balance[c], s.a);
                    __stcg(&db.c_ytd[c], s.b);
                    __stcg(&db.c_payment_cnt[c], s.c);
                }
                break;
            }
            case kItemStock: {
                s.b += sum;
                s.c += cnt;
                if (ends) {
                    const uint32_t r = cur.k - db.o_stock;
                    stg_cg(&db.s_quantity[r], (int32_t)s.q);
                    __stcg(&db.s_ytd[r], s.b);
                    stg_cg(&db.s_order_cnt[r], (int32_t)s.c);
                }
                break;
            }
            default: break;
            }
        }
        if (!more) break;
        carry.a = __shfl_sync(kFull, s.a, 31);
        carry.b = __shfl_sync(kFull, s.b, 31);
        carry.c = __shfl_sync(kFull, s.c, 31);
        carry.q = __shfl_sync(kFull, s.q, 31);
        prev = __shfl_sync(kFull, cur.k, 31);
        carried = true;
        cur = next;
        kind = next_kind;
        next = ahead;
        base += 32;
    }
}

}  // namespace

bool oe_only(const gputx_db *db)
{
    constexpr uint32_t oe = 1u << GPUTX_T_OE_NEW_ORDER | 1u << GPUTX_T_OE_PAYMENT | 1u << GPUTX_T_OE_ORDER_STATUS;
    return db->dev.registered && !(db->dev.registered & ~oe);
}

cudaError_t launch_items(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m, int shift)
{
    gputx_db *db = b->db;
    if (b->n == 0 || m == 0) return cudaSuccess;
    ItemArgs a;
    a.db = db->dev;
    a.b = make_dev_bulk(b, GPUTX_CONFLICT_PAPER);
    a.ctl = b->ctl;
    a.sk = sk;
    a.sv = sv;
    a.m = (uint32_t)m;
    a.shift = shift;
    const bool orders = db->dev.registered >> GPUTX_T_OE_NEW_ORDER & 1u;
    const unsigned grid = (unsigned)((m + kItemThreads - 1) / kItemThreads);
    if (orders) {
        const unsigned og = (unsigned)std::min<int64_t>((b->n * kGroup + kItemThreads - 1) / kItemThreads,
                                                        (int64_t)db->num_sms * 8);
        order_status_kernel<<<og, kItemThreads, 0, b->stream>>>(db->dev, a.b, b->ctl);
        count_launches(1);
    }
    items_kernel<false><<<grid, kItemThreads, 0, b->stream>>>(a);
    items_kernel<true><<<grid, kItemThreads, 0, b->stream>>>(a);
    count_launches(2);
    return cudaGetLastError();
}

}  // namespace gtx
