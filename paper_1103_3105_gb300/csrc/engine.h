// engine.h -- host-side state of a database and a bulk, and the launchers each
// translation unit provides.  Internal to the library.
#pragma once
#include <cuda_runtime.h>

#include <string>
#include <vector>

#include "common.cuh"

namespace gtx {

// Per-bulk control block in device memory (zeroed at submit).
struct BulkCtl {
    uint32_t err;          // ERR_* bits
    uint32_t depth;        // d: depth of the T-dependency graph
    uint32_t w0;           // 0-set size
    uint32_t last_level;   // largest entry of the level array (below d where blind increments do not order it)
    uint32_t cross;        // cross-partition transactions
    uint32_t npart;        // PART: non-empty partitions
    uint32_t claim;        // executors: next chunk to claim
    uint32_t n_live;       // fixed-capacity bulks: live transactions (the rest pad)
    InsertBase base;       // where this bulk's inserts start (copied from the cursor)
    InsertBase total;      // inserts this bulk reserves
    uint32_t rounds;       // exact-depth passes run (the dataflow pass: 1)
    uint32_t n_seg;        // segmented graph bulks: bulks in this segment (0 = one)
    uint32_t hot;          // TPL: operations before the last of the longest chain, if kTplHot at least (else 0)
    uint32_t chunk;        // relaxed TPL: next chunk to claim (claim counts commit tickets)
    uint32_t front;        // exact depth: chunks of transactions finished
    uint32_t rows_done;    // debit-credit rows: blocks finished
    uint32_t depth_err;    // launch_depths_aside: its ERR_* bits, which the execution beside it does not read
};

constexpr uint32_t kTplHot = 128;  // debit-credit TPL: a chain longer than this is served in lock order

// and where the bulk is this many times as long, a warp takes a run of 32s.  At
// 200,003 transactions, two 32s a warp, that line is where both are the same (16
// chains 858 us in runs, 834 with one 32; 32 445 / 447; 64 235 / 241; 128 133 /
// 135); at 2^20, seven a warp, runs are faster on both sides of it (16 chains 6.0
// ms against 12.3, 64 1.57 / 3.61, 256 0.42 / 1.04)
constexpr int kTplMany = 64;

constexpr int kScanAreas = 3;      // scans of a submitted bulk whose scratch its submission has cleared

constexpr int kSegMax = 64;        // bulks in one segment of a graph bulk, at most

// Scratch carved from one per-bulk allocation.
struct Scratch {
    uint32_t *keys_a, *vals_a, *keys_b, *vals_b;  // sort ping-pong, m entries each
    uint32_t *op_off;      // n+1 exclusive op offsets (non-uniform op counts)
    uint32_t *level;       // n
    uint32_t *rid;         // m: place in its run per sorted op (exact depth)
    unsigned long long *depths;   // n: a finished transaction's depth and level (exact depth)
    uint32_t *lock_key;    // m: TPL per-op object, indexed by op slot
    uint32_t *lock_ticket; // m
    uint32_t *level_off;   // n+2
    uint32_t *type_cut;    // 2 (n+2): per level, where types >= new-order, payment start
    uint32_t *chunk_off;   // n+2
    uint32_t *chunk_level; // n + n/min_block + 2
    uint32_t *done;        // n+1 per-level completion counters
    uint32_t *part_start;  // n
    uint32_t *pid_key, *pid_val, *pid_key2, *pid_val2;  // PART sort, n each (the op buffers: PART sorts no ops)
    int64_t *rec_params, *rec_ts;  // signatures gathered into execution order
    int32_t *rec_type;
    uint32_t *rec_t;
    uint32_t *slot_cf, *slot_ord, *slot_ol;   // n each
    uint32_t *slot_hist;   // n: history rows of debit-credit transactions in mixed databases
    uint32_t *sort_zero;   // a sort's tile counters, digit counts and look-back words, cleared by it at once
    uint64_t *scan_zero;   // kScanAreas times a scan's tile counter and look-back words, likewise
    uint64_t *scan_vals;   // 2 x tiles: per-tile values of 64-bit scans
    char *cleared;         // end of what the submission clears (from `status`)
    // graph bulks that carry a segment of several bulks
    uint32_t *seg_off;     // kSegMax + 1: first transaction of each bulk
    uint32_t *bulk_of;     // n: bulk of each transaction
    uint32_t *seg_depth;   // kSegMax: largest level of each bulk
    uint32_t *seg_base;    // kSegMax + 1: first global level of each bulk
    int64_t m_cap;         // op capacity
    int64_t sort_words, scan_tiles, chunk_cap;   // capacity of sort_zero (words), of the scans (tiles)
};

}  // namespace gtx

struct gputx_db {
    gtx::DevDB dev{};
    gputx_schema_desc schema{};
    gputx_config cfg{};
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int device = 0;
    int num_sms = 0;
    bool reads_host = false;               // kernels can read any host memory through the host's page tables
    std::string last_error;
    std::vector<void *> allocs;
    gtx::InsertBase *d_cursor = nullptr;   // device insert cursors
    uint32_t *d_done = nullptr;            // TPL per-object counters, kept zero between bulks
    gtx::LockSlots lock_slots{};           // item -> slot of d_done (32 x lines words)
    int kmax = 0;                          // largest op count of a registered type
    int uniform_k = 0;                     // every registered type has exactly this many ops (0 = no)
    bool need_fixpoint = false;            // a registered type's ops may leave one-pass ranks inexact
    int tbits = 0;                         // type bits in the level/type regroup key
    bool group_oe = false;                 // K-SET runs new-orders on 16-lane groups, orders are completed after it
    bool hist_by_type = false;             // debit-credit and other types: history rows for debit-credit only
    int obj_bits = 1;                      // key bits of object ids
    // Each bulk runs on a stream of this pool, so the analysis of one bulk
    // overlaps the execution of the one before; `last_done` orders the
    // database-touching tail of every bulk after that of its predecessor.
    static constexpr int kPool = 4;
    cudaStream_t pool[kPool] = {};
    // order-entry: the depths of a bulk on a pool stream are computed on its
    // side stream, beside the bulk's execution (created with the types)
    cudaStream_t side[kPool] = {};
    int next_pool = 0;
    cudaEvent_t last_done = nullptr;
    // relaxed PART: per-partition counters and their prefix-scan scratch,
    // allocated at first use (used only inside a bulk's ordered tail)
    uint32_t *part_cnt = nullptr;          // part_cnt_n counters, zero between bulks
    uint32_t *part_off = nullptr;          // part_cnt_n + 1 offsets
    int64_t part_cnt_n = 0;
    uint64_t *part_scan_status = nullptr;
    uint32_t *part_tile_ctr = nullptr;
};

struct gputx_bulk {
    gputx_db *db = nullptr;
    cudaStream_t stream = nullptr;          // this bulk's stream (from the database's pool)
    cudaEvent_t ev_in = nullptr;            // inputs ready on the database stream; later the side stream's fork and join
    bool aside = false;                     // work on the side stream that the bulk's stream has not waited for
    int64_t n = 0;
    int P = 0, R = 0;
    void *arena = nullptr;
    size_t arena_bytes = 0;
    int64_t *ts = nullptr;
    int32_t *type = nullptr;
    int64_t *params = nullptr;
    int32_t *status = nullptr;
    int64_t *out = nullptr;
    gtx::BulkCtl *ctl = nullptr;
    gtx::Scratch sc{};
    bool executed = false;
    bool synced = false;
    const uint32_t *serial_order = nullptr;   // relaxed strategies: the serial order executed
    bool graph = false;    // fixed capacity, padded with inactive transactions,
                           // no host synchronisation (capturable in a CUDA graph)
    int strategy_run = -1;
    int fallback = 0;
    int64_t fixpoint_rounds = 0;
    bool timing = false;
    cudaEvent_t ev[8] = {};
    gtx::BulkCtl host_ctl{};
    gtx::BulkCtl *pinned_ctl = nullptr;     // where the control block is copied as the bulk ends (or null)
    bool ctl_copied = false;                // that copy precedes ev[7]
    bool sort_clear = false;                // the sort scratch is as its submission cleared it
    int scans = gtx::kScanAreas;            // scans run so far, of those with a cleared area
    std::vector<uint32_t> level_off_host;   // K-SET level boundaries read back for launch planning
    std::vector<uint32_t> type_cut_host;    // and where the new-orders and payments start in each level
};

namespace gtx {

// analysis.cu
DevBulk make_dev_bulk(gputx_bulk *b, int mode);
cudaError_t launch_extract(gputx_bulk *b, int mode, int part_size, uint32_t *pid_key, uint32_t *pid_val,
                           bool write_ops, bool segmented = false);
// segmented graph bulks: bulk of each transaction; per-bulk depths and the
// global level numbering (bulk by bulk, levels in order)
int seg_bits(const gputx_db *db);
cudaError_t launch_seg_index(gputx_bulk *b);
cudaError_t launch_seg_levels(gputx_bulk *b);
// PART in a graph: flags a segment with cross-partition transactions (it
// then runs nothing and is re-run with TPL)
cudaError_t launch_part_fallback_check(gputx_bulk *b);
int64_t sort_scratch_words(int64_t count);   // scratch of a sort of up to `count` pairs
// single-operation bulks: keys and payloads by item (payload as launch_extract's)
// or by partition (payload = transaction), sorted; `deltas` (debit-credit-only
// bulks): each transaction's delta side by side, for launch_scan_exec
cudaError_t launch_group(gputx_bulk *b, int mode, int part_size, bool by_part, uint32_t *&keys, uint32_t *&vals,
                         uint32_t *&keys_alt, uint32_t *&vals_alt, int bits, int64_t *deltas = nullptr);
cudaError_t launch_sort(gputx_bulk *b, uint32_t *&keys, uint32_t *&vals, uint32_t *&keys_alt,
                        uint32_t *&vals_alt, int64_t count, int bits);
// `aside`: a wait that runs out is noted in depth_err, not in err
cudaError_t launch_rank_scan(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m, bool want_rid,
                             bool aside = false);
cudaError_t launch_ticket_scan(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m);
// d, w0 and the level array, exact; the rank scan's rid precedes it
cudaError_t launch_exact_depth(gputx_bulk *b, const uint32_t *sv, int64_t m, bool aside = false);
// d, w0 of the one-pass ranks
cudaError_t launch_level_stats(gputx_bulk *b);
cudaError_t launch_regroup_keys(gputx_bulk *b, uint32_t *keys, uint32_t *vals);
cudaError_t launch_level_tables(gputx_bulk *b, const uint32_t *skeys, int64_t depth, int block, bool chunks);
cudaError_t launch_insert_slots(gputx_bulk *b);
cudaError_t launch_part_heads(gputx_bulk *b, const uint32_t *skeys, int64_t n);
cudaError_t launch_tpl_reset(gputx_bulk *b, const uint32_t *skeys, int64_t m);
cudaError_t launch_gather(gputx_bulk *b, const uint32_t *order);
cudaError_t launch_begin(gputx_bulk *b);
cudaError_t launch_finish(gputx_bulk *b);

// exec.cu
cudaError_t launch_kset(gputx_bulk *b, int64_t nchunks, int block, bool atomic_add);
cudaError_t launch_kset_levels(gputx_bulk *b, const uint32_t *level_off_host, int64_t depth, int narrow_max,
                               bool atomic_add, const uint32_t *type_cut_host = nullptr);
// single-operation bulks, from the sorted operations: item by item, run by run
cudaError_t launch_kset_rounds(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, bool stats, bool atomic_add);
cudaError_t launch_part(gputx_bulk *b, const uint32_t *pkeys, int block, int64_t max_parts);
cudaError_t launch_tpl(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int block, bool atomic_add);
// after K-SET's levels, after TPL, after the items: the rows of the new orders,
// then what the order-statuses read of them.  `decided`: launch_items preceded
cudaError_t launch_orders(gputx_bulk *b, bool decided);
// a conflict-free bulk (a 0-set) in one launch
cudaError_t launch_independent(gputx_bulk *b, bool atomic_add);
// relaxed timestamps (Appendix G)
cudaError_t launch_tpl_relaxed(gputx_bulk *b, uint32_t *order, bool atomic_add);
cudaError_t launch_validate(gputx_bulk *b);
cudaError_t launch_part_count(gputx_bulk *b, int mode, int part_size, uint32_t *cnt, int64_t parts,
                              uint32_t *pid_of, uint32_t *key_of);
cudaError_t launch_part_offsets(gputx_bulk *b, const uint32_t *cnt, uint32_t *off, int64_t parts, uint64_t *status,
                                uint32_t *tile_ctr);
cudaError_t launch_part_scatter(gputx_bulk *b, const uint32_t *off, const uint32_t *pid_of, const uint32_t *key_of,
                                uint32_t *pkeys, uint32_t *order);
// debit-credit-only bulks: the account updates of transactions (vals >> vshift)
// grouped by branch or partition (exec_dc.cu), or by account (segmented prefix
// sums); then the history rows, statuses and teller and branch sums.  These take
// the place of the whole tail, launch_begin and launch_finish included: the
// bulk's rows start at the database's cursor, which launch_dc_rows moves on, and
// all fit or nothing runs (ERR_CAPACITY).  `stats`: the groups are the graph's
// paths, d and w0 are recorded
cudaError_t launch_dc_ranges(gputx_bulk *b, const uint32_t *keys, const uint32_t *vals, int vshift, bool stats);
// (the deltas launch_group left in sc.rec_ts)
cudaError_t launch_scan_exec(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m, bool stats);
cudaError_t launch_dc_rows(gputx_bulk *b);
bool dc_only(const gputx_db *db);
// order-entry-only bulks under K-SET, from the operations sorted by item (key >>
// shift), item by item (exec_oe.cu); launch_orders follows
bool oe_only(const gputx_db *db);
cudaError_t launch_items(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m, int shift);
// the rank scan and launch_exact_depth on the bulk's side stream, beside its
// execution, which needs neither: if a wait of theirs runs out, the bulk is
// applied all the same and the depths are reported as unknown.  join_depths makes
// the bulk's own stream wait for them (nothing to do if it has)
cudaError_t launch_depths_aside(gputx_bulk *b, const uint32_t *sk, const uint32_t *sv, int64_t m);
cudaError_t join_depths(gputx_bulk *b);
cudaError_t clear_outputs(gputx_bulk *b);
int exec_blocks_per_sm(int kind, int block);

// tables.cu
cudaError_t launch_fill_i64(int64_t *p, int64_t n, int64_t v, cudaStream_t s);
cudaError_t launch_fill_u64(unsigned long long *p, int64_t n, unsigned long long v, cudaStream_t s);

// kernels launched by this library since load (tracing)
void count_launches(int k);

inline int bits_for(uint64_t maxval)
{
    int b = 0;
    while (b < 32 && (maxval >> b) != 0) b++;
    return b;
}

}  // namespace gtx
