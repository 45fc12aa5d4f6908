// scan.cuh -- single-pass tile scans with decoupled look-back, and the LSD
// radix sort used by the dependency analysis (Section 4.2 steps
// 1 and 4: "a sort operation to perform grouping").
//
// Both follow published designs: decoupled look-back (Merrill & Garland,
// "Single-pass Parallel Prefix Scan with Decoupled Look-back", 2016) and the
// onesweep radix sort built on it (Adinets & Merrill, "Onesweep: A Faster
// Least Significant Digit Radix Sort for GPUs", 2022).  Tiles take their ids
// from an atomic counter, so every tile a look-back waits on has already
// started and publishes its aggregate before it waits on anyone: the waits
// always end.  They are bounded anyway (ERR_TIMEOUT) so that a fault never
// turns into a hang.
#pragma once
#include "common.cuh"

namespace gtx {

// ---------------------------------------------------------------------------
// relaxed gpu-scope accesses for look-back status words
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u32(uint32_t *p, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint64_t ld_relaxed_u64(const uint64_t *p)
{
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u64(uint64_t *p, uint64_t v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// ===========================================================================
// dual segmented sum: the scan state used by every analysis scan
// ===========================================================================
// 62-bit payload: [61] f1 [60:31] v1 (30 bits) [30] f2 [29:0] v2 (30 bits).
// Each (f, v) field is a segmented sum: a set flag starts a new segment.
// A field whose flag is never set is a plain prefix sum.
struct DualSeg {
    static constexpr uint64_t M30 = (1ull << 30) - 1;
    static constexpr uint64_t BOTH = (1ull << 61) | (1ull << 30);   // both flags
    __device__ __forceinline__ static uint64_t make(uint32_t f1, uint32_t v1, uint32_t f2, uint32_t v2)
    {
        return ((uint64_t)f1 << 61) | ((uint64_t)(v1 & M30) << 31) | ((uint64_t)f2 << 30) | (uint64_t)(v2 & M30);
    }
    __device__ __forceinline__ static uint32_t f1(uint64_t s) { return (uint32_t)(s >> 61) & 1u; }
    __device__ __forceinline__ static uint32_t v1(uint64_t s) { return (uint32_t)((s >> 31) & M30); }
    __device__ __forceinline__ static uint32_t f2(uint64_t s) { return (uint32_t)(s >> 30) & 1u; }
    __device__ __forceinline__ static uint32_t v2(uint64_t s) { return (uint32_t)(s & M30); }
    // a precedes b
    __device__ __forceinline__ static uint64_t combine(uint64_t a, uint64_t b)
    {
        const uint32_t fb1 = f1(b), fb2 = f2(b);
        return make(f1(a) | fb1, fb1 ? v1(b) : v1(a) + v1(b), f2(a) | fb2, fb2 ? v2(b) : v2(a) + v2(b));
    }
};

constexpr uint64_t LB_INVALID = 0, LB_AGG = 1, LB_INC = 2;
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

// Look-back by warp 0 of a tile: returns the exclusive prefix of `tile`.
// status[t] = flag << 62 | payload.  Called by all 32 lanes of warp 0.
// A tile in which both fields start a segment needs nothing from before it to
// know its inclusive value: it publishes that at once, so the chain of
// look-backs is cut there (a scan over groups shorter than a tile has none).
__device__ __forceinline__ uint64_t lookback_prefix(uint64_t *status, uint32_t tile, uint64_t tile_agg,
                                                    uint32_t *err, uint64_t spin_limit_ns)
{
    const int lane = threadIdx.x & 31;
    if (tile == 0) {
        if (lane == 0) st_relaxed_u64(&status[0], (LB_INC << 62) | tile_agg);
        return 0;
    }
    const bool closed = (tile_agg & DualSeg::BOTH) == DualSeg::BOTH;
    if (lane == 0) st_relaxed_u64(&status[tile], ((closed ? LB_INC : LB_AGG) << 62) | tile_agg);
    uint64_t running = 0;  // identity
    int64_t window_end = (int64_t)tile - 1;  // closest predecessor not yet folded
    const uint64_t t0 = globaltimer();
    while (true) {
        const int64_t t = window_end - lane;
        uint64_t s = 0;
        uint32_t flag;
        if (t >= 0) {
            while (true) {
                s = ld_relaxed_u64(&status[t]);
                flag = (uint32_t)(s >> 62);
                if (flag != LB_INVALID) break;
                if (globaltimer() - t0 > spin_limit_ns) { set_err(err, ERR_TIMEOUT); break; }
            }
        } else {
            flag = (uint32_t)LB_INC;  // before tile 0: behaves like an inclusive identity
            s = (LB_INC << 62);
        }
        const uint32_t inc_mask = __ballot_sync(0xffffffffu, flag == LB_INC);
        // lanes beyond the closest inclusive one contribute nothing
        const int stop = inc_mask ? __ffs(inc_mask) - 1 : 31;
        uint64_t v = (lane <= stop) ? (s & ((1ull << 62) - 1)) : 0;
        // fold farther (higher lane) before nearer (lower lane)
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            uint64_t other = __shfl_down_sync(0xffffffffu, v, off);
            if (lane + off < 32) v = DualSeg::combine(other, v);
        }
        v = __shfl_sync(0xffffffffu, v, 0);
        running = DualSeg::combine(v, running);
        if (inc_mask) break;
        window_end -= 32;
    }
    if (lane == 0 && !closed) st_relaxed_u64(&status[tile], (LB_INC << 62) | DualSeg::combine(running, tile_agg));
    return running;
}

// Generic single-pass scan of a DualSeg state over [0, count).  Mode
// provides `uint64_t element(int64_t i)` and `void output(int64_t i,
// uint64_t inclusive)`; elements are produced and consumed in blocked order
// (thread t owns SCAN_ITEMS consecutive elements).  `err`: where the scan notes
// that it gave up; `before`: the errors of the steps before it (the same word, but
// for a scan beside an executor); `stop`: the bits of both that make it do
// nothing.  They are bits that only earlier work on its stream sets, or that the
// scan itself sets when it gives up: a bit that something running beside the scan
// may set would leave the tiles not yet started without their outputs.
template <class Mode>
__global__ void __launch_bounds__(SCAN_THREADS)
dualseg_scan_kernel(Mode mode, int64_t count, uint64_t *status, uint32_t *tile_ctr, uint32_t *err,
                    const uint32_t *before, uint32_t stop, uint64_t spin_limit_ns)
{
    __shared__ uint32_t s_tile;
    __shared__ uint64_t s_warp[SCAN_THREADS / 32];
    __shared__ uint64_t s_prefix;
    __shared__ uint32_t s_abort;
    // an earlier step failed: consume nothing (a block that returns here has
    // not taken a tile id, so no look-back waits on it); decided once per block
    if (threadIdx.x == 0) {
        s_abort = (*(volatile uint32_t *)err | *(const volatile uint32_t *)before) & stop;
        if (!s_abort) s_tile = atomicAdd(tile_ctr, 1u);
    }
    __syncthreads();
    if (s_abort) return;
    const uint32_t tile = s_tile;
    const int64_t base = (int64_t)tile * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    uint64_t incl[SCAN_ITEMS];
    uint64_t acc = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        const int64_t i = base + j;
        const uint64_t e = (i < count) ? mode.element(i) : 0;
        acc = j ? DualSeg::combine(acc, e) : e;
        incl[j] = acc;
    }
    // block scan of thread aggregates
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t x = acc;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        uint64_t o = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x = DualSeg::combine(o, x);
    }
    if (lane == 31) s_warp[warp] = x;
    uint64_t thread_excl = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0) thread_excl = 0;
    __syncthreads();
    if (warp == 0) {
        uint64_t w = (lane < SCAN_THREADS / 32) ? s_warp[lane] : 0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            uint64_t o = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w = DualSeg::combine(o, w);
        }
        const uint64_t tile_agg = __shfl_sync(0xffffffffu, w, SCAN_THREADS / 32 - 1);
        uint64_t wexcl = __shfl_up_sync(0xffffffffu, w, 1);
        if (lane == 0) wexcl = 0;
        if (lane < SCAN_THREADS / 32) s_warp[lane] = wexcl;
        const uint64_t pre = lookback_prefix(status, tile, tile_agg, err, spin_limit_ns);
        if (lane == 0) s_prefix = pre;
    }
    __syncthreads();
    const uint64_t prefix = DualSeg::combine(DualSeg::combine(s_prefix, s_warp[warp]), thread_excl);
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; j++) {
        const int64_t i = base + j;
        if (i < count) mode.output(i, DualSeg::combine(prefix, incl[j]));
    }
}

// ===========================================================================
// segmented 64-bit sums (wrapping): the scan state of the SCAN executor
// ===========================================================================
// (f, c, v): f set = a segment starts in this span, c and v = elements and sum
// since the last start (or since the beginning).  A 64-bit sum and the rest do
// not fit one status word, so a tile publishes its value first and then, with
// release semantics, a 32-bit status word with f and c (a bulk has at most
// 2^25 elements); readers acquire the status word before reading the value.
// Aggregate and inclusive values have separate slots, so a value a reader may
// still fetch is never overwritten.
struct Seg64 {
    uint32_t fc;   // c << 1 | f
    uint64_t v;
    __device__ __forceinline__ static Seg64 make(uint32_t f, uint64_t v) { return Seg64{2u | f, v}; }
    __device__ __forceinline__ static Seg64 identity() { return Seg64{0u, 0ull}; }
    __device__ __forceinline__ uint32_t count() const { return fc >> 1; }
    // a precedes b
    __device__ __forceinline__ static Seg64 combine(const Seg64 &a, const Seg64 &b)
    {
        return b.fc & 1u ? b : Seg64{a.fc + b.fc, a.v + b.v};
    }
};

__device__ __forceinline__ uint32_t ld_acquire_gpu_u32(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_gpu_u32(uint32_t *p, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ Seg64 shfl_down_seg(const Seg64 &x, int off)
{
    return Seg64{__shfl_down_sync(0xffffffffu, x.fc, off), __shfl_down_sync(0xffffffffu, x.v, off)};
}
__device__ __forceinline__ Seg64 shfl_up_seg(const Seg64 &x, int off)
{
    return Seg64{__shfl_up_sync(0xffffffffu, x.fc, off), __shfl_up_sync(0xffffffffu, x.v, off)};
}
__device__ __forceinline__ Seg64 shfl_seg(const Seg64 &x, int lane)
{
    return Seg64{__shfl_sync(0xffffffffu, x.fc, lane), __shfl_sync(0xffffffffu, x.v, lane)};
}

struct Seg64Status {
    uint32_t *word;      // per tile: state (LB_*) | fc << 2
    uint64_t *agg, *inc; // per tile values
};

// Look-back by warp 0 of a tile; returns the exclusive prefix of `tile`.  A
// tile in which a segment starts publishes its inclusive value at once, as in
// lookback_prefix: uniform accounts never wait along a chain of tiles (2,048
// tiles at 2^22, 64 windows of 32 tiles one after another otherwise).
__device__ __forceinline__ Seg64 lookback_seg64(const Seg64Status &st, uint32_t tile, const Seg64 &tile_agg,
                                                uint32_t *err, uint64_t spin_limit_ns)
{
    const int lane = threadIdx.x & 31;
    const bool closed = tile == 0 || (tile_agg.fc & 1u);
    if (closed && lane == 0) {
        st.inc[tile] = tile_agg.v;
        st_release_gpu_u32(&st.word[tile], (uint32_t)LB_INC | (tile_agg.fc << 2));
    }
    if (tile == 0) return Seg64::identity();
    if (!closed && lane == 0) {
        st.agg[tile] = tile_agg.v;
        st_release_gpu_u32(&st.word[tile], (uint32_t)LB_AGG | (tile_agg.fc << 2));
    }
    Seg64 running = Seg64::identity();
    int64_t window_end = (int64_t)tile - 1;
    const uint64_t t0 = globaltimer();
    while (true) {
        const int64_t t = window_end - lane;
        uint32_t w = (uint32_t)LB_INC;
        Seg64 x = Seg64::identity();
        if (t >= 0) {
            while (true) {
                w = ld_acquire_gpu_u32(&st.word[t]);
                if ((w & 3u) != (uint32_t)LB_INVALID) break;
                if (globaltimer() - t0 > spin_limit_ns) {
                    set_err(err, ERR_TIMEOUT);
                    w = (uint32_t)LB_INC;   // give up: fold nothing more
                    break;
                }
            }
            if ((w & 3u) == (uint32_t)LB_INC) x = Seg64{w >> 2, ld_volatile_u64(&st.inc[t])};
            else if ((w & 3u) == (uint32_t)LB_AGG) x = Seg64{w >> 2, ld_volatile_u64(&st.agg[t])};
        }
        const uint32_t inc_mask = __ballot_sync(0xffffffffu, (w & 3u) == (uint32_t)LB_INC);
        const int stop = inc_mask ? __ffs(inc_mask) - 1 : 31;
        Seg64 v = (lane <= stop) ? x : Seg64::identity();
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const Seg64 other = shfl_down_seg(v, off);
            if (lane + off < 32) v = Seg64::combine(other, v);
        }
        v = shfl_seg(v, 0);
        running = Seg64::combine(v, running);
        if (inc_mask) break;
        window_end -= 32;
    }
    if (lane == 0 && !closed) {
        const Seg64 incl = Seg64::combine(running, tile_agg);
        st.inc[tile] = incl.v;
        st_release_gpu_u32(&st.word[tile], (uint32_t)LB_INC | (incl.fc << 2));
    }
    return running;
}

// ===========================================================================
// LSD radix sort of (u32 key, u32 value) pairs
// ===========================================================================
// Up to SMALL_SORT pairs: one CTA sorts them in shared memory, one launch.
// Above: a histogram of every digit, then one onesweep pass per digit.
//
// What bounds a pass is the latency of a tile (claim, load, rank, look back,
// reorder, store), not bandwidth: 2^22 pairs are 67 MB, 10 us at the copy
// rate, and a pass takes 46 us; 200,000 pairs take 10 us.  Hence
//   * tiles of 2,048 pairs up to 2^19 pairs, where they are what fills the
//     chip (a pass over 200,000 pairs: 10.1 us, 14.9 with tiles of 8,192;
//     over 20,000: 7.5 and 13.7), and of 8,192 above, where longer runs per
//     digit make the stores cheaper (2^22: 46 us, 58 with tiles of 2,048);
//   * 10-bit digits where they save a pass (9-10, 17-20, 25-30 key bits): a
//     10-bit pass costs 1.4 to 1.6 of an 8-bit one (2^22: 67 us against two
//     passes of 47, 200,000: 16 against 20), and it is a launch less;
//   * each pass scans its digit counts itself instead of a launch between.
// (internal linkage: each translation unit that includes this header gets
// its own copy of these kernels)
namespace {
constexpr int SORT_THREADS = 512;
constexpr int SORT_WARPS = SORT_THREADS / 32;
constexpr int64_t SORT_WIDE_FROM = 1 << 19;   // pairs above which a tile holds 16 per thread, not 4
constexpr int SMALL_SORT_ITEMS = 4;
constexpr int SMALL_SORT = 1024 * SMALL_SORT_ITEMS;
constexpr uint32_t ST_AGG = 1u << 30, ST_INC = 2u << 30, ST_VAL = (1u << 30) - 1;

struct SortShape {
    int digit_bits, passes, items;
    int64_t tiles;
    __host__ __device__ int digits() const { return 1 << digit_bits; }
};
inline SortShape sort_shape(int64_t count, int bits)
{
    const int p8 = (bits + 7) / 8, p10 = (bits + 9) / 10;
    SortShape s;
    s.digit_bits = p10 < p8 ? 10 : 8;
    s.passes = p10 < p8 ? p10 : p8;
    s.items = count <= SORT_WIDE_FROM ? 4 : 16;
    s.tiles = (count + (int64_t)SORT_THREADS * s.items - 1) / ((int64_t)SORT_THREADS * s.items);
    return s;
}

// lanes of the warp whose digit is this lane's (`ok` lanes only)
template <int RB> __device__ __forceinline__ uint32_t digit_peers(uint32_t d, bool ok)
{
    uint32_t peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int b = 0; b < RB; b++) {
        const uint32_t m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        peers &= ((d >> b) & 1u) ? m : ~m;
    }
    return peers;
}

// The stable rank of each of this lane's items among its warp's items of the
// same digit; wh[digit] ends as the warp's count.  Items are striped over the
// warp: item j of lane l is element 32 j + l.
template <int RB, int ITEMS>
__device__ __forceinline__ void warp_digit_ranks(const uint32_t (&key)[ITEMS], int shift, uint32_t wbase, uint32_t n,
                                                 uint16_t *wh, uint16_t (&rank)[ITEMS])
{
    const uint32_t lt = lanemask_lt();
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const bool ok = wbase + j * 32 < n;
        const uint32_t d = (key[j] >> shift) & ((1u << RB) - 1u);
        const uint32_t peers = digit_peers<RB>(d, ok);
        uint32_t prior = 0;
        if (ok) prior = wh[d];
        __syncwarp();
        rank[j] = (uint16_t)(prior + __popc(peers & lt));
        if (ok && (peers & lt) == 0) wh[d] = (uint16_t)(prior + __popc(peers));
        __syncwarp();
    }
}

// every digit position of up to T * SMALL_SORT_ITEMS pairs in one CTA: the pairs
// live in registers, each digit reorders them through shared memory (T = 256
// for up to 1,024 pairs: fewer warps to add up per digit, 5.4 us for 1,000
// pairs of 24 bits against 12)
template <int T>
__global__ void __launch_bounds__(T, 1)
radix_small_kernel(const uint32_t *__restrict__ kin, const uint32_t *__restrict__ vin, uint32_t *__restrict__ kout,
                   uint32_t *__restrict__ vout, uint32_t n, int bits, const uint32_t *err)
{
    constexpr int ITEMS = SMALL_SORT_ITEMS, D = 256, W = T / 32;
    __shared__ uint32_t s_kv[T * ITEMS];
    __shared__ uint16_t s_whist[W * D];
    __shared__ uint32_t s_start[D], s_w[D / 32], s_abort;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_abort = *(volatile const uint32_t *)err;
    const uint32_t wbase = warp * 32 * ITEMS + lane;
    uint32_t key[ITEMS], val[ITEMS];
    uint16_t rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const uint32_t i = wbase + j * 32;
        key[j] = i < n ? kin[i] : 0xffffffffu;
        val[j] = i < n ? vin[i] : 0u;
    }
    __syncthreads();
    if (s_abort) return;
    uint16_t *wh = s_whist + warp * D;
    for (int shift = 0; shift < bits; shift += 8) {
        for (int i = lane; i < D / 2; i += 32) ((uint32_t *)wh)[i] = 0;
        __syncwarp();
        warp_digit_ranks<8, ITEMS>(key, shift, wbase, n, wh, rank);
        __syncthreads();
        uint32_t cnt = 0, x = 0;
        if (tid < D) {
            uint16_t c[W];
#pragma unroll
            for (int w = 0; w < W; w++) c[w] = s_whist[w * D + tid];
#pragma unroll
            for (int w = 0; w < W; w++) {
                s_whist[w * D + tid] = (uint16_t)cnt;
                cnt += c[w];
            }
            x = cnt;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, x, off);
                if (lane >= off) x += o;
            }
            if (lane == 31) s_w[warp] = x;
        }
        __syncthreads();
        if (tid < D) {
            uint32_t a = x - cnt;
            for (int w = 0; w < warp; w++) a += s_w[w];
            s_start[tid] = a;
        }
        __syncthreads();
        uint32_t pos[ITEMS];
#pragma unroll
        for (int j = 0; j < ITEMS; j++) {
            const uint32_t d = (key[j] >> shift) & (D - 1);
            pos[j] = s_start[d] + wh[d] + rank[j];
        }
        // keys, then values, through one buffer
#pragma unroll
        for (int j = 0; j < ITEMS; j++)
            if (wbase + j * 32 < n) s_kv[pos[j]] = key[j];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; j++)
            if (wbase + j * 32 < n) key[j] = s_kv[wbase + j * 32];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; j++)
            if (wbase + j * 32 < n) s_kv[pos[j]] = val[j];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; j++)
            if (wbase + j * 32 < n) val[j] = s_kv[wbase + j * 32];
    }
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const uint32_t i = wbase + j * 32;
        if (i < n) {
            kout[i] = key[j];
            vout[i] = val[j];
        }
    }
}

// Histograms of every digit position in one pass over the keys.
template <int RB>
__global__ void __launch_bounds__(256) radix_hist_kernel(const uint32_t *__restrict__ keys, int64_t n, int passes,
                                                         uint32_t *hist, const uint32_t *err)
{
    constexpr int D = 1 << RB, MAXP = (32 + RB - 1) / RB;
    __shared__ uint32_t sh[MAXP * D];
    __shared__ uint32_t s_abort;
    if (threadIdx.x == 0) s_abort = *(volatile const uint32_t *)err;
    for (int i = threadIdx.x; i < passes * D; i += blockDim.x) sh[i] = 0;
    __syncthreads();
    if (s_abort) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = keys[i];
        for (int p = 0; p < passes; p++) atomicAdd(&sh[p * D + ((k >> (RB * p)) & (D - 1))], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * D; i += blockDim.x)
        if (sh[i]) atomicAdd(&hist[i], sh[i]);
}

template <int RB, int ITEMS> constexpr size_t radix_smem()
{
    return (size_t)SORT_THREADS * ITEMS * 8 + (size_t)SORT_WARPS * (1 << RB) * sizeof(uint16_t);
}

// One stable counting pass on digit (key >> shift); hist = the digit's counts
// over all keys.
template <int RB, int ITEMS>
__global__ void __launch_bounds__(SORT_THREADS, 2)
radix_pass_kernel(const uint32_t *__restrict__ kin, const uint32_t *__restrict__ vin, uint32_t *__restrict__ kout,
                  uint32_t *__restrict__ vout, uint32_t n, int shift, const uint32_t *__restrict__ hist,
                  uint32_t *status, uint32_t *tile_ctr, uint32_t *err, uint64_t spin_limit_ns)
{
    constexpr int D = 1 << RB, TILE = SORT_THREADS * ITEMS;
    constexpr int DPT = (D + SORT_THREADS - 1) / SORT_THREADS;   // digits per thread
    constexpr int LOOK = 4;                                      // predecessors per look
    extern __shared__ __align__(16) uint32_t smem[];
    uint32_t *s_keys = smem;
    uint32_t *s_vals = smem + TILE;
    uint16_t *s_whist = (uint16_t *)(smem + 2 * TILE);  // [SORT_WARPS][D]: at most 32 ITEMS a warp
    __shared__ uint32_t s_tile, s_abort;
    __shared__ uint32_t s_start[D];          // tile-local start of each digit
    __shared__ uint32_t s_gbase[D];          // its global position minus that start (modulo 2^32)
    __shared__ uint32_t s_wt[SORT_WARPS], s_wg[SORT_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {   // block-uniform abort decision, see dualseg_scan_kernel
        s_abort = *(volatile uint32_t *)err;
        if (!s_abort) s_tile = atomicAdd(tile_ctr, 1u);
    }
    for (int i = tid; i < SORT_WARPS * D / 2; i += SORT_THREADS) ((uint32_t *)s_whist)[i] = 0;
    __syncthreads();
    if (s_abort) return;
    const uint32_t tile = s_tile;
    const uint32_t base = tile * TILE;
    const uint32_t wbase = base + (uint32_t)warp * 32 * ITEMS + lane;
    uint32_t key[ITEMS], val[ITEMS];
    uint16_t rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const uint32_t i = wbase + j * 32;
        const bool ok = i < n;
        key[j] = ok ? kin[i] : 0xffffffffu;
        val[j] = ok ? vin[i] : 0u;
    }
    uint32_t all[DPT];                       // the digit counts over all keys
#pragma unroll
    for (int q = 0; q < DPT; q++) all[q] = tid * DPT < D ? __ldg(&hist[tid * DPT + q]) : 0u;
    uint16_t *wh = s_whist + warp * D;
    warp_digit_ranks<RB, ITEMS>(key, shift, wbase, n, wh, rank);
    __syncthreads();

    // per digit: exclusive prefix over warps, tile count, look-back
    uint32_t cnt[DPT], excl[DPT], tsum = 0, gsum = 0;
#pragma unroll
    for (int q = 0; q < DPT; q++) cnt[q] = excl[q] = 0;
    if (tid * DPT < D) {
#pragma unroll
        for (int q = 0; q < DPT; q++) {
            const int d = tid * DPT + q;
            uint16_t c[SORT_WARPS];
#pragma unroll
            for (int w = 0; w < SORT_WARPS; w++) c[w] = s_whist[w * D + d];
            uint32_t a = 0;
#pragma unroll
            for (int w = 0; w < SORT_WARPS; w++) {
                s_whist[w * D + d] = (uint16_t)a;
                a += c[w];
            }
            cnt[q] = a;
            st_relaxed_u32(status + (size_t)tile * D + d, (tile == 0 ? ST_INC : ST_AGG) | a);
            tsum += a;
            gsum += all[q];
        }
    }
    // exclusive scans over the digits: the tile's counts and those of all keys
    uint32_t xt = tsum, xg = gsum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t ot = __shfl_up_sync(0xffffffffu, xt, off), og = __shfl_up_sync(0xffffffffu, xg, off);
        if (lane >= off) {
            xt += ot;
            xg += og;
        }
    }
    if (lane == 31) {
        s_wt[warp] = xt;
        s_wg[warp] = xg;
    }
    if (tid * DPT < D && tile > 0) {
#pragma unroll
        for (int q = 0; q < DPT; q++) {
            const int d = tid * DPT + q;
            int64_t t = (int64_t)tile - 1;
            const uint64_t t0 = globaltimer();
            bool done = false;
            while (!done) {
                uint32_t s[LOOK];
#pragma unroll
                for (int u = 0; u < LOOK; u++)
                    s[u] = t - u >= 0 ? ld_relaxed_u32(status + (size_t)(t - u) * D + d) : ST_INC;
                int used = 0;                // nearest first, up to the first not yet published
#pragma unroll
                for (int u = 0; u < LOOK; u++) {
                    if (done || used < u || !(s[u] & (ST_INC | ST_AGG))) continue;
                    excl[q] += s[u] & ST_VAL;
                    used = u + 1;
                    done = (s[u] & ST_INC) != 0;
                }
                t -= used;
                if (!done && !used && globaltimer() - t0 > spin_limit_ns) {
                    set_err(err, ERR_TIMEOUT);
                    done = true;
                }
            }
            st_relaxed_u32(status + (size_t)tile * D + d, ST_INC | (excl[q] + cnt[q]));
        }
    }
    __syncthreads();
    if (tid * DPT < D) {
        uint32_t at = xt - tsum, ag = xg - gsum;
        for (int w = 0; w < warp; w++) {
            at += s_wt[w];
            ag += s_wg[w];
        }
#pragma unroll
        for (int q = 0; q < DPT; q++) {
            const int d = tid * DPT + q;
            s_start[d] = at;
            s_gbase[d] = ag + excl[q] - at;
            at += cnt[q];
            ag += all[q];
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        if (wbase + j * 32 < n) {
            const uint32_t d = (key[j] >> shift) & (D - 1);
            const uint32_t pos = s_start[d] + wh[d] + rank[j];
            s_keys[pos] = key[j];
            s_vals[pos] = val[j];
        }
    }
    __syncthreads();
    const uint32_t tile_n = (n - base) < TILE ? (n - base) : TILE;
#pragma unroll
    for (int j = 0; j < ITEMS; j++) {
        const uint32_t i = tid + j * SORT_THREADS;
        if (i < tile_n) {
            const uint32_t k = s_keys[i];
            const uint32_t g = s_gbase[(k >> shift) & (D - 1)] + i;
            if (g < n) {
                kout[g] = k;
                vout[g] = s_vals[i];
            } else {
                set_err(err, ERR_BOUNDS);   // only after a timeout
            }
        }
    }
}

}  // namespace

}  // namespace gtx
