// Tile binning and depth sort (GS3LAM Sec. 3.2.1: Gaussians are blended in
// depth order; rasterisation is tile based).
//
// The result is the order of the 64-bit keys (tile << 32 | depth bits) with
// ties broken by item index.  Instead of radix-sorting 64-bit keys over all
// M instances (six 8-bit passes over M), the sort runs in two stages:
//   1. the visible items (tiles_touched > 0) are compacted in index order and
//      sorted by their 32-bit depth bits (four passes over the visible items);
//   2. instances are emitted in that depth order and stably sorted by their
//      tile id (one pass per 8 bits of tile id, two for up to 65536 tiles).
// A stable sort by tile of a depth-ordered, index-tie-broken stream is exactly
// the (tile, depth, index) order.
//
// The digit histograms of every pass are counted by the kernels that write the keys (the
// compaction for the depth keys, the emission for the tile keys) with shared-memory atomics.
// Each radix pass is one kernel: a block ranks its keys (1024 or 2048 in a depth pass, 4096 or 8192 in
// a tile pass) stably within the block (peer lanes of a digit from one ballot per digit bit + per-warp digit
// counters), publishes its per-digit
// counts, finds its global offsets by a chained look-back over earlier blocks,
// and scatters through shared memory.  Blocks take chunks of keys from an atomic
// counter until none is left, so a block only waits on chunks that a running block has taken; every wait
// is bounded and reports GS_ERR_TIMEOUT in the status word if it gives up.
#include <type_traits>

#include "common.cuh"

namespace gs {

// Counter slots in the workspace.
enum { CTR_NVIS = 0, CTR_M = 1, CTR_MRAW = 2, CTR_TILE = 8 };

namespace {

constexpr uint32_t kFlagAgg = 1u << 30;
constexpr uint32_t kFlagPre = 2u << 30;
constexpr uint32_t kValMask = (1u << 30) - 1;

// ----------------------------------------------------------- block scan helper
// Exclusive scan of one value per thread over a block of NT threads (256 unless given);
// returns the prefix and writes the block total to *total.  s_warp holds NT / 32 + 1 values.
template <int NT = 256>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t *total, uint32_t *s_warp) {
    constexpr int W = NT / 32;
    static_assert(NT % 32 == 0 && W <= 32, "block of at most 32 warps");
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) s_warp[w] = inc;
    __syncthreads();
    if (w == 0) {
        uint32_t t = lane < W ? s_warp[lane] : 0, ti = t;
#pragma unroll
        for (int o = 1; o < W; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        if (lane < W) s_warp[lane] = ti - t;
        if (lane == W - 1) s_warp[W] = ti;
    }
    __syncthreads();
    uint32_t r = s_warp[w] + inc - x;
    *total = s_warp[W];
    __syncthreads();
    return r;
}

// ------------------------------------------------ compaction of visible items
// Block b looks at items [b kScanBlock, (b + 1) kScanBlock), warp w of it at the 32 kScanIPT items from
// 32 kScanIPT w on, 32 consecutive ones at a time.
__device__ __forceinline__ int64_t scan_base() {
    return (int64_t)blockIdx.x * kScanBlock + (int64_t)(threadIdx.x >> 5) * (32 * kScanIPT) + (threadIdx.x & 31);
}

// What a binning accumulates into, zeroed by its first kernel.
struct BinState {
    uint32_t *ranges, *counters, *tile_counts, *emit_sums, *hist, *queue;
    uint4 *lookback;
    int64_t n_ranges, n_tiles, n_emit, n_lookback4;
    int64_t *n_inst;
    int32_t *status;
};

// First kernel of a binning: zeroes what the call accumulates into (the ranges, the counters, the instance
// count and status word, the queued forward's work counters, the tile counts, the emission's per-block
// instance counts, the digit histograms and the look-back flags, the last and largest in 16-byte stores over
// the whole grid; above kSortSmallItems items without the depth passes' flags) and counts the visible items of
// its scan block (grid: at least the count's scan blocks).
__global__ void __launch_bounds__(256) init_reduce_kernel(BinState b, const int32_t *touched, int64_t count,
                                                          uint32_t *block_sums) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    __shared__ uint32_t s_warp[8];
    const int64_t base = scan_base();
    bool f[kScanIPT];
#pragma unroll
    for (int k = 0; k < kScanIPT; ++k) f[k] = base + 32 * k < count && touched[base + 32 * k] > 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = i0; i < b.n_lookback4; i += stride) b.lookback[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int64_t i = i0; i < b.n_ranges; i += stride) b.ranges[i] = 0u;
    for (int64_t i = i0; i < b.n_tiles; i += stride) b.tile_counts[i] = 0u;
    for (int64_t i = i0; i < b.n_emit; i += stride) b.emit_sums[i] = 0u;
    for (int64_t i = i0; i < 8 * 256; i += stride) b.hist[i] = 0u;
    for (int64_t i = i0; i < 64; i += stride) b.counters[i] = 0u;
    if (i0 == 0) {
        *b.n_inst = 0;
        *b.status = 0;
        if (b.queue) b.queue[0] = b.queue[1] = 0u;
    }
    if ((int64_t)blockIdx.x * kScanBlock >= count) return;  // whole block
    uint32_t c = 0;
#pragma unroll
    for (int k = 0; k < kScanIPT; ++k) c += __popc(__ballot_sync(0xffffffffu, f[k]));
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t tot = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) tot += s_warp[w];
        block_sums[blockIdx.x] = tot;
    }
}

// Single-block exclusive scan of nb block sums; total -> counters[slot].
// If cap_slot >= 0 the total is also clamped to capacity into counters[cap_slot],
// the raw count goes to *n_inst and overflow sets the status word.
__global__ void __launch_bounds__(1024) blocksum_scan_kernel(uint32_t *block_sums, const uint32_t *nb_from,
                                                             int64_t nb_fixed, int items_per_block,
                                                             uint32_t *counters, int slot, int cap_slot,
                                                             int64_t capacity, int64_t *n_inst, int32_t *status) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    __shared__ uint32_t s_warp[33];
    const bool failed = binning_failed(status);
    int64_t nb = nb_from ? ((int64_t)*nb_from + items_per_block - 1) / items_per_block : nb_fixed;
    if (failed) return;  // whole block (the word is only written by earlier kernels)
    int64_t per = (nb + 1023) / 1024;
    int64_t b0 = (int64_t)threadIdx.x * per;
    uint32_t s = 0;
    for (int64_t i = b0; i < b0 + per && i < nb; ++i) s += block_sums[i];
    uint32_t total;
    uint32_t run = block_exclusive_scan<1024>(s, &total, s_warp);
    for (int64_t i = b0; i < b0 + per && i < nb; ++i) {
        uint32_t x = block_sums[i];
        block_sums[i] = run;
        run += x;
    }
    if (threadIdx.x == 0) {
        counters[slot] = total;
        if (cap_slot >= 0) {
            counters[cap_slot] = (int64_t)total > capacity ? (uint32_t)capacity : total;
            if (n_inst) *n_inst = total;
            if ((int64_t)total > capacity) set_status(status, GS_ERR_CAPACITY);
        }
    }
}

// Adds the `bits`-wide digits of passes [0, n_passes) of `key` (lanes with `valid`) to the block's
// shared histograms.  Every lane of the warp calls it.  Per pass: one atomic for the warp
// when all of its valid lanes have the same digit (the high digits of nearby keys), else one
// per lane (the low digits, mostly distinct, so the atomics rarely collide).
__device__ __forceinline__ void hist_add(uint32_t (*sh)[256], int n_passes, int bits, bool valid, uint32_t key) {
    const uint32_t mask = __ballot_sync(0xffffffffu, valid);
    if (!valid) return;
    const int lane = threadIdx.x & 31, first = __ffs(mask) - 1;
    for (int p = 0; p < n_passes; ++p) {
        const uint32_t d = (key >> (bits * p)) & ((1u << bits) - 1u);
        const uint32_t d0 = __shfl_sync(mask, d, first);
        if (__all_sync(mask, d == d0)) {
            if (lane == first) atomicAdd(&sh[p][d], (uint32_t)__popc(mask));
        } else {
            atomicAdd(&sh[p][d], 1u);
        }
    }
}

// Adds the block's shared histograms into the global ones (zero counts skipped).
__device__ __forceinline__ void hist_flush(uint32_t (*sh)[256], int n_passes, uint32_t *hist) {
    __syncthreads();
    for (int i = threadIdx.x; i < n_passes * 256; i += blockDim.x) {
        const uint32_t c = (&sh[0][0])[i];
        if (c) atomicAdd(&hist[i], c);
    }
}

// Order-preserving compaction of the visible items with their depth keys; also the digit
// histograms of the depth sort's four passes (no separate pass over the keys), counted over the
// block's visible keys gathered in shared memory, so that the warps count only visible keys
// (about a fifth of the items of a frame) in whole rounds of 32.  With lookback, it also clears
// the four passes' look-back flags, one row of 256 per chunk of visible keys: above kSortSmallItems items, where clearing
// them for every item there could be costs more than it delays this kernel (32 MB for eight frames of a 2M-Gaussian
// map: binning 0.860 -> 0.846 ms with the narrower rows of the tile passes; one frame of 1M: 0.138, 0.140 if cleared here).
__global__ void __launch_bounds__(256) vis_compact_kernel(const int32_t *touched, const float4 *uvdo, int64_t count,
                                                          const uint32_t *block_sums, uint32_t *keys, uint32_t *vals,
                                                          uint32_t *hist, const uint32_t *n_vis, uint4 *lookback,
                                                          int lb_tiles, int chunk) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    __shared__ uint32_t s_warp[8];
    __shared__ uint32_t sh[4][256];
    __shared__ uint32_t s_key[kScanBlock];  // the block's visible keys, in item order
    for (int i = threadIdx.x; i < 4 * 256; i += 256) (&sh[0][0])[i] = 0u;
    const int64_t base = scan_base();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    bool f[kScanIPT];
    uint32_t bal[kScanIPT];
#pragma unroll
    for (int k = 0; k < kScanIPT; ++k) f[k] = base + 32 * k < count && touched[base + 32 * k] > 0;
    uint32_t key[kScanIPT];
#pragma unroll
    for (int k = 0; k < kScanIPT; ++k) key[k] = f[k] ? __float_as_uint(uvdo[base + 32 * k].z) : 0u;
    const uint32_t block_off = block_sums[blockIdx.x];
    uint32_t c = 0;
#pragma unroll
    for (int k = 0; k < kScanIPT; ++k) {
        bal[k] = __ballot_sync(0xffffffffu, f[k]);
        c += __popc(bal[k]);
    }
    if (lane == 0) s_warp[w] = c;
    __syncthreads();
    uint32_t loc = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        loc += i < w ? s_warp[i] : 0u;
        tot += s_warp[i];
    }
#pragma unroll
    for (int k = 0; k < kScanIPT; ++k) {
        const uint32_t at = loc + __popc(bal[k] & lanemask_lt());
        if (f[k]) {
            keys[block_off + at] = key[k];
            vals[block_off + at] = (uint32_t)(base + 32 * k);
            s_key[at] = key[k];
        }
        loc += __popc(bal[k]);
    }
    __syncthreads();
    for (uint32_t i0 = threadIdx.x - lane; i0 < tot; i0 += 256) {  // warp-uniform rounds
        const uint32_t i = i0 + lane;
        hist_add(sh, 4, 8, i < tot, i < tot ? s_key[i] : 0u);
    }
    hist_flush(sh, 4, hist);
    if (!lookback) return;
    const int64_t row4 = (int64_t)((*n_vis + chunk - 1) / chunk) * 64;  // 16-byte words of a pass
    for (int p = 0; p < 4; ++p)
        for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < row4; i += (int64_t)gridDim.x * 256)
            lookback[(int64_t)p * lb_tiles * 64 + i] = make_uint4(0u, 0u, 0u, 0u);
}

// ------------------------------------------------------------ instance emission
constexpr int kEmitBlock = 256;  // sorted items per block of the emission kernels

// One thread per sorted item computes its instance offset; the block's instances are then
// split evenly over its warps, 32 consecutive instances per warp round.  A round knows the item that
// owns its first instance; the next 32 items' offsets say at which lanes the following ones begin, so
// one shared-memory read and one reduction give every lane its owner (a binary search per lane took
// eight dependent reads).  Every store is coalesced, and a few long items (large splats) do not
// keep one warp of the block busy while the others idle.  The grid is bounded and its blocks
// stride over the sorted items, so a batch whose items are mostly out of view launches no blocks for them.
// Also the digit histograms of the tile sort's n_passes passes over the written keys.
__global__ void __launch_bounds__(kEmitBlock) emit_kernel(ViewTable vt, const uint32_t *sorted_items,
                                                          const int32_t *touched, const float4 *uvdo,
                                                          const float4 *conic, const uint32_t *counters,
                                                          const uint32_t *block_sums, int64_t capacity,
                                                          uint32_t *tile_keys, uint32_t *inst_vals, int n_passes,
                                                          int bits, uint32_t *hist, int64_t vn, const int32_t *status) {
    pdl_wait();  // the previous kernel's results (no trigger: see pdl_trigger)
    __shared__ uint32_t s_warp[9];
    __shared__ uint32_t sh[4][256];
    __shared__ uint32_t s_off[kEmitBlock];  // exclusive instance offset of each item in the block
    __shared__ uint4 s_rect[kEmitBlock];    // (first tile, width, tiles per row, item)
    // whole block (the word is only written by earlier kernels): after a failed depth sort or an
    // overflow nothing is emitted
    const bool failed = binning_failed(status);
    const int64_t count = counters[CTR_NVIS];
    if (failed || (int64_t)blockIdx.x * kEmitBlock >= count) return;  // whole block: no barrier is skipped
    for (int i = threadIdx.x; i < 4 * 256; i += kEmitBlock) (&sh[0][0])[i] = 0u;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int64_t blk = blockIdx.x; blk * kEmitBlock < count; blk += gridDim.x) {
        const int64_t i = blk * kEmitBlock + threadIdx.x;
        uint32_t item = 0, c = 0, first = 0, w = 1, tx = 1;
        if (i < count && sorted_items[i] < vn) {
            item = sorted_items[i];
            c = (uint32_t)touched[item];
            const int v = (int)(item / (uint32_t)vt.n);
            const float4 rec = uvdo[item];
            int x0, y0, x1, y1;
            tile_rect(rec.x, rec.y, (int)conic[item].w, vt.TX[v], vt.TY[v], x0, y0, x1, y1);
            w = (uint32_t)max(x1 - x0, 1);
            tx = (uint32_t)vt.TX[v];
            first = (uint32_t)vt.tile_off[v] + (uint32_t)y0 * tx + (uint32_t)x0;
        }
        const uint32_t bbase = block_sums[blk];
        uint32_t tot;
        const uint32_t excl = block_exclusive_scan(c, &tot, s_warp);
        s_off[threadIdx.x] = excl;
        s_rect[threadIdx.x] = make_uint4(first, w, tx, item);
        __syncthreads();
        // warp wid takes instances [q_lo, q_hi) of the block, in whole rounds of 32
        const uint32_t per = ((tot + 32u * (kEmitBlock / 32) - 1) / (32u * (kEmitBlock / 32))) * 32u;
        const uint32_t q_lo = min(tot, (uint32_t)wid * per), q_hi = min(tot, q_lo + per);
        // the owner of the warp's first instance: the last item whose offset is <= q_lo
        int own = 0;
#pragma unroll
        for (int step = kEmitBlock / 2; step >= 1; step >>= 1)
            if (s_off[own + step] <= q_lo) own += step;
        for (uint32_t q0 = q_lo; q0 < q_hi; q0 += 32) {
            const uint32_t q = q0 + lane;
            // bit b: an item after `own` begins at instance q0 + b (every sorted item has instances)
            const int nx = own + 1 + lane;
            const uint32_t at = nx < kEmitBlock ? s_off[nx] - q0 : 32u;
            const uint32_t begins = __reduce_or_sync(0xffffffffu, at < 32u ? 1u << at : 0u);
            const int owner = min(own + __popc(begins & ((2u << lane) - 1u)), kEmitBlock - 1);
            own = min(own + __popc(begins), kEmitBlock - 1);
            const int64_t off = (int64_t)bbase + q;
            const bool write = q < q_hi && off < capacity;
            uint32_t key = 0u;
            if (write) {
                const uint4 rc = s_rect[owner];
                const uint32_t k = q - s_off[owner];
                // row of instance k: floor(k / width), by a reciprocal where its rounding (4e-7 relative)
                // cannot reach the half instance that (k + 1/2) / width is away from a whole number
                const uint32_t ky = k < (1u << 20) ? (uint32_t)(((float)k + 0.5f) * __fdividef(1.f, (float)rc.y)) : k / rc.y;
                key = rc.x + ky * rc.z + (k - ky * rc.y);
                tile_keys[off] = key;
                inst_vals[off] = rc.w;
            }
            hist_add(sh, n_passes, bits, write, key);
        }
        __syncthreads();  // the block's offsets and rectangles are read before the next items' are written
    }
    hist_flush(sh, n_passes, hist);
}

// ------------------------------------------------------------------ radix sort
// Shared memory of a radix-pass block of NT threads with IPT keys each (dynamic: 51 KB for 512 x 8).
template <int NT, int IPT>
struct SortSmem {
    uint32_t keys[NT * IPT];
    uint32_t vals[NT * IPT];
    uint32_t whist[NT / 32][256];
    uint32_t excl[256];   // block-local exclusive digit offsets
    uint32_t glob[256];   // global destination of the digit's first key in this block
    uint32_t dbase[256];  // global exclusive digit base of the pass
    uint32_t warp[2][8];
    uint32_t tile;
    int failed;
};

// One radix pass over BITS-wide digits, NT threads per block and IPT keys per thread: 256 threads for the
// depth passes over the visible items, 512 with 8 or 16 keys for the tile passes over the instances.
// Resident blocks per SM the register allocation must allow: four depth-pass blocks of 8 keys a
// thread (64 registers), six of 4 (40); three tile-pass blocks of 8 (40 registers, 56 to 60 bytes spilled), two of
// 16 (64 registers, 152 bytes spilled).  Whole binning in ms with tile-pass blocks of 512 x 8 keys at three per
// SM, 1024 x 8 at two, 512 x 16 at two, 256 x 16 at four: 0.143 / 0.149 / 0.146 / 0.149 (1M Gaussians at 1200x680,
// 1.7M instances), 0.091 / 0.098 / 0.096 / 0.096 (300k at 811x607), 0.87 / 0.91 / 0.86 / 0.85 (2M, eight
// keyframes, 22M instances).
template <int NT, int IPT> constexpr int sort_min_blocks() {
    return NT == 256 ? (IPT >= 8 ? 4 : 6) : (IPT >= 16 ? 2 : 3);
}

// Lanes of the warp with the same digit (among the lanes in `valid`), by one ballot per bit: a fraction of the
// time of match.any, which takes the distinct values one after another (the ranking of a depth pass's 1,024
// keys took 2.2 of the block's 8.7 us with it, and takes 0.8).
template <int BITS>
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, uint32_t valid) {
    uint32_t peers = valid;
#pragma unroll
    for (int b = 0; b < BITS; ++b) {
        const bool set = (d >> b) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, set);
        peers &= set ? m : ~m;
    }
    return peers;
}

template <int NT, int IPT, int BITS>
__global__ void __launch_bounds__(NT, sort_min_blocks<NT, IPT>()) onesweep_kernel(const uint32_t *keys_in, const uint32_t *vals_in,
                                                      uint32_t *keys_out, uint32_t *vals_out,
                                                      const uint32_t *count_ptr, int shift,
                                                      const uint32_t *pass_hist, uint32_t *tile_ctr,
                                                      uint32_t *lookback, int32_t *status, int spin_limit,
                                                      uint32_t *tile_counts, uint32_t n_tiles,
                                                      const int32_t *emit_touched, uint32_t *emit_sums,
                                                      uint32_t emit_vn) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    constexpr int W = NT / 32, TILE = NT * IPT, BINS = 1 << BITS;
    static_assert(NT >= BINS && BINS >= 32 && BITS <= 8, "one thread per digit");
    extern __shared__ __align__(16) unsigned char sort_smem[];
    SortSmem<NT, IPT> &S = *reinterpret_cast<SortSmem<NT, IPT> *>(sort_smem);
    uint32_t *s_keys = S.keys, *s_vals = S.vals, *s_excl = S.excl, *s_glob = S.glob, *s_dbase = S.dbase;
    uint32_t(*s_whist)[256] = S.whist;

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // chunks of TILE keys until none is left: a chunk's number comes from the counter, so every chunk
    // before it has been taken by a block that runs (or has run)
    for (;;) {
    __syncthreads();  // the previous chunk's reads of shared memory are done
    if (tid == 0) {
        S.tile = atomicAdd(tile_ctr, 1u);
        S.failed = binning_failed(status);
    }
    for (int i = tid; i < W * BINS; i += NT) s_whist[i / BINS][i % BINS] = 0;
    __syncthreads();
    const uint32_t tile = S.tile;
    const uint32_t n = *count_ptr;  // below 2^30
    if ((uint64_t)tile * TILE >= n) return;
    const uint32_t base = tile * TILE;
    if (S.failed) {
        // an earlier wait gave up (or the count overflowed): this pass's output is not used.  The
        // block still publishes an inclusive prefix (0: never more than the true one, so a block
        // that adds it scatters in bounds) so that no running block waits for it.
        if (tid < BINS) st_relaxed(lookback + (size_t)tile * BINS + tid, kFlagPre);
        return;
    }

    const uint32_t mine = base + (uint32_t)w * (IPT * 32) + lane;  // this thread's keys: mine + 32 r
    uint32_t key[IPT], val[IPT], rank2[IPT / 2];  // ranks below TILE <= 2^16, two to a register
    static_assert(TILE <= 1 << 16 && IPT % 2 == 0, "16-bit ranks");
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const bool valid = mine + 32 * r < n;
        key[r] = valid ? keys_in[mine + 32 * r] : 0u;
        val[r] = valid ? vals_in[mine + 32 * r] : 0u;
    }
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const bool valid = mine + 32 * r < n;
        const uint32_t d = (key[r] >> shift) & (BINS - 1u);
        const uint32_t peers = digit_peers<BITS>(d, __ballot_sync(0xffffffffu, valid));
        // every lane reads its digit's count so far; the last lane of the digit adds the round's
        const uint32_t b = s_whist[w][d];
        const uint32_t rank = b + __popc(peers & lanemask_lt());
        if (r % 2) rank2[r / 2] |= rank << 16;
        else rank2[r / 2] = rank;
        __syncwarp();
        if (valid && (peers >> lane) == 1u) s_whist[w][d] = b + __popc(peers);
        __syncwarp();
    }
    __syncthreads();

    // per-digit (thread d < BINS): warp-exclusive offsets and the block's count, published at once
    // for later chunks; then the block-exclusive digit offsets and the pass's digit bases, two scans over the
    // digits that share their barriers
    const int d = tid;
    uint32_t cnt = 0, hist_d = 0;
    uint32_t *my = lookback + (size_t)tile * BINS + (d & (BINS - 1));
    uint32_t ci = 0, hi = 0;
    if (d < BINS) {
        hist_d = pass_hist[d];
#pragma unroll
        for (int ww = 0; ww < W; ++ww) {
            uint32_t c = s_whist[ww][d];
            s_whist[ww][d] = cnt;
            cnt += c;
        }
        st_relaxed(my, (tile == 0 ? kFlagPre : kFlagAgg) | cnt);
        ci = cnt;
        hi = hist_d;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, ci, o), y = __shfl_up_sync(0xffffffffu, hi, o);
            if (lane >= o) {
                ci += x;
                hi += y;
            }
        }
        if (lane == 31) {
            S.warp[0][w] = ci;
            S.warp[1][w] = hi;
        }
    }
    __syncthreads();
    if (d < BINS) {
        for (int ww = 0; ww < w; ++ww) {
            ci += S.warp[0][ww];
            hi += S.warp[1][ww];
        }
        s_excl[d] = ci - cnt;
        s_dbase[d] = hi - hist_d;
    }
    __syncthreads();

    // local scatter by digit into shared memory (the keys leave the registers before the wait)
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        if (mine + 32 * r < n) {
            const uint32_t dd = (key[r] >> shift) & (BINS - 1u);
            const uint32_t pos = s_excl[dd] + s_whist[w][dd] + (r % 2 ? rank2[r / 2] >> 16 : rank2[r / 2] & 0xffffu);
            s_keys[pos] = key[r];
            s_vals[pos] = val[r];
        }
    }

    // chained look-back over earlier tiles for digit d: kWin of their flags are read at a time
    // (all tiles start together, so the chain is as long as the tile number over kWin); spin
    // (bounded) only on a tile that has not published its count yet
    uint32_t prefix = 0;
    if (tile != 0 && d < BINS) {
        constexpr int kWin = 8;
        int t = (int)tile - 1;
        bool done = false, timeout = false;
        while (!done && t >= 0) {
            uint32_t w[kWin];
#pragma unroll
            for (int i = 0; i < kWin; ++i) w[i] = t - i >= 0 ? ld_relaxed(lookback + (size_t)(t - i) * BINS + d) : 0u;
#pragma unroll
            for (int i = 0; i < kWin; ++i) {
                if (done) continue;
                if (t - i < 0 || spin_limit < 0) {  // the first tile passed; or the test hook: give up at once
                    timeout = spin_limit < 0;
                    done = true;
                    continue;
                }
                uint32_t vv = w[i];
                if ((vv & ~kValMask) == 0u) {
                    const uint32_t *pp = lookback + (size_t)(t - i) * BINS + d;
                    int spin = 0;
                    while ((vv & ~kValMask) == 0u && spin < spin_limit) {
                        if (++spin > 64) __nanosleep(64);
                        vv = ld_relaxed(pp);
                    }
                    if ((vv & ~kValMask) == 0u) {
                        timeout = true;
                        done = true;
                        continue;
                    }
                }
                prefix += vv & kValMask;
                if ((vv & ~kValMask) == kFlagPre) done = true;
            }
            t -= kWin;
        }
        if (timeout) set_status(status, GS_ERR_TIMEOUT);
        st_relaxed(my, kFlagPre | (prefix + cnt));
    }
    if (d < BINS) s_glob[d] = s_dbase[d] + prefix;
    __syncthreads();

    // coalesced-by-run global writes, in warp-uniform rounds of 32 consecutive keys
    const int tile_n = (int)min((uint32_t)TILE, n - base);
    for (int i0 = tid - lane; i0 < tile_n; i0 += NT) {
        const int i = i0 + lane;
        const bool ok = i < tile_n;
        uint32_t dst = 0u, v = 0u;
        if (ok) {
            const uint32_t k = s_keys[i];
            const uint32_t dd = (k >> shift) & (BINS - 1u);
            dst = s_glob[dd] + (uint32_t)i - s_excl[dd];
            v = s_vals[i];
            keys_out[dst] = k;
            vals_out[dst] = v;
            // last pass of the tile sort: the block's keys are sorted by tile here, so each run of one
            // tile adds its length to the tile's count (end + 1 from its last key, -start from its first)
            if (tile_counts && k < n_tiles) {
                if (i == 0 || s_keys[i - 1] != k) atomicAdd(&tile_counts[k], 0u - (uint32_t)i);
                if (i == tile_n - 1 || s_keys[i + 1] != k) atomicAdd(&tile_counts[k], (uint32_t)i + 1u);
            }
        }
        if (emit_sums) {
            // last pass of the depth sort: the instances of each block of kEmitBlock sorted items,
            // which the emission scans.  dst increases with i in a block (digits in order, each
            // digit's keys at consecutive places), so the lanes of one emission block are
            // consecutive: a segmented sum over the warp and one atomic per segment.
            const uint32_t seg = ok ? dst / (uint32_t)kEmitBlock : 0xffffffffu;
            uint32_t c = ok && v < emit_vn ? (uint32_t)emit_touched[v] : 0u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, c, o);
                const uint32_t sy = __shfl_up_sync(0xffffffffu, seg, o);
                if (lane >= o && sy == seg) c += y;
            }
            const uint32_t s_next = __shfl_down_sync(0xffffffffu, seg, 1);
            if (ok && (lane == 31 || s_next != seg) && c) atomicAdd(&emit_sums[seg], c);
        }
    }
    }
}

// The optional 64-bit keys (tile << 32 | depth bits) of the sorted instances.  Tile ids and
// items are checked against their counts: only a sort that gave up (status set, so nothing
// runs here) could leave other values, but an access out of bounds must not be possible.
__global__ void __launch_bounds__(256) keys64_kernel(const uint32_t *tile_keys, const uint32_t *vals,
                                                     const uint32_t *counters, const float4 *uvdo, uint64_t *keys64,
                                                     int64_t n_tiles, int64_t vn, const int32_t *status) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    const bool failed = binning_failed(status);
    int64_t m = counters[CTR_M];
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (failed || j >= m) return;
    const uint32_t t = tile_keys[j], it = vals[j];
    keys64[j] = t < n_tiles && it < vn ? ((uint64_t)t << 32) | __float_as_uint(uvdo[it].z) : ~0ull;
}

struct SortBufs {
    uint32_t *k0, *v0, *k1, *v1;
};

// Stable LSD sort of (key, val) pairs by `n_passes` digits of BITS bits from bit 0, given the
// digit histograms of every pass (hist [n_passes][256], written by the kernel that
// produced the keys).  Input in (k0, v0); output lands in (k0, v0) if n_passes is even,
// else (k1, v1).  The last pass also adds the tile runs to tile_counts and, with emit_sums,
// emit_touched[val] to the count of its kEmitBlock-item block of the output (either optional).
// The grid is at most one resident wave, whose blocks take chunks until none is left: max_count is the
// most there can be (every item, the capacity), often several times what there is.
template <int NT, int IPT, int BITS>
gs_status radix_sort(SortBufs b, const uint32_t *count_ptr, int64_t max_count, int n_passes, const uint32_t *hist,
                     uint32_t *lookback, int lb_tiles, uint32_t *tile_ctrs, int32_t *status, int spin_limit,
                     cudaStream_t st, uint32_t *tile_counts = nullptr, uint32_t n_tiles = 0,
                     const int32_t *emit_touched = nullptr, uint32_t *emit_sums = nullptr, uint32_t emit_vn = 0) {
    if (max_count <= 0 || n_passes <= 0) return GS_OK;
    constexpr size_t smem = sizeof(SortSmem<NT, IPT>);
    if (smem > 48 * 1024) {
        // above the static limit: opted in once per device
        static bool opted[64] = {false};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return GS_ERR_CUDA;
        if (dev < 0 || dev >= 64 || !opted[dev]) {
            if (cudaFuncSetAttribute(onesweep_kernel<NT, IPT, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem) != cudaSuccess)
                return GS_ERR_CUDA;
            if (dev >= 0 && dev < 64) opted[dev] = true;
        }
    }
    const int grid = std::min(ceil_div(max_count, (int64_t)NT * IPT), kSMs * sort_min_blocks<NT, IPT>());
    uint32_t *ki = b.k0, *vi = b.v0, *ko = b.k1, *vo = b.v1;
    for (int p = 0; p < n_passes; ++p) {
        const gs_status s = launch_pdl(onesweep_kernel<NT, IPT, BITS>, grid, NT, smem, st, ki, vi, ko, vo, count_ptr,
                                       BITS * p, hist + 256 * p, tile_ctrs + p, lookback + ((size_t)p * lb_tiles << BITS),
                                       status, spin_limit, p == n_passes - 1 ? tile_counts : nullptr, n_tiles, emit_touched,
                                       p == n_passes - 1 ? emit_sums : nullptr, emit_vn);
        if (s) return s;
        uint32_t *tk = ki, *tv = vi;
        ki = ko; vi = vo; ko = tk; vo = tv;
    }
    return last_launch();
}

}  // namespace
}  // namespace gs

namespace gs {
namespace {

// Per-tile ranges and the launch order of the blend kernels' tiles, from the instance count of
// every tile (counted by the last tile-sort pass).  One CTA of 1024 threads.
//   ranges: an exclusive scan of the counts (each thread scans a contiguous chunk of tiles),
//   [0, 0) for an empty tile;
//   order: decreasing instance count, so the longest tiles start first and the short ones fill
//   in behind them (longest-processing-time-first; the order within a count bucket is
//   arbitrary): a counting sort on a bucket of the count (exact below 1024 instances,
//   64-instance steps above, saturating at 50,112), buckets taken high to low.
// After a failed binning the ranges stay empty and every count is taken as 0.
__device__ __forceinline__ int order_bucket(uint32_t c) {
    return c < 1024u ? (int)(c >> 2) : (int)min(256u + ((c - 1024u) >> 6), 1023u);
}

// Exclusive scan of one value per thread over the 1024-thread block; returns the prefix and the total.
__device__ __forceinline__ uint32_t scan1024(uint32_t x, uint32_t *total, uint32_t *s_warp) {
    return block_exclusive_scan<1024>(x, total, s_warp);
}

__global__ void __launch_bounds__(1024) ranges_order_kernel(const uint32_t *counts, int n_tiles, uint32_t *ranges,
                                                            uint32_t *order, const int32_t *status) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    __shared__ uint32_t hist[1024];
    __shared__ uint32_t warp_tot[33];
    const int tid = threadIdx.x;
    const bool failed = binning_failed(status);
    hist[tid] = 0u;
    __syncthreads();
    // 1,024 consecutive tiles at a time (coalesced), with the running total carried from one to the next
    uint32_t carry = 0u;
    for (int t0 = 0; t0 < n_tiles; t0 += 1024) {
        const int t = t0 + tid;
        const uint32_t c = t < n_tiles && !failed ? counts[t] : 0u;
        uint32_t total;
        const uint32_t run = carry + scan1024(c, &total, warp_tot);
        if (t < n_tiles) {
            if (!failed) {
                ranges[2 * t] = c ? run : 0u;  // empty tiles: [0, 0)
                ranges[2 * t + 1] = c ? run + c : 0u;
            }
            if (order) atomicAdd(&hist[order_bucket(c)], 1u);
        }
        carry += total;
    }
    if (!order) return;  // whole block
    __syncthreads();
    // exclusive scan over buckets from the highest down: thread i takes bucket 1023 - i
    const uint32_t h = hist[1023 - tid];
    uint32_t all;
    const uint32_t before = scan1024(h, &all, warp_tot);
    hist[1023 - tid] = before;  // first slot of bucket 1023 - tid
    __syncthreads();
    for (int t = tid; t < n_tiles; t += 1024) {
        const uint32_t pos = atomicAdd(&hist[order_bucket(failed ? 0u : counts[t])], 1u);
        order[pos] = (uint32_t)t;
    }
}

gs_status write_ranges_order(const uint32_t *counts, const gs_binning *out, int64_t total_tiles, cudaStream_t st) {
    return launch_pdl(ranges_order_kernel, 1, 1024, 0, st, counts, (int)total_tiles, out->ranges, out->tile_order,
                      out->status);
}

}  // namespace
}  // namespace gs

extern "C" gs_status gs_bin_sort(int64_t n, const gs_projected *proj, const gs_camera *cams, int n_views,
                                 const gs_raster_params *p, void *ws, size_t ws_bytes, gs_binning *out,
                                 gs_stream stream) {
    GS_NVTX_RANGE("gs_bin_sort");
    using namespace gs;
    cudaStream_t st = (cudaStream_t)stream;
    ViewTable vt;
    Params prm;
    if (!proj || !out || n < 0) return GS_ERR_ARG;
    if (!make_view_table(cams, n_views, n, &vt) || !make_params(p, &prm)) return GS_ERR_ARG;
    if (out->capacity < 0 || out->capacity >= ((int64_t)1 << 30) || n * n_views >= ((int64_t)1 << 30)) return GS_ERR_ARG;
    if (!out->vals || !out->ranges || !out->n_inst || !out->status || !ws) return GS_ERR_ARG;
    WsLayout L = ws_layout(n, n_views, out->capacity, &vt);
    if (ws_bytes < L.bin_end || (reinterpret_cast<uintptr_t>(ws) & 255)) return GS_ERR_ARG;
    char *w = static_cast<char *>(ws);
    uint32_t *counters = reinterpret_cast<uint32_t *>(w + L.counters);
    uint32_t *block_sums = reinterpret_cast<uint32_t *>(w + L.scan_blocks);
    uint32_t *emit_sums = reinterpret_cast<uint32_t *>(w + L.emit_sums);
    uint32_t *hist = reinterpret_cast<uint32_t *>(w + L.hist);
    uint32_t *lookback = reinterpret_cast<uint32_t *>(w + L.lookback);
    uint32_t *tile_counts = reinterpret_cast<uint32_t *>(w + L.tile_counts);
    int64_t total_tiles = vt.tile_off[n_views];
    int64_t vn = n * n_views;

    if (vn > 0 && (!proj->uvdo || !proj->conic || !proj->tiles_touched)) return GS_ERR_ARG;

    // Every kernel of the binning is launched with programmatic stream serialization: it is
    // scheduled while its predecessor drains and waits for it (pdl_wait) before reading.
    gs_status s;
    int tile_bits = 1;
    while (((int64_t)1 << tile_bits) < total_tiles) ++tile_bits;
    // the fewest passes of at most 8 bits, and digits no wider than those passes need: fewer digits mean
    // fewer ballots, counters and look-back words per block and longer runs to write (1200x680: two passes
    // of 6 bits)
    const int tile_passes = (tile_bits + 7) / 8;
    const int digit_bits = std::max(5, (tile_bits + tile_passes - 1) / tile_passes);
    // Chunks of 16 keys a thread where several passes have 8-bit digits (more than 16,384 tiles: large
    // batches, where they are as fast), of 8 elsewhere: the look-back rows, as wide as the digits, then fit in the
    // workspace's 768 words per 8,192 instances.
    const bool wide = digit_bits == 8 && tile_passes > 1;
    const int lb_tiles = ceil_div(out->capacity, wide ? 2 * kSortTileInst : kSortTileInst);
    uint32_t *tile_lookback = lookback + (size_t)4 * L.lb_tiles_depth * 256;
    // look-back flags that the first kernel clears: of all passes (the depth passes' come first), or above
    // kSortSmallItems items of the tile passes, the compaction clearing the others
    const bool clear_first = vn <= kSortSmallItems;
    const int64_t n_lb4 = vn > 0 ? (((int64_t)tile_passes * lb_tiles << digit_bits) / 4 +
                                    (clear_first ? 4 * (int64_t)L.lb_tiles_depth * 64 : 0))
                                 : 0;
    const int64_t nbe = ceil_div(vn, kEmitBlock);  // emission blocks
    const int nb = ceil_div(vn, kScanBlock);       // scan blocks
    const int init_grid = std::max<int>({1, nb, (int)std::min<int64_t>((n_lb4 + 255) / 256, kSMs * 8)});
    const BinState state{out->ranges, counters, tile_counts, emit_sums, hist, out->queue,
                         reinterpret_cast<uint4 *>(clear_first ? lookback : tile_lookback),
                         2 * total_tiles, total_tiles, nbe + 1, n_lb4, out->n_inst, out->status};
    // 1. the call's state; the visible items of every scan block
    if ((s = launch_pdl(init_reduce_kernel, init_grid, 256, 0, st, state, proj->tiles_touched, vn, block_sums))) return s;
    if (vn == 0) return write_ranges_order(tile_counts, out, total_tiles, st);

    const float4 *uvdo = reinterpret_cast<const float4 *>(proj->uvdo);
    const float4 *conic = reinterpret_cast<const float4 *>(proj->conic);
    uint32_t *dk_a = reinterpret_cast<uint32_t *>(w + L.dkeys_a), *dv_a = reinterpret_cast<uint32_t *>(w + L.dvals_a);
    uint32_t *dk_b = reinterpret_cast<uint32_t *>(w + L.dkeys_b), *dv_b = reinterpret_cast<uint32_t *>(w + L.dvals_b);

    // compact visible items in index order, keyed by depth bits
    if ((s = launch_pdl(blocksum_scan_kernel, 1, 1024, 0, st, block_sums, nullptr, (int64_t)nb, kScanBlock, counters,
                        (int)CTR_NVIS, -1, (int64_t)0, nullptr, nullptr)))
        return s;
    if ((s = launch_pdl(vis_compact_kernel, nb, 256, 0, st, proj->tiles_touched, uvdo, vn, block_sums, dk_a, dv_a,
                        hist, counters + CTR_NVIS,
                        clear_first ? (uint4 *)nullptr : reinterpret_cast<uint4 *>(lookback), L.lb_tiles_depth,
                        depth_sort_tile(vn))))
        return s;

    // 2. stable sort of the visible items by depth (4 passes: result in dk_a/dv_a); the last pass
    //    also counts the instances of every emission block of the sorted items
    auto depth_sort = [&](auto ipt) {
        return radix_sort<kSortThreads, decltype(ipt)::value, 8>(
            {dk_a, dv_a, dk_b, dv_b}, counters + CTR_NVIS, vn, 4, hist, lookback, L.lb_tiles_depth, counters + CTR_TILE,
            out->status, prm.spin_limit, st, nullptr, 0, proj->tiles_touched, emit_sums, (uint32_t)vn);
    };
    s = vn <= kSortSmallItems ? depth_sort(std::integral_constant<int, kSortIPTSmall>())
                              : depth_sort(std::integral_constant<int, kSortIPTLarge>());
    if (s) return s;
    const uint32_t *sorted_items = dv_a;

    // 3. emit instances in depth order; instance count -> n_inst (clamped copy for the sort)
    uint32_t *tk_a = reinterpret_cast<uint32_t *>(w + L.tkeys_a), *tk_b = reinterpret_cast<uint32_t *>(w + L.tkeys_b);
    uint32_t *tv_b = reinterpret_cast<uint32_t *>(w + L.tvals_b);
    // the emitted values go where the final pass must not land: out->vals ends the sort
    uint32_t *emit_vals = (tile_passes % 2 == 0) ? out->vals : tv_b;
    uint32_t *other_vals = (tile_passes % 2 == 0) ? tv_b : out->vals;
    if ((s = launch_pdl(blocksum_scan_kernel, 1, 1024, 0, st, emit_sums, counters + CTR_NVIS, (int64_t)0, kEmitBlock,
                        counters, (int)CTR_MRAW, (int)CTR_M, out->capacity, out->n_inst, out->status)))
        return s;
    if ((s = launch_pdl(emit_kernel, (int)std::min<int64_t>(nbe, kSMs * 8), kEmitBlock, 0, st, vt, sorted_items,
                        proj->tiles_touched, uvdo, conic, counters, emit_sums, out->capacity, tk_a, emit_vals, tile_passes,
                        digit_bits, hist + 4 * 256, vn, out->status)))
        return s;
    if (out->capacity == 0) return write_ranges_order(tile_counts, out, total_tiles, st);

    // 4. stable sort of the instances by tile id
    auto tile_sort = [&](auto ipt, auto bits) {
        return radix_sort<kSortThreadsInst, decltype(ipt)::value, decltype(bits)::value>(
            {tk_a, emit_vals, tk_b, other_vals}, counters + CTR_M, out->capacity, tile_passes, hist + 4 * 256,
            tile_lookback, lb_tiles, counters + CTR_TILE + 4, out->status, prm.spin_limit, st, tile_counts,
            (uint32_t)total_tiles);
    };
    constexpr std::integral_constant<int, kSortIPTInst> keys8;
    s = digit_bits == 5   ? tile_sort(keys8, std::integral_constant<int, 5>())
        : digit_bits == 6 ? tile_sort(keys8, std::integral_constant<int, 6>())
        : digit_bits == 7 ? tile_sort(keys8, std::integral_constant<int, 7>())
        : !wide           ? tile_sort(keys8, std::integral_constant<int, 8>())
                          : tile_sort(std::integral_constant<int, 2 * kSortIPTInst>(), std::integral_constant<int, 8>());
    if (s) return s;
    const uint32_t *sorted_tiles = (tile_passes % 2 == 0) ? tk_a : tk_b;

    // 5. per-tile ranges from the tile counts, the launch order, and the 64-bit keys if requested
    if ((s = write_ranges_order(tile_counts, out, total_tiles, st))) return s;
    if (out->keys) {
        if ((s = launch_pdl(keys64_kernel, ceil_div(out->capacity, 256), 256, 0, st, sorted_tiles, out->vals, counters,
                            uvdo, out->keys, total_tiles, vn, out->status)))
            return s;
    }
    return GS_OK;
}
