// Forward blend (GS3LAM Eq. 4-7 and 10): one CTA per 16x16 tile, NP pixels per
// thread.  Splats of the tile are staged 128 at a time in shared memory (one
// record per thread load) and read back as broadcasts; a warp tests 32 splats at
// a time (one per lane, one ballot) for whether their alpha >= alpha_min ellipse
// reaches its pixel box, and walks only those that do; every pixel walks the
// rest front to back and stops at the T_min threshold; the CTA leaves as soon
// as all of its pixels are done.  With a blend mask, each warp also records, per
// 8x4 pixel group and 32-instance word, which splats any pixel of it blended.
#include <type_traits>

#include "raster.cuh"

namespace gs {
namespace {

// Resident CTAs per SM the register allocation must allow, per feature width and
// pixels per thread: the blend loop is issue-bound, so warps resident matter
// more than the few values ptxas would otherwise keep live across the mask flush.  At D = 16 with one
// pixel per thread four CTAs rather than five (64 registers, 48): with 48 the loads of the two splats
// evaluated together are taken apart (0.054 -> 0.044 ms at 320x240, 0.067 -> 0.056 at 64x48).  At D = 16 with two
// pixels per thread six CTAs (80 registers) spill 20 bytes, 36 in 16-bit storage; five take 0.241 ms
// against 0.232 (1M Gaussians at 1200x680).
constexpr int fwd_min_blocks(int D, int NP) {
    return NP == 1 ? (D == 0 ? 8 : D <= 4 ? 6 : D <= 8 ? 5 : D <= 16 ? 4 : 3) : NP == 2 ? (D <= 16 ? 6 : 4) : 6;
}

// A staged splat is one record of 3 + D / 4 16-byte words: geometry (two), colour and depth, the
// features.  One base address serves all of a splat's reads, and the odd word counts of D = 0, 8, 16
// and 32 keep eight threads that write neighbouring records in different banks.
template <int D> constexpr int kRecWords = 3 + D / 4;

__device__ __forceinline__ SplatGeo geo_of(const float4 *rec) {
    const float4 a = rec[0], b = rec[1];
    return SplatGeo{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
}
__device__ __forceinline__ void put_geo(float4 *rec, const SplatGeo &s) {
    rec[0] = make_float4(s.u, s.v, s.ulo, s.vlo);
    rec[1] = make_float4(s.qa, s.qb, s.qc, s.o);
}

// Splats evaluated together: four with two pixels per thread (forward of 1M Gaussians at 1200x680, D =
// 16: 0.231 ms, against 0.233 with two and 0.254 with one; D = 32 at 640x480: 0.163, 0.175, 0.192),
// two with one pixel, whose kernels have half the registers (D = 8: 0.075, 0.077 with four or one).
constexpr int walk_splats(int NP) { return NP == 2 ? 4 : NP == 1 ? 2 : 1; }

// The pixels of one thread while they are blended: position, transmittance, whether the pixel is done
// (stopped, or outside the image) and the blended sums.  The sums are kept as packed pairs of channels ((r, g), (b, depth), the
// features), which match the 16-byte words of the staged records, so a splat costs (4 + D) / 2
// packed multiply-adds per pixel instead of 4 + D scalar ones, with the same rounding.
//
// The kernel is bound by instruction issue (74 % of cycles at D = 16) and by the latency of the
// staging between its barriers.  One base address per record, packed multiply-adds and the exact
// ellipse test alone (the rectangle test before it cost a logarithm, two roots and two divisions per
// staged splat and culled little more, blended pixels of long thin splats among it) took the forward
// from 0.266 to 0.246 ms (room, 1M Gaussians, D = 16, 1200x680), 0.230 to 0.190 ms (1M, D = 32, 640x480),
// 4.33 to 3.26 ms (2M, D = 32, 16-bit storage, 8 keyframes) and 0.107 to 0.075 ms (300k, D = 8,
// 811x607), with the same images on these scenes.  Measured and slower: the next batch's records copied
// (cp.async) into a second buffer while the current one is walked (0.339 ms with 128-splat batches,
// 0.282 with 64: the second buffer takes the L1 that serves the gathers of neighbouring tiles), and the
// box tests done once by the staging thread for all four warps (0.262 against 0.237 ms: they then sit
// between the loads and the barrier).
template <int D, int NP>
struct BlendPixels {
    using SH = Shape<NP, true>;  // horizontal pixel pairs
    static constexpr int NL = SH::PIX_GROUPS ? NP : 1;  // mask bit registers per thread
    static constexpr int D4 = D / 4, F4 = D4 > 0 ? D4 : 1;
    static constexpr int kWalk = walk_splats(NP);
    float pxc[NP], pyc[NP], T[NP], as[NP];
    bool done[NP];
    float2 acc[NP][2], af[NP][2 * F4];
    int last[NP], blended[NP];

    __device__ __forceinline__ void init(const ViewTable &vt, const Params &prm, int v, int tx, int ty, int tid) {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            int lx, ly;
            SH::pixel(tid, p, lx, ly);
            const int px = tx * kTile + lx, py = ty * kTile + ly;
            pxc[p] = (float)px + 0.5f;
            pyc[p] = (float)py + 0.5f;
            T[p] = 1.f;
            done[p] = !(px < vt.W[v] && py < vt.H[v]);
            as[p] = 0.f;
            acc[p][0] = acc[p][1] = make_float2(0.f, 0.f);
#pragma unroll
            for (int q = 0; q < 2 * F4; ++q) af[p][q] = make_float2(0.f, 0.f);
            last[p] = blended[p] = 0;
        }
    }
    __device__ __forceinline__ bool all_done() const {
        bool a = true;
#pragma unroll
        for (int p = 0; p < NP; ++p) a = a && done[p];
        return a;
    }
    // The splat's alpha at each of the thread's pixels, which does not depend on what is in front.
    __device__ __forceinline__ void evaluate(const Params &prm, const float4 *rec, PairEval (&e)[NP]) const {
        const SplatGeo s = geo_of(rec);
#pragma unroll
        for (int p = 0; p < NP; ++p) e[p] = eval_pair(s, pxc[p], pyc[p], prm.alpha_min, prm.alpha_max);
    }
    // Blends one evaluated splat (its record, list position pos, mask bit `bit`) into the thread's pixels.
    template <bool CNT>
    __device__ __forceinline__ void blend(const Params &prm, const PairEval (&ev)[NP], const float4 *rec, int pos,
                                          uint32_t bit, uint32_t (&lbits)[NL]) {
        float wgt[NP];
        bool any = false;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const PairEval &e = ev[p];
            const float Tn = T[p] * (1.f - e.alpha);
            const bool ok = !e.skip && !done[p];
            const bool stop = ok && Tn < prm.T_min;
            const bool b = ok && !stop;
            done[p] = done[p] || stop;
            wgt[p] = b ? e.alpha * T[p] : 0.f;
            T[p] = b ? Tn : T[p];
            last[p] = b ? pos : last[p];
            if constexpr (CNT) blended[p] += b ? 1 : 0;
            any = any || b;
            if (SH::PIX_GROUPS) lbits[p % NL] |= b ? bit : 0u;
        }
        if (!SH::PIX_GROUPS) lbits[0] |= any ? bit : 0u;
        if (!any) return;
        const float4 c = rec[2];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float2 w = make_float2(wgt[p], wgt[p]);
            as[p] += wgt[p];
            acc[p][0] = fma2(w, make_float2(c.x, c.y), acc[p][0]);
            acc[p][1] = fma2(w, make_float2(c.z, c.w), acc[p][1]);
        }
#pragma unroll
        for (int q = 0; q < D4; ++q) {
            const float4 f = rec[3 + q];
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 w = make_float2(wgt[p], wgt[p]);
                af[p][2 * q] = fma2(w, make_float2(f.x, f.y), af[p][2 * q]);
                af[p][2 * q + 1] = fma2(w, make_float2(f.z, f.w), af[p][2 * q + 1]);
            }
        }
    }
    // Walks the splats of `todo` (bit k: record k of the chunk, list position pos0 + k) front to back
    // and sets the bits of those blended; true once all of the warp's pixels are done.  kWalk splats
    // are evaluated together before they are blended in order, so their loads and exponentials
    // overlap; whether the warp is done is looked at every fourth splat (a later exit only runs
    // splats whose pairs blend nothing).
    template <bool CNT>
    __device__ __forceinline__ bool walk(const Params &prm, const float4 *chunk, uint32_t todo, int pos0,
                                         uint32_t (&lbits)[NL]) {
        constexpr int REC = kRecWords<D>;
        for (int run = 0; todo; run += kWalk) {
            if ((run & 3) == 0 && __all_sync(0xffffffffu, all_done())) return true;
            int k[kWalk];
            bool has[kWalk];
            PairEval e[kWalk][NP];
#pragma unroll
            for (int u = 0; u < kWalk; ++u) {
                has[u] = todo != 0u;  // warp-uniform
                k[u] = has[u] ? __ffs(todo) - 1 : k[u > 0 ? u - 1 : 0];
                todo &= todo - 1u;
                evaluate(prm, chunk + k[u] * REC, e[u]);
            }
#pragma unroll
            for (int u = 0; u < kWalk; ++u)
                if (u == 0 || has[u]) blend<CNT>(prm, e[u], chunk + k[u] * REC, pos0 + k[u], 1u << k[u], lbits);
        }
        return false;
    }
    __device__ __forceinline__ void write(const ViewTable &vt, const Params &prm, int v, int tx, int ty, int tid, int64_t P,
                                          float *o_rgb, float *o_depth, float *o_sil, float *o_feat, float *o_T,
                                          int32_t *o_nc, int32_t *o_nb) const {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            int lx, ly;
            SH::pixel(tid, p, lx, ly);
            const int px = tx * kTile + lx, py = ty * kTile + ly;
            if (px >= vt.W[v] || py >= vt.H[v]) continue;
            const int64_t pix = vt.pix_off[v] + (int64_t)py * vt.W[v] + px;
            o_rgb[pix] = acc[p][0].x + T[p] * prm.bg[0];
            o_rgb[P + pix] = acc[p][0].y + T[p] * prm.bg[1];
            o_rgb[2 * P + pix] = acc[p][1].x + T[p] * prm.bg[2];
            o_depth[pix] = acc[p][1].y;
            o_sil[pix] = as[p];
#pragma unroll
            for (int q = 0; q < D / 2; ++q) {
                o_feat[(2 * q) * P + pix] = af[p][q].x;
                o_feat[(2 * q + 1) * P + pix] = af[p][q].y;
            }
            o_T[pix] = T[p];
            o_nc[pix] = last[p];
            if (o_nb) o_nb[pix] = blended[p];
        }
    }
};

// One 16x16 tile gt of the blend, by the whole CTA (every exit is uniform over the CTA), staging
// BATCH splats per round; with CNT it also counts each pixel's blended splats (o_nb).
template <int D, int NP, typename RT, typename FT, int BATCH, bool CNT>
__device__ __forceinline__ void fwd_tile(
    const ViewTable &vt, const Params &prm, const float4 *__restrict__ uvdo, const float2 *__restrict__ uv_lo,
    const float4 *__restrict__ conic, const RT *__restrict__ rgb, const FT *__restrict__ feat,
    const uint32_t *__restrict__ vals, const uint32_t *__restrict__ ranges, int64_t P, float *o_rgb, float *o_depth,
    float *o_sil, float *o_feat, float *o_T, int32_t *o_nc, int32_t *o_nb, uint32_t *bmask, int64_t bm_stride,
    const int gt, int32_t *status, int64_t capacity) {
    using SH = Shape<NP, true>;  // horizontal pixel pairs
    constexpr int NT = SH::THREADS, REC = kRecWords<D>, D4 = D / 4;
    constexpr int NL = SH::PIX_GROUPS ? NP : 1;  // mask bit registers per thread
    __shared__ float4 s_rec[BATCH * REC];  // the batch's records
    __shared__ float4 s_cull[BATCH];       // their culling constants

    if (gt < 0 || gt >= vt.tile_off[vt.n_views]) return;  // not a permutation of the tiles: leave the tile
    const int v = view_of_tile(vt, gt);
    const int t = gt - vt.tile_off[v];
    const int tx = t % vt.TX[v], ty = t / vt.TX[v];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t start = ranges[2 * gt], end = ranges[2 * gt + 1];
    checked_range(start, end, capacity, status);
    const int64_t voff = (int64_t)v * vt.n;
    int bx0, by0;
    SH::warp_origin(warp, bx0, by0);
    const float bcx = (float)(tx * kTile + bx0) + 0.5f * SH::BW, bcy = (float)(ty * kTile + by0) + 0.5f * SH::BH;
    const float hx = 0.5f * (SH::BW - 1), hy = 0.5f * (SH::BH - 1);

    BlendPixels<D, NP> px;
    px.init(vt, prm, v, tx, ty, tid);

    bool finished = false;
    // every warp stays in the batch loop (it stages splats and meets the CTA
    // barriers); a warp whose pixels are all done only skips the splat loop
    for (uint32_t b0 = start & ~31u; b0 < end; b0 += BATCH) {
        if (__syncthreads_and(px.all_done())) break;
        for (int i = tid; i < BATCH; i += NT) {
            const uint32_t j = b0 + i;
            if (j >= start && j < end) {
                const uint32_t item = checked_item(vals[j], voff, vt.n, status);
                const int64_t g = (int64_t)item - voff;
                const float4 a = uvdo[item];
                const SplatGeo sg = make_geo(a, uv_lo[item], conic[item]);
                float4 *rec = s_rec + i * REC;
                put_geo(rec, sg);
                s_cull[i] = ellipse_cull(sg, prm.alpha_min);
                rec[2] = load_rgbd(rgb, g, a.z);
#pragma unroll
                for (int q = 0; q < D4; ++q) rec[3 + q] = load_feat4(feat, g * D + 4 * q);
            }
        }
        __syncthreads();
        for (int c0 = 0; c0 < BATCH && !finished; c0 += 32) {
            // the chunk's splats that can reach the warp's box, lane k testing splat c0 + k
            const uint32_t j = b0 + c0 + lane;
            const float4 *chunk = s_rec + c0 * REC;
            const bool reach = j >= start && j < end &&
                               reaches_box_exact(geo_of(chunk + lane * REC), s_cull[c0 + lane], bcx, bcy, hx, hy);
            const uint32_t todo = __ballot_sync(0xffffffffu, reach);
            if (todo == 0u) continue;
            // blend-mask bits: batches start on 32-instance boundaries, so each 32-splat chunk is one
            // word of the mask; a lane ORs "my pixel(s) of group j blended splat k" into a register
            // (one per group its pixels lie in) and the warp combines the lanes of each of its NP
            // groups at the end of the chunk
            uint32_t lbits[NL];
#pragma unroll
            for (int l = 0; l < NL; ++l) lbits[l] = 0u;
            const int pos0 = (int)(b0 + c0 - start) + 1;
            finished = px.template walk<CNT>(prm, chunk, todo, pos0, lbits);
            if (bmask) {
#pragma unroll
                for (int l = 0; l < NP; ++l) {
                    const uint32_t mine =
                        SH::PIX_GROUPS ? lbits[l % NL] : ((SH::lanes_of_group(l) >> lane) & 1u ? lbits[0] : 0u);
                    const uint32_t word = __reduce_or_sync(0xffffffffu, mine);
                    if (lane == 0 && word)
                        atomicOr(&bmask[(int64_t)SH::group(warp, l) * bm_stride + ((b0 + c0) >> 5)], word);
                }
            }
        }
    }
    px.write(vt, prm, v, tx, ty, tid, P, o_rgb, o_depth, o_sil, o_feat, o_T, o_nc, o_nb);
}

// With QUEUE, the grid is as many CTAs as fit on the GPU at once and each takes tiles, in the
// tile order, from the work counter queue[0] until none is left; the last CTA to finish
// (counted in queue[1]) sets both counters back to 0 for the next launch.  Nothing waits.
template <int D, int NP, typename RT, typename FT, bool QUEUE, int BATCH, bool CNT>
__global__ void __launch_bounds__(Shape<NP>::THREADS, fwd_min_blocks(D, NP)) raster_fwd_kernel(
    ViewTable vt, Params prm, const float4 *__restrict__ uvdo, const float2 *__restrict__ uv_lo,
    const float4 *__restrict__ conic, const RT *__restrict__ rgb, const FT *__restrict__ feat,
    const uint32_t *__restrict__ vals, const uint32_t *__restrict__ ranges, int64_t P, float *o_rgb, float *o_depth,
    float *o_sil, float *o_feat, float *o_T, int32_t *o_nc, int32_t *o_nb, uint32_t *bmask, int64_t bm_stride,
    const uint32_t *__restrict__ order, int32_t *status, int64_t capacity, uint32_t *queue) {
    pdl_wait();  // the previous kernel's results (no trigger: see pdl_trigger)
    const int n_tiles = vt.tile_off[vt.n_views];
    const bool failed = binning_failed(status);  // the binning overflowed or gave up: render nothing
    if constexpr (QUEUE) {
        __shared__ int s_idx;
        for (;;) {
            __syncthreads();  // the previous tile's reads of shared memory and s_idx are done
            if (threadIdx.x == 0) s_idx = failed ? n_tiles : (int)atomicAdd(queue, 1u);
            __syncthreads();
            const int idx = s_idx;
            if (idx >= n_tiles) break;
            fwd_tile<D, NP, RT, FT, BATCH, CNT>(vt, prm, uvdo, uv_lo, conic, rgb, feat, vals, ranges, P, o_rgb, o_depth, o_sil,
                                    o_feat, o_T, o_nc, o_nb, bmask, bm_stride, order ? (int)order[idx] : idx,
                                    status, capacity);
        }
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicAdd(queue + 1, 1u) == gridDim.x - 1) {  // every CTA has taken its last item
                queue[0] = 0u;
                queue[1] = 0u;
            }
        }
    } else {
        if (failed) return;
        fwd_tile<D, NP, RT, FT, BATCH, CNT>(vt, prm, uvdo, uv_lo, conic, rgb, feat, vals, ranges, P, o_rgb, o_depth, o_sil,
                                o_feat, o_T, o_nc, o_nb, bmask, bm_stride,
                                order ? (int)order[blockIdx.x] : (int)blockIdx.x, status, capacity);
    }
}

// The same blend with one 32-thread block per pixel group (an 8x4 group with one pixel
// per thread, an 8x8 block with two): the group stages the tile's splats 32 at a time in
// its own shared memory, so it never waits at a barrier for the tile's other groups, and
// it leaves as soon as its own pixels are done, freeing its registers and shared memory.
// Arithmetic, order and outputs are those of raster_fwd_kernel.
// Register caps: 80 registers with one pixel per thread, spill-free; with two, 80 at D = 16, where 20
// bytes spill, and 128 at D = 32, spill-free.
constexpr int fwd_group_min_blocks(int D, int NP) { return NP == 1 ? 24 : (D <= 16 ? 22 : 16); }

template <int D, int NP, typename RT, typename FT>
__global__ void __launch_bounds__(32, fwd_group_min_blocks(D, NP)) raster_fwd_group_kernel(
    ViewTable vt, Params prm, const float4 *__restrict__ uvdo, const float2 *__restrict__ uv_lo,
    const float4 *__restrict__ conic, const RT *__restrict__ rgb, const FT *__restrict__ feat,
    const uint32_t *__restrict__ vals, const uint32_t *__restrict__ ranges, int64_t P, float *o_rgb, float *o_depth,
    float *o_sil, float *o_feat, float *o_T, int32_t *o_nc, int32_t *o_nb, uint32_t *bmask, int64_t bm_stride,
    const uint32_t *__restrict__ order, int32_t *status, int64_t capacity, uint32_t * /*queue*/) {
    pdl_wait();  // the previous kernel's results (no trigger: see pdl_trigger)
    using SH = Shape<NP, true>;  // horizontal pixel pairs
    constexpr int D4 = D / 4;
    constexpr int NL = SH::PIX_GROUPS ? NP : 1;  // mask bit registers per thread
    constexpr int GW = SH::WARPS;  // pixel-group blocks per tile
    constexpr int REC = kRecWords<D>;
    __shared__ float4 s_rec[32 * REC];

    if (binning_failed(status)) return;  // the binning overflowed or gave up: render nothing
    const int rank = blockIdx.x / GW, grp = blockIdx.x % GW;
    const int gt = order ? (int)order[rank] : rank;
    if (gt < 0 || gt >= vt.tile_off[vt.n_views]) return;  // not a permutation of the tiles: leave the tile
    const int v = view_of_tile(vt, gt);
    const int t = gt - vt.tile_off[v];
    const int tx = t % vt.TX[v], ty = t / vt.TX[v];
    const int lane = threadIdx.x;
    const int tid = grp * 32 + lane;  // the thread's index in the tile kernel's numbering
    uint32_t start = ranges[2 * gt], end = ranges[2 * gt + 1];
    checked_range(start, end, capacity, status);
    const int64_t voff = (int64_t)v * vt.n;
    int bx0, by0;
    SH::warp_origin(grp, bx0, by0);
    const float bcx = (float)(tx * kTile + bx0) + 0.5f * SH::BW, bcy = (float)(ty * kTile + by0) + 0.5f * SH::BH;
    const float hx = 0.5f * (SH::BW - 1), hy = 0.5f * (SH::BH - 1);

    BlendPixels<D, NP> px;
    px.init(vt, prm, v, tx, ty, tid);
    for (uint32_t b0 = start & ~31u; b0 < end; b0 += 32) {
        if (__all_sync(0xffffffffu, px.all_done())) break;
        // lane k stages splat b0 + k and tests whether it can reach the group's box
        bool reach = false;
        {
            const uint32_t j = b0 + lane;
            if (j >= start && j < end) {
                const uint32_t item = checked_item(vals[j], voff, vt.n, status);
                const int64_t g = (int64_t)item - voff;
                const float4 a = uvdo[item];
                const SplatGeo sg = make_geo(a, uv_lo[item], conic[item]);
                float4 *rec = s_rec + lane * REC;
                put_geo(rec, sg);
                reach = reaches_box_exact(sg, ellipse_cull(sg, prm.alpha_min), bcx, bcy, hx, hy);
                rec[2] = load_rgbd(rgb, g, a.z);
#pragma unroll
                for (int q = 0; q < D4; ++q) rec[3 + q] = load_feat4(feat, g * D + 4 * q);
            }
        }
        const uint32_t todo = __ballot_sync(0xffffffffu, reach);
        __syncwarp();
        uint32_t lbits[NL];
#pragma unroll
        for (int j = 0; j < NL; ++j) lbits[j] = 0u;
        px.template walk<true>(prm, s_rec, todo, (int)(b0 - start) + 1, lbits);
        if (bmask) {
            // the chunk is one mask word; words at a tile's ends are shared with the
            // neighbouring tile's blocks, hence the atomic OR
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const uint32_t mine =
                    SH::PIX_GROUPS ? lbits[j % NL] : ((SH::lanes_of_group(j) >> lane) & 1u ? lbits[0] : 0u);
                const uint32_t word = __reduce_or_sync(0xffffffffu, mine);
                if (lane == 0 && word) atomicOr(&bmask[(int64_t)SH::group(grp, j) * bm_stride + (b0 >> 5)], word);
            }
        }
        __syncwarp();  // every lane is done with the staged chunk before the next one
    }
    px.write(vt, prm, v, tx, ty, tid, P, o_rgb, o_depth, o_sil, o_feat, o_T, o_nc, o_nb);
}

// One batch slot of the ring forward: B staged splat records.
template <int D, int B>
struct RingSlot {
    float4 rec[B * kRecWords<D>];
    float4 cull[B];
};

// The per-tile forward with its splats staged into a ring of NBUF batch slots of B records:
// the four warps stage each batch together (a quarter each) and walk the staged batches at
// their own pace, synchronised per slot by mbarriers instead of CTA barriers: slot full (every
// warp has staged its quarter) and slot empty (every warp has walked it), so a warp can run up
// to NBUF - 1 batches ahead of the slowest.  A warp whose pixels are all done still stages
// its quarters; once every warp's pixels are done, the next batch staged carries a stop flag
// and every warp leaves at that same batch.  Arithmetic, order and outputs are those of
// raster_fwd_kernel.  Every wait is bounded (prm.spin_limit polls); one that gives up sets
// GS_ERR_TIMEOUT in the status word and its warp leaves without writing its pixels.
template <int D, typename RT, typename FT, int B, int NBUF>
__global__ void __launch_bounds__(Shape<2, true>::THREADS, fwd_min_blocks(D, 2)) raster_fwd_ring_kernel(
    ViewTable vt, Params prm, const float4 *__restrict__ uvdo, const float2 *__restrict__ uv_lo,
    const float4 *__restrict__ conic, const RT *__restrict__ rgb, const FT *__restrict__ feat,
    const uint32_t *__restrict__ vals, const uint32_t *__restrict__ ranges, int64_t P, float *o_rgb, float *o_depth,
    float *o_sil, float *o_feat, float *o_T, int32_t *o_nc, int32_t *o_nb, uint32_t *bmask, int64_t bm_stride,
    const uint32_t *__restrict__ order, int32_t *status, int64_t capacity, uint32_t * /*queue*/) {
    pdl_wait();  // the previous kernel's results (no trigger: see pdl_trigger)
    constexpr int NP = 2;
    using SH = Shape<NP, true>;  // horizontal pixel pairs
    constexpr int NT = SH::THREADS, NW = SH::WARPS;
    constexpr int NL = SH::PIX_GROUPS ? NP : 1;
    constexpr int D4 = D / 4;
    constexpr int QB = B / NW;  // records a warp stages per batch
    static_assert(B % 32 == 0 && QB <= 32 && NBUF >= 2, "ring shape");
    __shared__ RingSlot<D, B> s_slot[NBUF];
    __shared__ __align__(8) uint64_t s_full[NBUF], s_empty[NBUF];
    __shared__ int s_stop[NBUF][NW];
    __shared__ int s_done;

    if (binning_failed(status)) return;  // the binning overflowed or gave up: render nothing
    const int gt = order ? (int)order[blockIdx.x] : (int)blockIdx.x;
    if (gt < 0 || gt >= vt.tile_off[vt.n_views]) return;  // not a permutation of the tiles: leave the tile
    const int v = view_of_tile(vt, gt);
    const int t = gt - vt.tile_off[v];
    const int tx = t % vt.TX[v], ty = t / vt.TX[v];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint32_t start = ranges[2 * gt], end = ranges[2 * gt + 1];
    checked_range(start, end, capacity, status);
    const int64_t voff = (int64_t)v * vt.n;
    if (tid < NBUF) {
        mbar_init(&s_full[tid], NT);
        mbar_init(&s_empty[tid], NT);
    }
    if (tid == 0) s_done = 0;
    __syncthreads();  // the barriers are initialised before any thread uses them

    const uint32_t first = start & ~31u;
    const int n_batch = end > first ? (int)((end - first + B - 1) / B) : 0;
    // warp `warp` stages records [warp QB, (warp + 1) QB) of batch j into its slot, with its
    // stop flag (every warp's pixels done when it staged), then arrives on the slot's full barrier
    auto stage = [&](int j) {
        RingSlot<D, B> &S = s_slot[j % NBUF];
        const uint32_t b0 = first + (uint32_t)j * B;
        if (lane < QB) {
            const int k = warp * QB + lane;
            const uint32_t jj = b0 + k;
            if (jj >= start && jj < end) {
                const uint32_t item = checked_item(vals[jj], voff, vt.n, status);
                const int64_t g = (int64_t)item - voff;
                const float4 a = uvdo[item];
                const SplatGeo sg = make_geo(a, uv_lo[item], conic[item]);
                float4 *rec = S.rec + k * kRecWords<D>;
                put_geo(rec, sg);
                S.cull[k] = ellipse_cull(sg, prm.alpha_min);
                rec[2] = load_rgbd(rgb, g, a.z);
#pragma unroll
                for (int q = 0; q < D4; ++q) rec[3 + q] = load_feat4(feat, g * D + 4 * q);
            }
        }
        if (lane == 0) s_stop[j % NBUF][warp] = *(volatile int *)&s_done == NW;
        mbar_arrive(&s_full[j % NBUF]);
    };

    int bx0, by0;
    SH::warp_origin(warp, bx0, by0);
    const float bcx = (float)(tx * kTile + bx0) + 0.5f * SH::BW, bcy = (float)(ty * kTile + by0) + 0.5f * SH::BH;
    const float hx = 0.5f * (SH::BW - 1), hy = 0.5f * (SH::BH - 1);
    BlendPixels<D, NP> px;
    px.init(vt, prm, v, tx, ty, tid);
    auto flush = [&](const uint32_t (&lbits)[NL], uint32_t word_idx) {
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            const uint32_t mine =
                SH::PIX_GROUPS ? lbits[j % NL] : ((SH::lanes_of_group(j) >> lane) & 1u ? lbits[0] : 0u);
            const uint32_t word = __reduce_or_sync(0xffffffffu, mine);
            if (lane == 0 && word) atomicOr(&bmask[(int64_t)SH::group(warp, j) * bm_stride + word_idx], word);
        }
    };

    // a wait the whole warp takes together (every lane sees the phase complete), bounded
    auto wait_warp = [&](uint64_t *bar, uint32_t parity) {
        for (int it = 0;; ++it) {
            if (__all_sync(0xffffffffu, mbar_test(bar, parity))) return true;
            if (prm.spin_limit < 0 || it >= prm.spin_limit) return false;
        }
    };
    for (int j = 0; j < NBUF - 1 && j < n_batch; ++j) stage(j);
    bool counted = false;  // this warp's pixels are all done and s_done counts it
    bool ok = true;
    for (int i = 0; i < n_batch; ++i) {
        const int slot = i % NBUF;
        if (!wait_warp(&s_full[slot], (uint32_t)(i / NBUF) & 1u)) {
            ok = false;
            break;
        }
        bool stop = false;
#pragma unroll
        for (int w = 0; w < NW; ++w) stop = stop || s_stop[slot][w];
        if (stop) break;  // the same batch for every warp: every pixel of the tile is done
        const RingSlot<D, B> &S = s_slot[slot];
        const uint32_t b0 = first + (uint32_t)i * B;
        if (!__all_sync(0xffffffffu, px.all_done())) {
            const int k_lo = b0 < start ? (int)(start - b0) : 0;
            const int nb = min((uint32_t)B, end - b0);
            bool finished = false;
            for (int c0 = k_lo & ~31; c0 < nb && !finished; c0 += 32) {
                uint32_t lbits[NL];
#pragma unroll
                for (int jj = 0; jj < NL; ++jj) lbits[jj] = 0u;
                const int kl = c0 + lane;
                bool reach = false;
                if (kl >= k_lo && kl < nb) {
                    const SplatGeo sg = geo_of(S.rec + kl * kRecWords<D>);
                    reach = reaches_box_exact(sg, S.cull[kl], bcx, bcy, hx, hy);
                }
                const uint32_t todo = __ballot_sync(0xffffffffu, reach);
                finished = px.template walk<true>(prm, S.rec + c0 * kRecWords<D>, todo, (int)(b0 - start) + c0 + 1, lbits);
                if (bmask) flush(lbits, (b0 + c0) >> 5);
            }
        }
        if (!counted && __all_sync(0xffffffffu, px.all_done())) {
            counted = true;
            if (lane == 0) atomicAdd(&s_done, 1);
        }
        __syncwarp();
        mbar_arrive(&s_empty[slot]);
        // batch i + NBUF - 1 goes into the slot batch i - 1 used, once every warp has walked it
        const int jn = i + NBUF - 1;
        if (jn < n_batch) {
            if (i >= 1 && !wait_warp(&s_empty[jn % NBUF], (uint32_t)((i - 1) / NBUF) & 1u)) {
                ok = false;
                break;
            }
            stage(jn);
        }
    }
    if (!ok) {
        set_status(status, GS_ERR_TIMEOUT);
        return;  // this warp's pixels stay unwritten; the status word says so
    }
    px.write(vt, prm, v, tx, ty, tid, P, o_rgb, o_depth, o_sil, o_feat, o_T, o_nc, o_nb);
}

template <int D, int NP, typename RT, typename FT>
gs_status launch(const ViewTable &vt, const Params &prm, const gs_gaussians *g, const gs_projected *proj,
                 const gs_binning *bins, gs_images *out, cudaStream_t st) {
    const int tiles = vt.tile_off[vt.n_views];
    const int64_t P = vt.pix_off[vt.n_views];
    auto args = [&](auto kern, int blocks, int threads, size_t smem) -> gs_status {
        return launch_pdl(
            kern, blocks, threads, smem, st, vt, prm, reinterpret_cast<const float4 *>(proj->uvdo),
            reinterpret_cast<const float2 *>(proj->uv_lo), reinterpret_cast<const float4 *>(proj->conic),
            static_cast<const RT *>(g->rgb), static_cast<const FT *>(g->feat), bins->vals, bins->ranges, P, out->rgb,
            out->depth, out->sil, out->feat, out->T_final, out->n_contrib, out->n_blended, out->blend_mask,
            bins->capacity / 32 + 1, bins->tile_order, bins->status, bins->capacity, bins->queue);
    };
    if constexpr (NP <= 2) {
        if (prm.fwd_group) {
            return args(raster_fwd_group_kernel<D, NP, RT, FT>, tiles * Shape<NP>::WARPS, 32, 0);
        }
    }
    if (prm.fwd_ring) {
        // batch slots within the 48 KB of static shared memory: two of 128 or four of 64 records
        // at D = 16, three of 64 at D = 32
        if constexpr (NP == 2 && D == 16) {
            if (prm.fwd_batch == 128)
                return args(raster_fwd_ring_kernel<D, RT, FT, 128, 2>, tiles, Shape<2, true>::THREADS, 0);
            if (prm.fwd_batch == 64)
                return args(raster_fwd_ring_kernel<D, RT, FT, 64, 4>, tiles, Shape<2, true>::THREADS, 0);
        }
        if constexpr (NP == 2 && D == 32)
            if (prm.fwd_batch == 64)
                return args(raster_fwd_ring_kernel<D, RT, FT, 64, 3>, tiles, Shape<2, true>::THREADS, 0);
        return GS_ERR_UNSUPPORTED;
    }
    // the per-tile forward with BATCH splats staged per round; batches other than 128 are built
    // for the two-pixel shape: 64 at feature widths 16 and 32, 256 at 16
    // (the blended-splat count is compiled in only for a caller that asks for it)
    auto per_tile_cnt = [&](auto batch_c, auto cnt_c) -> gs_status {
        constexpr int B = decltype(batch_c)::value;
        constexpr bool C = decltype(cnt_c)::value;
        if (prm.fwd_queue) {
            // one wave: as many CTAs as are resident at once
            static int res = 0;  // this kernel instance: SMs x resident CTAs per SM
            if (res == 0) {
                int dev = 0, sms = 0, per_sm = 0;
                if (cudaGetDevice(&dev) != cudaSuccess ||
                    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
                    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, raster_fwd_kernel<D, NP, RT, FT, true, B, C>,
                                                                  Shape<NP>::THREADS, 0) != cudaSuccess)
                    return GS_ERR_CUDA;
                res = sms * (per_sm > 0 ? per_sm : 1);
            }
            return args(raster_fwd_kernel<D, NP, RT, FT, true, B, C>, tiles < res ? tiles : res, Shape<NP>::THREADS,
                        0);
        }
        return args(raster_fwd_kernel<D, NP, RT, FT, false, B, C>, tiles, Shape<NP>::THREADS, 0);
    };
    auto per_tile = [&](auto batch_c) -> gs_status {
        return out->n_blended ? per_tile_cnt(batch_c, std::true_type()) : per_tile_cnt(batch_c, std::false_type());
    };
    if (prm.fwd_batch == 128) return per_tile(std::integral_constant<int, 128>());
    if constexpr (NP == 2 && D >= 16)
        if (prm.fwd_batch == 64) return per_tile(std::integral_constant<int, 64>());
    if constexpr (NP == 2 && D == 16)  // 256 records of D = 32 would not fit the 48 KB of static shared memory
        if (prm.fwd_batch == 256) return per_tile(std::integral_constant<int, 256>());
    return GS_ERR_UNSUPPORTED;
}

template <int D, typename RT, typename FT>
gs_status by_np(int np, const ViewTable &vt, const Params &prm, const gs_gaussians *g, const gs_projected *proj,
                const gs_binning *bins, gs_images *out, cudaStream_t st) {
    if (np == 1) return launch<D, 1, RT, FT>(vt, prm, g, proj, bins, out, st);
    if constexpr (D >= 16) {
        if (np == 2) return launch<D, 2, RT, FT>(vt, prm, g, proj, bins, out, st);
        if constexpr (D <= 16)
            if (np == 4) return launch<D, 4, RT, FT>(vt, prm, g, proj, bins, out, st);
    }
    return GS_ERR_UNSUPPORTED;
}

}  // namespace

bool storage_ok(const gs_gaussians *g) {
    bool plain = g->rgb_dtype == GS_F32 && g->feat_dtype == GS_F32;
    bool half = g->rgb_dtype == GS_F16 && g->feat_dtype == GS_BF16 && (g->feat_dim == 16 || g->feat_dim == 32);
    return (plain || half) && feat_dim_ok(g->feat_dim) && g->rgb && (g->feat || g->feat_dim == 0);
}

}  // namespace gs

extern "C" gs_status gs_render_fwd(const gs_gaussians *g, const gs_projected *proj, const gs_binning *bins,
                                   const gs_camera *cams, int n_views, const gs_raster_params *p, gs_images *out,
                                   gs_stream stream) {
    GS_NVTX_RANGE("gs_render_fwd");
    using namespace gs;
    if (!g || !proj || !bins || !out || g->n < 0) return GS_ERR_ARG;
    ViewTable vt;
    Params prm;
    if (!make_view_table(cams, n_views, g->n, &vt) || !make_params(p, &prm)) return GS_ERR_ARG;
    if (!feat_dim_ok(g->feat_dim)) return GS_ERR_UNSUPPORTED;
    if (!out->rgb || !out->depth || !out->sil || !out->T_final || !out->n_contrib || (g->feat_dim && !out->feat) ||
        !bins->ranges)
        return GS_ERR_ARG;
    if (g->n > 0 && (!storage_ok(g) || !bins->vals || !proj->uvdo || !proj->uv_lo || !proj->conic)) {
        return storage_ok(g) ? GS_ERR_ARG : GS_ERR_UNSUPPORTED;
    }
    if (g->feat_dim && (reinterpret_cast<uintptr_t>(g->feat) & 15)) return GS_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if (out->blend_mask) {
        const gs_status s = cuda_status(cudaMemsetAsync(
            out->blend_mask, 0, sizeof(uint32_t) * kGroups * (size_t)(bins->capacity / 32 + 1), st));
        if (s) return s;
    }
    int np = prm.fwd_np ? prm.fwd_np : default_fwd_np(g->feat_dim);
    // The default at D = 16 and 32 is two pixels per thread, and one where the image has too few tiles for
    // that: up to two waves of the two-pixel CTAs (six per SM at D = 16, four at D = 32) twice as many warps
    // hide more latency.  Measured, one against two pixels per thread: D = 16: 0.044 / 0.058 ms at 320x240, 0.068
    // / 0.084 at 640x480, then 0.103 / 0.098 at 880x600 and 0.237 / 0.218 at 1200x680; D = 32: 0.053 / 0.063
    // at 320x240, 0.148 / 0.163 at 640x480, but 0.114 / 0.109 at 811x607.  A scanned map, whose splats are
    // small, would take one pixel further: 0.145 / 0.156 at 800x600, which 1,900 tiles put just above the line of
    // 1,824.  The images do not depend on it.
    if (!prm.fwd_np && g->feat_dim >= 16 && prm.fwd_blocks == GS_BWD_BLOCKS_DEFAULT && prm.fwd_batch == kBatch &&
        vt.tile_off[n_views] <= kSMs * (g->feat_dim == 16 ? 12 : 8))
        np = 1;
    prm.fwd_group = prm.fwd_blocks == GS_BWD_BLOCKS_GROUP;
    prm.fwd_queue = prm.fwd_blocks == GS_BLOCKS_QUEUE;
    prm.fwd_ring = prm.fwd_blocks == GS_BLOCKS_RING;
    if (prm.fwd_ring && np != 2) return GS_ERR_UNSUPPORTED;
    if (prm.fwd_group && np > 2) return GS_ERR_UNSUPPORTED;
    if (prm.fwd_queue && !bins->queue) return GS_ERR_ARG;
    if (g->rgb_dtype == GS_F16) {
        if (g->feat_dim == 16) return by_np<16, __half, __nv_bfloat16>(np, vt, prm, g, proj, bins, out, st);
        return by_np<32, __half, __nv_bfloat16>(np, vt, prm, g, proj, bins, out, st);
    }
    switch (g->feat_dim) {
        case 0: return by_np<0, float, float>(np, vt, prm, g, proj, bins, out, st);
        case 4: return by_np<4, float, float>(np, vt, prm, g, proj, bins, out, st);
        case 8: return by_np<8, float, float>(np, vt, prm, g, proj, bins, out, st);
        case 16: return by_np<16, float, float>(np, vt, prm, g, proj, bins, out, st);
        case 32: return by_np<32, float, float>(np, vt, prm, g, proj, bins, out, st);
        default: return GS_ERR_UNSUPPORTED;
    }
}
