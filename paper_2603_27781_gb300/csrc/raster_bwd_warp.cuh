// Blend backward (Eq. 4-7 differentiated) with one single-warp block per pixel
// group, D 16 or 32, with the forward's blend mask: map mode (every parameter's
// sums) and pose-only mode (the six sums the projection backward needs for the
// twist).
//
// The tile kernel's eight warps share one staged splat batch and meet at a CTA
// barrier per batch, so a tile's warps all wait for whichever of them has the
// longest masked list, and the CTA holds its registers and shared memory until
// its slowest warp ends.  Here each pixel group (an 8x4 group, or an 8x8 block of
// two with two pixels per thread) is its own 32-thread block: it builds its own
// list of the instances its pixels blended (back to front, from the mask words),
// stages a few splat records at a time in its own shared memory and runs the
// per-pixel recurrence on them.  Nothing waits on another warp, and a finished
// group frees its resources at once.
//
// Every per-splat sum is deferred.  While it walks a stage of splats, each pixel only records, per
// splat, its weight w = alpha T (the factor of the depth, colour and feature gradients; in pose mode w
// times the pixel's depth gradient) and dpow = o G dL/dalpha (zero where alpha is clamped), the factor
// of every geometric gradient: with (dx, dy) the pixel centre from the splat centre, the centre and
// conic gradients need only the moments
//   S1, Sx, Sy, Sxx, Sxy, Syy = sum over pixels of dpow (1, dx, dy, dx^2, dx dy, dy^2),
// and the opacity gradient is S1 / o.  After the stage, lanes (pixel column, slot pair) contract the
// slots with the block's per-pixel terms (weights against the gradients of depth, colour and features;
// dpow against the row's dy, the column's dx scaling the column sums afterwards) in packed FP32
// multiply-adds, the eight columns are combined by one transpose reduction per stage, and each slot's
// sums go out as 16-byte L2 reductions.  No warp reduction runs per splat.
//
// What bounds it: the shared-memory pipe (every 16-byte read returns 512 bytes to a warp, four cycles,
// broadcast or not; about 57 cycles per splat and block at D = 16 with two pixels per thread) and
// instruction issue, both near 70 %.  Packed multiply-adds for g.x, the contraction, z = W f and W^T z,
// weight and dpow as one 8-byte pair, moments about the splat centre (no expansion afterwards, nothing
// cancels) and a first reduction level without selects took the map mode from 0.417 to 0.391 ms (1M
// Gaussians, D = 16, 1200x680) and 0.217 to 0.207 (1M, D = 32, 640x480), and the pose mode, which before
// reduced six values over the warp for every splat, from 0.355 to 0.241 ms (300k scanned Gaussians).
//
// Factored feature gradients.  When the image gradient of the features comes from
// a linear decoder (Eq. 8 read as a 1x1 convolution), g_feat = W^T e with e the
// gradient of the K logits.  Then g_feat . f = e . (W f) and sum_p w_p g_feat,p =
// W^T sum_p w_p e_p, so the kernel stages z = W f (K values) per splat, evaluates
// the K-term dot product per pixel and contracts K terms, and multiplies by W^T once
// per splat: the same sums, in fewer operations when K < D.
#pragma once

#include "raster_bwd.cuh"

namespace gs {

// Feature-like gradient channels per pixel in the factored form: the K <= kFactorK logit
// gradients (zero beyond K).
constexpr int kFactorK = 8;

// Layout of the deferred sums: SL slots (splats staged and contracted together).  In the contraction
// lane (column c, slot group jg) sums, for the SPL slots of group jg, the NWT weighted terms (map mode)
// and the moments of dpow over the ROWS pixels of column c; the eight columns are then added by
// shuffles.  In the epilogue LPS = 32 / SL lanes serve each slot.
template <int D, int NP, bool MAP, int KF, int SL>
struct WarpLayout {
    static constexpr int F = KF ? KF : D;
    static constexpr int PXW = 32 * NP;         // pixels of the block, 8 wide
    static constexpr int ROWS = PXW / 8;
    static constexpr int LPS = 32 / SL;
    static constexpr int SPL = SL / 4;          // slots per lane in the contraction
    static constexpr int NWT = MAP ? 4 + F : 0; // weighted terms: depth, r, g, b, F
    static constexpr int GROW = NWT;            // a pixel's row of weighted terms
    // a slot's sums: the terms, then S1, Sx, Sy, Sxx, Sxy, Syy (map mode), or Sx, Sy, Sxx, Sxy, Syy and
    // the depth gradient (pose mode)
    static constexpr int NSV = NWT + 6;
    // The contraction runs in up to four chunks of terms so that a lane's running sums fit in
    // its registers (at most 2 CAPS values): the first chunk [0, T1) carries the moments,
    // then [T1, T2), [T2, T3) and [T3, NWT).
    static constexpr int CAPS = KF ? 28 : NP == 2 ? 18 : D == 32 ? 20 : 12;
    static constexpr int TC = CAPS / 4 * 4;
    static constexpr int T1 = NWT < (CAPS - 6) / 4 * 4 ? NWT : (CAPS - 6) / 4 * 4;
    static constexpr int T2 = NWT < T1 + TC ? NWT : T1 + TC;
    static constexpr int T3 = NWT < T2 + TC ? NWT : T2 + TC;
    static_assert(NWT <= T3 + TC, "four chunks cover the terms");
    // a slot's row of per-pixel pairs: 8 words beyond a multiple of 32, which spreads the contraction's
    // reads (two slots a group, taken in opposite order by even and odd columns) over all banks
    static constexpr int WROW = PXW + 4;
    static_assert(NWT % 4 == 0 && SL % 8 == 0 && SPL % 2 == 0 && (!MAP || D % (4 * LPS) == 0),
                  "16-byte rows; lanes divide the work");
};

template <int V> struct IntC { static constexpr int value = V; };

// Slots per stage: 8 (four lanes per slot) keeps the per-slot arrays small enough for more
// resident blocks (pose mode, 300k scanned Gaussians at 1200x680: 0.241 ms, 0.265 with 16).
constexpr int kSlots = 8;

// Resident blocks per SM the register allocation must allow.  With two pixels per thread 16 in map mode (128
// registers), except with the features themselves at D = 32, whose 19 KB of shared memory allow 11
// anyway; in pose mode 18 at D = 16 (96 registers: 0.243 -> 0.232 ms, 300k scanned Gaussians at 1200x680; 0.240 with
// 14, 0.237 with 20) and 14 at D = 32 (factored form, 0.151 -> 0.147 ms, 1M Gaussians at 640x480).  With
// one pixel per thread, which small images take, 16 as well in map mode, so that the contraction runs
// in fewer chunks (20 and 18 blocks before: factored form, 0.066 -> 0.060 ms at 64x48, 0.093 -> 0.082 at 640x320;
// features themselves at D = 32, 0.076 -> 0.067 at 320x240), but 20 with the features themselves at D = 16 (0.098 ms,
// 0.101 with 16, at 600x384) and, in pose mode, 24 at D = 16 (0.069, 0.072) and 20 at D = 32 (0.050 with 24, 0.047 at
// 320x240).
template <int D, int NP, bool MAP, int KF> constexpr int warp_bwd_min_blocks() {
    if (NP == 1) return !MAP ? (D == 16 ? 24 : 20) : (D == 16 && KF == 0) ? 20 : 16;
    if (!MAP) return D == 16 ? 18 : 14;
    return D == 32 && KF == 0 ? 11 : 16;
}

template <int D, int NP, bool MAP, int KF, typename RT, typename FT>
__global__ void __launch_bounds__(32, warp_bwd_min_blocks<D, NP, MAP, KF>())
    raster_bwd_warp_kernel(ViewTable vt, Params prm, BwdArgs A) {
    pdl_wait();  // the previous kernel's results (no trigger: see pdl_trigger)
    using SH = Shape<NP>;
    constexpr int STAGE = kSlots;
    using WL = WarpLayout<D, NP, MAP, KF, STAGE>;
    constexpr int F = WL::F;
    constexpr int F4 = F / 4;
    constexpr int NC2 = 2 + F / 2;        // channel pairs: (r, g), (b, depth), then F
    constexpr int GW = SH::WARPS;         // pixel-group blocks per tile
    constexpr int PARTS = 32 / STAGE;     // lanes per staged splat
    static_assert(F % 4 == 0 && (KF == 0 || KF % PARTS == 0), "staged values in float4 / lane parts");
    __shared__ SplatGeo s_geo[STAGE];
    __shared__ float4 s_rgbd[STAGE];
    __shared__ __align__(16) float s_feat[STAGE * F];  // features, or z = W f in the factored form
    __shared__ uint32_t s_item[STAGE];
    __shared__ int s_pos[STAGE];
    __shared__ uint32_t s_list[64];
    __shared__ float2 s_ctr[STAGE];                                   // splat centre from the block's
    __shared__ float2 s_wp[STAGE * WL::WROW];                         // [slot][pixel] weight, dpow
    __shared__ __align__(16) float s_g[MAP ? WL::PXW * WL::GROW : 4]; // [pixel][term] gradients
    __shared__ float s_t[STAGE * WL::NSV];                            // [slot][sum] sums
    // W, K x D (rows >= K zero), rows padded by 4 so that the four lane parts, which read rows
    // k = part (K / 4) + kk, fall in different banks
    constexpr int BROW = D + 4;
    __shared__ __align__(16) float s_basis[KF ? KF * BROW : 4];
    // raw records of two stages (the next one is copied while the current one is processed):
    // centre / depth / opacity, conic / radius, centre low parts, colour (f32 storage), features
    constexpr bool RGB32 = sizeof(RT) == 4;
    constexpr int FB = D * (int)sizeof(FT);   // feature bytes per Gaussian
    constexpr int FCH = FB / 16;              // their 16-byte chunks
    // a staged slot's feature row, padded to an odd number of 16-byte chunks so that the eight
    // slots' rows start in different banks (the copies and the reads of one chunk index are
    // then conflict-free)
    constexpr int FBP = FCH % 2 == 0 ? FB + 16 : FB;
    constexpr int NCOPY = 3 + (RGB32 ? 3 : 0) + FCH;
    static_assert(FB % 16 == 0, "features in 16-byte chunks");
    __shared__ float4 r_a[2][STAGE], r_c[2][STAGE];
    __shared__ float2 r_lo[2][STAGE];
    __shared__ float r_rgb[2][STAGE][4];
    __shared__ __align__(16) unsigned char r_f[2][STAGE * FBP];
    const RT *rgb = static_cast<const RT *>(A.rgb);
    const FT *feat = static_cast<const FT *>(A.feat);

    if (binning_failed(A.status)) return;  // the binning overflowed or gave up
    const int rank = blockIdx.x / GW, grp = blockIdx.x % GW;
    const int gt = A.order ? (int)A.order[rank] : rank;
    if (gt < 0 || gt >= vt.tile_off[vt.n_views]) return;  // not a permutation of the tiles: leave the tile
    const int v = view_of_tile(vt, gt);
    const int t = gt - vt.tile_off[v];
    const int tx = t % vt.TX[v], ty = t / vt.TX[v];
    const int lane = threadIdx.x;
    const int tid = grp * 32 + lane;  // the thread's index in the tile kernel's numbering
    const uint32_t start = A.ranges[2 * gt];
    const int64_t voff = (int64_t)v * vt.n;
    const int64_t P = A.P;
    int bx0, by0;
    SH::warp_origin(grp, bx0, by0);
    // block centre: pixel (lx, ly) of the block sits at (lx - 3.5, ly + 0.5 - ROWS / 2) from it
    const float bcx = (float)(tx * kTile + bx0) + 4.f, bcy = (float)(ty * kTile + by0) + 0.5f * WL::ROWS;

    if constexpr (KF > 0) {
        for (int i = lane; i < KF * D; i += 32)
            s_basis[(i / D) * BROW + i % D] = i < A.feat_rank * D ? A.feat_basis[i] : 0.f;
    }

    float2 gch[NP][NC2];  // gradients of the channel pairs
    float gsil[NP], T[NP], gS[NP], pxc[NP], pyc[NP];
    int last[NP];
    int my_max = 0;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        int lx, ly;
        SH::pixel(tid, p, lx, ly);
        const int px = tx * kTile + lx, py = ty * kTile + ly;
        pxc[p] = (float)px + 0.5f;
        pyc[p] = (float)py + 0.5f;
        T[p] = 1.f;
        last[p] = 0;
#pragma unroll
        for (int c = 0; c < NC2; ++c) gch[p][c] = make_float2(0.f, 0.f);
        gsil[p] = 0.f;
        if (px < vt.W[v] && py < vt.H[v]) {
            const int64_t pix = vt.pix_off[v] + (int64_t)py * vt.W[v] + px;
            T[p] = A.T_final[pix];
            last[p] = A.n_contrib[pix];
            gch[p][0] = make_float2(A.g_rgb[pix], A.g_rgb[P + pix]);
            gch[p][1] = make_float2(A.g_rgb[2 * P + pix], A.g_depth[pix]);
            gsil[p] = A.g_sil ? A.g_sil[pix] : 0.f;
#pragma unroll
            for (int c = 0; c < F / 2; ++c) {
                if constexpr (KF > 0)
                    gch[p][2 + c] = make_float2(2 * c < A.feat_rank ? A.feat_coef[2 * c * P + pix] : 0.f,
                                                2 * c + 1 < A.feat_rank ? A.feat_coef[(2 * c + 1) * P + pix] : 0.f);
                else
                    gch[p][2 + c] = make_float2(A.g_feat[2 * c * P + pix], A.g_feat[(2 * c + 1) * P + pix]);
            }
        }
        gS[p] = gch[p][0].x * prm.bg[0] + gch[p][0].y * prm.bg[1] + gch[p][1].x * prm.bg[2];
        my_max = max(my_max, last[p]);
    }
    const int wmax = checked_last(start, A.ranges, gt, __reduce_max_sync(0xffffffffu, my_max), A.capacity, A.status);
    if (wmax == 0) return;  // no pixel of the group blended anything (warp-uniform)
    if constexpr (MAP) {
        // pixel q = p * 32 + lane of the block: its weighted terms (depth, r, g, b, F), part by part
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float4 *row = reinterpret_cast<float4 *>(s_g + (p * 32 + lane) * WL::GROW);
            row[0] = make_float4(gch[p][1].y, gch[p][0].x, gch[p][0].y, gch[p][1].x);
#pragma unroll
            for (int c = 0; c < F4; ++c)
                row[1 + c] = make_float4(gch[p][2 + 2 * c].x, gch[p][2 + 2 * c].y, gch[p][3 + 2 * c].x, gch[p][3 + 2 * c].y);
        }
    }

    // After a stage: lane (column col, slot group jg) sums, for its SPL slots, w times the weighted terms
    // [T0, T1) and (with MOM) dpow times (1, dy, dy^2) down the pixels of its column, dy from the
    // splat's own centre (so nothing cancels when the sums are formed), and scales the column sums by
    // the column's dx into the moments.  Lanes of odd columns take the two halves of their slots in
    // the opposite order, so that the first level of the transpose reduction over the eight columns
    // sends one half and keeps the other without selects; the next two levels split the values.
    auto contract_chunk = [&](auto t0c, auto t1c, auto momc) {
        constexpr int T0 = decltype(t0c)::value, T1 = decltype(t1c)::value;
        constexpr bool MOM = decltype(momc)::value != 0;
        constexpr int SPL = WL::SPL, NT = T1 - T0, CV = NT + (MOM ? 6 : 0);
        constexpr int HALF = SPL / 2 * CV, LEN = (HALF + 3) / 4 * 4;  // values kept after the first level
        const int col = lane & 7, jg = lane >> 3;
        const bool odd = col & 1;
        float2 acc[SPL][NT / 2 > 0 ? NT / 2 : 1];
        float s1[SPL], sy[SPL], syy[SPL], sd[SPL], dy[SPL], dx[SPL];
        const float2 *wp[SPL];
#pragma unroll
        for (int sj = 0; sj < SPL; ++sj) {
            const int j = jg * SPL + (odd ? (sj + SPL / 2) % SPL : sj);
            wp[sj] = s_wp + j * WL::WROW + col;
#pragma unroll
            for (int c = 0; c < NT / 2; ++c) acc[sj][c] = make_float2(0.f, 0.f);
            s1[sj] = sy[sj] = syy[sj] = sd[sj] = 0.f;
            if constexpr (MOM) {
                const float2 ctr = s_ctr[j];
                dx[sj] = (float)col - 3.5f - ctr.x;
                dy[sj] = 0.5f - 0.5f * WL::ROWS - ctr.y;
            }
        }
#pragma unroll 4
        for (int ly = 0; ly < WL::ROWS; ++ly) {
            float2 e[SPL];
#pragma unroll
            for (int sj = 0; sj < SPL; ++sj) {
                e[sj] = wp[sj][ly * 8];
                if constexpr (MOM) {
                    const float d = dy[sj] + (float)ly, t = d * e[sj].y;
                    s1[sj] += e[sj].y;
                    sy[sj] += t;
                    syy[sj] = fmaf(d, t, syy[sj]);
                    if constexpr (!MAP) sd[sj] += e[sj].x;
                }
            }
            const float4 *g4 = reinterpret_cast<const float4 *>(s_g + (ly * 8 + col) * WL::GROW + T0);
#pragma unroll
            for (int c = 0; c < NT / 4; ++c) {
                const float4 gv = g4[c];
#pragma unroll
                for (int sj = 0; sj < SPL; ++sj) {
                    const float2 w = make_float2(e[sj].x, e[sj].x);
                    acc[sj][2 * c] = fma2(w, make_float2(gv.x, gv.y), acc[sj][2 * c]);
                    acc[sj][2 * c + 1] = fma2(w, make_float2(gv.z, gv.w), acc[sj][2 * c + 1]);
                }
            }
        }
        float v[LEN];
#pragma unroll
        for (int i = 0; i < LEN; ++i) v[i] = 0.f;
#pragma unroll
        for (int sj = 0; sj < SPL; ++sj) {
            float x[CV];
#pragma unroll
            for (int c = 0; c < NT / 2; ++c) {
                x[2 * c] = acc[sj][c].x;
                x[2 * c + 1] = acc[sj][c].y;
            }
            if constexpr (MOM) {
                constexpr int M = MAP ? NT + 1 : 0;
                if constexpr (MAP) x[NT] = s1[sj];
                else x[5] = sd[sj];
                const float sx = dx[sj] * s1[sj];
                x[M] = sx;
                x[M + 1] = sy[sj];
                x[M + 2] = dx[sj] * sx;
                x[M + 3] = dx[sj] * sy[sj];
                x[M + 4] = syy[sj];
            }
            // slots of the second half go to the neighbouring column, whose second half arrives here
#pragma unroll
            for (int i = 0; i < CV; ++i) {
                const int at = (sj % (SPL / 2)) * CV + i;
                if (sj < SPL / 2) v[at] += x[i];
                else v[at] += __shfl_xor_sync(0xffffffffu, x[i], 1);
            }
        }
#pragma unroll
        for (int sft = 2, len = LEN; sft <= 4; sft <<= 1, len >>= 1) {
            const bool up = col & sft;
#pragma unroll
            for (int i = 0; i < len / 2; ++i) {
                const float send = up ? v[i] : v[i + len / 2];
                const float keep = up ? v[i + len / 2] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, sft);
            }
        }
        const int first = (col & 2 ? LEN / 2 : 0) + (col & 4 ? LEN / 4 : 0);
#pragma unroll
        for (int i = 0; i < LEN / 4; ++i) {
            const int q = first + i, sj = q / CV, t = q % CV;
            if (q < HALF)
                s_t[(jg * SPL + (odd ? SPL / 2 : 0) + sj) * WL::NSV + (t < NT ? T0 + t : WL::NWT + t - NT)] = v[i];
        }
    };
    // Then lanes (slot j, part) send slot j's sums to the splat's accumulators.
    auto contract = [&](const int cnt) {
        __syncwarp();
        contract_chunk(IntC<0>(), IntC<WL::T1>(), IntC<1>());
        if constexpr (WL::T2 > WL::T1) contract_chunk(IntC<WL::T1>(), IntC<WL::T2>(), IntC<0>());
        if constexpr (WL::T3 > WL::T2) contract_chunk(IntC<WL::T2>(), IntC<WL::T3>(), IntC<0>());
        if constexpr (WL::NWT > WL::T3) contract_chunk(IntC<WL::T3>(), IntC<WL::NWT>(), IntC<0>());
        __syncwarp();
        const int j = lane % STAGE, part = lane / STAGE;
        if (j < cnt) {
            const int64_t item = s_item[j];
            // slot j's sums: the terms (depth, r, g, b, F) then the moments about the splat centre
            const float *tj = s_t + j * WL::NSV, *mj = tj + WL::NWT + (MAP ? 1 : 0);
            if (part == 0) {
                const SplatGeo sg = s_geo[j];
                const float du = (-1.f / kLog2e) * fmaf(2.f * sg.qa, mj[0], sg.qb * mj[1]);
                const float dv = (-1.f / kLog2e) * fmaf(2.f * sg.qc, mj[1], sg.qb * mj[0]);
                const float4 val = MAP ? make_float4(du, dv, tj[WL::NWT] / sg.o, tj[0]) : make_float4(du, dv, 0.f, mj[5]);
                if (val.x != 0.f || val.y != 0.f || val.z != 0.f || val.w != 0.f) atomicAdd(A.acc_uvod + item, val);
            } else if (part == 1) {
                const float4 val = make_float4(-0.5f * mj[2], -mj[3], -0.5f * mj[4], 0.f);
                if (val.x != 0.f || val.y != 0.f || val.z != 0.f) atomicAdd(A.acc_conic + item, val);
            }
            if constexpr (MAP) {
                const int64_t g = item - voff;
                if (part == (WL::LPS > 2 ? 2 : 0)) {
                    const float4 val = make_float4(tj[1], tj[2], tj[3], 0.f);
                    if (val.x != 0.f || val.y != 0.f || val.z != 0.f) atomicAdd(A.acc_rgb + g, val);
                }
                // features [part D / LPS, (part + 1) D / LPS): the summed feature terms, or W^T times the
                // summed logit terms
                constexpr int DP = D / WL::LPS;
                float *fo = A.d_feat + g * D + part * DP;
#pragma unroll
                for (int c4 = 0; c4 < DP / 4; ++c4) {
                    const int c = part * DP + 4 * c4;
                    float4 val;
                    if constexpr (KF > 0) {
                        float2 lo = make_float2(0.f, 0.f), hi = lo;
#pragma unroll
                        for (int k = 0; k < KF; ++k) {
                            const float4 b = *reinterpret_cast<const float4 *>(s_basis + k * BROW + c);
                            const float2 z = make_float2(tj[4 + k], tj[4 + k]);
                            lo = fma2(z, make_float2(b.x, b.y), lo);
                            hi = fma2(z, make_float2(b.z, b.w), hi);
                        }
                        val = make_float4(lo.x, lo.y, hi.x, hi.y);
                    } else {
                        val = make_float4(tj[4 + c], tj[5 + c], tj[6 + c], tj[7 + c]);
                    }
                    if (val.x != 0.f || val.y != 0.f || val.z != 0.f || val.w != 0.f)
                        atomicAdd(reinterpret_cast<float4 *>(fo) + c4, val);
                }
            }
        }
        __syncwarp();
    };

    // Every listed splat was blended by a pixel of the group, so no box culling is needed.
    auto process = [&](const int k, const float *sfeat, const int fstride) {
        const int pos = s_pos[k];
        const SplatGeo s = s_geo[k];
        // the mask listed this splat because a pixel of the group blended it, so some lane
        // contributes: no vote is needed before the work
        PairEval e[NP];
        bool contrib[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            e[p] = eval_pair(s, pxc[p], pyc[p], prm.alpha_min, prm.alpha_max);
            contrib[p] = pos < last[p] && !e[p].skip;
        }
        float2 x[NC2];
        {
            const float4 c = s_rgbd[k];
            x[0] = make_float2(c.x, c.y);
            x[1] = make_float2(c.z, c.w);
            const float4 *sf = reinterpret_cast<const float4 *>(sfeat + k * fstride);
#pragma unroll
            for (int q = 0; q < F4; ++q) {
                const float4 f = sf[q];
                x[2 + 2 * q] = make_float2(f.x, f.y);
                x[3 + 2 * q] = make_float2(f.z, f.w);
            }
        }
        // Branch-free over the lanes: a pixel that did not blend the splat runs the same
        // instructions with alpha 0 and keeps its state, and every value it records is 0.
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float a = contrib[p] ? e[p].alpha : 0.f;
            const float Tb = __fdividef(T[p], 1.f - a);
            // g.x as four interleaved partial sums, two packed (a short dependent chain)
            float2 ga = make_float2(gsil[p], 0.f), gb = make_float2(0.f, 0.f);
#pragma unroll
            for (int c = 0; c < NC2; c += 2) {
                ga = fma2(gch[p][c], x[c], ga);
                gb = fma2(gch[p][c + 1], x[c + 1], gb);
            }
            const float gx = (ga.x + ga.y) + (gb.x + gb.y);
            const float da = Tb * (gx - gS[p]);
            gS[p] = fmaf(a, gx - gS[p], gS[p]);
            T[p] = contrib[p] ? Tb : T[p];
            const bool free_alpha = contrib[p] && e[p].oG < prm.alpha_max;
            const float w = a * Tb;
            s_wp[k * WL::WROW + p * 32 + lane] =
                make_float2(MAP ? w : w * gch[p][1].y, free_alpha ? e[p].oG * da : 0.f);
        }
    };

    // Stages and walks list entries [0, cnt) (instance indices, back to front; cnt <= 32), STAGE at
    // a time: the batch's items are loaded once (one per lane), each stage's records are copied
    // into shared memory asynchronously, the next stage's while the current one is processed,
    // and in map mode each stage's slots are contracted after it.
    auto run_batch = [&](const int cnt) {
        const int si = lane % STAGE, part = lane / STAGE;
        const uint32_t my_ii = lane < cnt ? s_list[lane] : 0u;
        const uint32_t my_item = lane < cnt ? checked_item(A.vals[my_ii], voff, vt.n, A.status) : (uint32_t)voff;
        const int n_st = (cnt + STAGE - 1) / STAGE;
        auto issue = [&](const int st) {
            const int e = st * STAGE + si, b = st & 1;
            const uint32_t item = __shfl_sync(0xffffffffu, my_item, e & 31);
            if (e < cnt) {
                const int64_t g = (int64_t)item - voff;
#pragma unroll
                for (int c = part; c < NCOPY; c += PARTS) {
                    if (c == 0) cp_async16(&r_a[b][si], A.uvdo + item);
                    else if (c == 1) cp_async16(&r_c[b][si], A.conic + item);
                    else if (c == 2) cp_async8(&r_lo[b][si], A.uv_lo + item);
                    else if (RGB32 && c < 6) cp_async4(&r_rgb[b][si][c - 3], rgb + 3 * g + (c - 3));
                    else {
                        const int q = c - (RGB32 ? 6 : 3);
                        cp_async16(&r_f[b][si * FBP + 16 * q], reinterpret_cast<const unsigned char *>(feat + g * D) + 16 * q);
                    }
                }
            }
            cp_async_commit();
        };
        issue(0);
        for (int st = 0; st < n_st; ++st) {
            const int b = st & 1, c_cnt = min(STAGE, cnt - st * STAGE);
            if (st + 1 < n_st) {
                issue(st + 1);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncwarp();
            // the stage's working records from the raw ones
            const int e = st * STAGE + si;
            const uint32_t ii = __shfl_sync(0xffffffffu, my_ii, e & 31);
            const uint32_t item = __shfl_sync(0xffffffffu, my_item, e & 31);
            if (si < c_cnt) {
                const int64_t g = (int64_t)item - voff;
                if (part == 0) {
                    const float4 a = r_a[b][si];
                    const float2 l = r_lo[b][si];
                    s_geo[si] = make_geo(a, l, r_c[b][si]);
                    s_ctr[si] = make_float2(__fadd_rn(__fsub_rn(a.x, bcx), l.x), __fadd_rn(__fsub_rn(a.y, bcy), l.y));
                    s_rgbd[si] = RGB32 ? make_float4(r_rgb[b][si][0], r_rgb[b][si][1], r_rgb[b][si][2], a.z)
                                       : load_rgbd(rgb, g, a.z);
                    s_item[si] = item;
                    s_pos[si] = (int)(ii - start);
                }
                const FT *fr = reinterpret_cast<const FT *>(&r_f[b][si * FBP]);
                if constexpr (KF > 0) {
                    // z = W f for this part's K / PARTS logits
#pragma unroll
                    for (int kk = 0; kk < KF / PARTS; ++kk) {
                        const int k = part * (KF / PARTS) + kk;
                        float2 za = make_float2(0.f, 0.f), zb = za;
#pragma unroll
                        for (int q = 0; q < D / 4; ++q) {
                            const float4 f4 = load_feat4(fr, 4 * q);
                            const float4 w4 = reinterpret_cast<const float4 *>(s_basis + k * BROW)[q];
                            za = fma2(make_float2(w4.x, w4.y), make_float2(f4.x, f4.y), za);
                            zb = fma2(make_float2(w4.z, w4.w), make_float2(f4.z, f4.w), zb);
                        }
                        s_feat[si * F + k] = (za.x + za.y) + (zb.x + zb.y);
                    }
                } else if (!RGB32 || sizeof(FT) != 4) {
                    // half storage: the features widened to f32
                    for (int q = part; q < D / 4; q += PARTS)
                        reinterpret_cast<float4 *>(s_feat + si * F)[q] = load_feat4(fr, 4 * q);
                }
            }
            __syncwarp();
            // f32 features are read where they landed; the others from the widened copy
            constexpr bool IN_PLACE = KF == 0 && sizeof(FT) == 4;
            const float *sfeat = IN_PLACE ? reinterpret_cast<const float *>(r_f[b]) : s_feat;
            // two splats at a time overlap their loads and exponentials, where the registers allow
            constexpr int kTogether = KF > 0 ? 2 : 1;
#pragma unroll kTogether
            for (int k = 0; k < c_cnt; ++k) process(k, sfeat, IN_PLACE ? FBP / 4 : F);
            contract(c_cnt);
            __syncwarp();
        }
    };

    // the group's blended instances, back to front: the mask words are read 32 at a time (lane
    // l holds word wc - l), each word appends its set bits (highest first) to the list, and every
    // 32 entries are staged and processed
    const int64_t lo_i = start, hi_i = (int64_t)start + wmax;
    const int64_t w_lo = lo_i >> 5;
    int n = 0;  // entries in the list (warp-uniform, < 32 between words)
    for (int64_t wc = (hi_i - 1) >> 5; wc >= w_lo; wc -= 32) {
        const int64_t wl = wc - lane;
        uint32_t mw = 0u;
        if (wl >= w_lo) {
#pragma unroll
            for (int j = 0; j < NP; ++j) mw |= A.bmask[(int64_t)SH::group(grp, j) * A.bm_stride + wl];
            const int64_t base = wl << 5;
            if (base < lo_i) mw &= ~0u << (int)(lo_i - base);
            if (hi_i - base < 32) mw &= (1u << (int)(hi_i - base)) - 1u;
        }
        const int nw = wc - w_lo + 1 < 32 ? (int)(wc - w_lo + 1) : 32;
        for (int t = 0; t < nw; ++t) {
            const uint32_t m = __shfl_sync(0xffffffffu, mw, t);
            if (m == 0u) continue;
            const int64_t base = (wc - t) << 5;
            const int b = 31 - lane;
            const int above = lane == 0 ? 0 : __popc(m >> (32 - lane));  // set bits above bit b
            if ((m >> b) & 1u) s_list[n + above] = (uint32_t)(base + b);
            n += __popc(m);
            __syncwarp();
            if (n >= 32) {
                run_batch(32);
                if (lane < n - 32) s_list[lane] = s_list[32 + lane];
                __syncwarp();
                n -= 32;
            }
        }
    }
    if (n > 0) run_batch(n);
}

template <int D, int NP, bool MAP, int KF, typename RT, typename FT>
gs_status launch_bwd_warp(const ViewTable &vt, const Params &prm, const BwdArgs &A, cudaStream_t st) {
    const int n_tiles = vt.tile_off[vt.n_views];
    return launch_pdl(raster_bwd_warp_kernel<D, NP, MAP, KF, RT, FT>, n_tiles * Shape<NP>::WARPS, 32, 0, st, vt, prm,
                      A);
}

// The warp-block form: D 16 or 32, 1 or 2 pixels per thread, blend mask present; factored
// feature gradients (A.feat_basis) with at most kFactorK logits.
template <bool MAP, typename RT, typename FT>
gs_status dispatch_bwd_warp_typed(int D, int np, const ViewTable &vt, const Params &prm, const BwdArgs &A,
                                  cudaStream_t st) {
    if (!A.bmask) return GS_ERR_UNSUPPORTED;
    const bool fact = A.feat_basis != nullptr;
    if (fact && (A.feat_rank < 1 || A.feat_rank > kFactorK || !A.feat_coef)) return GS_ERR_UNSUPPORTED;
#define GS_BWD_WARP(DD, NN)                                                                              \
    if (D == DD && np == NN)                                                                             \
        return fact ? launch_bwd_warp<DD, NN, MAP, kFactorK, RT, FT>(vt, prm, A, st)                     \
                    : launch_bwd_warp<DD, NN, MAP, 0, RT, FT>(vt, prm, A, st);
    GS_BWD_WARP(16, 1) GS_BWD_WARP(16, 2) GS_BWD_WARP(32, 1) GS_BWD_WARP(32, 2)
#undef GS_BWD_WARP
    return GS_ERR_UNSUPPORTED;
}

}  // namespace gs
