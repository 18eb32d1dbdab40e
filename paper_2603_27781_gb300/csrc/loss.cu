// Losses and reductions around the blend:
//   - decoder + L1 colour/depth + semantic cross-entropy with image gradients
//     (Eq. 8, 15-17) and the tracking mask M_obs (Eq. 21), whose depth-error
//     median is found by a 4-pass 8-bit radix select over f32 bit patterns;
//   - depth-adaptive scale regularisation (Eq. 12);
//   - the reduction of the pose-twist contributions (supplementary B.1);
//   - the Adam + SE(3) exponential pose step (Sec. 3.4, supplementary C.1).
//
// Reductions are two-level and deterministic: a bounded grid of blocks writes
// per-block partials (f32 sums inside a thread, f64 across threads and
// blocks), and a finishing step sums the partials in a fixed order.  GB300's
// f64 rate is a small fraction of its f32 rate, so f64 is kept to the
// cross-thread sums.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "common.cuh"

namespace gs {
namespace {

constexpr int kMaxK = 32;
constexpr int kMedianThreads = 512, kMedianPx = 4;  // of a block of the median's passes; pixels per thread

// Lower median (element floor((n-1)/2) in sorted order) of view v, as the f32
// bit pattern selected digit by digit from the per-pass histograms
// hist[p][v][256] (p < passes), by one warp: lane l holds digits [8 l, 8 l + 8) of every pass, loaded
// together (the passes' counts do not depend on one another once written), and each pass takes
// one scan over the lanes.  Valid in every lane.
__device__ __forceinline__ uint32_t warp_select(const uint32_t *hist, int n_views, int v, int passes) {
    const int lane = threadIdx.x & 31;
    uint32_t h[4][8];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const uint4 *src = reinterpret_cast<const uint4 *>(hist + ((size_t)p * n_views + v) * 256 + 8 * lane);
        const uint4 z = make_uint4(0u, 0u, 0u, 0u), a = p < passes ? src[0] : z, b = p < passes ? src[1] : z;
        h[p][0] = a.x; h[p][1] = a.y; h[p][2] = a.z; h[p][3] = a.w;
        h[p][4] = b.x; h[p][5] = b.y; h[p][6] = b.z; h[p][7] = b.w;
    }
    uint32_t k = 0u, prefix = 0u;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        uint32_t sum = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i) sum += h[p][i];
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (p == 0) {
            const uint32_t n = __shfl_sync(0xffffffffu, inc, 31);
            if (n == 0u) return 0u;  // no pixel with depth
            k = (n - 1u) / 2u;
        }
        if (p >= passes) break;
        // the lane whose digits hold element k, the digit, and the elements below it
        uint32_t below = inc - sum, digit = 0u, rest = 0u;
        const uint32_t owner = __ballot_sync(0xffffffffu, k >= below && k < inc);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (k >= below && k < below + h[p][i]) {
                digit = 8u * lane + i;
                rest = below;
            }
            below += h[p][i];
        }
        const int src = __ffs(owner) - 1;
        digit = __shfl_sync(0xffffffffu, digit, src);
        k -= __shfl_sync(0xffffffffu, rest, src);
        prefix |= digit << (24 - 8 * p);
    }
    return prefix;
}

// The same for a block (every thread of it takes part).
__device__ __forceinline__ uint32_t block_select(const uint32_t *hist, int n_views, int v, int passes) {
    __shared__ uint32_t s_prefix;
    if (threadIdx.x < 32) {
        const uint32_t x = warp_select(hist, n_views, v, passes);
        if (threadIdx.x == 0) s_prefix = x;
    }
    __syncthreads();
    return s_prefix;
}

__device__ __forceinline__ float depth_error(float d, float dgt) { return fabsf(__fsub_rn(d, dgt)); }

// One pass of the median's selection: the histogram of digit `pass` over the pixels whose higher digits
// are the median's.  What bounds a pass is its chain of latencies: the images' pixels, the choice among the
// pass before's counts (block_select), the shared and the global additions.  So a thread takes
// kMedianPx pixels at once, whose loads and differences do not wait for the pass before (the images were
// complete before that one passed its own wait), and few blocks add to the global histogram: 1024 blocks
// with a pixel a turn spent 16 us a pass at 640x480, most of it on finding the lanes of equal digits
// (the lanes of no digit among them), which the additions of a constant do better by themselves.
__global__ void __launch_bounds__(kMedianThreads) median_hist_kernel(ViewTable vt, int pass,
                                                                     const float *__restrict__ depth,
                                                                     const float *__restrict__ tdepth,
                                                                     uint32_t *hist) {
    __shared__ uint32_t s_hist[256];
    const int v = blockIdx.y, tid = threadIdx.x;
    const int64_t Pv = (int64_t)vt.W[v] * vt.H[v], base = (int64_t)blockIdx.x * (kMedianThreads * kMedianPx) + tid;
    if (pass == 0) pdl_wait();  // the first pass reads what the kernels before it wrote
    uint32_t bits[kMedianPx];
    bool valid[kMedianPx];
#pragma unroll
    for (int u = 0; u < kMedianPx; ++u) {
        const int64_t i = base + u * kMedianThreads;
        const bool in = i < Pv;
        const float dgt = in ? tdepth[vt.pix_off[v] + i] : 0.f, d = in ? depth[vt.pix_off[v] + i] : 0.f;
        valid[u] = dgt > 0.f;
        bits[u] = __float_as_uint(depth_error(d, dgt));
    }
    if (tid < 256) s_hist[tid] = 0u;
    if (pass > 0) pdl_wait();  // the previous pass's histogram
    pdl_trigger();             // the next kernel may be scheduled now
    const uint32_t prefix = pass > 0 ? block_select(hist, vt.n_views, v, pass) : 0u;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kMedianPx; ++u)
        if (valid[u] && (pass == 0 || ((bits[u] ^ prefix) >> (32 - 8 * pass)) == 0u))
            atomicAdd(&s_hist[(bits[u] >> (24 - 8 * pass)) & 255u], 1u);
    __syncthreads();
    const uint32_t c = tid < 256 ? s_hist[tid] : 0u;
    if (c) atomicAdd(&hist[((size_t)pass * vt.n_views + v) * 256 + tid], c);
}

// The four passes of the median's histograms (hist zeroed here), each launched while its predecessor
// drains.
gs_status launch_median(const ViewTable &vt, const float *depth, const float *tdepth, uint32_t *hist,
                        cudaStream_t st) {
    gs_status s = cuda_status(cudaMemsetAsync(hist, 0, sizeof(uint32_t) * 4 * 256 * vt.n_views, st));
    int64_t maxPv = 1;
    for (int v = 0; v < vt.n_views; ++v) maxPv = std::max<int64_t>(maxPv, (int64_t)vt.W[v] * vt.H[v]);
    const dim3 grid(ceil_div(maxPv, kMedianThreads * kMedianPx), vt.n_views);
    for (int pass = 0; pass < 4 && !s; ++pass)
        s = launch_pdl(median_hist_kernel, grid, kMedianThreads, 0, st, vt, pass, depth, tdepth, hist);
    return s;
}

struct LossP {
    float color, depth, sem, tau_obs;  // color: weight of the L1 part
    int mask_mode, K;
    float ssim_coef;                   // lambda_c lambda of Eq. 15 (0: no SSIM term)
    float *ssim_maps;
};

// Sums of N per-thread f32 values over the block in f64 (thread i's value x[n], rounding error lo[n]
// subtracted where LO), in a fixed order; out[n] valid in every thread.  The values go through
// shared memory and one warp adds each sum: NT / 32 additions and five shuffle steps for 32 threads
// instead of five steps for all of them, since the GPU adds two f64 a cycle and SM (the loss kernel's
// three sums with a division in every thread kept its blocks for 7 of 45 us).
template <int NT, bool LO, int N>
__device__ __forceinline__ void block_sums_f64(const float (&x)[N], const float *lo, double (&out)[N]) {
    __shared__ float s_x[LO ? 2 : 1][N][NT];
    __shared__ double s_sum[N];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    __syncthreads();
#pragma unroll
    for (int n = 0; n < N; ++n) {
        s_x[0][n][tid] = x[n];
        if constexpr (LO) s_x[LO][n][tid] = lo[n];
    }
    __syncthreads();
    for (int n = w; n < N; n += NT / 32) {
        double t = 0.0;
#pragma unroll
        for (int i = 0; i < NT / 32; ++i) {
            t += (double)s_x[0][n][i * 32 + lane];
            if constexpr (LO) t -= (double)s_x[LO][n][i * 32 + lane];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) s_sum[n] = t;
    }
    __syncthreads();
#pragma unroll
    for (int n = 0; n < N; ++n) out[n] = s_sum[n];
}

// Sum over the block (any multiple of 32 threads, up to 1024) in f64; valid in thread 0.
__device__ __forceinline__ double block_sum_f64(double x, double *s_red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) s_red[w] = x;
    __syncthreads();
    double t = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += s_red[i];
    return t;
}

// Blocks [off[v], off[v + 1]) of the loss kernel's grid work on view v.
struct LossGrid {
    int off[kMaxViews + 1];
};

// Per-pixel losses and image gradients; per-block partials of the decoder
// gradient (f32 [nblk][K*D + K]) and of the three loss sums (f64 [nblk][3]).
//
// KC is a compile-time bound on the class count (K <= KC, a multiple of 8).  What bounds the kernel
// is the shared-memory pipe (a 16-byte read costs a warp four cycles even as a broadcast) and its
// FMAs, so that each word read serves as many of them as registers allow:
//  - a thread takes NPX pixels at a time, so each row of W read for z = W f and W^T dz serves
//    NPX of them, in packed multiply-adds along d;
//  - the decoder gradient dW[k][d] = sum_px dz_k f_d, db[k] = sum_px dz_k is a contraction over pixels:
//    each warp stages dz and f of 32 pixels in shared memory, and every lane keeps an 8 x 4 tile
//    of dW in registers for the whole grid-stride loop (TILES lanes cover K x D, GROUPS such
//    sets of lanes each take their share of the 32 pixels): 12 words read for 32 multiply-adds.
//    The sums reach the block's shared ones once, at the end.
// Loss step (this kernel and the finish), before and now: 0.054 -> 0.047 ms (D = 16, K = 8, 1200x680),
// 0.433 -> 0.25 (D = 32, K = 8, eight keyframes of two sizes), 0.167 -> 0.096 (D = 16, K = 20, 1200x680, with
// the features' gradient).  Two pixels a thread where 128 registers hold them with at most 8 bytes
// spilled (D = 16, K = 8); K = 20: 0.101 with two, 0.096 with one.
template <int D, int KC>
struct LossShape {
    static constexpr int NT = 128;                        // keeps the static shared memory < 48 KB
    static constexpr int NPX = KC + D <= 32 ? 2 : 1;      // pixels a thread has in flight
    // resident blocks the register allocation must allow (128 registers, 168 for the widest)
    static constexpr int BLOCKS = KC + D > 40 || (NPX == 2 && KC >= 16 && KC + D >= 28) ? 3 : 4;
    static constexpr int WARPS = NT / 32;
    static constexpr int DD = D > 0 ? D : 1;
    static constexpr int D4 = D / 4 > 0 ? D / 4 : 1;
    static constexpr int FROW = D > 0 ? D + 4 : 4;        // staged rows, padded: eight lanes' 16-byte
    static constexpr int ZROW = KC + 4;                   // words of neighbouring rows fall in different banks
    static constexpr int TILES = KC / 8 * D4;
    static constexpr int GROUPS = TILES <= 4 ? 8 : TILES <= 8 ? 4 : TILES <= 16 ? 2 : 1;
    static_assert(KC % 8 == 0 && D % 4 == 0 && TILES * GROUPS <= 32, "8 x 4 tiles of dW");
};

template <int D, int KC>
__global__ void __launch_bounds__(LossShape<D, KC>::NT, LossShape<D, KC>::BLOCKS) loss_kernel(
    ViewTable vt, LossGrid lg, LossP lp, const float *__restrict__ rgb, const float *__restrict__ depth,
    const float *__restrict__ sil, const float *__restrict__ feat, const float *__restrict__ trgb,
    const float *__restrict__ tdepth, const uint8_t *__restrict__ label, const float *__restrict__ Wd,
    const float *__restrict__ bd, int64_t P, const uint32_t *__restrict__ med_hist, float *__restrict__ g_rgb,
    float *__restrict__ g_depth, float *__restrict__ g_sil, float *__restrict__ g_feat, float *__restrict__ g_coef,
    float *__restrict__ part_f, double *__restrict__ part_d, float *__restrict__ mask_out,
    float *__restrict__ median_out) {
    pdl_wait();  // the previous kernel's results (no trigger: see pdl_trigger)
    using SH = LossShape<D, KC>;
    constexpr int NT = SH::NT, NPX = SH::NPX, DD = SH::DD, TILES = SH::TILES, GROUPS = SH::GROUPS;
    __shared__ __align__(16) float s_W[KC * DD];
    __shared__ float s_b[KC];
    __shared__ float s_dW[KC * DD + KC];
    __shared__ __align__(16) float s_dz[SH::WARPS][32][SH::ZROW];
    __shared__ __align__(16) float s_f[SH::WARPS][32][SH::FROW];
    __shared__ float s_med;
    const int blk = blockIdx.x;
    int v = 0;
    while (v + 1 < vt.n_views && blk >= lg.off[v + 1]) ++v;
    const int bx = blk - lg.off[v], nbx = lg.off[v + 1] - lg.off[v];
    const int64_t Pv = (int64_t)vt.W[v] * vt.H[v];
    const int K = lp.K, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nval = K * D + K;
    for (int i = tid; i < KC * D; i += NT) s_W[i] = i < K * D ? Wd[i] : 0.f;
    for (int i = tid; i < K; i += NT) s_b[i] = bd[i];
    for (int i = tid; i < nval; i += NT) s_dW[i] = 0.f;
    if (wid == 0) {
        const float med = lp.mask_mode == 1 ? __uint_as_float(warp_select(med_hist, vt.n_views, v, 4)) : 0.f;
        if (lane == 0) {
            s_med = med;
            if (median_out && bx == 0) median_out[v] = med;
        }
    }
    __syncthreads();
    // the view's planes: uniform base addresses, so that a pixel's 32-bit index addresses every plane
    const int64_t o = vt.pix_off[v];
    rgb += o; depth += o; sil += o; trgb += o; tdepth += o; label += o; g_rgb += o; g_depth += o; g_sil += o;
    if (D > 0) feat += o;
    if (g_feat) g_feat += o;
    if (g_coef) g_coef += o;
    if (mask_out) mask_out += o;
    const uint32_t n_px = (uint32_t)Pv;
    const float invP = 1.f / (float)Pv;
    float lc = 0.f, ld = 0.f, ls = 0.f;  // per-thread partial sums (a thread sees few pixels)
    // this lane's tile of the decoder gradient: classes [k0, k0 + 8), features [d0, d0 + 4), pixel group grp
    const int tile = lane % TILES, grp = lane / TILES;
    const int k0 = tile / SH::D4 * 8, d0 = tile % SH::D4 * 4;
    float2 accW[8][2], accb[4];
#pragma unroll
    for (int k = 0; k < 8; ++k) accW[k][0] = accW[k][1] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 4; ++k) accb[k] = make_float2(0.f, 0.f);

    for (uint32_t base = (uint32_t)bx * (NT * NPX); base < n_px; base += (uint32_t)nbx * (NT * NPX)) {
        float f[NPX][DD], dz[NPX][KC];
        int lab[NPX];
        float m[NPX];
        // loads first: colours, depths, labels and features of the thread's pixels
#pragma unroll
        for (int p = 0; p < NPX; ++p) {
            const uint32_t i = base + p * NT + tid;
            lab[p] = 255;
            m[p] = 1.f;
#pragma unroll
            for (int d = 0; d < DD; ++d) f[p][d] = 0.f;
            if (i < n_px) {
#pragma unroll
                for (int d = 0; d < D; ++d) f[p][d] = (feat + d * P)[i];
                lab[p] = label[i];
                const float dgt = tdepth[i], dd = depth[i];
                if (lp.mask_mode == 1)
                    m[p] = (sil[i] > lp.tau_obs && dgt > 0.f && depth_error(dd, dgt) < 10.f * s_med) ? 1.f : 0.f;
                if (mask_out) mask_out[i] = m[p];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float r = (rgb + c * P)[i] - (trgb + c * P)[i];
                    lc += m[p] * fabsf(r);
                    (g_rgb + c * P)[i] = m[p] * lp.color * (r > 0.f ? 1.f : (r < 0.f ? -1.f : 0.f)) * invP;
                }
                float gd = 0.f;
                if (dgt > 0.f) {
                    const float r = dd - dgt;
                    ld += m[p] * fabsf(r);
                    gd = m[p] * lp.depth * (r > 0.f ? 1.f : (r < 0.f ? -1.f : 0.f)) * invP;
                }
                g_depth[i] = gd;
                g_sil[i] = 0.f;
            }
        }
        if (K == 0) {
            if (!g_coef) {
#pragma unroll
                for (int p = 0; p < NPX; ++p) {
                    const uint32_t i = base + p * NT + tid;
#pragma unroll
                    for (int d = 0; d < D; ++d)
                        if (i < n_px) (g_feat + d * P)[i] = 0.f;
                }
            }
            continue;
        }
        // z = W f + b, each row summed in four partial sums (two packed)
#pragma unroll
        for (int k = 0; k < KC; ++k) {
            if (k < K) {
                float2 a[NPX][2];
#pragma unroll
                for (int p = 0; p < NPX; ++p) a[p][0] = a[p][1] = make_float2(0.f, 0.f);
                if constexpr (D > 0) {
                    const float4 *wr = reinterpret_cast<const float4 *>(s_W + k * D);
#pragma unroll
                    for (int q = 0; q < D / 4; ++q) {
                        const float4 w4 = wr[q];
#pragma unroll
                        for (int p = 0; p < NPX; ++p) {
                            a[p][0] = fma2(make_float2(w4.x, w4.y), make_float2(f[p][4 * q], f[p][4 * q + 1]), a[p][0]);
                            a[p][1] = fma2(make_float2(w4.z, w4.w), make_float2(f[p][4 * q + 2], f[p][4 * q + 3]), a[p][1]);
                        }
                    }
                }
#pragma unroll
                for (int p = 0; p < NPX; ++p) dz[p][k] = s_b[k] + ((a[p][0].x + a[p][0].y) + (a[p][1].x + a[p][1].y));
            } else {
#pragma unroll
                for (int p = 0; p < NPX; ++p) dz[p][k] = 0.f;
            }
        }
        // softmax from one exponential per class: p_k = e_k / sum_j e_j, e_k = exp(z_k - zmax)
#pragma unroll
        for (int p = 0; p < NPX; ++p) {
            const bool on = lab[p] != 255 && lab[p] < K;
            float zmax = -INFINITY, se = 0.f, zl = 0.f;
#pragma unroll
            for (int k = 0; k < KC; ++k)
                if (k < K) {
                    zmax = fmaxf(zmax, dz[p][k]);
                    if (k == lab[p]) zl = dz[p][k];
                }
#pragma unroll
            for (int k = 0; k < KC; ++k)
                if (k < K) {
                    dz[p][k] = expf(dz[p][k] - zmax);
                    se += dz[p][k];
                }
            if (on) ls += m[p] * (zmax + logf(se) - zl);
            const float scale = m[p] * lp.sem * invP;
            const float inv_se = 1.f / se;
#pragma unroll
            for (int k = 0; k < KC; ++k)
                if (k < K) dz[p][k] = on ? scale * (dz[p][k] * inv_se - (k == lab[p] ? 1.f : 0.f)) : 0.f;
        }
        // the decoder gradient: the warp's dz and f of 32 pixels staged, each lane's tile summed over its
        // group's share of them
#pragma unroll
        for (int p = 0; p < NPX; ++p) {
            float4 *zr = reinterpret_cast<float4 *>(&s_dz[wid][lane][0]);
#pragma unroll
            for (int q = 0; q < KC / 4; ++q)
                zr[q] = make_float4(dz[p][4 * q], dz[p][4 * q + 1], dz[p][4 * q + 2], dz[p][4 * q + 3]);
            if constexpr (D > 0) {
                float4 *fr = reinterpret_cast<float4 *>(&s_f[wid][lane][0]);
#pragma unroll
                for (int q = 0; q < D / 4; ++q)
                    fr[q] = make_float4(f[p][4 * q], f[p][4 * q + 1], f[p][4 * q + 2], f[p][4 * q + 3]);
            }
            __syncwarp();
            if (grp < GROUPS) {
#pragma unroll 2
                for (int it = 0; it < 32 / GROUPS; ++it) {
                    const int px = grp * (32 / GROUPS) + it;
                    const float4 za = *reinterpret_cast<const float4 *>(&s_dz[wid][px][k0]);
                    const float4 zb = *reinterpret_cast<const float4 *>(&s_dz[wid][px][k0 + 4]);
                    if constexpr (D > 0) {
                        const float4 fv = *reinterpret_cast<const float4 *>(&s_f[wid][px][d0]);
                        const float z8[8] = {za.x, za.y, za.z, za.w, zb.x, zb.y, zb.z, zb.w};
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            accW[k][0] = fma2(make_float2(z8[k], z8[k]), make_float2(fv.x, fv.y), accW[k][0]);
                            accW[k][1] = fma2(make_float2(z8[k], z8[k]), make_float2(fv.z, fv.w), accW[k][1]);
                        }
                    }
                    accb[0] = __fadd2_rn(accb[0], make_float2(za.x, za.y));
                    accb[1] = __fadd2_rn(accb[1], make_float2(za.z, za.w));
                    accb[2] = __fadd2_rn(accb[2], make_float2(zb.x, zb.y));
                    accb[3] = __fadd2_rn(accb[3], make_float2(zb.z, zb.w));
                }
            }
            __syncwarp();
        }
        // the gradient of the logits (the factored form; W^T dz is left to the backward) or of the features
        if (g_coef) {
#pragma unroll
            for (int p = 0; p < NPX; ++p) {
                const uint32_t i = base + p * NT + tid;
#pragma unroll
                for (int k = 0; k < KC; ++k)
                    if (k < K && i < n_px) (g_coef + k * P)[i] = dz[p][k];
            }
        } else if constexpr (D > 0) {
            float2 gf[NPX][D / 2];
#pragma unroll
            for (int p = 0; p < NPX; ++p)
#pragma unroll
                for (int d = 0; d < D / 2; ++d) gf[p][d] = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < KC; ++k) {
                if (k < K) {
                    const float4 *wr = reinterpret_cast<const float4 *>(s_W + k * D);
#pragma unroll
                    for (int q = 0; q < D / 4; ++q) {
                        const float4 w4 = wr[q];
#pragma unroll
                        for (int p = 0; p < NPX; ++p) {
                            const float2 z = make_float2(dz[p][k], dz[p][k]);
                            gf[p][2 * q] = fma2(make_float2(w4.x, w4.y), z, gf[p][2 * q]);
                            gf[p][2 * q + 1] = fma2(make_float2(w4.z, w4.w), z, gf[p][2 * q + 1]);
                        }
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < NPX; ++p) {
                const uint32_t i = base + p * NT + tid;
                if (i < n_px) {
    #pragma unroll
                    for (int d = 0; d < D / 2; ++d) {
                        (g_feat + 2 * d * P)[i] = gf[p][d].x;
                        (g_feat + (2 * d + 1) * P)[i] = gf[p][d].y;
                    }
                }
            }
        }
    }
    // the groups' tiles by shuffles, then the warps' in warp order (one warp at a time), so the decoder
    // gradient is the same bits on every run and through every entry point
    if (K > 0) {
#pragma unroll
        for (int g = 1; g < GROUPS; ++g) {
            const int src = (lane + g * TILES) & 31;
#pragma unroll
            for (int k = 0; k < 8; ++k)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float x = __shfl_sync(0xffffffffu, accW[k][h].x, src), y = __shfl_sync(0xffffffffu, accW[k][h].y, src);
                    if (grp == 0) accW[k][h] = __fadd2_rn(accW[k][h], make_float2(x, y));
                }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float x = __shfl_sync(0xffffffffu, accb[k].x, src), y = __shfl_sync(0xffffffffu, accb[k].y, src);
                if (grp == 0) accb[k] = __fadd2_rn(accb[k], make_float2(x, y));
            }
        }
    }
    for (int w = 0; w < SH::WARPS; ++w) {
        if (K > 0 && wid == w && grp == 0) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k0 + k >= K) continue;
                if constexpr (D > 0) {
                    float *o = s_dW + (k0 + k) * D + d0;
                    o[0] += accW[k][0].x;
                    o[1] += accW[k][0].y;
                    o[2] += accW[k][1].x;
                    o[3] += accW[k][1].y;
                }
                if (d0 == 0) s_dW[K * D + k0 + k] += k % 2 ? accb[k / 2].y : accb[k / 2].x;
            }
        }
        __syncthreads();
    }
    // per-block partials, weighted and normalised by the view's pixel count
    const float x[3] = {lc, ld, ls};
    double sums[3];
    block_sums_f64<NT, false>(x, nullptr, sums);
    for (int j = tid; j < nval; j += NT) part_f[(size_t)blk * nval + j] = s_dW[j];
    if (tid < 3) {
        const double w = tid == 0 ? lp.color : tid == 1 ? lp.depth : lp.sem;
        part_d[3 * blk + tid] = (tid == 0 ? sums[0] : tid == 1 ? sums[1] : sums[2]) * w / (double)Pv;
    }
}

// Sums the per-block partials in a fixed order (nblk rows of decoder partials, nrows_d rows
// of loss-term partials: the loss blocks, then any SSIM tiles).  A warp sums each decoder gradient
// column (no barrier: the few hundred rows are one round of loads); the last block sums the three loss
// terms and their total.
constexpr int kFinishThreads = 256;
__global__ void __launch_bounds__(kFinishThreads) loss_finish_kernel(int nblk, int nrows_d, int K, int D, const float *part_f,
                                                                     const double *part_d, float *dW, float *db,
                                                                     double *loss_out) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    const int nval = K * D + K, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (blockIdx.x + 1 < gridDim.x) {
        const int j = blockIdx.x * (kFinishThreads / 32) + w;
        if (j >= nval) return;
        double x = 0;
#pragma unroll 8
        for (int b = lane; b < nblk; b += 32) x += (double)part_f[(size_t)b * nval + j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) {
            if (j < K * D) dW[j] = (float)x;
            else db[j - K * D] = (float)x;
        }
        return;
    }
    __shared__ double s_red[3][kFinishThreads / 32];
    double x[3] = {0, 0, 0};
#pragma unroll 4
    for (int b = threadIdx.x; b < nrows_d; b += kFinishThreads)
#pragma unroll
        for (int c = 0; c < 3; ++c) x[c] += part_d[3 * (size_t)b + c];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x[c] += __shfl_xor_sync(0xffffffffu, x[c], o);
        if (lane == 0) s_red[c][w] = x[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t[3] = {0, 0, 0};
        for (int c = 0; c < 3; ++c)
            for (int i = 0; i < kFinishThreads / 32; ++i) t[c] += s_red[c][i];
        loss_out[0] = t[0] + t[1] + t[2];
        for (int c = 0; c < 3; ++c) loss_out[1 + c] = t[c];
    }
}

// --------------------------------------------------------------------- DSR
// Compensated (Kahan) f32 accumulation inside a thread.
struct Kahan {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float y = x - c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

constexpr int kRedBlocks = 512;

// Calls f(i, x[i]) for the elements of x this thread owns: block b owns a contiguous range
// (a multiple of 4 long), which its threads read as float4 with four loads in flight per
// iteration (scalar loads if x is not 16-byte aligned); a fixed assignment, so per-thread
// sums are reproducible.
template <typename F>
__device__ __forceinline__ void for_my_elements(int64_t m, const float *x, F f) {
    const int64_t per = ((m + gridDim.x - 1) / gridDim.x + 3) / 4 * 4;
    const int64_t b0 = (int64_t)blockIdx.x * per, b1 = min(m, b0 + per);
    if (b0 >= b1) return;
    if (reinterpret_cast<uintptr_t>(x) & 15) {
        for (int64_t e = b0 + threadIdx.x; e < b1; e += blockDim.x) f(e, x[e]);
        return;
    }
    const int64_t n4 = (b1 - b0) / 4;
    const float4 *x4 = reinterpret_cast<const float4 *>(x + b0);
    for (int64_t i = threadIdx.x; i < n4; i += 4 * (int64_t)blockDim.x) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t j = i + u * (int64_t)blockDim.x;
            v[u] = j < n4 ? x4[j] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t j = i + u * (int64_t)blockDim.x;
            if (j < n4) {
                const int64_t e = b0 + 4 * j;
                f(e, v[u].x);
                f(e + 1, v[u].y);
                f(e + 2, v[u].z);
                f(e + 3, v[u].w);
            }
        }
    }
    for (int64_t e = b0 + 4 * n4 + threadIdx.x; e < b1; e += blockDim.x) f(e, x[e]);
}


// True in the block that finishes last (its partial and every other block's are written
// and visible); that block then resets *ctr for the next call.
__device__ bool last_block(uint32_t *ctr) {
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(ctr, 1u) == gridDim.x - 1;
    __syncthreads();
    return s_last;
}

// Sum of a strided f64 partial column written by other blocks of this grid (read past L1).
__device__ double sum_partials_cg(const double *part, int stride, int col, int nb, double *s_red) {
    double x = 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) x += __ldcg(part + (size_t)b * stride + col);
    return block_sum_f64(x, s_red);
}

// Pass 1 of Eq. 12: per-block sums of s and s^2 over the 3N scales; the last block turns
// them into the population mean and deviation, out[1], out[2] (detached constants).
__global__ void __launch_bounds__(256) dsr_stats_kernel(int64_t m, const float *ls, double *part, double *out,
                                                        uint32_t *ctr) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    __shared__ double s_red[8];
    Kahan s1, s2;
    for_my_elements(m, ls, [&](int64_t, float l) {
        const float s = expf(l);
        s1.add(s);
        s2.add(s * s);
    });
    const float x[2] = {s1.s, s2.s}, lo[2] = {s1.c, s2.c};
    double t[2];
    block_sums_f64<256, true>(x, lo, t);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = t[0];
        part[2 * blockIdx.x + 1] = t[1];
    }
    if (!last_block(ctr)) return;
    const double u1 = sum_partials_cg(part, 2, 0, gridDim.x, s_red);
    const double u2 = sum_partials_cg(part, 2, 1, gridDim.x, s_red);
    if (threadIdx.x == 0) {
        const double mu = u1 / (double)m, var = u2 / (double)m - mu * mu;
        out[1] = mu;
        out[2] = sqrt(var > 0 ? var : 0.0);
        *ctr = 0u;
    }
}

// Thresholds mu +- 2 sigma in f32, formed the same way by both passes that compare against them.
__device__ __forceinline__ float2 dsr_bounds(const double *out) {
    return make_float2((float)(out[1] + 2.0 * out[2]), (float)(out[1] - 2.0 * out[2]));
}

// Pass 2: per-block sizes and sums of the two sets; the last block forms their means and
// the regulariser's value, out = (lam_big L_big + lam_small L_small, mu, sigma, n_big,
// n_small, L_big, L_small, 0).
__global__ void __launch_bounds__(256) dsr_mask_kernel(int64_t m, const float *ls, double *out, double *mask_part,
                                                       float lam_big, float lam_small, uint32_t *ctr) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    __shared__ double s_red[8];
    const float2 bd = dsr_bounds(out);
    Kahan sb, ss;
    int nb = 0, ns = 0;
    for_my_elements(m, ls, [&](int64_t, float l) {
        const float s = expf(l);
        if (s > bd.x) { sb.add(s); ++nb; }
        if (s < bd.y) { ss.add(-l); ++ns; }
    });
    // a thread's counts are far below 2^24: exact in f32
    const float x[4] = {sb.s, (float)nb, ss.s, (float)ns}, lo[4] = {sb.c, 0.f, ss.c, 0.f};
    double t[4];
    block_sums_f64<256, true>(x, lo, t);
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; ++k) mask_part[4 * blockIdx.x + k] = t[k];
    if (!last_block(ctr)) return;
    double u[4];
    for (int k = 0; k < 4; ++k) u[k] = sum_partials_cg(mask_part, 4, k, gridDim.x, s_red);
    if (threadIdx.x == 0) {
        const double Lb = u[1] > 0 ? u[0] / u[1] : 0.0, Ls = u[3] > 0 ? u[2] / u[3] : 0.0;
        out[0] = (double)lam_big * Lb + (double)lam_small * Ls;
        out[3] = u[1];
        out[4] = u[3];
        out[5] = Lb;
        out[6] = Ls;
        out[7] = 0.0;
        *ctr = 0u;
    }
}

__global__ void __launch_bounds__(256) dsr_grad_kernel(int64_t m, const float *ls, float lam_big, float lam_small,
                                                       const double *out, float *d_ls) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    const float2 bd = dsr_bounds(out);
    const double nb = out[3], ns = out[4];
    const float gb = nb > 0 ? (float)(lam_big / nb) : 0.f;
    const float gsm = ns > 0 ? (float)(lam_small / ns) : 0.f;
    for_my_elements(m, ls, [&](int64_t i, float l) {
        const float s = expf(l);
        float g = 0.f;
        if (s > bd.x) g += gb * s;
        if (s < bd.y) g -= gsm;
        if (g != 0.f) d_ls[i] += g;
    });
}

// ------------------------------------------------------------ pose reduction
// Block (x, vk) sums a contiguous slice of component vk in compensated f32 and
// adds its f64 total into d_twist[vk] (at most kPoseBlocks adds per value).
constexpr int kPoseBlocks = 128;

__global__ void __launch_bounds__(256) pose_reduce_kernel(int64_t n, const float *pose_part, double *d_twist) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    const int vk = blockIdx.y;  // view * 6 + component
    const float *p = pose_part + (int64_t)vk * n;
    Kahan s;
    for_my_elements(n, p, [&](int64_t, float x) { s.add(x); });
    const float x[1] = {s.s}, lo[1] = {s.c};
    double t[1];
    block_sums_f64<256, true>(x, lo, t);
    if (threadIdx.x == 0 && t[0] != 0) atomicAdd(&d_twist[vk], t[0]);
}

// ------------------------------------------------------------------ pose step
// bc1 < 0 selects the device step counter: adam[12 * n_views] holds the number
// of steps taken so far (as a double); this step is that number + 1 and the
// bias corrections 1 - beta^step are formed here.
// One block, 16 threads per view: the six Adam components, then the SE(3) exponential
// (one thread for theta and its sin/cos, nine for the 3x3 products, sixteen for T <- E T).
constexpr int kPoseLanes = 16;

__global__ void pose_step_kernel(int n_views, const double *grad, double *Tst, double *adam, double bc1, double bc2,
                                 double lr0, double lr1, double lr2, double lr3, double lr4, double lr5, double b1,
                                 double b2, double lb1, double lb2, double eps, float *pose_f32) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    __shared__ double s_bc[2];
    __shared__ double s_dl[kMaxViews][6], s_abc[kMaxViews][3], s_R[kMaxViews][9], s_V[kMaxViews][9];
    __shared__ double s_t[kMaxViews][3];
    const int v = threadIdx.x / kPoseLanes, j = threadIdx.x % kPoseLanes;
    const bool active = v < n_views;
    if (threadIdx.x == 0) {
        double c1 = bc1, c2 = bc2;
        if (bc1 < 0.0) {  // device step count: this step is the stored count + 1
            const double step = adam[12 * n_views] + 1.0;
            // beta^step as exp(step ln beta), ln beta from the host (one exp instead of a pow)
            c1 = 1.0 - exp(step * lb1);
            c2 = 1.0 - exp(step * lb2);
            adam[12 * n_views] = step;
        }
        s_bc[0] = c1;
        s_bc[1] = c2;
    }
    __syncthreads();
    if (active && j < 6) {
        const double lr[6] = {lr0, lr1, lr2, lr3, lr4, lr5};
        double *m = adam + 12 * v, *vv = m + 6;
        const double g = grad[6 * v + j];
        m[j] = b1 * m[j] + (1 - b1) * g;
        vv[j] = b2 * vv[j] + (1 - b2) * g * g;
        const double mh = m[j] / s_bc[0], vh = vv[j] / s_bc[1];
        s_dl[v][j] = -lr[j] * mh / (sqrt(vh) + eps);
    }
    __syncthreads();
    // SE(3) exponential of (rho, phi) = dl
    if (active && j == 0) {
        const double *ph = s_dl[v] + 3;
        const double th = sqrt(ph[0] * ph[0] + ph[1] * ph[1] + ph[2] * ph[2]);
        double a, b, c;
        if (th < 0.05) {
            // a = sin(th)/th, b = (1 - cos th)/th^2, c = (th - sin th)/th^3 by their Taylor series in
            // t = th^2 up to t^4: the next terms are below 1e-20 here, and the series avoids the
            // cancellation of 1 - cos th (the rotation increments of a tracking step are ~1e-3)
            const double t = th * th;
            a = 1.0 + t * (-1.0 / 6 + t * (1.0 / 120 + t * (-1.0 / 5040 + t * (1.0 / 362880))));
            b = 0.5 + t * (-1.0 / 24 + t * (1.0 / 720 + t * (-1.0 / 40320 + t * (1.0 / 3628800))));
            c = 1.0 / 6 + t * (-1.0 / 120 + t * (1.0 / 5040 + t * (-1.0 / 362880 + t * (1.0 / 39916800))));
        } else {
            const double sn = sin(th), cs = cos(th);
            a = sn / th;
            b = (1 - cs) / (th * th);
            c = (th - sn) / (th * th * th);
        }
        s_abc[v][0] = a;
        s_abc[v][1] = b;
        s_abc[v][2] = c;
    }
    __syncthreads();
    if (active && j < 9) {
        const double *ph = s_dl[v] + 3;
        const double K[9] = {0, -ph[2], ph[1], ph[2], 0, -ph[0], -ph[1], ph[0], 0};
        const int i = j / 3, jj = j % 3;
        const double K2 = K[3 * i] * K[jj] + K[3 * i + 1] * K[3 + jj] + K[3 * i + 2] * K[6 + jj];
        const double id = (j % 4 == 0) ? 1.0 : 0.0;
        s_R[v][j] = id + s_abc[v][0] * K[j] + s_abc[v][1] * K2;
        s_V[v][j] = id + s_abc[v][1] * K[j] + s_abc[v][2] * K2;
    }
    __syncthreads();
    if (active && j < 3) {
        const double *V = s_V[v], *dl = s_dl[v];
        s_t[v][j] = V[3 * j] * dl[0] + V[3 * j + 1] * dl[1] + V[3 * j + 2] * dl[2];
    }
    __syncthreads();
    double out = 0.0;
    double *T = Tst + 16 * v;
    if (active) {
        const int i = j / 4, c = j % 4;
        const double E[4] = {i < 3 ? s_R[v][3 * i] : 0.0, i < 3 ? s_R[v][3 * i + 1] : 0.0,
                             i < 3 ? s_R[v][3 * i + 2] : 0.0, i < 3 ? s_t[v][i] : 1.0};
        for (int k = 0; k < 4; ++k) out += E[k] * T[4 * k + c];
    }
    __syncthreads();  // every thread has read T before any writes it
    if (active) {
        T[j] = out;
        if (pose_f32) pose_f32[16 * v + j] = (float)out;
    }
}

// The loss kernel's blocks: at most one resident wave (resident = blocks per SM x SMs of the current
// device; 0 = unknown) and at most kLossBlocks in all, shared among the views in proportion to their
// pixels (each view at least one), so that views of different sizes finish together: on eight keyframes of
// 1200x680 and 640x363 in turn, equal shares left the blocks of the small views idle for most of
// the kernel.
LossGrid loss_grid(const ViewTable &vt, int resident, int pixels_per_block) {
    const int64_t P = vt.pix_off[vt.n_views];
    const int total = std::max(vt.n_views, resident > 0 ? std::min(resident, kLossBlocks) : kLossBlocks);
    LossGrid g;
    g.off[0] = 0;
    for (int v = 0; v < vt.n_views; ++v) {
        const int64_t Pv = (int64_t)vt.W[v] * vt.H[v];
        const int64_t share = (int64_t)(total - vt.n_views) * Pv / P + 1;  // the shares' sum is at most total
        g.off[v + 1] = g.off[v] + (int)std::min<int64_t>(share, (Pv + pixels_per_block - 1) / pixels_per_block);
    }
    return g;
}

template <typename K>
int resident_blocks(K kernel, int threads) {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess) return 0;
    return per_sm * sms;
}

template <int D, int KC>
gs_status launch_loss_kernel(const ViewTable &vt, const LossP &lp, const gs_images *img, const gs_targets *tgt,
                             const float *W, const float *b, int64_t P, const uint32_t *mh, gs_image_grads_out *g,
                             float *part_f, double *part_d, float *mask_out, float *median_out, cudaStream_t st,
                             int *rows) {
    using SH = LossShape<D, KC>;
    const LossGrid lg = loss_grid(vt, resident_blocks(loss_kernel<D, KC>, SH::NT), SH::NT * SH::NPX);
    *rows = lg.off[vt.n_views];
    return launch_pdl(loss_kernel<D, KC>, *rows, SH::NT, 0, st, vt, lg, lp, img->rgb, img->depth, img->sil, img->feat,
                      tgt->rgb, tgt->depth, tgt->label, W, b, P, mh, g->rgb, g->depth, g->sil, g->feat, g->feat_coef,
                      part_f, part_d, mask_out, median_out);
}

template <int D>
gs_status launch_loss(const ViewTable &vt, const LossP &lp, const gs_images *img, const gs_targets *tgt,
                      const float *W, const float *b, int64_t P, const uint32_t *mh, gs_image_grads_out *g,
                      float *part_f, double *part_d, float *dW, float *db, double *loss_out, float *mask_out,
                      float *median_out, cudaStream_t st) {
    int rows_f = 0;
    auto launch = [&](auto kc) {
        return launch_loss_kernel<D, decltype(kc)::value>(vt, lp, img, tgt, W, b, P, mh, g, part_f, part_d, mask_out,
                                                          median_out, st, &rows_f);
    };
    // the class bound in steps of 8: registers, shared memory and the unrolled work follow it
    const gs_status ls = lp.K <= 8    ? launch(std::integral_constant<int, 8>())
                         : lp.K <= 16 ? launch(std::integral_constant<int, 16>())
                         : lp.K <= 24 ? launch(std::integral_constant<int, 24>())
                                      : launch(std::integral_constant<int, 32>());
    if (ls) return ls;
    int rows = rows_f;
    if (lp.ssim_coef != 0.f) {
        // the SSIM tiles add their colour-term shares as further partial rows
        const gs_status s = launch_ssim(vt, lp.ssim_coef, img->rgb, tgt->rgb, lp.ssim_maps, part_d + 3 * (size_t)rows,
                                        g->rgb, st);
        if (s) return s;
        rows += ssim_blocks(vt);
    }
    return launch_pdl(loss_finish_kernel, ceil_div(lp.K * D + lp.K, kFinishThreads / 32) + 1, kFinishThreads, 0, st, rows_f,
                      rows, lp.K, D, part_f, part_d, dW, db, loss_out);
}

}  // namespace
}  // namespace gs

extern "C" gs_status gs_loss_fwd_bwd(const gs_camera *cams, int n_views, int feat_dim, const gs_images *img,
                                     const gs_targets *tgt, const float *dec_W, const float *dec_b,
                                     const gs_loss_params *lp, void *ws, size_t ws_bytes, gs_image_grads_out *grad,
                                     float *d_dec_W, float *d_dec_b, double *loss_out, float *mask_out,
                                     float *median_out, gs_stream stream) {
    GS_NVTX_RANGE("gs_loss_fwd_bwd");
    using namespace gs;
    cudaStream_t st = (cudaStream_t)stream;
    ViewTable vt;
    if (!img || !tgt || !lp || !grad || !loss_out || !make_view_table(cams, n_views, 0, &vt)) return GS_ERR_ARG;
    if (!feat_dim_ok(feat_dim)) return GS_ERR_UNSUPPORTED;
    if (lp->n_classes < 0 || lp->n_classes > kMaxK || (lp->mask_mode != 0 && lp->mask_mode != 1)) return GS_ERR_ARG;
    if (!img->rgb || !img->depth || !img->sil || (feat_dim && !img->feat) || !tgt->rgb || !tgt->depth ||
        !tgt->label || !grad->rgb || !grad->depth || !grad->sil || (feat_dim && !grad->feat && !grad->feat_coef))
        return GS_ERR_ARG;
    if (lp->n_classes > 0 && (!dec_W || !dec_b || !d_dec_W || !d_dec_b)) return GS_ERR_ARG;
    if (!(lp->ssim >= 0.f && lp->ssim <= 1.f) || (lp->ssim > 0.f && lp->mask_mode != 0)) return GS_ERR_ARG;
    WsLayout L = ws_layout(0, n_views, 0, &vt);
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255) || ws_bytes < L.misc_end) return GS_ERR_ARG;
    char *w = static_cast<char *>(ws);
    uint32_t *mh = reinterpret_cast<uint32_t *>(w + L.med_hist);
    float *part_f = reinterpret_cast<float *>(w + L.loss_part_f);
    double *part_d = reinterpret_cast<double *>(w + L.loss_part_d);
    const int64_t P = vt.pix_off[n_views];
    gs_status s;
    if (lp->mask_mode == 1) {
        if ((s = launch_median(vt, img->depth, tgt->depth, mh, st))) return s;
    }
    // Eq. 15: the L1 part weighted lambda_c (1 - lambda), the SSIM part lambda_c lambda
    LossP q{lp->color * (1.f - lp->ssim), lp->depth, lp->sem, lp->tau_obs, lp->mask_mode, lp->n_classes,
            lp->color * lp->ssim, reinterpret_cast<float *>(w + L.ssim_maps)};
#define GS_LOSS(DD)                                                                                              \
    case DD:                                                                                                     \
        return launch_loss<DD>(vt, q, img, tgt, dec_W, dec_b, P, mh, grad, part_f, part_d, d_dec_W, d_dec_b,     \
                               loss_out, mask_out, median_out, st);
    switch (feat_dim) {
        GS_LOSS(0) GS_LOSS(4) GS_LOSS(8) GS_LOSS(16) GS_LOSS(32)
        default: return GS_ERR_UNSUPPORTED;
    }
#undef GS_LOSS
}

namespace gs {
namespace {
static_assert(6 * kRedBlocks * sizeof(double) + 2 * sizeof(uint32_t) <= GS_DSR_SCRATCH_BYTES,
              "the DSR partials and their arrival counters fit the scratch");

// The value of Eq. 12 into out, with its partials (and two arrival counters after them) in part.
gs_status dsr_value(int64_t n, const float *log_scales, float lam_big, float lam_small, double *part, double *out,
                    cudaStream_t st) {
    if (n == 0) return cuda_status(cudaMemsetAsync(out, 0, 8 * sizeof(double), st));
    const int64_t m = 3 * n;
    const int grid = std::min(ceil_div(m, 256), kRedBlocks);
    // the arrival counters are zeroed here; each finishing block resets its own
    uint32_t *ctr = reinterpret_cast<uint32_t *>(part + 6 * kRedBlocks);
    gs_status s;
    if ((s = cuda_status(cudaMemsetAsync(ctr, 0, 2 * sizeof(uint32_t), st)))) return s;
    if ((s = launch_pdl(dsr_stats_kernel, grid, 256, 0, st, m, log_scales, part, out, ctr))) return s;
    return launch_pdl(dsr_mask_kernel, grid, 256, 0, st, m, log_scales, out, part + 2 * kRedBlocks, lam_big, lam_small,
                      ctr + 1);
}

gs_status dsr_grad(int64_t n, const float *log_scales, float lam_big, float lam_small, const double *out,
                   float *d_log_scales, cudaStream_t st) {
    if (n == 0) return GS_OK;
    const int64_t m = 3 * n;
    // no partials here: enough blocks for every thread to hold four 16-byte loads at a time
    return launch_pdl(dsr_grad_kernel, std::min(ceil_div(m, 256 * 16), kSMs * 16), 256, 0, st, m, log_scales, lam_big,
                      lam_small, out, d_log_scales);
}
}  // namespace
}  // namespace gs

extern "C" gs_status gs_dsr(int64_t n, const float *log_scales, float lam_big, float lam_small, void *ws,
                            size_t ws_bytes, float *d_log_scales, double *out, gs_stream stream) {
    GS_NVTX_RANGE("gs_dsr");
    using namespace gs;
    cudaStream_t st = (cudaStream_t)stream;
    if (n < 0 || !out || !ws || (reinterpret_cast<uintptr_t>(ws) & 255)) return GS_ERR_ARG;
    WsLayout L = ws_layout(0, 1, 0);
    if (ws_bytes < L.misc_end) return GS_ERR_ARG;
    if (n > 0 && (!log_scales || !d_log_scales)) return GS_ERR_ARG;
    double *part = reinterpret_cast<double *>(static_cast<char *>(ws) + L.dsr_part);
    gs_status s;
    if ((s = dsr_value(n, log_scales, lam_big, lam_small, part, out, st))) return s;
    return dsr_grad(n, log_scales, lam_big, lam_small, out, d_log_scales, st);
}

extern "C" gs_status gs_dsr_value(int64_t n, const float *log_scales, float lam_big, float lam_small, void *scratch,
                                  double *out, gs_stream stream) {
    GS_NVTX_RANGE("gs_dsr_value");
    using namespace gs;
    if (n < 0 || !out || !scratch || (reinterpret_cast<uintptr_t>(scratch) & 255) || (n > 0 && !log_scales))
        return GS_ERR_ARG;
    return dsr_value(n, log_scales, lam_big, lam_small, static_cast<double *>(scratch), out, (cudaStream_t)stream);
}

extern "C" gs_status gs_dsr_grad(int64_t n, const float *log_scales, float lam_big, float lam_small, const double *out,
                                 float *d_log_scales, gs_stream stream) {
    GS_NVTX_RANGE("gs_dsr_grad");
    using namespace gs;
    if (n < 0 || !out || (n > 0 && (!log_scales || !d_log_scales))) return GS_ERR_ARG;
    return dsr_grad(n, log_scales, lam_big, lam_small, out, d_log_scales, (cudaStream_t)stream);
}

extern "C" gs_status gs_pose_grad(int64_t n, int n_views, const float *pose_part, double *d_twist, gs_stream stream) {
    GS_NVTX_RANGE("gs_pose_grad");
    using namespace gs;
    cudaStream_t st = (cudaStream_t)stream;
    if (n < 0 || n_views < 1 || n_views > kMaxViews || !d_twist) return GS_ERR_ARG;
    gs_status s;
    if ((s = cuda_status(cudaMemsetAsync(d_twist, 0, sizeof(double) * 6 * n_views, st)))) return s;
    if (n == 0) return GS_OK;
    if (!pose_part) return GS_ERR_ARG;
    dim3 grid(std::min(ceil_div(n, 256 * 8), kPoseBlocks), 6 * n_views);
    return launch_pdl(pose_reduce_kernel, grid, 256, 0, st, n, pose_part, d_twist);
}

extern "C" gs_status gs_pose_step(int n_views, const double *d_twist, double *T_state, double *adam, int step,
                                  const double *lr, double beta1, double beta2, double eps, float *pose_f32,
                                  gs_stream stream) {
    GS_NVTX_RANGE("gs_pose_step");
    using namespace gs;
    if (n_views < 1 || n_views > kMaxViews || !d_twist || !T_state || !adam || !lr || step < 0) return GS_ERR_ARG;
    // Adam bias corrections 1 - beta^step: on the host for a given step, on the
    // device (from the counter after the moments) for step 0
    const double bc1 = step ? 1.0 - pow(beta1, step) : -1.0, bc2 = step ? 1.0 - pow(beta2, step) : -1.0;
    return launch_pdl(pose_step_kernel, 1, kPoseLanes * n_views, 0, (cudaStream_t)stream, n_views, d_twist, T_state,
                      adam, bc1, bc2, lr[0], lr[1], lr[2], lr[3], lr[4], lr[5], beta1, beta2, log(beta1),
                      log(beta2), eps, pose_f32);
}

// ------------------------------------------------- allocation-free loss entry
// Same computation as gs_loss_fwd_bwd for callers that cannot allocate device
// memory: the scratch (median histograms of up to kNoAllocMaxViews views and the
// per-block partials) lives in one file-scope device array that every GPU which
// loads the library holds until the process exits.
namespace gs {
namespace {

constexpr int kNoAllocMaxViews = 16;
constexpr size_t kNoAllocHistBytes = sizeof(uint32_t) * 4 * 256 * kNoAllocMaxViews;          //    65,536
constexpr size_t kNoAllocPartFBytes = sizeof(float) * (size_t)kLossBlocks * (kMaxK * 32 + kMaxK);  // 4,325,376
constexpr size_t kNoAllocPartDBytes = sizeof(double) * (size_t)kLossBlocks * 3;                //    24,576
constexpr size_t kNoAllocBytes = kNoAllocHistBytes + kNoAllocPartFBytes + kNoAllocPartDBytes;   // 4,415,488

static __device__ __align__(256) unsigned char g_noalloc_loss_scratch[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 256;
std::atomic<void *> g_noalloc_scratch_addr[kNoAllocMaxDevices];

// Device address of the scratch array on the current device (host code only sees a
// host-side stand-in for the symbol).  Outside a stream capture it is looked up on every
// call (cheap once the module is loaded), so a context torn down and created again gets
// its own address; during a capture, where the lookup is not attempted, the address of the
// last call outside a capture on this device is used.
gs_status noalloc_scratch(cudaStream_t st, char **out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return GS_ERR_CUDA;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return GS_ERR_UNSUPPORTED;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool capturing = cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
    (void)cudaGetLastError();  // a refused query must not linger as the sticky last error
    void *p = nullptr;
    if (!capturing) {
        if (cudaGetSymbolAddress(&p, g_noalloc_loss_scratch) != cudaSuccess || !p) return GS_ERR_CUDA;
        g_noalloc_scratch_addr[dev].store(p, std::memory_order_release);
    } else {
        p = g_noalloc_scratch_addr[dev].load(std::memory_order_acquire);
        if (!p) return GS_ERR_UNSUPPORTED;  // first call on this device inside a capture
    }
    *out = static_cast<char *>(p);
    return GS_OK;
}

}  // namespace
}  // namespace gs

extern "C" gs_status gs_loss_fwd_bwd_noalloc(const gs_camera *cams, int n_views, int feat_dim, const gs_images *img,
                                             const gs_targets *tgt, const float *dec_W, const float *dec_b,
                                             const gs_loss_params *lp, gs_image_grads_out *grad, float *d_dec_W,
                                             float *d_dec_b, double *loss_out, float *mask_out, float *median_out,
                                             gs_stream stream) {
    GS_NVTX_RANGE("gs_loss_fwd_bwd_noalloc");
    using namespace gs;
    cudaStream_t st = (cudaStream_t)stream;
    ViewTable vt;
    if (!img || !tgt || !lp || !grad || !loss_out || !make_view_table(cams, n_views, 0, &vt)) return GS_ERR_ARG;
    if (n_views > kNoAllocMaxViews) return GS_ERR_UNSUPPORTED;
    if (!feat_dim_ok(feat_dim)) return GS_ERR_UNSUPPORTED;
    if (lp->n_classes < 0 || lp->n_classes > kMaxK || (lp->mask_mode != 0 && lp->mask_mode != 1)) return GS_ERR_ARG;
    if (!img->rgb || !img->depth || !img->sil || (feat_dim && !img->feat) || !tgt->rgb || !tgt->depth ||
        !tgt->label || !grad->rgb || !grad->depth || !grad->sil || (feat_dim && !grad->feat && !grad->feat_coef))
        return GS_ERR_ARG;
    if (lp->n_classes > 0 && (!dec_W || !dec_b || !d_dec_W || !d_dec_b)) return GS_ERR_ARG;
    if (!(lp->ssim >= 0.f && lp->ssim <= 1.f) || (lp->ssim > 0.f && lp->mask_mode != 0)) return GS_ERR_ARG;
    if (lp->ssim != 0.f) return GS_ERR_UNSUPPORTED;  // the SSIM maps need per-pixel scratch
    // every argument is checked: only now is the shared array touched
    char *w = nullptr;
    gs_status s;
    if ((s = noalloc_scratch(st, &w))) return s;
    uint32_t *mh = reinterpret_cast<uint32_t *>(w);
    float *part_f = reinterpret_cast<float *>(w + kNoAllocHistBytes);
    double *part_d = reinterpret_cast<double *>(w + kNoAllocHistBytes + kNoAllocPartFBytes);
    const int64_t P = vt.pix_off[n_views];
    if (lp->mask_mode == 1) {
        // the histograms keep the previous call's counts: clear them first
        if ((s = launch_median(vt, img->depth, tgt->depth, mh, st))) return s;
    }
    LossP q{lp->color, lp->depth, lp->sem, lp->tau_obs, lp->mask_mode, lp->n_classes};
#define GS_LOSS(DD)                                                                                              \
    case DD:                                                                                                     \
        return launch_loss<DD>(vt, q, img, tgt, dec_W, dec_b, P, mh, grad, part_f, part_d, d_dec_W, d_dec_b,     \
                               loss_out, mask_out, median_out, st);
    switch (feat_dim) {
        GS_LOSS(0) GS_LOSS(4) GS_LOSS(8) GS_LOSS(16) GS_LOSS(32)
        default: return GS_ERR_UNSUPPORTED;
    }
#undef GS_LOSS
}

// ---------------------------------------------------- adaptive Gaussian expansion
// Eq. 11: M_unobs = (o_hat < tau) or (d_hat > d_gt and |d_gt - d_hat| > 50 median) on pixels with
// d_gt > 0, the median being the view's lower median of |d - d_gt| over d_gt > 0 (the same radix
// selection as the tracking mask).  One new Gaussian per masked pixel, in pixel order per view,
// views in order: a count per 256-pixel chunk, an ordered scan of the counts, then an emit pass
// that ranks the chunk's masked pixels by ballots.  A warp takes a chunk, eight pixels a lane, so that a
// block finds the median once for 2048 pixels, and its loads do not wait for the kernel before it. The
// new Gaussians of a chunk have consecutive ranks: its warp copies their features as one run (a
// thread copying a Gaussian's row by itself wrote 64 bytes apart from its neighbours').
// Median, count, scan and emission at 1200x680 with 10% of the pixels unobserved: 99 -> 46 us.
namespace gs {
namespace {

__device__ __forceinline__ bool unobserved(float sil, float d, float dgt, float med, float tau) {
    if (!(dgt > 0.f)) return false;
    return sil < tau || (d > dgt && depth_error(d, dgt) > 50.f * med);
}

constexpr int kChunkRounds = 8;  // rounds of 32 pixels of a warp's 256-pixel chunk

// The lane's eight pixels of the warp's chunk: rendered silhouette and depth, observed depth.
struct ChunkPixels {
    int64_t chunk, first;  // the chunk of the view, its first pixel in the view
    float sil[kChunkRounds], d[kChunkRounds], dgt[kChunkRounds];
};

__device__ __forceinline__ void load_chunk(ChunkPixels &c, const ViewTable &vt, const float *__restrict__ sil,
                                           const float *__restrict__ depth, const float *__restrict__ tdepth) {
    const int v = blockIdx.y;
    const int64_t Pv = (int64_t)vt.W[v] * vt.H[v];
    c.chunk = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    c.first = c.chunk * (32 * kChunkRounds);
#pragma unroll
    for (int u = 0; u < kChunkRounds; ++u) {
        const int64_t i = c.first + 32 * u + (threadIdx.x & 31), pix = vt.pix_off[v] + i;
        const bool in = i < Pv;
        c.sil[u] = in ? sil[pix] : 0.f;
        c.d[u] = in ? depth[pix] : 0.f;
        c.dgt[u] = in ? tdepth[pix] : 0.f;  // no depth: not an unobserved pixel
    }
}

// chunks: 256-pixel chunks of a view's row of counts.
__global__ void __launch_bounds__(256) expand_count_kernel(ViewTable vt, const float *sil, const float *depth,
                                                           const float *tdepth, const uint32_t *hist, float tau,
                                                           int chunks, uint32_t *counts) {
    ChunkPixels c;
    load_chunk(c, vt, sil, depth, tdepth);  // the images were complete before the median's last pass began
    pdl_wait();                             // the median's histograms
    pdl_trigger();
    const int v = blockIdx.y;
    // every thread of the block takes part in the selection (it synchronises the block)
    const float med = __uint_as_float(block_select(hist, vt.n_views, v, 4));
    uint32_t n = 0;
#pragma unroll
    for (int u = 0; u < kChunkRounds; ++u)
        n += __popc(__ballot_sync(0xffffffffu, unobserved(c.sil[u], c.d[u], c.dgt[u], med, tau)));
    if ((threadIdx.x & 31) == 0 && c.chunk < chunks) counts[(int64_t)v * chunks + c.chunk] = n;
}

// One block: exclusive scan of the counts in order (views, then blocks); the total to *n_new.
__global__ void __launch_bounds__(1024) expand_scan_kernel(const uint32_t *counts, int64_t n, uint32_t *offsets,
                                                           int64_t *n_new) {
    __shared__ uint32_t s_warp[32];
    __shared__ uint64_t s_carry;
    pdl_wait();  // the counts
    pdl_trigger();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < n; base += 1024) {
        const int64_t i = base + threadIdx.x;
        const uint32_t c = i < n ? counts[i] : 0u;
        uint32_t x = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) s_warp[w] = x;
        __syncthreads();
        if (w == 0) {
            uint32_t t = s_warp[lane];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, t, d);
                if (lane >= d) t += y;
            }
            s_warp[lane] = t;
        }
        __syncthreads();
        const uint64_t before = s_carry + (w > 0 ? s_warp[w - 1] : 0u) + x - c;
        if (i < n) offsets[i] = (uint32_t)before;
        __syncthreads();
        if (threadIdx.x == 0) s_carry += s_warp[31];
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_new = (int64_t)s_carry;
}

struct ExpandOut {
    float *means, *quats, *log_scales, *logits, *rgb, *feat;
    int64_t *src_pix;
};

__global__ void __launch_bounds__(256) expand_emit_kernel(ViewTable vt, const float *sil, const float *depth,
                                                          const float *__restrict__ trgb, const float *tdepth,
                                                          const uint32_t *hist, float tau, int chunks,
                                                          const uint32_t *offsets, int64_t room, int64_t P, int D,
                                                          const float *__restrict__ feat_init, ExpandOut o,
                                                          int32_t *status) {
    ChunkPixels c;
    load_chunk(c, vt, sil, depth, tdepth);
    pdl_wait();  // the offsets
    const int v = blockIdx.y, lane = threadIdx.x & 31;
    // every thread of the block takes part in the selection (it synchronises the block)
    const float med = __uint_as_float(block_select(hist, vt.n_views, v, 4));
    if (c.chunk >= chunks) return;
    const int64_t begin = offsets[(int64_t)v * chunks + c.chunk];
    int64_t first = begin;  // rank of the round's first new Gaussian
#pragma unroll
    for (int u = 0; u < kChunkRounds; ++u) {
        const float d = c.dgt[u];
        const bool m = unobserved(c.sil[u], c.d[u], d, med, tau);
        const uint32_t bal = __ballot_sync(0xffffffffu, m);
        if (!bal) continue;
        const int64_t rank = first + __popc(bal & ((1u << lane) - 1u));
        first += __popc(bal);
        if (!m) continue;
        if (rank >= room) {
            set_status(status, GS_ERR_CAPACITY);
            continue;
        }
        const int64_t i = c.first + 32 * u + lane, pix = vt.pix_off[v] + i;
        const int x = (int)(i % vt.W[v]), y = (int)(i / vt.W[v]);
        // the pixel centre unprojected at d_gt: camera point, then world = R^T (p_c - t)
        const float pc[3] = {((float)x + 0.5f - vt.cx[v]) / vt.fx[v] * d, ((float)y + 0.5f - vt.cy[v]) / vt.fy[v] * d,
                             d};
        const float *T = vt.T[v];
        const float q[3] = {pc[0] - T[3], pc[1] - T[7], pc[2] - T[11]};
#pragma unroll
        for (int j = 0; j < 3; ++j) o.means[3 * rank + j] = T[j] * q[0] + T[4 + j] * q[1] + T[8 + j] * q[2];
        o.quats[4 * rank] = 1.f;
        o.quats[4 * rank + 1] = o.quats[4 * rank + 2] = o.quats[4 * rank + 3] = 0.f;
        const float ls = logf(d / vt.fx[v]);
#pragma unroll
        for (int j = 0; j < 3; ++j) o.log_scales[3 * rank + j] = ls;
        o.logits[rank] = 0.f;                       // opacity 0.5
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) o.rgb[3 * rank + ch] = trgb[ch * P + pix];
        if (o.src_pix) o.src_pix[rank] = pix;
    }
    // the features of the chunk's Gaussians: one run of the array
    const int64_t f0 = begin * D, f1 = min(first, room) * D;
    float *__restrict__ feat = o.feat;
#pragma unroll 8
    for (int64_t k = f0 + lane; k < f1; k += 32) feat[k] = feat_init[k];
}

}  // namespace
}  // namespace gs

extern "C" gs_status gs_expand(const gs_camera *cams, int n_views, const gs_images *img, const gs_targets *tgt,
                               float tau_unobs, const float *feat_init, int64_t n_existing, gs_field_mut *field,
                               int64_t *n_new, int64_t *src_pix, int32_t *status, void *ws, size_t ws_bytes,
                               gs_stream stream) {
    GS_NVTX_RANGE("gs_expand");
    using namespace gs;
    ViewTable vt;
    if (!img || !tgt || !field || !n_new || !status || !make_view_table(cams, n_views, 0, &vt)) return GS_ERR_ARG;
    if (!feat_dim_ok(field->feat_dim)) return GS_ERR_UNSUPPORTED;
    const int64_t capacity = field->n;  // rows of the field's arrays
    if (n_existing < 0 || capacity < n_existing || !img->sil || !img->depth || !tgt->rgb || !tgt->depth ||
        !field->means || !field->quats || !field->log_scales || !field->opacity_logits || !field->rgb ||
        (field->feat_dim && (!field->feat || !feat_init)) || !(tau_unobs >= 0.f))
        return GS_ERR_ARG;
    WsLayout L = ws_layout(0, n_views, 0, &vt);
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255) || ws_bytes < L.misc_end) return GS_ERR_ARG;
    char *w = static_cast<char *>(ws);
    uint32_t *mh = reinterpret_cast<uint32_t *>(w + L.med_hist);
    const int bx = expand_blocks_x(vt);
    uint32_t *counts = reinterpret_cast<uint32_t *>(w + L.expand_counts);
    uint32_t *offsets = counts + (size_t)n_views * bx;
    cudaStream_t st = (cudaStream_t)stream;
    gs_status s;
    if ((s = cuda_status(cudaMemsetAsync(status, 0, sizeof(int32_t), st)))) return s;
    if ((s = launch_median(vt, img->depth, tgt->depth, mh, st))) return s;
    const dim3 grid(ceil_div(bx, 8), n_views);  // eight warps of a chunk each
    if ((s = launch_pdl(expand_count_kernel, grid, 256, 0, st, vt, img->sil, img->depth, tgt->depth, mh, tau_unobs,
                        bx, counts)))
        return s;
    if ((s = launch_pdl(expand_scan_kernel, 1, 1024, 0, st, counts, (int64_t)n_views * bx, offsets, n_new))) return s;
    const int64_t D = field->feat_dim;
    ExpandOut o{field->means + 3 * n_existing, field->quats + 4 * n_existing, field->log_scales + 3 * n_existing,
                field->opacity_logits + n_existing, field->rgb + 3 * n_existing,
                D ? field->feat + D * n_existing : nullptr, src_pix};
    return launch_pdl(expand_emit_kernel, grid, 256, 0, st, vt, img->sil, img->depth, tgt->rgb, tgt->depth, mh,
                      tau_unobs, bx, offsets, capacity - n_existing, vt.pix_off[n_views], (int)D, feat_init, o, status);
}
