// SSIM term of the mapping colour loss (Eq. 15, read as lambda_c lambda (1 - SSIM)):
// per view, channel and pixel the window moments over an 11x11 Gaussian window
// (sigma 1.5, zero outside the image), S = (2 mx my + C1)(2 sxy + C2) /
// ((mx^2 + my^2 + C1)(sx + sy + C2)), averaged over the view's 3 P_v positions.
//
// Two passes over 32x32-pixel tiles of one channel (one CTA each, 256 threads):
//   forward: the tile and a 5-pixel halo of the rendered and observed colour in
//     shared memory, the separable window (rows, then columns) applied to x, y,
//     x^2, y^2, x y; per pixel S and the partials A = dS/dmx - 2 mx dS/dsx -
//     my dS/dsxy, B = dS/dsx, C = dS/dsxy (stored, f32), and the tile's sum of S
//     (f64 partial, fixed order);
//   backward: dS/dx(q) = sum_p w(q - p) (A(p) + 2 B(p) x(q) + C(p) y(q)), the
//     same separable window over A, B and C, added to the colour gradient.
//
// Bound by instruction issue and shared-memory reads, not by its 144 bytes a pixel, so each thread slides the
// window over four neighbouring outputs (14 values read for 44 taps) and carries (x, y), (x^2, y^2)
// and (A, B) as packed pairs: three (two) multiply-adds a tap instead of seven (three) with two (three)
// reads.  In the row pass a warp's lanes are 32 rows of one column group, in the column pass 32 columns; the odd
// row pitches keep both free of bank conflicts.  Loss step with the term over a 1200x680 frame: 0.153 -> 0.114
// ms (0.049 without the term).
#include "common.cuh"

namespace gs {
namespace {

constexpr int kSW = 32, kSH = 32, kR = 5;                 // tile and window radius
constexpr int kTaps = 2 * kR + 1, kOut = 4;               // window taps, outputs a thread slides over
constexpr int kIW = kSW + 2 * kR, kIH = kSH + 2 * kR;     // tile with halo: 42 x 42
constexpr int kSThreads = 256;
static_assert(kSThreads / 32 * kOut == kSW && kSThreads / 32 * kOut == kSH && kSW == 32, "a warp per group of outputs");

struct SsimTable {
    int off[kMaxViews + 1];  // first CTA of each view (3 channels x tiles)
    int tx[kMaxViews];       // tiles per row
    float g[11];             // normalised 1D window
    float coef;              // lambda_c * lambda
};

__device__ __forceinline__ void locate(const ViewTable &vt, const SsimTable &t, int &v, int &ch, int &x0, int &y0) {
    const int b = blockIdx.x;
    v = 0;
    while (v + 1 < vt.n_views && b >= t.off[v + 1]) ++v;
    const int tiles = (t.off[v + 1] - t.off[v]) / 3;
    const int r = b - t.off[v];
    ch = r / tiles;
    const int k = r - ch * tiles;
    x0 = (k % t.tx[v]) * kSW;
    y0 = (k / t.tx[v]) * kSH;
}

// Loads N channel planes' tile with halo (zero outside the image) through put(n, row, column, value).
template <int N, typename F>
__device__ __forceinline__ void load_halo(const float *const (&src)[N], int W, int H, int x0, int y0, F put) {
    for (int i = threadIdx.x; i < kIW * kIH; i += kSThreads) {
        const int r = i / kIW, c = i - r * kIW;
        const int gy = y0 + r - kR, gx = x0 + c - kR;
        const bool in = gy >= 0 && gy < H && gx >= 0 && gx < W;
#pragma unroll
        for (int n = 0; n < N; ++n) put(n, r, c, in ? src[n][(int64_t)gy * W + gx] : 0.f);
    }
}

// sum += x, with what the f32 addition rounds away added to lo (an infinite sum stays one).
__device__ __forceinline__ void add_exact(float x, float &sum, float &lo) {
    float e;
    two_sum(sum, x, sum, e);
    lo += isfinite(e) ? e : 0.f;
}

// Five resident blocks per SM (48 registers), as many as its 44 KB of shared memory allow.
__global__ void __launch_bounds__(kSThreads, 5) ssim_fwd_kernel(ViewTable vt, SsimTable t, const float *rgb,
                                                             const float *trgb, int64_t P, float *maps,
                                                             double *part) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    __shared__ float2 s_xy[kIH][kIW + 1];
    __shared__ float2 s_m[kIH][kSW + 1], s_q[kIH][kSW + 1];  // row sums of (x, y), (x^2, y^2) and x y
    __shared__ float s_c[kIH][kSW + 1];
    __shared__ float s_sum[2][kSThreads];
    int v, ch, x0, y0;
    locate(vt, t, v, ch, x0, y0);
    const int W = vt.W[v], H = vt.H[v], lane = threadIdx.x & 31, o0 = threadIdx.x / 32 * kOut;
    const int64_t base = ch * P + vt.pix_off[v];
    const float *const src[2] = {rgb + base, trgb + base};
    load_halo(src, W, H, x0, y0, [&](int n, int r, int c, float x) { (n ? s_xy[r][c].y : s_xy[r][c].x) = x; });
    __syncthreads();
    for (int r = lane; r < kIH; r += 32) {
        float2 m[kOut], q[kOut];
        float c[kOut];
#pragma unroll
        for (int j = 0; j < kOut; ++j) {
            m[j] = q[j] = make_float2(0.f, 0.f);
            c[j] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < kOut + kTaps - 1; ++i) {
            const float2 a = s_xy[r][o0 + i], aa = __fmul2_rn(a, a);
            const float ab = a.x * a.y;
#pragma unroll
            for (int j = 0; j < kOut; ++j)
                if (i - j >= 0 && i - j < kTaps) {
                    const float w = t.g[i - j];
                    m[j] = fma2(make_float2(w, w), a, m[j]);
                    q[j] = fma2(make_float2(w, w), aa, q[j]);
                    c[j] = fmaf(w, ab, c[j]);
                }
        }
#pragma unroll
        for (int j = 0; j < kOut; ++j) {
            s_m[r][o0 + j] = m[j];
            s_q[r][o0 + j] = q[j];
            s_c[r][o0 + j] = c[j];
        }
    }
    __syncthreads();
    constexpr float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
    const int64_t Pv = (int64_t)W * H;
    float2 m[kOut], q[kOut];
    float c[kOut], ssum = 0.f, slo = 0.f;  // the thread's sum of S and what its additions rounded away
#pragma unroll
    for (int j = 0; j < kOut; ++j) {
        m[j] = q[j] = make_float2(0.f, 0.f);
        c[j] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < kOut + kTaps - 1; ++i) {
        const float2 a = s_m[o0 + i][lane], b = s_q[o0 + i][lane];
        const float d = s_c[o0 + i][lane];
#pragma unroll
        for (int j = 0; j < kOut; ++j)
            if (i - j >= 0 && i - j < kTaps) {
                const float w = t.g[i - j];
                m[j] = fma2(make_float2(w, w), a, m[j]);
                q[j] = fma2(make_float2(w, w), b, q[j]);
                c[j] = fmaf(w, d, c[j]);
            }
    }
#pragma unroll
    for (int j = 0; j < kOut; ++j) {
        const int py = y0 + o0 + j, px = x0 + lane;
        if (py >= H || px >= W) continue;
        const float mx = m[j].x, my = m[j].y;
        const float sx = q[j].x - mx * mx, sy = q[j].y - my * my, sxy = c[j] - mx * my;
        const float N1 = 2.f * mx * my + C1, N2 = 2.f * sxy + C2;
        const float D1 = mx * mx + my * my + C1, D2 = sx + sy + C2;
        const float inv = 1.f / (D1 * D2);
        const float S = N1 * N2 * inv;
        const float dS_dmx = 2.f * my * N2 * inv - S * 2.f * mx / D1;
        const float dS_dsx = -S / D2;
        const float dS_dsxy = 2.f * N1 * inv;
        const int64_t o = (int64_t)py * W + px;
        // maps of (channel, view): 3 planes of P_v floats at 3 (ch P + pix_off(v))
        const int64_t mb = (int64_t)3 * (ch * P + vt.pix_off[v]);
        maps[mb + o] = dS_dmx - 2.f * mx * dS_dsx - my * dS_dsxy;
        maps[mb + Pv + o] = dS_dsx;
        maps[mb + 2 * Pv + o] = dS_dsxy;
        add_exact(S, ssum, slo);
    }
    // the tile's sum by one warp, in f64 at the end (f64 additions are slow, see the loss's block sums; f32
    // sums of values near 1 alone would round away what 1 - SSIM is made of)
    s_sum[0][threadIdx.x] = ssum;
    s_sum[1][threadIdx.x] = slo;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    ssum = slo = 0.f;
#pragma unroll
    for (int i = 0; i < kSThreads / 32; ++i) {
        add_exact(s_sum[0][i * 32 + lane], ssum, slo);
        slo += s_sum[1][i * 32 + lane];
    }
    double tot = (double)ssum + (double)slo;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0) {
        // colour-term share of this tile: coef (1 - S_sum / (3 P_v)) summed over the view's tiles
        double val = -(double)t.coef * tot / (3.0 * (double)Pv);
        if (blockIdx.x == t.off[v]) val += (double)t.coef;
        part[3 * blockIdx.x] = val;
        part[3 * blockIdx.x + 1] = 0.0;
        part[3 * blockIdx.x + 2] = 0.0;
    }
}

__global__ void __launch_bounds__(kSThreads) ssim_bwd_kernel(ViewTable vt, SsimTable t, const float *rgb,
                                                             const float *trgb, int64_t P, const float *maps,
                                                             float *g_rgb) {
    pdl_wait();     // the previous kernel's results
    pdl_trigger();  // the next kernel may be scheduled now
    __shared__ float2 s_ab[kIH][kIW + 1], s_hab[kIH][kSW + 1];  // (A, B) and their row sums
    __shared__ float s_c[kIH][kIW + 1], s_hc[kIH][kSW + 1];
    int v, ch, x0, y0;
    locate(vt, t, v, ch, x0, y0);
    const int W = vt.W[v], H = vt.H[v], lane = threadIdx.x & 31, o0 = threadIdx.x / 32 * kOut;
    const int64_t Pv = (int64_t)W * H;
    const float *mb = maps + (int64_t)3 * (ch * P + vt.pix_off[v]);
    const float *const src[3] = {mb, mb + Pv, mb + 2 * Pv};
    load_halo(src, W, H, x0, y0,
              [&](int n, int r, int c, float x) { (n == 2 ? s_c[r][c] : n ? s_ab[r][c].y : s_ab[r][c].x) = x; });
    __syncthreads();
    for (int r = lane; r < kIH; r += 32) {
        float2 f[kOut];
        float c[kOut];
#pragma unroll
        for (int j = 0; j < kOut; ++j) {
            f[j] = make_float2(0.f, 0.f);
            c[j] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < kOut + kTaps - 1; ++i) {
            const float2 a = s_ab[r][o0 + i];
            const float d = s_c[r][o0 + i];
#pragma unroll
            for (int j = 0; j < kOut; ++j)
                if (i - j >= 0 && i - j < kTaps) {
                    const float w = t.g[i - j];
                    f[j] = fma2(make_float2(w, w), a, f[j]);
                    c[j] = fmaf(w, d, c[j]);
                }
        }
#pragma unroll
        for (int j = 0; j < kOut; ++j) {
            s_hab[r][o0 + j] = f[j];
            s_hc[r][o0 + j] = c[j];
        }
    }
    __syncthreads();
    float2 f[kOut];
    float c[kOut];
#pragma unroll
    for (int j = 0; j < kOut; ++j) {
        f[j] = make_float2(0.f, 0.f);
        c[j] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < kOut + kTaps - 1; ++i) {
        const float2 a = s_hab[o0 + i][lane];
        const float d = s_hc[o0 + i][lane];
#pragma unroll
        for (int j = 0; j < kOut; ++j)
            if (i - j >= 0 && i - j < kTaps) {
                const float w = t.g[i - j];
                f[j] = fma2(make_float2(w, w), a, f[j]);
                c[j] = fmaf(w, d, c[j]);
            }
    }
    const float scale = -t.coef / (3.f * (float)Pv);
    const int64_t base = ch * P + vt.pix_off[v];
#pragma unroll
    for (int j = 0; j < kOut; ++j) {
        const int py = y0 + o0 + j, px = x0 + lane;
        if (py >= H || px >= W) continue;
        const int64_t pix = base + (int64_t)py * W + px;
        const float grad = f[j].x + 2.f * rgb[pix] * f[j].y + trgb[pix] * c[j];
        g_rgb[pix] = fmaf(scale, grad, g_rgb[pix]);
    }
}

}  // namespace

int ssim_blocks(const ViewTable &vt) {
    int b = 0;
    for (int v = 0; v < vt.n_views; ++v) b += 3 * ((vt.W[v] + kSW - 1) / kSW) * ((vt.H[v] + kSH - 1) / kSH);
    return b;
}

// Adds the SSIM term to the loss partials (rows part[0 .. ssim_blocks) of f64 [.][3], colour
// column) and its gradient to g_rgb.  maps: f32 scratch [9 P].
gs_status launch_ssim(const ViewTable &vt, float coef, const float *rgb, const float *trgb, float *maps,
                      double *part, float *g_rgb, cudaStream_t st) {
    SsimTable t;
    t.off[0] = 0;
    for (int v = 0; v < vt.n_views; ++v) {
        t.tx[v] = (vt.W[v] + kSW - 1) / kSW;
        t.off[v + 1] = t.off[v] + 3 * t.tx[v] * ((vt.H[v] + kSH - 1) / kSH);
    }
    double g[11], gs = 0.0;
    for (int k = 0; k < 11; ++k) {
        g[k] = exp(-(double)((k - 5) * (k - 5)) / (2.0 * 1.5 * 1.5));
        gs += g[k];
    }
    for (int k = 0; k < 11; ++k) t.g[k] = (float)(g[k] / gs);
    t.coef = coef;
    const int blocks = t.off[vt.n_views];
    if (blocks == 0) return GS_OK;
    const int64_t P = vt.pix_off[vt.n_views];
    const gs_status s = launch_pdl(ssim_fwd_kernel, blocks, kSThreads, 0, st, vt, t, rgb, trgb, P, maps, part);
    if (s) return s;
    return launch_pdl(ssim_bwd_kernel, blocks, kSThreads, 0, st, vt, t, rgb, trgb, P, maps, g_rgb);
}

}  // namespace gs
