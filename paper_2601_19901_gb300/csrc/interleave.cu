// Elemental image array construction (Sec. 4): optional angular tent
// reconstruction of the 2N supersampled views, optional +-1 crosstalk mixing,
// then the slanted-lens subpixel interleave.
//
// Every panel pixel samples one view pixel (nearest, pixel centres) of the
// views its three subpixels select, and neighbouring subpixels select
// different views, so reading views straight from global memory is a gather
// touching a new sector per byte. k_interleave_tile instead takes one view
// row and a strip of 1024 panel columns: it stages the strip's source
// segment of that row for every rendered view in shared memory with
// coalesced loads, then forms every panel row that samples that view row,
// one thread per 4 adjacent panel pixels and one 16-byte store per row.
// k_interleave_tent stages the tent's display views instead.
// k_interleave (the direct gather) serves displays whose tile would not fit, or
// of whose view pixels the panel shows too few (tent_pays).
// k_interleave_gauss is the Gaussian reconstruction of Sec. 4 (recon 2, 3):
// per subpixel the mean of the caller's samples, each the nearest rendered
// view to the subpixel's phase plus the sample's angular offset at the view
// pixel holding its spatially offset position: up to 72 view searches and
// gathers a pixel with crosstalk and eight samples. The searches go through a
// table of thresholds in shared memory, and a warp's lanes take panel columns
// a stride apart at which the lens phase repeats, so that they mostly gather
// from the same view (see there); k_interleave_gauss_plain serves what is too
// little for a table.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "lfdpr_internal.cuh"

namespace lfdpr {
namespace {

// View pixel channel as stored: global views [view][H][W][RGBA8].
struct GlobalTexels {
    const uint8_t* __restrict__ views;
    uint64_t npix, pix;
    __device__ __forceinline__ uint32_t byte(int view, int ch) const {
        return __ldg(views + ((uint64_t)view * npix + pix) * 4u + ch);
    }
    __device__ __forceinline__ float operator()(int view, int ch) const { return float(byte(view, ch)); }
};

// The same from a staged row segment: s[view * stride + i], RGBA8 words.
struct SharedTexels {
    const uint32_t* s;
    int stride, i;
    __device__ __forceinline__ uint32_t byte(int view, int ch) const {
        return (s[view * stride + i] >> (8 * ch)) & 255u;
    }
    __device__ __forceinline__ float operator()(int view, int ch) const { return float(byte(view, ch)); }
};

// Display view k, channel ch, as binary32 before rounding.
template <class T>
__device__ __forceinline__ float display_value(const DispConst& c, const T& tex, int k, int ch) {
    if (c.recon != 1) return tex(k, ch);
    float acc = 0.0f, ws = 0.0f;
#pragma unroll
    for (int q = 0; q < 3; q++) {
        const int m = 2 * k - 1 + q;
        if (m < 0 || m >= c.nr) continue;
        const float w = q == 1 ? 0.5f : 0.25f;
        acc = fmaf(w, tex(m, ch), acc);
        ws += w;
    }
    return __fdiv_rn(acc, ws);
}

// Lens phase of subpixel (x, y, ch) on the display-view axis, [0, N).
__device__ __forceinline__ float subpixel_phase(const DispConst& c, int x, int y, int ch) {
    const float third = ch == 0 ? (float)(1.0 / 6.0) : (ch == 1 ? 0.5f : (float)(5.0 / 6.0));
    const float cx = float(x) + third;
    const float a = fmaf(c.slant, float(y), cx);
    const float ph = fmaf(a, c.inv_pitch, c.phase_offset);
    const float fr = ph - floorf(ph);
    return fr * float(c.n_views);
}

// floor of the phase, below N (one addition rounded down onto 2^23: the
// conversion instruction runs at a quarter of the rate); 0 where the phase is
// no number (slant or pitch overflow).
__device__ __forceinline__ int view_of_subpixel(const DispConst& c, int x, int y, int ch) {
    const uint32_t N = uint32_t(c.n_views);
    const uint32_t k = __float_as_uint(__fadd_rd(subpixel_phase(c, x, y, ch), 8388608.0f)) - 0x4b000000u;
    return int(k > N ? 0u : min(k, N - 1u));
}

// Panel pixel (x, y) as RGBA8 (alpha 255) from its view pixel's texels.
template <class T>
__device__ __forceinline__ uint32_t panel_pixel(const DispConst& c, const T& tex, int x, int y) {
    uint32_t o = 0xff000000u;
    if (c.recon != 1 && !(c.xtalk > 0.0f)) {
        // each subpixel shows its view's byte as it is (a byte converted to
        // binary32 and rounded back is the byte)
#pragma unroll
        for (int ch = 0; ch < 3; ch++) o |= tex.byte(view_of_subpixel(c, x, y, ch), ch) << (8 * ch);
        return o;
    }
#pragma unroll
    for (int ch = 0; ch < 3; ch++) {
        const int k = view_of_subpixel(c, x, y, ch);
        float val;
        if (c.xtalk > 0.0f) {
            const int km = k == 0 ? c.n_views - 1 : k - 1;
            const int kp = k == c.n_views - 1 ? 0 : k + 1;
            float acc = display_value(c, tex, k, ch) * c.xtalk_c;
            acc = fmaf(c.xtalk, display_value(c, tex, km, ch), acc);
            acc = fmaf(c.xtalk, display_value(c, tex, kp, ch), acc);
            val = acc;
        } else {
            val = display_value(c, tex, k, ch);
        }
        o |= uint32_t(round_u8(val)) << (8 * ch);
    }
    return o;
}

// Nearest view pixel of panel column x (row y): pixel centres aligned. In
// 32 bits: (2 x + 1) W < 2^31 for panels up to 32768 and views up to 16384.
__device__ __forceinline__ int source_x(const DispConst& c, int x) {
    return int((2u * uint32_t(x) + 1u) * uint32_t(c.W) / (2u * uint32_t(c.Wp)));
}
__device__ __forceinline__ int source_y(const DispConst& c, int y) {
    return int((2u * uint32_t(y) + 1u) * uint32_t(c.H) / (2u * uint32_t(c.Hp)));
}

__device__ __forceinline__ void store4(const DispConst& c, uint8_t* __restrict__ panel, int xg, int y,
                                       const uint32_t* px) {
    if (!LFDPR_IN_BOUNDS(uint32_t(y), uint32_t(c.Hp), 21) || !LFDPR_IN_BOUNDS(uint32_t(xg), uint32_t(c.Wp), 21)) return;
    uint8_t* dst = panel + ((uint64_t)y * c.Wp + xg) * 4u;
    if (xg + 4 <= c.Wp && ((reinterpret_cast<uintptr_t>(dst) & 15u) == 0)) {
        *reinterpret_cast<uint4*>(dst) = make_uint4(px[0], px[1], px[2], px[3]);
    } else {
        for (int e = 0; e < 4 && xg + e < c.Wp; e++) reinterpret_cast<uint32_t*>(dst)[e] = px[e];
    }
}

constexpr int kTileThreads = 256, kTentThreads = 128;
constexpr int kTileCols = 4 * kTileThreads;   // panel columns per tile
constexpr int kTentCols = 4 * kTentThreads;
constexpr int kStageCols = 4;                 // 32-column runs of a row segment loaded together

// Rendered views from which a tile is staged run after run of all views, two
// views' loads in flight a warp; fewer leave a warp one view, and its whole segment,
// where it is longer than a run, is loaded in turn (48 views of 1024x768 to 1920x1080: 62.8 us run after run, 71.2
// view after view; 5 of 4000x1000 to 1000x500: 21.8 and 13.8).
constexpr int kTileManyViews = 16;

// The first panel row sampling view row sy; false if none does.
__device__ __forceinline__ bool first_row_of(const DispConst& c, int sy, int& y) {
    y = max(0, int(uint32_t(sy) * uint32_t(c.Hp) / uint32_t(c.H)) - 1);
    while (y < c.Hp && source_y(c, y) < sy) y++;
    return y < c.Hp && source_y(c, y) == sy;
}

// Block (strip bx, view row sy): view pixels sx_lo..sx_lo + n - 1 of row sy
// for every rendered view, then the panel rows whose source row is sy.
// InTurn: view after view. (A kernel for each order: with both in one, at five blocks
// an SM a frame of 61 views of 341x143 took 68.6 us instead of 65.5, and held to six
// one of 65 of 174x182 to a host panel 130.7 instead of 126.6.)
template <bool InTurn>
__global__ void __launch_bounds__(kTileThreads) k_interleave_tile(DispConst c, const uint8_t* __restrict__ views,
                                                                  uint8_t* __restrict__ panel, int cols, int stride) {
    wait_previous_kernel();
    allow_next_kernel();
    extern __shared__ uint32_t s_row[];
    const int sy = blockIdx.y;
    const int x0 = blockIdx.x * cols;
    const int x1 = min(x0 + cols, c.Wp);   // exclusive
    int y;
    if (!first_row_of(c, sy, y)) return;
    const int sx_lo = source_x(c, x0), n = source_x(c, x1 - 1) - sx_lo + 1;
    const uint64_t npix = (uint64_t)c.W * c.H;
    const uint32_t* v32 = reinterpret_cast<const uint32_t*>(views);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kWarps = kTileThreads / 32;
    if constexpr (InTurn) {
        for (int m = warp; m < c.nr; m += kWarps) {
            const uint32_t* src = v32 + (uint64_t)m * npix + (uint64_t)sy * c.W + sx_lo;
            for (int i = lane; i < n; i += 32)
                if (LFDPR_IN_BOUNDS(uint32_t(sx_lo + i), uint32_t(c.W), 20) && LFDPR_IN_BOUNDS(i, stride, 20))
                    s_row[m * stride + i] = __ldg(src + i);
        }
    } else {
        for (int i0 = lane; i0 < n; i0 += 32 * kStageCols)
#pragma unroll 2
            for (int m = warp; m < c.nr; m += kWarps) {
                const uint32_t* src = v32 + (uint64_t)m * npix + (uint64_t)sy * c.W + sx_lo;
#pragma unroll
                for (int q = 0; q < kStageCols; q++) {
                    const int i = i0 + 32 * q;
                    if (i < n && LFDPR_IN_BOUNDS(uint32_t(sx_lo + i), uint32_t(c.W), 20) && LFDPR_IN_BOUNDS(i, stride, 20))
                        s_row[m * stride + i] = __ldg(src + i);
                }
            }
    }
    __syncthreads();
    const int xg = x0 + 4 * threadIdx.x;
    if (xg >= x1) return;
    int sxi[4];
#pragma unroll
    for (int e = 0; e < 4; e++) sxi[e] = min(source_x(c, min(xg + e, x1 - 1)) - sx_lo, n - 1);
    for (; y < c.Hp && source_y(c, y) == sy; y++) {
        uint32_t px[4];
#pragma unroll
        for (int e = 0; e < 4; e++) px[e] = panel_pixel(c, SharedTexels{s_row, stride, sxi[e]}, xg + e, y);
        store4(c, panel, xg, y, px);
    }
}

// The same for tent reconstruction (recon 1). The block stages the display
// views instead of the rendered ones: four times display view k is
// r[2k-1] + 2 r[2k] + r[2k+1], a 10-bit sum per channel, so a pixel's three
// channels fit one word and a subpixel reads one word per display view (three
// with crosstalk) where it read three times as many rendered views and divided
// each sum by its weight. The values are the specified ones exactly: the
// weights 1/4 and 1/2 times bytes add without rounding, a sum of weights of 1
// divides to the sum itself, and the factor 4 is taken back from the crosstalk
// weights (a power of two). Display view 0 has no view before it, so its
// weights sum to 3/4: its quotients are staged as binary32 (4 times each).
// 96 views of 420x560 to a 2560x1600 panel with crosstalk: 0.222 ms reading the
// rendered views' bytes and dividing, 0.049 now (90 MB of views read: 0.014 at
// the copy rate); bound by issue, some 45 instructions a subpixel, and by the
// staging's loads. Blocks of 128 threads: 256 leave fewer blocks to cover each
// other's staging (0.057). Six registers spill to keep ten blocks per SM
// (0.055 without).
__device__ __forceinline__ uint32_t tent_word(uint32_t a, uint32_t b, uint32_t d) {
    const uint32_t m = 0x00ff00ffu;
    const uint32_t e = (a & m) + 2u * (b & m) + (d & m);                                        // channels 0 and 2
    const uint32_t o = ((a >> 8) & 255u) + 2u * ((b >> 8) & 255u) + ((d >> 8) & 255u);   // channel 1
    return (e & 0x3ffu) | (o << 10) | ((e >> 16) << 20);
}
template <bool XT>
__global__ void __launch_bounds__(kTentThreads, 10) k_interleave_tent(DispConst c, const uint8_t* __restrict__ views,
                                                                  uint8_t* __restrict__ panel, int cols, int stride) {
    wait_previous_kernel();
    allow_next_kernel();
    // [1 + n_views + 1][stride] words (view N - 1 again before view 0, and view
    // 0 after view N - 1, as crosstalk wraps), then [3][stride] view 0
    extern __shared__ uint32_t s_tent[];
    const int N = c.n_views;
    float* s_view0 = reinterpret_cast<float*>(s_tent + (N + 2) * stride);
    const int sy = blockIdx.y;
    const int x0 = blockIdx.x * cols;
    const int x1 = min(x0 + cols, c.Wp);   // exclusive
    int y;
    if (!first_row_of(c, sy, y)) return;
    const int sx_lo = source_x(c, x0), n = source_x(c, x1 - 1) - sx_lo + 1;
    const uint64_t npix = (uint64_t)c.W * c.H;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(views) + (uint64_t)sy * c.W + sx_lo;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // a warp takes a run of display views, so that view 2k + 1 serves k + 1 too
    const int k0 = N * warp / (kTentThreads / 32), k1 = N * (warp + 1) / (kTentThreads / 32);
    for (int i0 = lane; i0 < n && k0 < k1; i0 += 32 * kStageCols) {
        const uint32_t* p = src + i0 + (uint64_t)(2 * k0) * npix;
        uint32_t a[kStageCols];
        bool on[kStageCols];
#pragma unroll
        for (int q = 0; q < kStageCols; q++) {
            const int i = i0 + 32 * q;
            on[q] = i < n && LFDPR_IN_BOUNDS(uint32_t(sx_lo + i), uint32_t(c.W), 20) && LFDPR_IN_BOUNDS(i, stride, 20);
            a[q] = on[q] && k0 > 0 ? __ldg(p + 32 * q - npix) : 0u;
        }
#pragma unroll 2
        for (int k = k0; k < k1; k++, p += 2 * npix) {
            uint32_t b[kStageCols], d[kStageCols];
#pragma unroll
            for (int q = 0; q < kStageCols; q++) {
                b[q] = on[q] ? __ldg(p + 32 * q) : 0u;
                d[q] = on[q] ? __ldg(p + 32 * q + npix) : 0u;
            }
#pragma unroll
            for (int q = 0; q < kStageCols; q++) {
                const int i = i0 + 32 * q;
                const uint32_t w = tent_word(a[q], b[q], d[q]);
                if (on[q]) s_tent[(k + 1) * stride + i] = w;
                if (XT && k == N - 1 && on[q]) s_tent[i] = w;
                if (XT && k == 0 && on[q]) s_tent[(N + 1) * stride + i] = w;
                if (k == 0 && on[q])
#pragma unroll
                    for (int ch = 0; ch < 3; ch++)
                        s_view0[ch * stride + i] = 4.0f * __fdiv_rn(0.25f * float((w >> (10 * ch)) & 0x3ffu), 0.75f);
                a[q] = d[q];
            }
        }
    }
    __syncthreads();
    const int xg = x0 + 4 * threadIdx.x;
    if (xg >= x1) return;
    const float xc4 = 0.25f * c.xtalk_c, x4 = 0.25f * c.xtalk;
    const uint32_t pitch = 4u * uint32_t(stride), view0 = uint32_t(N + 2) * pitch;
    // four times the display view in row `at` of the words (column and channel
    // as given, byte offsets); view 0's are the binary32 ones
    auto value4 = [&](uint32_t at, uint32_t col, int ch, bool first) -> float {
        const uint32_t off = first ? view0 + uint32_t(ch) * pitch + col : at;
        const uint32_t w = *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(s_tent) + off);
        // 2^23 + the sum, by its bits
        const float t = __uint_as_float(((w >> (10 * ch)) & 0x3ffu) | 0x4b000000u) - 8388608.0f;
        return first ? __uint_as_float(w) : t;
    };
    uint32_t col[4];
#pragma unroll
    for (int e = 0; e < 4; e++) col[e] = 4u * uint32_t(min(source_x(c, min(xg + e, x1 - 1)) - sx_lo, n - 1));
    for (; y < c.Hp && source_y(c, y) == sy; y++) {
        uint32_t px[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            uint32_t o = 0xff000000u;
#pragma unroll
            for (int ch = 0; ch < 3; ch++) {
                const int k = view_of_subpixel(c, xg + e, y, ch);
                const uint32_t at = col[e] + uint32_t(k) * pitch;   // view k - 1's row
                float val;
                if constexpr (XT) {
                    val = value4(at + pitch, col[e], ch, k == 0) * xc4;
                    val = fmaf(x4, value4(at, col[e], ch, k == (N > 1 ? 1 : 0)), val);
                    val = fmaf(x4, value4(at + 2u * pitch, col[e], ch, k == N - 1), val);
                } else {
                    val = 0.25f * value4(at + pitch, col[e], ch, k == 0);
                }
                // round half to even (0 <= val < 255.5): the low byte of 1.5 2^23 + val
                o |= (__float_as_uint(val + 12582912.0f) & 255u) << (8 * ch);
            }
            px[e] = o;
        }
        store4(c, panel, xg, y, px);
    }
}

__global__ void __launch_bounds__(256) k_interleave(DispConst c, const uint8_t* __restrict__ views,
                                                     uint8_t* __restrict__ panel) {
    wait_previous_kernel();
    allow_next_kernel();
    const uint64_t npix = (uint64_t)c.W * c.H;
    const int groups_x = (c.Wp + 3) >> 2;
    const uint64_t total = (uint64_t)groups_x * c.Hp;
    for (uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total;
         g += (uint64_t)gridDim.x * blockDim.x) {
        const int y = int(g / groups_x);
        const int xg = int(g - (uint64_t)y * groups_x) * 4;
        const int sy = source_y(c, y);
        uint32_t px[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int x = min(xg + e, c.Wp - 1);
            uint64_t pix = (uint64_t)sy * c.W + source_x(c, x);
            if (!LFDPR_IN_BOUNDS(pix, npix, 22)) pix = 0;
            px[e] = panel_pixel(c, GlobalTexels{views, npix, pix}, x, y);
        }
        store4(c, panel, xg, y, px);
    }
}

// Rendered view nearest a on the display-view axis (positions pos[], ties to
// the later view), from the window of four views around it.
__device__ __forceinline__ int nearest_view(const float* pos, int nr, float r, float a) {
    // clamped as binary32: an offset of any size converts to an index
    int lo = int(fminf(fmaxf(floorf(r * a), 0.0f), float(nr))) - 2;
    lo = lo > nr - 4 ? nr - 4 : lo;
    lo = lo < 0 ? 0 : lo;
    const int hi = lo + 3 < nr - 1 ? lo + 3 : nr - 1;
    int m = lo;
    float best = fabsf(pos[lo] - a);
#pragma unroll
    for (int q = 1; q < 4; q++) {
        if (lo + q > hi) break;
        const float dq = fabsf(pos[lo + q] - a);
        if (dq <= best) {
            best = dq;
            m = lo + q;
        }
    }
    return m;
}

// Panel pixel (x, y) under Gaussian reconstruction (+ crosstalk): for each
// channel the mean over the samples of the rendered view nearest phi + dphi
// at the view pixel holding (vx + dx, vy + dy), clamped; with crosstalk the
// same at phi - 1 and phi + 1 (wrapping) mixed in. The samples are the outer
// loop (each sample's pixel is found once); each of the nine sums still adds
// its samples in order.
__device__ __forceinline__ uint32_t gauss_pixel(const DispConst& c, const uint32_t* __restrict__ v32, const float* pos,
                                                const float* smp, int ns, int x, int y, float sxw, float syh) {
    const int nr = c.nr, W = c.W, H = c.H;
    const uint64_t npix = (uint64_t)W * H;
    const float r = float(nr / c.n_views), N = float(c.n_views);
    const float vx = (float(x) + 0.5f) * sxw, vy = (float(y) + 0.5f) * syh;
    const bool xt = c.xtalk > 0.0f;
    float phi[3][3];   // [channel][own, -1, +1]
#pragma unroll
    for (int ch = 0; ch < 3; ch++) {
        const float p0 = subpixel_phase(c, x, y, ch);
        float pm = p0 - 1.0f, pp = p0 + 1.0f;
        if (pm < 0.0f) pm += N;
        if (pp >= N) pp -= N;
        phi[ch][0] = p0;
        phi[ch][1] = pm;
        phi[ch][2] = pp;
    }
    float acc[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
    for (int s = 0; s < ns; s++) {
        int px = int(floorf(vx + smp[3 * s])), py = int(floorf(vy + smp[3 * s + 1]));
        px = px < 0 ? 0 : (px >= W ? W - 1 : px);
        py = py < 0 ? 0 : (py >= H ? H - 1 : py);
        const uint32_t* row = v32 + (uint64_t)py * W + px;
        const float dphi = smp[3 * s + 2];
#pragma unroll
        for (int ch = 0; ch < 3; ch++)
#pragma unroll
            for (int k = 0; k < 3; k++) {
                if (k > 0 && !xt) continue;
                int m = nearest_view(pos, nr, r, phi[ch][k] + dphi);
                if (!LFDPR_IN_BOUNDS(uint32_t(m), uint32_t(nr), 23)) m = 0;
                acc[ch][k] += float((__ldg(row + (uint64_t)m * npix) >> (8 * ch)) & 255u);
            }
    }
    uint32_t o = 0xff000000u;
#pragma unroll
    for (int ch = 0; ch < 3; ch++) {
        float v = acc[ch][0] / float(ns);
        if (xt) {
            float t = v * c.xtalk_c;
            t = fmaf(c.xtalk, acc[ch][1] / float(ns), t);
            t = fmaf(c.xtalk, acc[ch][2] / float(ns), t);
            v = t;
        }
        o |= uint32_t(round_u8(v)) << (8 * ch);
    }
    return o;
}

// The nearest view by a table. On the axis of a = phase + angular offset the
// nearest view changes at the midpoints of neighbouring positions, which lie
// at least a quarter of a view apart (a view stays in its interval of half a
// display view), so a bin an eighth of a view wide holds at most one change:
// view v below a threshold, v + 1 from it on. A search is then one 8-byte
// shared load, a comparison and an addition, instead of four positions loaded
// and compared.
//
// The table gives what nearest_view gives, bit for bit. Its thresholds are
// found with nearest_view itself: the smallest a at which it returns the
// later view, a few floats around the rounded midpoint (near a midpoint the
// rounded distances still move one way each, so the answer changes once).
// That needs neighbouring positions further apart than rounding can confuse:
// where two views around a bin are less than kGaussApart apart (views placed
// on the same border of their intervals), or the few steps do not settle a
// threshold, the block keeps to nearest_view for every pixel.
constexpr int kGaussBins = 8;          // bins per display view
constexpr float kGaussApart = 0x1p-12f;
constexpr int kGaussSteps = 16;
constexpr int kGaussMaxStride = 64;    // largest column stride between a warp's lanes

struct __align__(8) GaussBin {
    float from;       // the next view's bytes start here (+inf: not in this bin)
    uint32_t off;     // byte offset of the bin's first view
};

__host__ __device__ __forceinline__ int gauss_bins(int n_views) { return kGaussBins * (n_views + 2 * kGaussMargin) + 1; }

// Bin b: a in [b / 8 - 4, (b + 1) / 8 - 4). False if it has no single threshold.
__device__ __forceinline__ bool gauss_bin(const float* pos, int nr, float r, int b, uint32_t view_bytes, GaussBin& o) {
    const float lo = float(b) * (1.0f / kGaussBins) - float(kGaussMargin), hi = lo + 1.0f / kGaussBins;
    int m0 = nearest_view(pos, nr, r, lo);
    const int m1 = nearest_view(pos, nr, r, hi);
    if (!LFDPR_IN_BOUNDS(uint32_t(m0), uint32_t(nr), 23) || !LFDPR_IN_BOUNDS(uint32_t(m1), uint32_t(nr), 23)) m0 = m1;
    o.from = INFINITY;
    o.off = uint32_t(m0) * view_bytes;
    bool ok = m1 == m0 || m1 == m0 + 1;
    for (int m = max(m0 - 1, 0); m <= min(m1, nr - 2); m++) ok &= pos[m + 1] - pos[m] >= kGaussApart;
    if (!ok || m1 == m0) return ok;
    float t = 0.5f * (pos[m0] + pos[m1]);   // positive: the positions are apart and not negative
    int step = 0;
    if (nearest_view(pos, nr, r, t) >= m1) {
        for (; step < kGaussSteps; step++) {
            const float q = __uint_as_float(__float_as_uint(t) - 1u);
            if (nearest_view(pos, nr, r, q) < m1) break;
            t = q;
        }
    } else {
        for (; step < kGaussSteps; step++) {
            t = __uint_as_float(__float_as_uint(t) + 1u);
            if (nearest_view(pos, nr, r, t) >= m1) break;
        }
    }
    o.from = t;
    return step < kGaussSteps;
}

// Panel pixel (x, y) as gauss_pixel, its views found in the table (bins, in
// shared memory): the same view bytes, summed as integers (exact, as the sums of at most 32 bytes are in binary32).
// The bin number is floor(8 a) + 32, the low bits of one fma rounded down
// onto 1.5 2^23. mean: 1 / ns where ns is a power of two (the product is then
// the quotient), else 0.
constexpr float kGaussMagic = 12582912.0f;              // 1.5 2^23
constexpr uint32_t kGaussMagicBits = 0x4b400000u;
template <bool XT>
__device__ __forceinline__ uint32_t gauss_pixel_table(const DispConst& c, const uint8_t* __restrict__ views,
                                                      const GaussBin* bins, uint32_t view_bytes, const float4* smp, int ns,
                                                      float mean, int x, int y, float sxw, float syh) {
    constexpr int K = XT ? 3 : 1;
    const int W = c.W, H = c.H;
    const float N = float(c.n_views);
    const float vx = (float(x) + 0.5f) * sxw, vy = (float(y) + 0.5f) * syh;
    float phi[3][K];   // [channel][own, -1, +1]
#pragma unroll
    for (int ch = 0; ch < 3; ch++) {
        const float p0 = subpixel_phase(c, x, y, ch);
        phi[ch][0] = p0;
        if constexpr (XT) {
            float pm = p0 - 1.0f, pp = p0 + 1.0f;
            if (pm < 0.0f) pm += N;
            if (pp >= N) pp -= N;
            phi[ch][1] = pm;
            phi[ch][2] = pp;
        }
    }
    uint32_t acc[3][K];
#pragma unroll
    for (int ch = 0; ch < 3; ch++)
#pragma unroll
        for (int k = 0; k < K; k++) acc[ch][k] = 0u;
    for (int s = 0; s < ns; s++) {
        const float4 q = smp[s];
        int px = int(floorf(vx + q.x)), py = int(floorf(vy + q.y));
        px = px < 0 ? 0 : (px >= W ? W - 1 : px);
        py = py < 0 ? 0 : (py >= H ? H - 1 : py);
        const uint8_t* at = views + 4u * (uint32_t(py) * uint32_t(W) + uint32_t(px));
#pragma unroll
        for (int ch = 0; ch < 3; ch++)
#pragma unroll
            for (int k = 0; k < K; k++) {
                const float a = phi[ch][k] + q.z;
                const uint32_t n = __float_as_uint(__fmaf_rd(a, float(kGaussBins), kGaussMagic + float(kGaussBins * kGaussMargin)));
                const GaussBin b = bins[n - kGaussMagicBits];
                uint32_t off = b.off;
                if (a >= b.from) off += view_bytes;
                uint64_t p;   // at + off in one instruction
                asm("mad.wide.u32 %0, %1, 1, %2;" : "=l"(p) : "r"(off), "l"(at));
                acc[ch][k] += __ldg(reinterpret_cast<const uint8_t*>(p) + ch);
            }
    }
    uint32_t o = 0xff000000u;
#pragma unroll
    for (int ch = 0; ch < 3; ch++) {
        float m[K];
#pragma unroll
        for (int k = 0; k < K; k++)
            m[k] = mean > 0.0f ? float(acc[ch][k]) * mean : __fdiv_rn(float(acc[ch][k]), float(ns));
        float v = m[0];
        if constexpr (XT) {
            float t = v * c.xtalk_c;
            t = fmaf(c.xtalk, m[1], t);
            t = fmaf(c.xtalk, m[2], t);
            v = t;
        }
        o |= uint32_t(round_u8(v)) << (8 * ch);
    }
    return o;
}

// A block's tile is one panel row of 32 S columns; warp w's lanes take columns
// j, j + S, j + 2 S, ... for j = w, w + 8, ... < S. With S a multiple of the
// lens pitch the lanes see the same lens phase, so each gather's 32 bytes lie
// in one view's row, S W / Wp pixels apart: two 128-byte lines for the 48-view
// display (S = 8) instead of the eight views of 32 neighbouring columns, and
// the gathers' lines are what the kernel would otherwise wait for (gauss_stride
// picks S). Blocks take runs of consecutive rows of a column tile, which share
// view rows in L1; a finished row is written from shared memory in order.
// 96 views of 420x560 to a 2560x1600 panel, 8 samples, crosstalk: 0.646 ms with
// four positions compared per search and 32 neighbouring columns a warp, 0.182
// now, bound by issue (two thirds of the slots; 72 searches and gathers of
// about a dozen instructions) and the L1 wavefronts of the gathers (half their
// rate). 64 registers and four blocks per SM: five at 48 registers take 0.195.
// The views' bytes fit 32-bit offsets (gauss_table). Whether every sample's angular
// offset lies within the table's margin is checked here: a captured launch may
// meet other samples than it was recorded with.
constexpr int kGaussThreads = 256;
template <bool XT>
__global__ void __launch_bounds__(kGaussThreads, 4) k_interleave_gauss(DispConst c, const uint8_t* __restrict__ views,
                                                                    const float* __restrict__ pos,
                                                                    const float* __restrict__ samples, int ns,
                                                                    uint8_t* __restrict__ panel, int S, int n_bins) {
    wait_previous_kernel();
    allow_next_kernel();
    extern __shared__ __align__(16) uint8_t s_dyn[];
    GaussBin* s_bins = reinterpret_cast<GaussBin*>(s_dyn);
    uint32_t* s_row = reinterpret_cast<uint32_t*>(s_bins + n_bins);   // [2][32 S] finished rows
    __shared__ float s_pos[kMaxRenderViews];
    __shared__ float s_smp[3 * 32];
    __shared__ float4 s_smp4[32];
    const uint32_t view_bytes = 4u * uint32_t(c.W) * uint32_t(c.H);
    bool slow = false;
    for (int i = threadIdx.x; i < c.nr; i += kGaussThreads) s_pos[i] = pos[i];
    for (int i = threadIdx.x; i < 3 * ns; i += kGaussThreads) s_smp[i] = samples[i];
    for (int i = threadIdx.x; i < ns; i += kGaussThreads) {
        const float4 q = make_float4(samples[3 * i], samples[3 * i + 1], samples[3 * i + 2], 0.0f);
        s_smp4[i] = q;
        slow |= !(fabsf(q.z) <= float(kGaussMargin));
    }
    __syncthreads();
    for (int b = threadIdx.x; b < n_bins; b += kGaussThreads) {
        GaussBin o;
        slow |= !gauss_bin(s_pos, c.nr, float(c.nr / c.n_views), b, view_bytes, o);
        s_bins[b] = o;
    }
    slow = __syncthreads_or(slow);
    const float mean = (ns & (ns - 1)) == 0 ? 1.0f / float(ns) : 0.0f;
    const float sxw = float(c.W) / float(c.Wp), syh = float(c.H) / float(c.Hp);
    const uint32_t* v32 = reinterpret_cast<const uint32_t*>(views);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cols = 32 * S, n_strips = (c.Wp + cols - 1) / cols;
    const uint32_t total = uint32_t(n_strips) * uint32_t(c.Hp);
    // this block's run of rows, strip after strip
    const uint32_t i0 = uint32_t((uint64_t)total * blockIdx.x / gridDim.x);
    const uint32_t i1 = uint32_t((uint64_t)total * (blockIdx.x + 1u) / gridDim.x);
    uint32_t* row = s_row;
    for (uint32_t i = i0; i < i1; i++, row = row == s_row ? s_row + cols : s_row) {
        const int strip = int(i / uint32_t(c.Hp)), y = int(i - uint32_t(strip) * uint32_t(c.Hp));
        const int x0 = strip * cols;
        for (int j = warp; j < S; j += kGaussThreads / 32) {
            const int x = x0 + j + S * lane;
            if (x >= c.Wp) continue;
            bool exact = slow;   // (a phase is no number where slant or pitch overflow)
#pragma unroll
            for (int ch = 0; ch < 3; ch++) {
                const float p0 = subpixel_phase(c, x, y, ch);
                exact |= !(p0 >= 0.0f && p0 <= float(c.n_views));
            }
            row[j + S * lane] = exact ? gauss_pixel(c, v32, s_pos, s_smp, ns, x, y, sxw, syh)
                                      : gauss_pixel_table<XT>(c, views, s_bins, view_bytes, s_smp4, ns, mean, x, y, sxw, syh);
        }
        __syncthreads();   // the row is complete; the other buffer's readers are past their barrier
        uint32_t* dst = reinterpret_cast<uint32_t*>(panel) + (uint64_t)y * c.Wp + x0;
        for (int q = threadIdx.x; q < cols && x0 + q < c.Wp; q += kGaussThreads) dst[q] = row[q];
    }
}

// The same a thread a pixel, each search among four positions: where a table's
// making costs more than it saves, for views beyond its 32-bit offsets and for
// angular offsets beyond its margin (gauss_table).
__global__ void __launch_bounds__(kGaussThreads) k_interleave_gauss_plain(DispConst c, const uint8_t* __restrict__ views,
                                                                          const float* __restrict__ pos,
                                                                          const float* __restrict__ samples, int ns,
                                                                          uint8_t* __restrict__ panel) {
    wait_previous_kernel();
    allow_next_kernel();
    __shared__ float s_pos[kMaxRenderViews];
    __shared__ float s_smp[3 * 32];
    for (int i = threadIdx.x; i < c.nr; i += kGaussThreads) s_pos[i] = pos[i];
    for (int i = threadIdx.x; i < 3 * ns; i += kGaussThreads) s_smp[i] = samples[i];
    __syncthreads();
    const uint64_t total = (uint64_t)c.Wp * c.Hp;
    const float sxw = float(c.W) / float(c.Wp), syh = float(c.H) / float(c.Hp);
    const uint32_t* v32 = reinterpret_cast<const uint32_t*>(views);
    for (uint64_t i = (uint64_t)blockIdx.x * kGaussThreads + threadIdx.x; i < total; i += (uint64_t)gridDim.x * kGaussThreads) {
        const int y = int(i / c.Wp), x = int(i - (uint64_t)y * c.Wp);
        reinterpret_cast<uint32_t*>(panel)[i] = gauss_pixel(c, v32, s_pos, s_smp, ns, x, y, sxw, syh);
    }
}

// Whether the table pays. Every block makes it, bins / 256 of them a thread with
// several searches each, and it saves most of a search per look-up: of a thread's
// look-ups, 3 a pixel and sample (9 with crosstalk) for at least one pixel. 256
// views to a panel of 256x256, one sample: 5.2 us a thread a pixel, 10.6 with the
// table; of 32 samples 28.9 and 14.6. 96 views to 512x512: one sample 6.9 and 10.1,
// four 13.4 and 11.9. near: every sample's angular offset lies within the table's
// margin (beyond it the kernel would search as the plain one does, a fifth slower).
bool gauss_table(const DispConst& c, int ns, bool near, int sms) {
    if (!near || (uint64_t)c.nr * c.W * c.H * 4u > 0xffffffffull) return false;
    const double pixels = std::max(1.0, double(c.Wp) * c.Hp / (4.0 * kGaussThreads * sms));
    return pixels * ns * (c.xtalk > 0.0f ? 9.0 : 3.0) > 3.2 * gauss_bins(c.n_views) / kGaussThreads;
}

// The column stride between a warp's lanes: of the multiples of 8 (one warp
// of the block per column between) the one whose gathers touch the fewest
// lines, counting up to the strip's width past the panel as work. A gather's
// lines are estimated from the lanes' views (the stride in lens periods) and
// columns; below three lines the kernel no longer waits for them.
int gauss_stride(const DispConst& c) {
    int best = 8;
    double least = 1e30;
    for (int S = 8; S <= kGaussMaxStride; S += 8) {
        int lines = 0;
        int last_view = -1, last_line = -1;
        for (int l = 0; l < 32; l++) {
            const double ph = double(l) * S * double(c.inv_pitch);
            // half a view up, so that a stride of whole periods stays in one view whatever its
            // rounding; no number where the pitch's reciprocal overflows
            const int view = std::isfinite(ph) ? int((ph - std::floor(ph)) * c.nr + 0.5) % c.nr : 0;
            const int line = int(double(l) * S * c.W / c.Wp) / 32;
            lines += view != last_view || line != last_line;
            last_view = view;
            last_line = line;
        }
        const int cols = 32 * S;
        const double cost = std::max(3, lines) * (double((c.Wp + cols - 1) / cols) * cols / c.Wp);
        if (cost < least) {
            least = cost;
            best = S;
        }
    }
    return best;
}

// Whether the tent's tiles, of `bytes` of shared memory and `blocks` in all, are
// faster than the direct gather. The tiles stage every rendered view's rows,
// whatever share of them the panel shows: they pay with the panel pixels per view
// pixel staged, and with the blocks that an SM holds to cover each other's staging
// (128 threads each, 10 at most); less where a staged row feeds one panel row.
// Over seventeen pairs of view and panel sizes and 1 to 256 views, tiles against
// gather: with crosstalk (nine views a pixel to gather instead of three) 48 views
// of 420x560 to 2560x1600 46 against 172 us, 128 123 against 179, 200 280 against
// 186, 96 of 333x251 to 1277x719 45 against 36; without, 48 39 against 68, 96 90
// against 73, 256 466 against 76, 48 of 640x480 to 640x480 108 against 11. At the
// lines they are mostly within a fifth of each other. Without crosstalk a panel of
// few tiles (100x50 to 400x2000) is left to the gather too, 12.7 against 15.8.
bool tent_pays(const DispConst& c, int64_t bytes, int64_t blocks, int sms, int smem_sm) {
    const double shown = double(c.Wp) * c.Hp / (double(c.nr) * c.W * std::min(c.H, c.Hp));
    const double resident = double(std::min<int64_t>(10, smem_sm / (bytes + 1024)));
    const bool xt = c.xtalk > 0.0f;
    const double line = c.Hp > c.H ? (xt ? 1.25 : 7.9) : (xt ? 15.0 : 60.0);
    return shown * resident * resident >= line && (xt || 2 * blocks >= sms);
}

}  // namespace

namespace {

// One 2 x 2 box of RGBA8 texels: (a + b + c + d + 2) >> 2 per channel, two
// channels at a time in 16-bit fields (a sum is at most 1022).
__device__ __forceinline__ uint32_t box4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    constexpr uint32_t m = 0x00ff00ffu, half = 0x00020002u;
    const uint32_t even = ((a & m) + (b & m) + (c & m) + (d & m) + half) >> 2;
    const uint32_t odd = ((a >> 8 & m) + (b >> 8 & m) + (c >> 8 & m) + (d >> 8 & m) + half) >> 2;
    return (even & m) | (odd & m) << 8;
}

// Mip level L (1 or 2) of every rendered view (Sec. 5.1: with spatial
// supersampling a mipmap of each view is built): L times the 2 x 2 box of the
// level above, with the texture mips' rounding. W and H are multiples of 2^L, so
// the views stack to one image of nr H rows, and row r of all views' level L comes
// from its rows 2^L r on: no view or row index is divided out. A warp takes a
// stretch of a row, kMipTexels texels a lane 32 apart, and has the 2^L vector loads
// of each in flight together. Bound by DRAM: level 1 of 96 views of 840x1120 122 us
// with a thread a texel (two 64-bit divisions each), about 67 now (451 MB; a copy of
// as much takes 66); with four texels a lane 72, with eight 68.
constexpr int kMipTexels = 2;
template <int L>
__global__ void __launch_bounds__(256) k_view_mip(const uint8_t* __restrict__ src, uint32_t W, uint32_t H,
                                                  uint32_t nr, uint8_t* __restrict__ dst) {
    wait_previous_kernel();
    allow_next_kernel();
    constexpr int K = 1 << L, T = kMipTexels / L;
    using Vec = typename std::conditional<L == 1, uint2, uint4>::type;
    const uint32_t wl = W >> L, hl = H >> L, segs = (wl + 32u * T - 1u) / (32u * T);
    const uint64_t rows = (uint64_t)hl * nr, tasks = rows * segs, warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    const uint32_t lane = threadIdx.x & 31u;
    uint64_t task = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    // row and stretch of the task, and their steps to the warp's next one
    uint64_t r = task / segs;
    uint32_t seg = uint32_t(task - r * segs);
    const uint64_t dr = warps / segs;
    const uint32_t dseg = uint32_t(warps - dr * segs);
    for (; task < tasks; task += warps) {
        const uint32_t* base = reinterpret_cast<const uint32_t*>(src) + r * K * W;
        uint32_t* out = reinterpret_cast<uint32_t*>(dst) + r * wl;
        Vec q[T][K];
        bool ok[T];
#pragma unroll
        for (int k = 0; k < T; k++) {
            const uint32_t x = (seg * T + k) * 32u + lane;
            ok[k] = x < wl && LFDPR_IN_BOUNDS((r * K + K - 1) * W + x * K + K - 1, (uint64_t)W * H * nr, 24);
            if (ok[k]) {
#pragma unroll
                for (int dy = 0; dy < K; dy++)
                    q[k][dy] = __ldg(reinterpret_cast<const Vec*>(base + (uint64_t)dy * W) + x);
            }
        }
#pragma unroll
        for (int k = 0; k < T; k++) {
            if (!ok[k]) continue;
            const uint32_t x = (seg * T + k) * 32u + lane;
            uint32_t v;
            if constexpr (L == 1) {
                v = box4(q[k][0].x, q[k][0].y, q[k][1].x, q[k][1].y);
            } else {
                v = box4(box4(q[k][0].x, q[k][0].y, q[k][1].x, q[k][1].y),
                         box4(q[k][0].z, q[k][0].w, q[k][1].z, q[k][1].w),
                         box4(q[k][2].x, q[k][2].y, q[k][3].x, q[k][3].y),
                         box4(q[k][2].z, q[k][2].w, q[k][3].z, q[k][3].w));
            }
            out[x] = v;
        }
        r += dr;
        seg += dseg;
        if (seg >= segs) {
            seg -= segs;
            r++;
        }
    }
}

}  // namespace

LFDPR_CHECK_READER(checks_interleave)

void prefer_view_mip_split() {
    for (const void* k : {reinterpret_cast<const void*>(k_view_mip<1>), reinterpret_cast<const void*>(k_view_mip<2>)})
        if (cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, kViewsSplit) != cudaSuccess)
            cudaGetLastError();
}

cudaError_t launch_view_mip(const uint8_t* views, int W, int H, int nr, int level, uint8_t* out, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (level == 1)
        return launch_after_previous(k_view_mip<1>, dim3(sms * 8), dim3(256), 0, s, views, uint32_t(W), uint32_t(H),
                                     uint32_t(nr), out);
    if (level == 2)
        return launch_after_previous(k_view_mip<2>, dim3(sms * 8), dim3(256), 0, s, views, uint32_t(W), uint32_t(H),
                                     uint32_t(nr), out);
    return cudaErrorInvalidValue;
}

cudaError_t launch_interleave(const DispConst& dc, const uint8_t* views, const float* pos, const float* samples,
                              int n_samples, bool near, uint8_t* panel, cudaStream_t s) {
    int dev = 0, sms = 0, smem_max = 0, smem_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (dc.recon == 2 || dc.recon == 3) {
        if (n_samples < 1 || n_samples > 32) return cudaErrorInvalidValue;
        if (!gauss_table(dc, n_samples, near, sms))
            return launch_after_previous(k_interleave_gauss_plain, dim3(sms * 16), dim3(kGaussThreads), 0, s, dc, views, pos,
                                         samples, n_samples, panel);
        const int S = gauss_stride(dc);
        const int bins = gauss_bins(dc.n_views);
        const size_t bytes = sizeof(GaussBin) * bins + 2u * 32u * S * 4u;
        const uint64_t rows = (uint64_t)((dc.Wp + 32 * S - 1) / (32 * S)) * dc.Hp;
        const int grid = int(std::min<uint64_t>(rows, uint64_t(sms) * 4u));
        return launch_after_previous(dc.xtalk > 0.0f ? k_interleave_gauss<true> : k_interleave_gauss<false>, dim3(grid),
                                     dim3(kGaussThreads), bytes, s, dc, views, pos, samples, n_samples, panel, S, bins);
    }
    // the widest source segment of a strip: (cols - 1) W / Wp + 2 pixels
    const bool tent = dc.recon == 1;
    const int cols = tent ? kTentCols : kTileCols;
    const int64_t seg = ((int64_t)(cols - 1) * dc.W) / dc.Wp + 2;
    const int64_t words = tent ? dc.n_views + 5 : dc.nr, bytes = words * seg * 4;
    const dim3 tiles((dc.Wp + cols - 1) / cols, dc.H);
    if (bytes <= smem_max / 2 && (!tent || tent_pays(dc, bytes, int64_t(tiles.x) * tiles.y, sms, smem_sm))) {
        const bool in_turn = dc.nr < kTileManyViews && seg > 32 * kStageCols + 1;
        const auto kernel = !tent            ? in_turn ? k_interleave_tile<true> : k_interleave_tile<false>
                            : dc.xtalk > 0.0f ? k_interleave_tent<true>
                                              : k_interleave_tent<false>;
        // the most that a tile takes, not this one's: another thread's tile may need more
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max / 2);
        if (e != cudaSuccess) return e;
        return launch_after_previous(kernel, tiles, dim3(tent ? kTentThreads : kTileThreads), size_t(bytes), s, dc, views,
                                     panel, cols, int(seg));
    }
    return launch_after_previous(k_interleave, dim3(sms * 8), dim3(256), 0, s, dc, views, panel);
}

}  // namespace lfdpr
