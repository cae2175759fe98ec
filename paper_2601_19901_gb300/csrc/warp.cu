// Depth-guided warp of rendered views to other eyes on the display's eye
// line: the base the learned angular reconstruction refines.
//
// Every eye lies on the line y = 0, z = D, and every view looks through the
// same focal rectangle at z = 0, so a surface point keeps its pixel row in
// every view and only moves along it. A point that view a sees at pixel
// centre x + 1/2 with ray parameter t (the depth key's high word; its depth
// is D (1 - t), the same t from every eye) is seen from eye E at
//     x + 1/2 + (1 - 1/t) (W / fw) (E - E_a)
// (the disparity of project_point: B = (1 - D / (D - z)) W / fw). For an
// output eye E between input eyes E_0 <= E <= E_1 (weight s = (E - E_0) /
// (E_1 - E_0) towards the second):
//  1. Forward: each input pixel of the row holding a depth key moves to E
//     and is kept at pixel floor(x'), the nearest point winning (smallest t,
//     then the first input, then the leftmost source pixel).
//  2. Backward: a pixel with a winner finds the point's position in each of
//     the two inputs and interpolates that input's row linearly there. An
//     input agrees if its own key at the pixel holding that position has a
//     t within 1 % of the winner's. The agreeing inputs are blended with
//     weights (1 - s, s), renormalised (times the reciprocal of their sum);
//     with none agreeing, the winner's own
//     source pixel is taken. A pixel with no winner (disoccluded, or beyond
//     every input's reach) takes the unshifted blend (1 - s) c_0 + s c_1.
// Colours are rounded half to even to 8 bits; alpha is 255. All arithmetic is
// binary32, one rounding per written operation (no contraction), so a plain
// CPU restatement gives the same bytes.
#include <algorithm>
#include <cmath>

#include "lfdpr_recon.h"
#include "objects.h"

namespace lfdpr {
namespace {

constexpr int kWarpThreads = 256;   // at most; see warp_threads
constexpr int kWarpViews = 4;       // output views a block takes at a time, at most
constexpr int kWarpPad = 4;         // pixels repeated before and after a staged row
constexpr uint64_t kNoKey = ~0ull;

struct WarpArgs {
    const uint8_t* views;     // [nin][H][W][4] RGBA8
    const uint64_t* keys;     // [nin][H][W] depth keys (t bits << 32 | point), all ones where empty
    const float* in_eyes;     // [nin] ascending
    const float* out_eyes;    // [nout]
    int nin, nout, W, H;
    float ipw;                // W / fw: view pixels per unit of x on the focal plane
    uint8_t* out;             // [nout][H][W][4] RGBA8
};

__device__ __forceinline__ bool key_depth(uint64_t key, float& t) {
    t = __uint_as_float(uint32_t(key >> 32));
    return key != kNoKey && t > 0.0f && isfinite(t);
}

__device__ __forceinline__ float channel(uint32_t rgba, int c) { return float((rgba >> (8 * c)) & 255u); }

// The input bracket of output eye E: j0 the last input eye at or before E
// (clamped to [0, nin - 2]), s the weight towards input j0 + 1.
__device__ __forceinline__ int bracket(const WarpArgs& a, float E, float& s) {
    int j0 = 0;
    for (int j = 0; j < a.nin; j++)
        if (a.in_eyes[j] <= E) j0 = j;
    j0 = min(j0, a.nin - 2);
    const float e0 = a.in_eyes[j0], e1 = a.in_eyes[j0 + 1];
    s = e1 > e0 ? (E - e0) / (e1 - e0) : 0.0f;
    s = fminf(fmaxf(s, 0.0f), 1.0f);
    return j0;
}

// Views an interval block takes at a time, for view width W.
__host__ __device__ __forceinline__ int views_per_pass(int W) {
    const int v = 32768 / (8 * W);
    return v < 1 ? 1 : (v > kWarpViews ? kWarpViews : v);
}

// A staged row: its W pixels with the first and last repeated, so that the
// clamped positions below need no clamp on the index.
__host__ __device__ __forceinline__ int row_stride(int W) { return W + 2 * kWarpPad + 1; }

// Threads of a block: a row is swept in as many steps as 256 threads need, by
// as few warps as do it in that many (420 pixels: two steps of 224).
int warp_threads(int W) {
    const int steps = (W + kWarpThreads - 1) / kWarpThreads;
    return ((W + steps - 1) / steps + 31) / 32 * 32;
}

// A block takes (row y, input interval j) pairs, a grid's stride apart: every
// output view whose bracket is (j, j + 1), up to views_per_pass(W) of them at
// a time. The two input rows are staged in shared memory with each pixel's
// colour as binary32, its t and its disparity factor g = (1 - 1/t) W / fw
// (both NaN where it has no key). The nearest point per output pixel is the
// 64-bit minimum of (t bits, input, source pixel); a minimum is cleared for
// the next pass by the thread that has read it.
//
// Bound by issue and, beside the network's layers, by shared memory. Each
// pixel's two positions are floored by one addition rounded down onto 1.5 2^23
// (its low bits are the index), not by conversions (a quarter of the rate);
// the pixel holding a position follows from the fraction, and its t lies
// beside its colour; the rows' repeated ends take the place of index clamps;
// the reciprocal of the summed weights takes one of three values a view; a
// source pixel is read once for all views of a pass.
// 12 views of 420x560 to 48, alone, a block per pair: 0.117 -> 0.107 ms (117 M
// -> 82 M warp instructions). Beside the layers the blocks last, two per SM on
// shared memory that the layers leave free, the next pair's rows asked of L1:
// the forward pass takes 0.283 ms there, 0.242 without the warp (0.353 while
// the SMs' split between L1 and shared memory kept the two apart), and 0.156 ms
// against 0.149 at 333x251. The minimum as two 32-bit ones in two sweeps took
// 0.128 alone, and blocks of twice the threads 0.121.
__global__ void __launch_bounds__(kWarpThreads) k_warp_views(WarpArgs a) {
    extern __shared__ __align__(16) uint8_t s_raw[];
    const int W = a.W, V = views_per_pass(W), WS = row_stride(W);
    float4* s_px = reinterpret_cast<float4*>(s_raw);                        // [2][WS] colour, t
    float* s_g = reinterpret_cast<float*>(s_px + 2 * WS);                   // [2][WS] g
    unsigned long long* s_win = reinterpret_cast<unsigned long long*>(s_g + 2 * WS);   // [V][W] nearest point
    int* s_views = reinterpret_cast<int*>(s_win + size_t(V) * W);           // [nout] output views, interval by interval
    float* s_w = reinterpret_cast<float*>(s_views + a.nout);                // [nout] their weights
    float* s_E = s_w + a.nout;                                              // [nout] and eyes
    int* s_first = reinterpret_cast<int*>(s_E + a.nout);                    // [nin] first view of each interval, and the end
    const int step = blockDim.x, tid = threadIdx.x;
    const size_t npix = size_t(W) * a.H;
    const int n_intervals = a.nin - 1;

    // the output views sorted by interval
    for (int j = threadIdx.x; j <= n_intervals; j += blockDim.x) s_first[j] = 0;
    for (int q = threadIdx.x; q < V * W; q += blockDim.x) s_win[q] = kNoKey;
    __syncthreads();
    for (int k = threadIdx.x; k < a.nout; k += blockDim.x) {
        float s;
        atomicAdd(&s_first[bracket(a, a.out_eyes[k], s) + 1], 1);
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int j = 1; j <= n_intervals; j++) s_first[j] += s_first[j - 1];
    __syncthreads();
    // placed from each interval's end: s_first[j + 1] counts down to its first view
    for (int k = threadIdx.x; k < a.nout; k += blockDim.x) {
        float s;
        const float E = a.out_eyes[k];
        const int m = atomicSub(&s_first[bracket(a, E, s) + 1], 1) - 1;
        s_views[m] = k;
        s_w[m] = s;
        s_E[m] = E;
    }
    __syncthreads();
    // now interval j's views are [s_first[j + 1], s_first[j + 2]), the last's up to nout

    constexpr float kMagic = 12582912.0f;   // 1.5 2^23
    constexpr uint32_t kMagicBits = 0x4b400000u;
    const int total = a.H * n_intervals;
    for (int it = blockIdx.x; it < total; it += gridDim.x) {
        const int y = it / n_intervals, j = it - y * n_intervals;
        const size_t row = size_t(y) * W;
        const int first = s_first[j + 1], n_views = (j + 1 < n_intervals ? s_first[j + 2] : a.nout) - first;
        if (n_views == 0) continue;
#pragma unroll
        for (int src = 0; src < 2; src++) {
            const size_t o = size_t(j + src) * npix + row;
            for (int i = tid; i < WS; i += step) {
                const int x = min(max(i - kWarpPad, 0), W - 1);
                const uint32_t c = reinterpret_cast<const uint32_t*>(a.views)[o + x];
                float t;
                const bool ok = key_depth(a.keys[o + x], t);
                const float nan = __int_as_float(0x7fc00000);   // no key
                s_px[src * WS + i] = make_float4(channel(c, 0), channel(c, 1), channel(c, 2), ok ? t : nan);
                s_g[src * WS + i] = ok ? (1.0f - 1.0f / t) * a.ipw : nan;
            }
        }
        {   // the next pair's rows
            const int nx = it + gridDim.x;
            if (nx < total) {
                const int yn = nx / n_intervals, jn = nx - yn * n_intervals;
                for (int src = 0; src < 2; src++) {
                    const size_t o = size_t(jn + src) * npix + size_t(yn) * W;
                    for (int i = 16 * tid; i < W; i += 16 * step) prefetch_l1(a.keys + o + i);
                    for (int i = 32 * tid; i < W; i += 32 * step) prefetch_l1(a.views + 4 * (o + i));
                }
            }
        }
        __syncthreads();
        const float eye[2] = {a.in_eyes[j], a.in_eyes[j + 1]};
        for (int m0 = first; m0 < first + n_views; m0 += V) {
            const int nv = min(V, first + n_views - m0);
            // 1. forward: the nearest point landing on each pixel (t, then input,
            // then source pixel). A pixel without a key has g = NaN, and a
            // position that is no number lies in no row.
#pragma unroll
            for (int src = 0; src < 2; src++)
                for (int i = tid; i < W; i += step) {
                    const float g = s_g[src * WS + kWarpPad + i], t = s_px[src * WS + kWarpPad + i].w;
                    const float centre = float(i) + 0.5f;
                    const uint64_t key = (uint64_t(__float_as_uint(t)) << 32) | (uint64_t(src) << 16) | uint64_t(i);
#pragma unroll
                    for (int m = 0; m < kWarpViews; m++) {
                        if (m >= nv) break;
                        const float X = centre + g * (s_E[m0 + m] - eye[src]);
                        if (X >= 0.0f && X < float(W))
                            atomicMin(&s_win[m * W + int(__float_as_uint(__fadd_rd(X, kMagic)) - kMagicBits)], key);
                    }
                }
            __syncthreads();
            // 2. backward: every output pixel of the pass's views
            for (int m = 0; m < nv; m++) {
                const int k = s_views[m0 + m];
                const float E = s_E[m0 + m], s = s_w[m0 + m], s1 = 1.0f - s;
                // the reciprocal of the weights' sum where both inputs agree, the first, the second
                const float both = s1 + s;
                const float rb = both > 0.0f ? 1.0f / both : 0.0f, r0 = s1 > 0.0f ? 1.0f / s1 : 0.0f,
                            r1 = s > 0.0f ? 1.0f / s : 0.0f;
                const float shift[2] = {eye[0] - E, eye[1] - E};
                uint32_t* out = reinterpret_cast<uint32_t*>(a.out) + size_t(k) * npix + row;
                for (int p = tid; p < W; p += step) {
                    const uint64_t w = s_win[m * W + p];
                    s_win[m * W + p] = kNoKey;
                    float v[3];
                    if (w == kNoKey) {
                        const float4 c0 = s_px[kWarpPad + p], c1 = s_px[WS + kWarpPad + p];
                        v[0] = s1 * c0.x + s * c1.x;
                        v[1] = s1 * c0.y + s * c1.y;
                        v[2] = s1 * c0.z + s * c1.z;
                    } else {
                        const int from = (uint32_t(w) >> 16 ? WS : 0) + kWarpPad + int(uint32_t(w) & 0xffffu);
                        const float t = __uint_as_float(uint32_t(w >> 32)), g = s_g[from];
                        const float tol = 0.01f * t;
                        float4 vs[2];
                        bool agree[2];
#pragma unroll
                        for (int src = 0; src < 2; src++) {
                            const float xa = ((float(p) + 0.5f) + g * shift[src]) - 0.5f;
                            // a position beyond the row's ends reads the end pixel: both
                            // neighbours are that pixel there, whatever the fraction
                            const float q = __fadd_rd(fminf(fmaxf(xa, -float(kWarpPad)), float(W + kWarpPad - 1)), kMagic);
                            const float fr = xa - (q - kMagic);
                            const int i0 = src * WS + kWarpPad + int(__float_as_uint(q) - kMagicBits);
                            const float4 ca = s_px[i0], cb = s_px[i0 + 1];
                            vs[src] = make_float4(ca.x + fr * (cb.x - ca.x), ca.y + fr * (cb.y - ca.y),
                                                  ca.z + fr * (cb.z - ca.z), 0.0f);
                            // the pixel holding the position: the second neighbour from the
                            // half on (no key there: NaN)
                            agree[src] = fabsf((fr >= 0.5f ? cb.w : ca.w) - t) <= tol;
                        }
                        const float w0 = agree[0] ? s1 : 0.0f, w1 = agree[1] ? s : 0.0f;
                        if (w0 + w1 > 0.0f) {
                            const float rw = agree[0] ? (agree[1] ? rb : r0) : r1;
                            v[0] = (w0 * vs[0].x + w1 * vs[1].x) * rw;
                            v[1] = (w0 * vs[0].y + w1 * vs[1].y) * rw;
                            v[2] = (w0 * vs[0].z + w1 * vs[1].z) * rw;
                        } else {
                            const float4 cs = s_px[from];
                            v[0] = cs.x;
                            v[1] = cs.y;
                            v[2] = cs.z;
                        }
                    }
                    // blends of bytes: at most 255 up to rounding (a NaN counts as 0);
                    // rounded half to even by the low bits of 1.5 2^23 + v
                    uint32_t o = 0xff000000u;
#pragma unroll
                    for (int c = 0; c < 3; c++)
                        o |= (__float_as_uint(fmaxf(v[c], 0.0f) + kMagic) & 255u) << (8 * c);
                    out[p] = o;
                }
            }
            __syncthreads();   // this pass's minima are cleared, and the rows read
        }
    }
}

// The same for rows of few pixels and calls of few views a row (see warp_rows): a
// block per (row y, input interval j). Its 256 threads sweep (view, pixel) pairs
// of a pass as one range, so that a short row leaves none idle, and it picks its
// own interval's views out of all instead of sorting them.
constexpr int kMaxRowsWidth = 512;   // 39 KB of shared memory
__global__ void __launch_bounds__(kWarpThreads) k_warp_rows(WarpArgs a) {
    extern __shared__ __align__(16) uint8_t s_raw[];
    const int y = blockIdx.x, j = blockIdx.y, W = a.W, V = views_per_pass(W);
    float4* s_px = reinterpret_cast<float4*>(s_raw);                        // [2][W] colour, t
    float* s_g = reinterpret_cast<float*>(s_px + 2 * W);                    // [2][W] g
    unsigned long long* s_win = reinterpret_cast<unsigned long long*>(s_g + 2 * W);   // [V][W] nearest point
    __shared__ int s_views[kMaxRenderViews];
    __shared__ float s_w[kMaxRenderViews], s_E[kMaxRenderViews];
    __shared__ int s_n;
    if (threadIdx.x == 0) s_n = 0;
    const size_t npix = size_t(W) * a.H, row = size_t(y) * W;
    for (int q = threadIdx.x; q < 2 * W; q += kWarpThreads) {
        const int src = q >= W, i = q - src * W;
        const size_t o = size_t(j + src) * npix + row + i;
        const uint32_t c = reinterpret_cast<const uint32_t*>(a.views)[o];
        float t;
        const bool ok = key_depth(a.keys[o], t);
        const float nan = __int_as_float(0x7fc00000);   // no key
        s_px[q] = make_float4(channel(c, 0), channel(c, 1), channel(c, 2), ok ? t : nan);
        s_g[q] = ok ? (1.0f - 1.0f / t) * a.ipw : nan;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < a.nout; k += kWarpThreads) {
        float s;
        const float E = a.out_eyes[k];
        if (bracket(a, E, s) == j) {
            const int m = atomicAdd(&s_n, 1);
            s_views[m] = k;
            s_w[m] = s;
            s_E[m] = E;
        }
    }
    __syncthreads();
    const int n_views = s_n;
    const float eye[2] = {a.in_eyes[j], a.in_eyes[j + 1]};
    // (m, r) -> (m, r + step) over rows of length L
    auto advance = [](int& m, int& r, int step, int L) {
        r += step;
        while (r >= L) {
            r -= L;
            m++;
        }
    };
    for (int m0 = 0; m0 < n_views; m0 += V) {
        const int nv = min(V, n_views - m0);
        for (int q = threadIdx.x; q < nv * W; q += kWarpThreads) s_win[q] = kNoKey;
        __syncthreads();
        // 1. forward
        int m = 0, r = threadIdx.x;
        for (advance(m, r, 0, 2 * W); m < nv; advance(m, r, kWarpThreads, 2 * W)) {
            const int src = r >= W, i = r - src * W;
            const float X = (float(i) + 0.5f) + s_g[r] * (s_E[m0 + m] - eye[src]);
            if (X >= 0.0f && X < float(W))
                atomicMin(&s_win[m * W + int(X)],
                          (uint64_t(__float_as_uint(s_px[r].w)) << 32) | (uint64_t(src) << 16) | uint64_t(i));
        }
        __syncthreads();
        // 2. backward
        m = 0;
        r = threadIdx.x;
        for (advance(m, r, 0, W); m < nv; advance(m, r, kWarpThreads, W)) {
            const float E = s_E[m0 + m], s = s_w[m0 + m], s1 = 1.0f - s;
            const uint64_t w = s_win[m * W + r];
            float v[3];
            if (w == kNoKey) {
                const float4 c0 = s_px[r], c1 = s_px[W + r];
                v[0] = s1 * c0.x + s * c1.x;
                v[1] = s1 * c0.y + s * c1.y;
                v[2] = s1 * c0.z + s * c1.z;
            } else {
                const int from = (uint32_t(w) >> 16 ? W : 0) + int(uint32_t(w) & 0xffffu);
                const float t = __uint_as_float(uint32_t(w >> 32)), g = s_g[from];
                float4 vs[2];
                float wt[2];
#pragma unroll
                for (int src = 0; src < 2; src++) {
                    const float X = (float(r) + 0.5f) + g * (eye[src] - E), xa = X - 0.5f;
                    const float fl = floorf(xa), fr = xa - fl;
                    const int i0 = int(fminf(fmaxf(fl, 0.0f), float(W - 1)));
                    const int i1 = int(fminf(fmaxf(fl + 1.0f, 0.0f), float(W - 1)));
                    const int n = int(fminf(fmaxf(floorf(X), 0.0f), float(W - 1)));
                    const float4 ca = s_px[src * W + i0], cb = s_px[src * W + i1];
                    vs[src] = make_float4(ca.x + fr * (cb.x - ca.x), ca.y + fr * (cb.y - ca.y),
                                          ca.z + fr * (cb.z - ca.z), 0.0f);
                    const bool agree = fabsf(s_px[src * W + n].w - t) <= 0.01f * t;   // (no key there: NaN)
                    wt[src] = agree ? (src == 0 ? s1 : s) : 0.0f;
                }
                const float ws = wt[0] + wt[1];
                if (ws > 0.0f) {
                    const float rw = 1.0f / ws;
                    v[0] = (wt[0] * vs[0].x + wt[1] * vs[1].x) * rw;
                    v[1] = (wt[0] * vs[0].y + wt[1] * vs[1].y) * rw;
                    v[2] = (wt[0] * vs[0].z + wt[1] * vs[1].z) * rw;
                } else {
                    const float4 cs = s_px[from];
                    v[0] = cs.x;
                    v[1] = cs.y;
                    v[2] = cs.z;
                }
            }
            uint32_t o = 0xff000000u;
#pragma unroll
            for (int c = 0; c < 3; c++) o |= uint32_t(rintf(fminf(fmaxf(v[c], 0.0f), 255.0f))) << (8 * c);
            reinterpret_cast<uint32_t*>(a.out)[size_t(s_views[m0 + m]) * npix + row + r] = o;
        }
        __syncthreads();   // this pass's views are done with the minima
    }
}

// Whether a call of its own takes k_warp_rows: rows that leave k_warp_views' threads
// idle, or so few output views an interval that its sorting of them is most of the
// work. 64x64, 2 input views to 300 output views 114 us against 254, to 8 8.4 against
// 12.5; 160x120, 2 to 300 191 against 263, 4 to 48 17.6 against 20.6; 256x256, 48 to
// 48 51 against 85, 16 to 48 34 against 39, 4 to 48 33 against 30; 333x251, 4 to 1
// 6.6 against 8.3, 48 to 300 204 against 222, 3 to 300 263 against 216.
bool warp_rows(int nin, int nout, int W) {
    const double views = double(nout) / (nin - 1);   // an interval
    if (W <= 110 || (W <= 192 && nin <= 4) || (W <= 224 && nin <= 3)) return true;
    if (nin > 32) return W <= (views < 0.5 ? 256 : kMaxRowsWidth) && views < 8.0;
    return (W <= 256 && views < 4.5) || (W <= 400 && views < 2.0);
}

}  // namespace

// Shared memory: the two staged rows (colour and t, g), the pass's minima, the
// output views by interval.
size_t warp_smem(int nin, int nout, int W) {
    return 40u * size_t(row_stride(W)) + 8u * size_t(views_per_pass(W)) * size_t(W) + 12u * size_t(nout) +
           4u * size_t(nin) + 8u;
}

cudaError_t launch_warp_views(const uint8_t* views, const uint64_t* keys, const float* in_eyes, int nin,
                              const float* out_eyes, int nout, int W, int H, float ipw, uint8_t* out, int grid,
                              bool beside, cudaStream_t s) {
    if (nin < 2 || nout < 1 || W < 1 || H < 1 || W > kMaxWarpWidth || H > 65535 || nout > kMaxRenderViews || !(ipw > 0.0f))
        return cudaErrorInvalidValue;
    const WarpArgs a{views, keys, in_eyes, out_eyes, nin, nout, W, H, ipw, out};
    if (!beside && warp_rows(nin, nout, W)) {
        const size_t smem = (40u + 8u * size_t(views_per_pass(W))) * size_t(W);
        k_warp_rows<<<dim3(unsigned(H), unsigned(nin - 1)), kWarpThreads, smem, s>>>(a);
        return cudaGetLastError();
    }
    const size_t smem = warp_smem(nin, nout, W);
    cudaError_t e = cudaSuccess;
    // the split from L1 that the network's layers have, so that it runs beside them
    if (beside) e = cudaFuncSetAttribute(k_warp_views, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    if (smem > 48u * 1024u) {
        // the most that a row takes, not this one's: another thread's views may be wider
        e = cudaFuncSetAttribute(k_warp_views, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(warp_smem(kMaxRenderViews, kMaxRenderViews, kMaxWarpWidth)));
        if (e != cudaSuccess) return e;
    }
    k_warp_views<<<std::min(grid, H * (nin - 1)), warp_threads(W), smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace lfdpr

extern "C" lfdpr_status lfdpr_warp_views(const uint8_t* in_views, const uint64_t* in_keys, const float* in_eyes,
                                         int32_t in_count, const float* out_eyes, int32_t out_count, int32_t view_w,
                                         int32_t view_h, float pixels_per_unit, uint8_t* out_views, void* stream) {
    lfdpr::g_last_error[0] = 0;
    if (!in_views || !in_keys || !in_eyes || !out_eyes || !out_views)
        return lfdpr::fail(LFDPR_EINVAL, "warp_views: null argument");
    if (in_count < 2 || in_count > lfdpr::kMaxRenderViews || out_count < 1 || out_count > lfdpr::kMaxRenderViews)
        return lfdpr::fail(LFDPR_EINVAL, "warp_views: need 2..%d input and 1..%d output views", lfdpr::kMaxRenderViews,
                           lfdpr::kMaxRenderViews);
    if (view_w < 1 || view_h < 1 || view_w > lfdpr::kMaxWarpWidth || view_h > 16384)
        return lfdpr::fail(LFDPR_EINVAL, "warp_views: views must be 1..%d pixels wide, 1..16384 high",
                           lfdpr::kMaxWarpWidth);
    if (!(pixels_per_unit > 0.0f) || !std::isfinite(pixels_per_unit))
        return lfdpr::fail(LFDPR_EINVAL, "warp_views: pixels_per_unit must be positive and finite");
    if ((reinterpret_cast<uintptr_t>(in_views) & 3u) || (reinterpret_cast<uintptr_t>(out_views) & 3u) ||
        (reinterpret_cast<uintptr_t>(in_keys) & 7u) || (reinterpret_cast<uintptr_t>(in_eyes) & 3u) ||
        (reinterpret_cast<uintptr_t>(out_eyes) & 3u))
        return lfdpr::fail(LFDPR_EINVAL, "warp_views: views and eyes must be 4-byte aligned, keys 8-byte aligned");
    const cudaError_t e = lfdpr::launch_warp_views(in_views, in_keys, in_eyes, in_count, out_eyes, out_count, view_w,
                                                   view_h, pixels_per_unit, out_views, view_h * (in_count - 1), false,
                                                   static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return lfdpr::cuda_fail(e, "launch k_warp_views");
    return LFDPR_OK;
}
