// EPR splatting into every view (Sec. 3.2) with the 64-bit depth|id test
// (Sec. 5.1), and the per-view resolve of Eq. 8-9 (Sec. 3.3).
//
//   k_splat    a half-warp per point forms the candidate pixels of every view,
//              a warp's candidates of several points are pooled into 32-lane
//              passes: every pixel centre inside the point's projected cell
//              and its projected triangle, at a depth in [near, far], does
//              atomicMin(key, float_bits(t) << 32 | point id).
//   k_resolve  one thread per view pixel: the winning point's 32-byte resolve
//              record gives the splat's pixel area in this view
//              (|alpha + beta Ex| / 2), Eq. 8 the view's texture area, Eq. 9
//              interpolates tv_min..tv_max.
#include "lfdpr_internal.cuh"

namespace lfdpr {
namespace {

// A warp takes a unit of 2P points of the work list, neighbours or spread over it: for each of
// its P pairs, one half-warp (16 lanes) per point, each lane taking up to S
// views of the point (views g + 16 s + lane of a group g of 16 S views, S
// chosen so that one group holds every rendered view where it can).
//
// Candidates. Candidate rows are the pixel-centre rows inside both the
// cell's and the triangle's projected y-extent, the same in every view since
// every eye lies on y = 0, z = D. A lane forms each of its views' candidate
// columns between a lower and an upper line x = alpha + beta Ex for the cell
// and for the triangle, which bound each one's projected x-extent within the
// band of candidate rows (the row's exact crossings for most points with one
// row), widened by a small margin.
//
// Pooling. The unit's candidates are numbered in (lane, pair, view slot)
// order; the non-empty (point, view) segments of that numbering go to a
// per-warp list in shared memory with their first number, and the points'
// test constants beside it. Then every pass hands the warp's 32 lanes the
// next 32 candidates of the whole unit: a lane's segment is the last one
// starting at or before its number, found from the OR-reduction of the
// start bits that fall in the pass (segments are numbered in start order).
// Points with few candidates, most of the work list, thus share passes
// instead of each filling a pass on its own.
//
// Test. Each candidate takes the per-pixel test in the oracle's plane-space
// form: the pixel centre's ray from the eye meets the triangle's plane at t
// (the division also yields the depth key); the hit must lie in the half-open
// cell and in the closed triangle (2-D edge functions of the lattice frame),
// at a depth t D in [near, far]. A cell inside its triangle skips the triangle
// test. The margin of the candidate ranges only admits extra candidates; the
// test alone decides.
//
// Points whose cell or triangle reaches within near_z of the eyes' plane come
// with candidate bounds of their cell and triangle clipped to that limit
// (k_fetch) and take the same passes and test.
constexpr int kSplatWarps = 8;
// Units a warp takes before the splat asks for more than the blocks the SMs hold
// at once (a wave, four blocks an SM). Each block more costs its start; with few
// blocks the longest warp decides. 8, 24, 48 and 96 views on 5,000 to 10^6
// triangles, grids of 1 to 4 waves: the second wave pays from about 55,000 units
// on, the fourth from 230,000. Against a grid of four waves whatever the size:
// 5,000 triangles at 48 views 125 -> 116 us a frame, at 96 views 201 -> 182; twelve
// scenes of a batch 2.88 -> 2.77 ms; from 300,000 triangles on the same.
constexpr uint32_t kUnitsPerWarp = 14;
// Units a warp of a wave up to which they are spread over the list (see k_splat).
__host__ __device__ constexpr uint32_t spread_units(int S) { return S == 3 ? 40u : 20u; }

// The per-pixel test; every condition is evaluated (no early exits), so the
// lanes' different candidates do not diverge.
__device__ __forceinline__ bool pixel_test(const DispConst& c, float Ex, float num, float qEx, float qEy,
                                           float qEz, const float4& q1, const float4& q2, const float4& q3,
                                           const float4& q4, float ulo, float uhi, float vlo, float vhi,
                                           bool interior, bool depth_ok, int x, int y, float& t) {
    const float Fx = fmaf(float(x) + 0.5f, c.pw, c.x0);
    const float Fy = fmaf(float(y) + 0.5f, -c.ph, c.y0);
    const float dx = Fx - Ex, dy = Fy - 0.0f, dz = -c.D;
    const float den = dot3(q3.x, q3.y, q3.z, dx, dy, dz);
    t = __fdiv_rn(num, den);
    const float depth = t * c.D;
    const bool in_depth = depth_ok ? t > 0.0f : (depth >= c.near_z && depth <= c.far_z);
    const float hx = fmaf(t, dx, qEx), hy = fmaf(t, dy, qEy), hz = fmaf(t, dz, qEz);
    const float uq = dot3(hx, hy, hz, q1.x, q1.y, q1.z);
    const float vq = dot3(hx, hy, hz, q2.x, q2.y, q2.z);
    const float u = uq - q2.w, vv = vq - q3.w;
    const bool in_cell = u >= ulo && u < uhi && vv >= vlo && vv < vhi;
    const float w0 = edge_fn(q4.x, q4.y, q4.z, q4.w, uq, vq);
    const float w1 = edge_fn(q4.z, q4.w, 0.0f, 0.0f, uq, vq);
    const float w2 = edge_fn(0.0f, 0.0f, q4.x, q4.y, uq, vq);
    return (den != 0.0f) & in_depth & in_cell & (interior | inside_either(w0, w1, w2));
}

// Eye x of view v from the eye array at shared-memory address ex_s.
__device__ __forceinline__ float eye_x(uint32_t ex_s, int v) {
    float e;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(e) : "r"(ex_s + 4u * uint32_t(v)));
    return e;
}

// warp-aggregated count of depth-test writes (the atomics issued)
__device__ __forceinline__ void add_writes(Counters* ctr, uint32_t writes) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) writes += __shfl_xor_sync(0xffffffffu, writes, o);
    if ((threadIdx.x & 31) == 0 && writes) atomicAdd(&ctr->n_writes, writes);
}

// floor(r / n) for n >= 1: below 2^21 one approximate division of r + 1/2
// (its quotient stays at least 1 / (2n) from an integer, more than the 2-ulp
// error of __fdividef), else an integer division.
__device__ __forceinline__ uint32_t div_floor(uint32_t r, uint32_t n) {
    if (r < (1u << 21)) return uint32_t(__fdividef(float(r) + 0.5f, float(n)));
    return r / n;
}

// Units of 2P points per warp: pairs per unit for S view slots per lane. More
// points share the unit's scan and fill its passes better; more segments take
// more shared memory and registers, and a small mesh has fewer units to spread.
// Splat of 10^6 triangles (200 instances), P = 1 for S = 6 and 8, else 2, against
// these: 8 views (S = 1) 172 -> 106 us, 24 (S = 2) 220 -> 181, 48 (S = 3)
// 292 -> 273, 96 (S = 6) 557 -> 464. P = 4 for S = 1 gave 121 (and a frame of
// 2,048 triangles 0.4 us less); P = 5 for S = 2 223; P = 4 for S = 3 286 of 283;
// P = 3 for S = 4 350 of 353 but slower small frames. With S = 8 two pairs would
// leave an SM three blocks. (Smaller units for few points, coarse cells and small
// meshes: see k_splat and splat_one.)
__host__ __device__ constexpr int unit_pairs(int S) {
    return S == 1 ? 6 : S <= 2 ? 4 : S == 3 ? 3 : S <= 6 ? 2 : 1;
}

// Per-warp shared memory of the pooled splat: the unit's non-empty (point,
// view) segments in candidate order (first candidate number,
// x0 | n_columns << 14, view | point << 16, eye x) and its points' test
// constants: (P0.x, -P0.y, D - P0.z, point id), (u-hat, work meta word),
// (v-hat, u_min), (n-hat, v_min), the 2-D vertices, the cell's u and v bounds.
template <int S, int P>
struct SplatWarpSmem {
    static constexpr int kSegs = 32 * S * P;
    uint4 seg[kSegs];
    float4 pt[2 * P][6];
};

// Candidate rr of segment e: its pixel, the test, and the depth-test atomic.
template <int S, int P>
__device__ __forceinline__ void test_candidate(const DispConst& c, const SplatWarpSmem<S, P>& sm, const uint4& e,
                                               uint32_t rr, unsigned long long* keys, uint32_t npix,
                                               uint32_t& writes) {
    const float4* d = sm.pt[e.z >> 16];
    const float4 d0 = d[0], d1 = d[1], q2 = d[2], q3 = d[3], q4 = d[4], b = d[5];
    const uint32_t meta = __float_as_uint(d1.w), flags = meta >> 29;
    const uint32_t nx = e.y >> 14;
    // one row (most segments): no division
    const uint32_t ry = rr < nx ? 0u : div_floor(rr, nx);
    const int x = int(e.y & 0x3fffu) + int(rr - ry * nx), y = int(meta & 0x3fffu) + int(ry);
    const uint32_t vo = e.z & 0xffffu;
    const float Ex = __uint_as_float(e.w);
    const float qEx = Ex - d0.x, qEy = d0.y, qEz = d0.z;
    const float num = -dot3(q3.x, q3.y, q3.z, qEx, qEy, qEz);
    float t;
    if (!pixel_test(c, Ex, num, qEx, qEy, qEz, d1, q2, q3, q4, b.x, b.y, b.z, b.w, flags & kFlagInterior,
                    flags & kFlagDepthOk, x, y, t))
        return;
    if (!LFDPR_IN_BOUNDS(vo, c.nr, 10) || !LFDPR_IN_BOUNDS(uint32_t(x), c.W, 11) ||
        !LFDPR_IN_BOUNDS(uint32_t(y), c.H, 11))
        return;
    // a view holds at most 2^26 pixels: 32-bit offset within it
    atomicMin(keys + ((uint64_t)vo * npix + (uint32_t(y) * uint32_t(c.W) + uint32_t(x))),
              ((unsigned long long)__float_as_uint(t) << 32) | __float_as_uint(d0.w));
    writes++;
}

// The splat proper: n_warps warps stride through the units of the work list's n
// points. ex_s: shared-memory address of the eye positions.
template <int S, int P, bool kSpread>
__device__ __forceinline__ void splat_units(const FrameArgs& a, uint32_t n, uint32_t total_units, uint32_t n_warps,
                                            uint32_t ex_s, SplatWarpSmem<S, P>& sm) {
    // unit g: work points 2 P g + q, q < 2 P, or (spread over the list, of which it
    // may have fewer than 2 P) g + q total_units; those below n
    const uint32_t A = kSpread ? 1u : 2u * P, B = kSpread ? total_units : 1u;
    const int lane = threadIdx.x & 31, sub = lane & 15, half = lane >> 4;
    const uint32_t lanes_below = (1u << lane) - 1u;
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const DispConst& c = a.dc;
    const WorkRec* work = a.work;
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(a.keys);
    const uint32_t npix = uint32_t(c.W) * uint32_t(c.H);
    const int vlo = a.view_lo, vhi = a.view_hi;
    uint32_t writes = 0;

    for (uint32_t g = warp; g < total_units; g += n_warps) {
        const uint32_t k0 = A * g;   // the unit's first work point
        {
            const uint32_t kn = k0 + A * n_warps + B * uint32_t(lane);   // the next unit's records
            if (lane < 2 * P && kn < n) prefetch_l2(work + kn);
        }
        // the next unit's triangles: read their ids now (the
        // work records were asked for a unit ago), ask L1 for their records'
        // 128-byte lines once this unit's candidates are formed, so that the
        // next unit's staging finds them there
        uint32_t next_tri = 0xffffffffu;
        {
            const uint32_t kn = k0 + A * n_warps + B * uint32_t(lane);
            if (lane < 2 * P && kn < n) next_tri = __ldg(&work[kn].meta.z);
        }
        for (int g0 = vlo; g0 < vhi; g0 += 16 * S) {
            __syncwarp();   // the previous passes are done with sm
            // (formed after the candidates where the registers allow: 64 views 345 -> 337 us,
            // 48 views 270 -> 265; with six slots it costs 3 %)
            auto stage = [&] {
                if (g0 != vlo) return;
                // the unit's test constants, one float4 a lane and turn: number
                // 5 q + f is float4 f of point k0 + q (a point past the end takes
                // the unit's first record; it has no rows), and with the cell's
                // spacings (f = 0 and 1) go its u and its v bounds. Five numbers a
                // point, not six, are one turn for six points: 10^6 triangles at 48
                // views 285 -> 270 us, at 8 views 131 -> 121, at 96 467 -> 465.
#pragma unroll
                for (int z = 0; z < 10 * P; z += 32) {
                    const int q = (lane + z) / 5, f = lane + z - 5 * q;
                    if (q >= 2 * P) break;
                    const uint32_t k = k0 + B * uint32_t(q);
                    const uint4 meta = __ldg(&work[k < n ? k : k0].meta);
                    float4 v = __ldg(&a.rec[meta.z].q[f]);
                    if (f < 2) {
                        const uint32_t ij = f == 0 ? meta.y & 0xffffu : meta.y >> 16;
                        reinterpret_cast<float2*>(&sm.pt[q][5])[f] = make_float2(float(int(ij)) * v.w, float(int(ij) + 1) * v.w);
                        v.w = __uint_as_float(f == 0 ? meta.w : meta.x);
                    }
                    if (f == 0) {
                        v.y = 0.0f - v.y;
                        v.z = c.D - v.z;
                    }
                    sm.pt[q][f] = v;
                }
            };
            if constexpr (S > 4) stage();
            uint32_t pk[P][S], ny[P];
            float ex[S];   // the lane's views' eyes, the same for every pair
            uint32_t cnt = 0, nz = 0;   // the lane's candidates and non-empty (point, view) segments
#pragma unroll
            for (int p = 0; p < P; p++) {
                // a half past the end takes the unit's first record, with no rows
                const uint32_t k = k0 + B * uint32_t(2 * p + half);
                const WorkRec* wr = work + (k < n ? k : k0);
                const float4 l0 = __ldg(&wr->L0), l1 = __ldg(&wr->L1);
                const uint4 meta = __ldg(&wr->meta);
                ny[p] = k < n ? (meta.x >> 14) & 0x7fffu : 0u;
                // branch-free: every slot computes its range, an empty or
                // absent one is masked to zero
#pragma unroll
                for (int sl = 0; sl < S; sl++) {
                    const int v = g0 + 16 * sl + sub;
                    if (p == 0) ex[sl] = eye_x(ex_s, v < vhi ? v : vlo);
                    const float Ex = ex[sl];
                    const float lo = fmaxf(fmaf(l0.y, Ex, l0.x), fmaf(l1.y, Ex, l1.x));
                    const float hi = fminf(fmaf(l0.w, Ex, l0.z), fmaf(l1.w, Ex, l1.z));
                    const int ix0 = max(__float2int_ru(lo), 0);
                    const int ix1 = min(__float2int_rd(hi), int(c.W) - 1);
                    const bool ok = v < vhi && ix0 <= ix1 && ny[p] > 0u;
                    const uint32_t nx = ok ? uint32_t(ix1 - ix0) + 1u : 0u;
                    pk[p][sl] = ok ? uint32_t(ix0) | (nx << 14) : 0u;
                    cnt += nx * ny[p];
                    nz += ok ? 1u : 0u;
                }
            }
            if constexpr (S <= 4) stage();
            // a segment holds at most 2^26 candidates (one view), so lanes
            // below the limit (at most 2^24) keep the unit's numbering below 2^32
            const bool big = __any_sync(0xffffffffu, cnt >= a.splat_lane_limit);
            // the unit's candidates and segments numbered in (lane, pair, slot)
            // order: one scan of both counts, the candidates in the high word
            // (wrapping as 32-bit sums would, only when the unit is walked)
            // and the segments (at most 32 S P) in the low one
            unsigned long long incl = ((unsigned long long)cnt << 32) | nz;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            const unsigned long long all = __shfl_sync(0xffffffffu, incl, 31);
            const uint32_t total = uint32_t(all >> 32), nseg = uint32_t(all);
            uint32_t first = uint32_t(incl >> 32) - cnt, rank = uint32_t(incl) - nz;
#pragma unroll
            for (int p = 0; p < P; p++)
#pragma unroll
                for (int sl = 0; sl < S; sl++) {
                    const bool ok = pk[p][sl] != 0u;
                    if (ok)
                        sm.seg[rank] = make_uint4(first, pk[p][sl], uint32_t(g0 + 16 * sl + sub) | uint32_t(2 * p + half) << 16,
                                                  __float_as_uint(ex[sl]));
                    rank += ok ? 1u : 0u;
                    first += (pk[p][sl] >> 14) * ny[p];
                }
            if (next_tri != 0xffffffffu && g0 == vlo) prefetch_l1(a.rec + next_tri);
            __syncwarp();
            if (big) {
                // huge cells: each lane walks whole segments
                for (uint32_t s = uint32_t(lane); s < nseg; s += 32) {
                    const uint4 e = sm.seg[s];
                    const uint32_t ny = (__float_as_uint(sm.pt[e.z >> 16][1].w) >> 14) & 0x7fffu;
                    const uint32_t m = (e.y >> 14) * ny;
                    for (uint32_t rr = 0; rr < m; rr++) test_candidate<S, P>(c, sm, e, rr, keys, npix, writes);
                }
                continue;
            }
            uint32_t before = 0;   // segments starting before the pass
            for (uint32_t pass = 0; pass < total; pass += 32) {
                const uint32_t kw = before + uint32_t(lane);
                const uint32_t st = kw < nseg ? sm.seg[kw].x : 0xffffffffu;
                const uint32_t off = st - pass;   // starts from `before` on are >= pass
                const uint32_t smask = __reduce_or_sync(0xffffffffu, off < 32u ? 1u << off : 0u);
                const uint32_t own = before + uint32_t(__popc(smask & (lanes_below | (1u << lane)))) - 1u;
                before += uint32_t(__popc(smask));
                const uint32_t q = pass + uint32_t(lane);
                if (q < total) {
                    const uint4 e = sm.seg[own];
                    test_candidate<S, P>(c, sm, e, q - e.x, keys, npix, writes);
                }
            }
        }
    }
    add_writes(a.ctr, writes);
}

// Cells of a sampling bias of eight pixels and more.
__host__ __device__ __forceinline__ bool coarse_cells(const DispConst& c) { return c.bias_h * c.bias_v >= 8.0f; }

// Whether a splat takes no more blocks than its units fill (else every block).
template <int S, int P>
__host__ __device__ __forceinline__ bool fills_blocks(const DispConst& c) {
    return P == unit_pairs(S) && !(S == 8 && coarse_cells(c));
}

template <int S, int P>
__global__ void __launch_bounds__(kSplatWarps * 32, 4) k_splat(FrameArgs a) {
    // With more than two slots the resolve is let in only when this block is
    // done: its blocks waiting on the SMs cost a splat with 40 KB or more of shared
    // memory a block a sixth of its time (96 views: 0.47 -> 0.56 ms). With fewer they
    // cost nothing, and a small frame is 3 us shorter for them.
    constexpr bool kLate = S > 2;
    wait_previous_kernel();
    if constexpr (!kLate) allow_next_kernel();
    extern __shared__ __align__(16) uint8_t s_dyn[];
    __shared__ float s_ex[kMaxRenderViews];
    for (int v = threadIdx.x; v < a.dc.nr; v += blockDim.x) s_ex[v] = a.ex[v];
    if (a.ctr->overflow) return;
    // (the reductions of one value keep it in a uniform register: of the kernel's 64
    // registers one more for the warps costs 96 views 3 %)
    const uint32_t n = __reduce_max_sync(0xffffffffu, a.ctr->n_work);
    const uint32_t wave = 4u * uint32_t(a.sm_count);
    const bool coarse = coarse_cells(a.dc);
    uint32_t unit = 2u * P;
    // few points, often of large cells, whose units are long, and coarse cells: a unit
    // for every warp (2,048 points of 18,000 pixels over 48 views: 8.2 -> 1.9 ms a
    // frame; 11,000 points at bias 32 over 8 and 48 views: 49 -> 38 and 97 -> 78 us).
    // The units of small cells are cheap, and with one slot shorter than the passes
    // that they fill: two points at least (15,000 points of two pixels at 8 views: 35
    // us a frame with units of one, 33 so; four would be better there, 31, and worse
    // where textures of few texels leave large cells, 69 -> 70).
    if (S <= 3 && (coarse || n < 2u * wave * kSplatWarps))
        unit = min(unit, max(S == 1 && !coarse ? 2u : 1u, n / (wave * kSplatWarps)));
    const uint32_t units = (n + unit - 1u) / unit;
    // Neighbouring points are alike, and a unit of the coarse ones of a mesh is much
    // longer than the others: of few units, each takes its points from all over the
    // list. Of many it takes neighbours, which share triangles. (Meshes of 20,000 and
    // 110,000 triangles with textures of 256 texels a side: at 16 views 98 -> 72 and
    // 160 -> 144 us a frame, at 48 views 182 -> 146 and 284 -> 258; 200,000 triangles,
    // 10^6 points, 40 and 48 views 357 -> 340 and 394 -> 374, the line at 40 units a warp
    // instead of 20; 10^6 triangles at 48 views 572 us with neighbours, 587 with points
    // from all over, at 24 views 443 and 455.)
    const bool spread = S <= 3 && units <= wave * kSplatWarps * spread_units(S);
    uint32_t blocks = gridDim.x;
    if (fills_blocks<S, P>(a.dc)) blocks = min(blocks, wave * (1u + units / (wave * kSplatWarps * kUnitsPerWarp)));
    if (blockIdx.x >= blocks) return;
    __syncthreads();
    const uint32_t n_warps = __reduce_max_sync(0xffffffffu, blocks * kSplatWarps);
    const uint32_t ex_s = uint32_t(__cvta_generic_to_shared(s_ex));
    SplatWarpSmem<S, P>& sm = reinterpret_cast<SplatWarpSmem<S, P>*>(s_dyn)[threadIdx.x >> 5];
    if (S <= 3 && spread)
        splat_units<S, P, true>(a, n, __reduce_max_sync(0xffffffffu, units), n_warps, ex_s, sm);
    else
        splat_units<S, P, false>(a, n, units, n_warps, ex_s, sm);
    if constexpr (kLate) allow_next_kernel();
}

// Eq. 8's interpolation weight for one view pixel whose depth test kept the
// point with resolve record (ra, rb): the splat's pixel area in view Ex is
// the shoelace area of its cell corners projected from the eye,
// |alpha + beta Ex| / 2. The colour it weights is held to the oracle within
// one level of 255, so both quotients take the hardware's approximate
// division (relative error near 1e-7: a colour moves by far less than a
// level, and changes level only where it lies within that of a rounding
// boundary); the divisors are at most 1 and a ratio of texture areas.
__device__ __forceinline__ float eq8_weight(float Ex, const float4& ra, const uint4& rb) {
    const float area_px = 0.5f * fabsf(fmaf(ra.y, Ex, ra.x));
    const float vmin = ra.w, vmax = __uint_as_float(rb.x);
    const float size_vse = __fdividef(ra.z, fminf(1.0f, area_px));
    const float size_vs = fminf(fmaxf(size_vse, vmin), vmax);
    return vmax > vmin ? __fdividef(size_vs - vmin, vmax - vmin) : 0.0f;
}

__device__ __forceinline__ uint32_t resolve_pixel(float Ex, const float4& ra, const uint4& rb) {
    const float w = eq8_weight(Ex, ra, rb);
    uint32_t out = 0u;
#pragma unroll
    for (int ch = 0; ch < 4; ch++) {
        const float lo = float((rb.y >> (8 * ch)) & 255u), hi = float((rb.z >> (8 * ch)) & 255u);
        out |= uint32_t(round_u8(fmaf(w, hi - lo, lo))) << (8 * ch);
    }
    return out;
}

// kResolvePix view pixels per thread, 256 apart (grid: pixel blocks x
// views): every key is loaded, then every winner's record, so each thread
// keeps that many dependent gathers in flight. A record is one 32-byte load
// (48 views of 420x560: 45 us; as two of 16 bytes 47).
constexpr int kResolvePix = 2;
__global__ void __launch_bounds__(256) k_resolve(FrameArgs a) {
    wait_previous_kernel();
    allow_next_kernel();
    const DispConst& c = a.dc;
    const uint32_t npix = uint32_t(c.W) * uint32_t(c.H);
    const uint32_t p0 = blockIdx.x * (256u * kResolvePix) + threadIdx.x;
    const int v = a.view_lo + int(blockIdx.y);
    const uint64_t o0 = (uint64_t)v * npix;
    unsigned long long key[kResolvePix];
#pragma unroll
    for (int k = 0; k < kResolvePix; k++) {
        const uint32_t p = p0 + 256u * k;
        key[k] = p < npix ? a.keys[o0 + p] : ~0ull;
    }
    float4 ra[kResolvePix];
    uint4 rb[kResolvePix];
#pragma unroll
    for (int k = 0; k < kResolvePix; k++) {
        if (key[k] != ~0ull && !LFDPR_IN_BOUNDS(uint32_t(key[k]), a.max_points, 12)) key[k] = ~0ull;
        if (key[k] != ~0ull) {
            load32(a.rrec + uint32_t(key[k]), ra[k], rb[k]);
        }
    }
    const float Ex = __ldg(a.ex + v);
#pragma unroll
    for (int k = 0; k < kResolvePix; k++) {
        const uint32_t p = p0 + 256u * k;
        if (p < npix && LFDPR_IN_BOUNDS(uint32_t(v), uint32_t(c.nr), 13))
            reinterpret_cast<uint32_t*>(a.views)[o0 + p] = key[k] != ~0ull ? resolve_pixel(Ex, ra[k], rb[k]) : 0u;
    }
}

// ---------------------------------------------------------------------------
// Physically based resolve of a mesh of materials
// ---------------------------------------------------------------------------

// Outgoing linear RGB of one surface sample (unit n, v, l): metallic-roughness
// microfacet BRDF, GGX distribution D = a^2 / (pi ((n.h)^2 (a^2 - 1) + 1)^2),
// a = r^2 (r >= 0.045), Schlick-GGX visibility G1(x) = x / (x (1 - k) + k),
// k = (r + 1)^2 / 8, Schlick Fresnel F = F0 + (1 - F0)(1 - v.h)^5, F0 = 0.04
// (1 - m) + albedo m, diffuse (1 - F)(1 - m) albedo / pi:
//   rgb = (diffuse + D G F / (4 n.l n.v)) light n.l + ambient albedo.
__device__ __forceinline__ float3 pbr_shade(const float3& albedo, float rough, float metal, const float3& n,
                                            const float3& v, const float3& l, const Shading& sh) {
    const float3 h = normalized(f3(l.x + v.x, l.y + v.y, l.z + v.z));
    const float nl = fmaxf(dot(n, l), 0.0f), nv = fmaxf(dot(n, v), 1e-4f);
    const float nh = fmaxf(dot(n, h), 0.0f), vh = fmaxf(dot(v, h), 0.0f);
    const float r = fmaxf(rough, 0.045f);
    const float a = r * r, a2 = a * a;
    const float dn = fmaf(nh * nh, a2 - 1.0f, 1.0f);
    const float Dg = __fdividef(a2, 3.14159265358979f * dn * dn);
    const float k = (r + 1.0f) * (r + 1.0f) * 0.125f;
    const float G = __fdividef(nl, fmaf(nl, 1.0f - k, k)) * __fdividef(nv, fmaf(nv, 1.0f - k, k));
    const float om = 1.0f - vh;
    const float f5 = (om * om) * (om * om) * om;
    const float den = fmaxf(4.0f * nl * nv, 1e-4f);
    const float spec_dg = __fdividef(Dg * G, den);
    const float alb[3] = {albedo.x, albedo.y, albedo.z};
    float o[3];
#pragma unroll
    for (int ch = 0; ch < 3; ch++) {
        const float F0 = fmaf(alb[ch], metal, 0.04f * (1.0f - metal));
        const float F = fmaf(1.0f - F0, f5, F0);
        const float diffuse = (1.0f - F) * (1.0f - metal) * alb[ch] * 0.318309886183791f;   // 1 / pi
        o[ch] = fmaf((diffuse + spec_dg * F) * sh.rgb[ch], nl, sh.amb[ch] * alb[ch]);
    }
    return f3(o[0], o[1], o[2]);
}

// One view pixel per thread: Eq. 8's weight as k_resolve; each map's value
// interpolated by Eq. 9 (unrounded); the surface point where the pixel
// centre's ray meets the triangle (the key's t: P = E + t (F - E)); the
// shading normal = the normal map's (2 c / 255 - 1) vector in the triangle's
// frame (of k_fetch_mat, with the normal map's values in the point's record), flipped when
// the triangle faces away from the eye; RGB = pbr_shade clamped, times 255,
// rounded half to even, alpha 255. Bound by its gathers (a warp's 32 points are
// 32 places): two sectors a pixel, each by one 32-byte load. 48 views of 420x560:
// 158 us with the frame formed from the triangle's record by every pixel (nine
// loads in six sectors), 107 now, for 10 us more in k_fetch_mat.
__global__ void __launch_bounds__(256) k_resolve_pbr(FrameArgs a) {
    wait_previous_kernel();
    allow_next_kernel();
    const DispConst& c = a.dc;
    const uint32_t npix = uint32_t(c.W) * uint32_t(c.H);
    const uint32_t px = blockIdx.x * blockDim.x + threadIdx.x;
    if (px >= npix) return;
    const int v = a.view_lo + int(blockIdx.y);
    const uint64_t o = (uint64_t)v * npix + px;
    unsigned long long key = a.keys[o];
    if (key != ~0ull && !LFDPR_IN_BOUNDS(uint32_t(key), a.max_points, 12)) key = ~0ull;
    uint32_t out = 0u;
    if (key != ~0ull) {
        const uint32_t p = uint32_t(key);
        const float t = __uint_as_float(uint32_t(key >> 32));
        const float Ex = __ldg(a.ex + v);
        float4 ra, ma;
        uint4 rb, mb;
        load32(a.rrec + p, ra, rb);
        load32(a.mrec + p, ma, mb);
        const uint2 nm = make_uint2(mb.z, mb.w);
        const float w = eq8_weight(Ex, ra, rb);
        auto lerp8 = [w](uint32_t lo, uint32_t hi, int ch) {
            const float a0 = float((lo >> (8 * ch)) & 255u), b0 = float((hi >> (8 * ch)) & 255u);
            return fmaf(w, b0 - a0, a0);
        };
        const float3 albedo = f3(lerp8(rb.y, rb.z, 0) * (1.0f / 255.0f), lerp8(rb.y, rb.z, 1) * (1.0f / 255.0f),
                                 lerp8(rb.y, rb.z, 2) * (1.0f / 255.0f));
        const float3 nt = f3(fmaf(lerp8(nm.x, nm.y, 0), 2.0f / 255.0f, -1.0f), fmaf(lerp8(nm.x, nm.y, 1), 2.0f / 255.0f, -1.0f),
                             fmaf(lerp8(nm.x, nm.y, 2), 2.0f / 255.0f, -1.0f));
        const uint32_t rm = rb.w;
        const float rough = fmaf(w, float((rm >> 8) & 255u) - float(rm & 255u), float(rm & 255u)) * (1.0f / 255.0f);
        const float metal =
            fmaf(w, float(rm >> 24) - float((rm >> 16) & 255u), float((rm >> 16) & 255u)) * (1.0f / 255.0f);
        // surface point and view direction
        const int x = int(px % uint32_t(c.W)), y = int(px / uint32_t(c.W));
        const float Fx = fmaf(float(x) + 0.5f, c.pw, c.x0), Fy = fmaf(float(y) + 0.5f, -c.ph, c.y0);
        const float3 P = f3(fmaf(t, Fx - Ex, Ex), t * Fy, fmaf(-t, c.D, c.D));
        const float3 V = normalized(f3(Ex - P.x, -P.y, c.D - P.z));
        // the shading frame: N, the tangent and their cross product by its sign
        const float3 N = f3(ma.x, ma.y, ma.z), Tg = f3(ma.w, __uint_as_float(mb.x), __uint_as_float(mb.y));
        float3 Bt = f3(fmaf(N.y, Tg.z, -(N.z * Tg.y)), fmaf(N.z, Tg.x, -(N.x * Tg.z)), fmaf(N.x, Tg.y, -(N.y * Tg.x)));
        if (mb.z >> 24) Bt = f3(-Bt.x, -Bt.y, -Bt.z);
        float3 n = f3(fmaf(nt.x, Tg.x, fmaf(nt.y, Bt.x, nt.z * N.x)), fmaf(nt.x, Tg.y, fmaf(nt.y, Bt.y, nt.z * N.y)),
                      fmaf(nt.x, Tg.z, fmaf(nt.y, Bt.z, nt.z * N.z)));
        if (dot(n, n) == 0.0f) n = N;
        n = normalized(n);
        if (dot(N, V) < 0.0f) n = f3(-n.x, -n.y, -n.z);
        const float3 rgb = pbr_shade(albedo, rough, metal, n, V, f3(a.sh.l[0], a.sh.l[1], a.sh.l[2]), a.sh);
        out = 0xff000000u | (uint32_t(__float2uint_rn(__saturatef(rgb.x) * 255.0f))) |
              (uint32_t(__float2uint_rn(__saturatef(rgb.y) * 255.0f)) << 8) |
              (uint32_t(__float2uint_rn(__saturatef(rgb.z) * 255.0f)) << 16);
    }
    reinterpret_cast<uint32_t*>(a.views)[o] = out;
}

// Blocks per SM of a splat: all of them, and at most where the kernel takes as many
// as its units fill.
struct SplatGrid {
    int all, filled;
};

// Launch with the per-warp pooling buffers as dynamic shared memory. Beyond 48 KB
// (with the kernel's eye positions) the launch needs the attribute, which holds for
// the current device only: it is set at every such launch.
template <int S, int P>
cudaError_t splat_as(const FrameArgs& a, const SplatGrid& grid, cudaStream_t s) {
    constexpr size_t bytes = kSplatWarps * sizeof(SplatWarpSmem<S, P>);
    if (bytes + sizeof(float) * kMaxRenderViews > 48u * 1024u) {
        const cudaError_t e =
            cudaFuncSetAttribute(k_splat<S, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
        if (e != cudaSuccess) return e;
    }
    const int per_sm = fills_blocks<S, P>(a.dc) ? grid.filled : grid.all;
    return launch_after_previous(k_splat<S, P>, dim3(a.sm_count * per_sm), dim3(kSplatWarps * 32), bytes, s, a);
}

// Coarse cells fill the passes of small units and make large ones uneven: two pairs
// (one with more slots) and every block, as 48 views of 420x560 at bias 16: 50,000
// points 178 -> 158 us a frame, 310,000 points 369 -> 336; 128 views, whose units are
// of one pair anyway, 73,000 points 373 -> 338 with every block, 276,000 825 -> 788. Up
// to 16 views the large units are as good.
// With six slots so do those of meshes below 150,000 triangles, where the points
// of a unit are too unlike for one of two pairs (82 and 96 views; 110,000 triangles,
// textures of 256 texels 413 -> 367 and 458 -> 406 us a frame, of up to 4,096 423 ->
// 447; from 200,000 on two pairs gain: 10^6 triangles 912 -> 836), and with four
// below 50,000 (60 views, 20,000 triangles: 148 -> 139 and 193 -> 170). A sampling
// bias leaves fewer and coarser points to the same triangles: with six slots the
// line is their number over the root of the bias (200,000 triangles at 96 views,
// bias 2, 4 and 6: 568, 603 and 546 us with one pair, 573, 627 and 556 with two
// whatever the bias, 550, 587 and 533 now; 10^6 at bias 6 784 and 721).
template <int S>
cudaError_t splat_one(const FrameArgs& a, const SplatGrid& grid, cudaStream_t s) {
    constexpr int kFew = S <= 3 ? 2 : 1;
    if (S > 1 && coarse_cells(a.dc)) return splat_as<S, (S == 1 ? unit_pairs(S) : kFew)>(a, grid, s);
    const double tris = double(a.n_tris), bias = double(a.dc.bias_h) * a.dc.bias_v;
    if ((S == 6 && tris * tris < 150000.0 * 150000.0 * bias) || (S == 4 && a.n_tris < 50000u))
        return splat_as<S, (S == 4 || S == 6 ? kFew : unit_pairs(S))>(a, grid, s);
    return splat_as<S, unit_pairs(S)>(a, grid, s);
}

}  // namespace

LFDPR_CHECK_READER(checks_splat)

cudaError_t launch_splat(const FrameArgs& a, cudaStream_t s, int blocks_per_sm, int filled_per_sm, int max_slots) {
    // the fewest view slots per lane that hold every view of the range
    // [view_lo, view_hi) in one group (more than 16 max_slots views take
    // several groups)
    const int nr = a.view_hi - a.view_lo;
    const SplatGrid grid{blocks_per_sm, filled_per_sm};
    const int slots = min((nr + 15) / 16, max_slots);
    if (slots <= 1) return splat_one<1>(a, grid, s);
    if (slots <= 2) return splat_one<2>(a, grid, s);
    if (slots <= 3) return splat_one<3>(a, grid, s);
    if (slots <= 4) return splat_one<4>(a, grid, s);
    if (slots <= 6) return splat_one<6>(a, grid, s);
    return splat_one<8>(a, grid, s);
}

void prefer_resolve_split() {
    for (const void* k : {reinterpret_cast<const void*>(k_resolve), reinterpret_cast<const void*>(k_resolve_pbr)})
        if (cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, kViewsSplit) != cudaSuccess)
            cudaGetLastError();
}

cudaError_t launch_resolve(const FrameArgs& a, cudaStream_t s) {
    const uint32_t npix = uint32_t(a.dc.W) * uint32_t(a.dc.H);
    const uint32_t nv = uint32_t(a.view_hi - a.view_lo);
    const dim3 grid((npix + 255u) / 256u, nv);
    if (a.pbr) return launch_after_previous(k_resolve_pbr, grid, dim3(256), 0, s, a);
    return launch_after_previous(k_resolve, dim3((npix + 256u * kResolvePix - 1u) / (256u * kResolvePix), nv),
                                 dim3(256), 0, s, a);
}

}  // namespace lfdpr
