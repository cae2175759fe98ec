// The library's launch code (its own objects) against the stand-in runtime of
// fake_cudart.cpp; needs no GPU. Prints the failed checks and returns their number.
#include <cmath>
#include <cstdio>
#include <cstring>

#include "fake_cudart.h"
#include "objects.h"

namespace {
int g_failed = 0;

void check(bool ok, const char* what) {
    if (ok) return;
    printf("failed: %s\n", what);
    g_failed++;
}
}  // namespace

namespace lfdpr {
thread_local char g_last_error[512];
lfdpr_status fail(lfdpr_status s, const char*, ...) { return s; }
lfdpr_status cuda_fail(cudaError_t, const char*) { return LFDPR_ECUDA; }
}  // namespace lfdpr

using namespace lfdpr;

static cudaError_t splat(int views, uint32_t tris, float bias = 1.0f) {
    FrameArgs a{};
    a.n_tris = tris;
    a.sm_count = 152;
    a.dc.bias_h = bias;
    a.dc.bias_v = 1.0f;
    a.dc.nr = a.view_hi = views;
    return launch_splat(a, nullptr);
}

static DispConst display(int recon, int n, int w, int h, int panel_w, int panel_h, float xtalk) {
    DispConst c{};
    c.recon = recon;
    c.n_views = n;
    c.nr = recon == 1 || recon == 2 ? 2 * n : n;
    c.W = w;
    c.H = h;
    c.Wp = panel_w;
    c.Hp = panel_h;
    c.inv_pitch = 0.125f;
    c.xtalk = xtalk;
    return c;
}

static cudaError_t interleave(int recon, int n, int w, int panel_w) {
    return launch_interleave(display(recon, n, w, 64, panel_w, 640, 0.15f), nullptr, nullptr, nullptr, 0, true, nullptr, nullptr);
}

// which form a tent interleave takes: tiles (dynamic shared memory) or the gather
static void tent() {
    const struct {
        int n, w, h, pw, ph;
        float xtalk;
        bool tiles;
    } cases[] = {{1, 420, 560, 2560, 1600, 0.0f, true},     {48, 420, 560, 2560, 1600, 0.0f, true},
                 {96, 420, 560, 2560, 1600, 0.0f, false},   {256, 420, 560, 2560, 1600, 0.0f, false},
                 {128, 420, 560, 2560, 1600, 0.15f, true},  {256, 420, 560, 2560, 1600, 0.15f, false},
                 {24, 333, 251, 1277, 719, 0.0f, true},     {64, 333, 251, 1277, 719, 0.0f, false},
                 {64, 333, 251, 1277, 719, 0.15f, true},    {96, 333, 251, 1277, 719, 0.15f, false},
                 {1, 640, 480, 640, 480, 0.0f, false},      {48, 640, 480, 640, 480, 0.15f, false},
                 {2, 1200, 300, 200, 200, 0.0f, false},     {8, 128, 128, 512, 512, 0.0f, true},
                 {12, 840, 1120, 2560, 1600, 0.0f, true},   {64, 840, 1120, 2560, 1600, 0.15f, false},
                 {128, 100, 50, 400, 2000, 0.0f, false},    {8, 120, 640, 2560, 300, 0.0f, true},
                 {48, 120, 640, 2560, 300, 0.15f, true},    {48, 480, 360, 1920, 1080, 0.0f, true},    {8, 160, 120, 3840, 2160, 0.0f, true}};
    for (const auto& k : cases) {
        char what[96];
        snprintf(what, sizeof what, "%d views of %dx%d to %dx%d, crosstalk %g", k.n, k.w, k.h, k.pw, k.ph, k.xtalk);
        check(launch_interleave(display(1, k.n, k.w, k.h, k.pw, k.ph, k.xtalk), nullptr, nullptr, nullptr, 0, true, nullptr,
                                nullptr) == cudaSuccess &&
                  (g_last_smem > 0) == k.tiles,
              what);
    }
}

// which form a Gaussian interleave takes: with the table (dynamic shared memory) or plain
static void gauss() {
    const struct {
        int n, w, h, pw, ph, ns;
        float xtalk;
        bool near, table;
    } cases[] = {{48, 420, 560, 2560, 1600, 8, 0.15f, true, true},   {48, 420, 560, 2560, 1600, 8, 0.15f, false, false},
                 {48, 420, 560, 2560, 1600, 1, 0.0f, true, true},    {256, 64, 64, 256, 256, 1, 0.0f, true, false},
                 {256, 64, 64, 256, 256, 4, 0.0f, true, false},      {256, 64, 64, 256, 256, 32, 0.0f, true, true},
                 {96, 128, 128, 512, 512, 1, 0.0f, true, false},     {96, 128, 128, 512, 512, 4, 0.0f, true, true},
                 {256, 1000, 2200, 2560, 1600, 8, 0.15f, true, false}};   // beyond 32-bit offsets
    for (const auto& k : cases) {
        char what[96];
        snprintf(what, sizeof what, "%d views of %dx%d to %dx%d, %d samples", k.n, k.w, k.h, k.pw, k.ph, k.ns);
        check(launch_interleave(display(2, k.n, k.w, k.h, k.pw, k.ph, k.xtalk), nullptr, nullptr, nullptr, k.ns, k.near,
                                nullptr, nullptr) == cudaSuccess &&
                  (g_last_smem > 0) == k.table,
              what);
    }
}

// units of one or two pairs of points (shared memory) with four and six slots
static void units() {
    const struct {
        int views;
        uint32_t tris;
        float bias;
        bool two;
    } cases[] = {{49, 49999, 1.0f, false},   {49, 50000, 1.0f, true},   {64, 50000, 4.0f, true},   {64, 50000, 8.0f, false},
                 {65, 149999, 1.0f, false},  {65, 150000, 1.0f, true},  {96, 200000, 1.0f, true},  {96, 200000, 2.0f, false},
                 {96, 200000, 6.0f, false},  {96, 300000, 3.9f, true},  {82, 1000000, 6.0f, true}, {82, 1000000, 8.0f, false},
                 {96, 100000, 0.25f, true}};
    for (const auto& k : cases) {
        char what[96];
        snprintf(what, sizeof what, "units of %d views, %u triangles, bias %g", k.views, k.tris, k.bias);
        const int slots = k.views <= 64 ? 4 : 6;
        check(splat(k.views, k.tris, k.bias) == cudaSuccess && (g_last_smem >= 8u * 2u * 32u * slots * 16u) == k.two, what);
    }
}

// a lens pitch whose reciprocal overflows: the lens phase is no number
static void tiny_pitch() {
    for (int recon : {2, 3}) {
        DispConst c = display(recon, 8, 64, 64, 200, 200, 0.15f);   // (with the table)
        c.inv_pitch = INFINITY;
        check(launch_interleave(c, nullptr, nullptr, nullptr, 1, true, nullptr, nullptr) == cudaSuccess, "tiny pitch");
    }
}

static cudaError_t warp(int w) { return launch_warp_views(nullptr, nullptr, nullptr, 2, nullptr, 4, w, 64, 1.0f, nullptr, 1, false, nullptr); }

// every number of view slots a lane, and both unit sizes, on one device and then another
static void devices() {
    for (int dev = 0; dev < 2; dev++) {
        g_device = dev;
        for (int views : {1, 32, 48, 64, 96, 128})
            for (uint32_t tris : {1000u, 1000000u}) {
                char what[96];
                snprintf(what, sizeof what, "splat of %d views, %u triangles on device %d", views, tris, dev);
                check(splat(views, tris) == cudaSuccess, what);
            }
        check(interleave(0, 48, 420, 1000) == cudaSuccess && interleave(1, 100, 240, 1000) == cudaSuccess, "interleave");
        check(warp(4032) == cudaSuccess, "warp");
    }
}

// both resolves and both view mips ask for their split; a refusal is no error
static void splits() {
    prefer_resolve_split();
    prefer_view_mip_split();
    check(g_splits == 4, "splits of the kernels between splat and interleave");
    g_fail_attributes = 4;
    prefer_resolve_split();
    prefer_view_mip_split();
    check(splat(48, 1000u) == cudaSuccess && cudaGetLastError() == cudaSuccess, "a refused split");
}

// a call after a failed one
static void retry() {
    g_fail_attributes = 1;
    splat(96, 1000000u);
    g_fail_attributes = 0;
    check(splat(96, 1000000u) == cudaSuccess, "splat after a failed attribute call");
}

// two threads' displays of different sizes: the smaller one's call between the
// larger one's attribute and its launch
static void threads() {
    g_meanwhile = [] { check(interleave(0, 4, 420, 2560) == cudaSuccess, "small tile"); };
    check(interleave(0, 48, 420, 1000) == cudaSuccess, "large tile beside a small one");
    g_meanwhile = [] { check(interleave(1, 4, 420, 2560) == cudaSuccess, "small tent tile"); };
    check(interleave(1, 100, 240, 1000) == cudaSuccess, "large tent tile beside a small one");
    g_meanwhile = [] { check(warp(1200) == cudaSuccess, "narrower warp"); };
    check(warp(4000) == cudaSuccess, "wide warp beside a narrow one");
}

int main(int, char** argv) {
    if (!strcmp(argv[1], "devices")) devices();
    if (!strcmp(argv[1], "retry")) retry();
    if (!strcmp(argv[1], "threads")) threads();
    if (!strcmp(argv[1], "tiny_pitch")) tiny_pitch();
    if (!strcmp(argv[1], "tent")) tent();
    if (!strcmp(argv[1], "gauss")) gauss();
    if (!strcmp(argv[1], "units")) units();
    if (!strcmp(argv[1], "splits")) splits();
    check(g_launched > 0, "something was launched");
    return g_failed;
}
