// Geometry of wgrad3x3_strip_kernel (conv_simt.cu).  Host code can include it by itself: tests/test_strip_shapes_host.py holds the cases of the
// GPU tests against it.
#pragma once
#include "common.cuh"

struct WgStrip {
    int N, H, W, Ci, Co;
    int cq, oq, pairs, sl, nb, R;         // quads per pixel, pairs of quads; slices per warp, blocks of pairs, row groups
    int BH, strips, per_img, per_cta;
    int a_floats, g_floats;               // of a buffer
    FastDiv dcq, dw2, dpairs, dimg, dnb;  // by cq, by W + 2, by pairs, by per_img, by nb
};
constexpr int kWgStripThreads = 480;
// Most pairs of quads.  Above (56 channels and more) no two warps share a row and the implicit GEMM is as quick or quicker: 56 channels at
// 8x8, batch 128, 24.6 against 24.5 us; fp32 stored step of the 110-layer network at batch 23 7.42 against 7.74 ms.
constexpr int kWgStripPairs = 144;
constexpr int kWgStripRun = 33;           // products of a run; pieces of a row are multiples of the loop's three pixels
constexpr int kWgStripRow = 512;          // longest row
// The shape of a launch on a 3x3 stride-1 layer; false: not taken (more channels, rows too long for the shared memory, tensors too small).
// most: CTAs whose partials there is room for
static bool wg_strip_shape(int N, int H, int W, int Ci, int Co, int sm, int most, WgStrip &p, int &ctas, int &threads, int &smem) {
    if (Ci % 4 || Co % 4 || Ci > 64 || Co > 64 || W > kWgStripRow) return false;
    p.N = N; p.H = H; p.W = W; p.Ci = Ci; p.Co = Co;
    p.cq = Ci / 4; p.oq = Co / 4; p.pairs = p.cq * p.oq;
    if (p.pairs > kWgStripPairs) return false;
    p.sl = p.pairs <= 16 ? 32 / p.pairs : 1;
    p.nb = p.sl > 1 ? 1 : (p.pairs + 31) / 32;
    if (p.sl > p.H) p.sl = p.H;
    // strips: two buffers of as many rows, a multiple of the slices, as there is shared memory for; one round of the slices at least
    const size_t room = 200 * 1024;
    auto bytes_of = [&](int bh) { return 2 * ((size_t)(bh + 2) * (W + 2) * Ci + (size_t)bh * W * Co) * sizeof(float); };
    if (bytes_of(p.sl) > room) return false;
    // Groups of rows: as many as make about twelve warps.  Where those CTAs would not fill the SMs, the number that gives an SM the shortest run of
    // rows.  CTAs per SM: one, or two to five of fewer warps where their buffers fit side by side.  (An SM counts as idle in part below six warps)
    int fit = 0, side = 1;             // CTAs in all, CTAs side by side on an SM
    long long least = -1;
    for (int R = 4 / p.nb < 1 ? 1 : 4 / p.nb; R >= 1; R--) {
        const int sl = R * p.sl, n = 96 * p.nb * R;
        if (R > 1 && (sl > p.H || bytes_of(sl) > room)) continue;
        int per_sm = kWgStripThreads / n;
        while (per_sm > 1 && bytes_of(sl) > room / per_sm) per_sm--;
        const int f = most < sm * per_sm ? most : sm * per_sm, strips = p.N * ((p.H + sl - 1) / sl), ctas1 = strips < f ? strips : f;
        const int warps = 3 * p.nb * R * ((ctas1 + sm - 1) / sm);
        const long long cost = (long long)((strips + f - 1) / f) * (warps < 6 ? 6 : warps);
        if (least < 0 || cost < least) { least = cost; p.R = R; fit = f; side = per_sm; threads = n; }
        if (strips >= sm) break;
    }
    if (threads * side < 192) return false;          // (rows so long that an SM holds one warp per row tap)
    const int slices = p.R * p.sl;
    // (of the heights the one that gives a CTA the fewest rows, its strips' halos counted as one each)
    long long best = -1;
    for (int bh = slices;; bh += slices) {
        const int h = bh < p.H ? bh : p.H, strips = p.N * ((p.H + h - 1) / h);
        const long long cost = (long long)((strips + fit - 1) / fit) * (h + 1);
        if (best < 0 || cost <= best) { best = cost; p.BH = h; }
        if (h == p.H || bytes_of(bh + slices) > room / side) break;
    }
    p.a_floats = (p.BH + 2) * (W + 2) * Ci; p.g_floats = p.BH * W * Co;
    size_t bytes = bytes_of(p.BH);
    const size_t red = slices > 1 ? (size_t)slices * 9 * Ci * Co * 4 : 0;
    if (bytes < red) bytes = red;
    if (bytes > room) return false;                  // (a few rows beside a large reduction: fewer CTAs per SM than counted on)
    smem = (int)bytes;
    p.per_img = (p.H + p.BH - 1) / p.BH; p.strips = p.N * p.per_img;
    p.per_cta = (p.strips + fit - 1) / fit;          // the same number of strips each
    ctas = (p.strips + p.per_cta - 1) / p.per_cta;
    // Partials for too few SMs: the implicit GEMM spreads its tiles of dW as well.  Few channels gain most from strips: 24 channels, 40 images of 13x12,
    // 299 us with the GEMM against 286 with strips on 54 % of the SMs; 40 channels, 40 of 31x25, 692 against 714 on 65 %.
    if (most < sm && ctas * 4 <= sm * (p.pairs <= 36 ? 2 : 3)) return false;
    p.dcq = fast_div(p.cq); p.dw2 = fast_div(W + 2); p.dpairs = fast_div(p.pairs); p.dimg = fast_div(p.per_img); p.dnb = fast_div(p.nb);
    return true;
}
