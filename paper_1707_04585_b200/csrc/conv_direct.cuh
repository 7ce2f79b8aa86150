// Geometry of conv3x3_direct_kernel (conv_simt.cu): how a 3x3 stride-1 layer is cut into tiles, and which rows a lane stores.
// Host code can include it by itself: tests/test_direct_tiles_host.py checks every address against the tensors with it.
#pragma once
#include "common.cuh"

struct DirectGeom {
    int N, H, W, Ci, Co;                          // Ci: channels summed over, Co: produced
    int NW, gx, gy, gi, CB, kc, pitch;            // warps of a CTA, of a tile, channels per chunk, floats per staged pixel
    int tx, ty, tiles;                            // tiles of an image, of all
    FastDiv dtx, dty, dq, dcol, drow;             // by tx, ty, quads per chunk, staged columns, staged rows
};
// rows that the lane at output n, column x, first row y of image i stores (and reads of the coupling partner), zero or less for none:
// the lower warps of a tile may lie below the image altogether
__host__ __device__ inline int direct_live_rows(const DirectGeom &g, int n, int x, int y, int i) {
    if (n >= g.Co || x >= g.W || i >= g.N) return 0;
    return g.H - y < 8 ? g.H - y : 8;
}
// Tiles of a layer: false where less than half of their pixels would lie inside an image.  Four warps per CTA where eight would
// leave SMs without one.
static bool direct_shape(int N, int H, int W, int Ci, int Co, int sm, DirectGeom &g) {
    g.N = N; g.H = H; g.W = W; g.Ci = Ci; g.Co = Co;
    g.CB = Co > 16 ? 2 : 1;
    g.kc = Ci < 32 ? Ci : 32;
    g.pitch = (g.kc / 4) % 2 ? g.kc : g.kc + 4;
    for (g.NW = 8; g.NW >= 4; g.NW -= 4) {
        const int wpx = g.NW / g.CB, nbs = (Co + g.CB * 16 - 1) / (g.CB * 16);
        g.gx = W <= 4 ? 1 : (W <= 8 ? 2 : 4);
        if (g.gx > wpx) g.gx = wpx;
        g.gy = wpx / g.gx;
        while (g.gy > 1 && (g.gy >> 1) * 8 >= H) g.gy >>= 1;
        g.gi = wpx / (g.gx * g.gy);
        g.tx = (W + g.gx * 4 - 1) / (g.gx * 4); g.ty = (H + g.gy * 8 - 1) / (g.gy * 8);
        const long long tiles = (long long)g.tx * g.ty * ((N + g.gi - 1) / g.gi);
        if (tiles * wpx * 32 > 2ll * N * H * W || tiles > (1 << 28)) { if (g.NW == 8) continue; return false; }
        g.tiles = (int)tiles;
        if (tiles * nbs >= sm || g.NW == 4) break;
    }
    g.dtx = fast_div(g.tx); g.dty = fast_div(g.ty); g.dq = fast_div(g.kc / 4); g.dcol = fast_div(g.gx * 4 + 2); g.drow = fast_div(g.gy * 8 + 2);
    return true;
}
