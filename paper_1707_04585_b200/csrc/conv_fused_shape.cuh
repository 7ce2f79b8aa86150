// Geometry of conv_fused_kernel (conv_fused.cu): how the positions of a layer are cut into ranges, segments, tiles and pieces, and how the
// shared memory of a CTA is divided.  Host code can include it by itself: tests/test_fused_shapes_host.py asks it which paths a shape takes.
#pragma once
#include "common.cuh"
#include <string.h>

constexpr int kFullBars = 16;             // tiles the build may run ahead of the MMAs
constexpr int kRawSlots = 16;             // most pieces of the input in shared memory
constexpr int kAuxSlots = 8;              // most tiles of an epilogue warp's partner rows in shared memory
constexpr int kAccBufs = 4;               // most accumulators
constexpr int NC = 16;                    // columns per epilogue thread
constexpr int kAuxBytes = 32 * NC * 4;    // partner rows of an epilogue warp's part of a tile: 32 rows x 64 bytes
__host__ __device__ constexpr int fused_threads(int EW, int NBT) { return EW * 32 + 64 + NBT; }      // NBT: build threads

// What all layers of a launch share
struct FusedGeom {
    int k;                 // 1 or 3
    int cin, nch;          // valid input channels, their 8-channel chunks
    int KC;                // channels of a weight row in shared memory: 16, 32 or 64 (rows of 32 / 64 / 128 bytes, swizzled by TMA)
    int ksteps;            // MMA steps of 16 channels per tap
    int wpitch;            // channels per tap in the weight pack (cin rounded up to 16)
    int BN, groups;        // output columns per CTA; groups = BN / NC: warp groups that share a tile (1, 2 or 4)
    int nacc, acc_shift;   // accumulators (2 or 4) and the logarithm of that
    int wtile_bytes;       // one tap of the weights: BN rows of KC bf16, rounded up to 1024
    int N, H, W, P, pitch; // P: pixels; pitch: positions per image row (W + 1; 1x1: unused)
    int nit, RS;           // the build: threads per row, rows in work at a time
    int step_r, step_c;    // 3x3: RS positions as whole image rows and columns
    int halo;              // operand rows before a tile's first position (3x3: W + 2, else 0)
    int total;             // positions in all
    int chunk;             // positions per CTA
    int S, nseg;           // tiles per operand segment, segment buffers (1 or 2)
    int plane16, seg_bytes, op_bytes;     // plane stride in 16-byte units; bytes of a segment buffer, of the whole operand region
    int tab_bytes, tabs;   // 3x3: the build's table of pixels, one entry per row of a segment; tables (see build_table)
    int pps, pieces;       // pieces per full segment, in all
    int piece, rowb;       // positions per piece of the input (a multiple of RS), bytes of a pixel of one input tensor
    int raw_bytes, raw_slots;             // bytes of a piece's slot, slots
    int aux_slots;         // tiles of partner rows that an epilogue warp holds
    FastDiv dpitch, drows, dnit, dpps;    // by positions per image row, by rows per image (H + 1), by nit, by pps
};
// Input of a launch
//   kInFloat, kInFixed   float / fixed-point tensor through BN + ReLU
//   kInBf16              bf16 tensor as it is (the gradient entering a data gradient)
//   kInBwd               gradient and BN input of the layer behind, through that layer's BN + ReLU backward
enum { kInFloat = 0, kInBf16 = 1, kInFixed = 2, kInBwd = 3 };
struct __align__(16) FusedShared {
    uint64_t full[kFullBars], seg_empty[2], acc_full[kAccBufs], acc_empty[kAccBufs], w_full;
    uint64_t raw_full[kRawSlots], raw_empty[kRawSlots], aux_full[16 * kAuxSlots];
    int raw_px[kRawSlots];           // first pixel of a piece
    uint32_t tmem_base, failed;
    __align__(16) float cf[7][64];   // per input channel: BN scale and shift; kInBwd: also mean, rstd and the three coefficients of the backward
    union {
        struct { __align__(16) double red[256 * 4], tot[32 * 4]; };    // statistics records; done with when the coefficients are there
        struct {
            __align__(16) float4 coef[64];            // BN+ReLU backward: (scale, shift, mean, rstd) of each output column
            __align__(16) float sums[16][2 * NC];     // per epilogue warp: NC sums, then NC second sums
        };
    };
};

static inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

struct FusedShape { int n_tiles, ctas, smem, EW, NBT; FusedGeom g; };

// aux: the epilogue reads a partner tensor.  The CTAs' ranges depend on geo, cin, cout, k and sm_count alone wherever the memory suffices.
static inline bool fused_shape(Geom geo, int cin, int cout, int k, int sm_count, int in_mode, bool aux, FusedShape &s) {
    if ((k != 1 && k != 3) || cin % 8 || cout % 4 || cin < 8 || cin > 64) return false;
    FusedGeom &g = s.g;
    memset(&g, 0, sizeof g);
    g.k = k; g.cin = cin; g.nch = cin / 8; g.wpitch = round_up(cin, 16); g.ksteps = g.wpitch / 16;
    g.KC = cin <= 16 ? 16 : (cin <= 32 ? 32 : 64);
    const size_t total = k == 3 ? (size_t)geo.N * (geo.H + 1) * (geo.W + 1) : geo.P();
    if (total >= (1u << 30)) return false;
    g.N = geo.N; g.H = geo.H; g.W = geo.W; g.P = (int)geo.P(); g.pitch = geo.W + 1;
    g.dpitch = fast_div(geo.W + 1); g.drows = fast_div(geo.H + 1);
    g.nit = in_mode == kInBwd ? 2 * g.nch : g.nch; g.dnit = fast_div(g.nit);
    g.halo = k == 3 ? geo.W + 2 : 0;
    g.total = (int)total;
    // pieces of about 12 KB
    const int tensors = in_mode == kInBwd ? 2 : 1;
    g.rowb = cin * (in_mode == kInBf16 ? 2 : 4);
    const int cout_pad = round_up(cout, 16), tiles = (g.total + 127) / 128, nchp = (g.nch + 1) & ~1;
    g.BN = cout_pad <= 16 ? 16 : (cout_pad <= 32 ? 32 : 64);
    // few tiles (late stages): split the output channels so that more SMs take part
    while (g.BN > 16 && tiles * ((cout_pad + g.BN - 1) / g.BN) * 2 <= sm_count) g.BN /= 2;
    bool tight = false;          // (very long rows: one shortest piece of the input at a time leaves the most to the operand)
    for (;; tight ? (void)0 : (void)(g.BN /= 2)) {
        s.n_tiles = (cout_pad + g.BN - 1) / g.BN;
        g.groups = g.BN / NC;
        s.EW = g.BN == 64 ? 16 : 8;
        g.nacc = g.BN == 64 ? 2 : 4; g.acc_shift = g.BN == 64 ? 1 : 2;
        int ctas = sm_count / s.n_tiles; if (ctas < 1) ctas = 1;
        // A contiguous range of positions per CTA, a tile at least.  (Half tiles would put a small layer on every SM, but take as long and
        // leave none to the launches of other streams beside it: 38-layer step 1680 -> 1635 us, 110-layer 4542 -> 4429, odd-sized basic block 153 -> 143
        // with whole ones.)  A layer of so few tiles that half ones leave half of the SMs takes those: 24 channels, 8 images of 9x17, block forward
        // 32.5 -> 31.2 us.
        const int least_chunk = tiles * 4 * s.n_tiles <= sm_count ? 64 : 128;
        g.chunk = round_up((g.total + ctas - 1) / ctas, 8); if (g.chunk < least_chunk) g.chunk = least_chunk;
        s.ctas = (g.total + g.chunk - 1) / g.chunk;
        // Six build warps, or ten where a CTA has a tile at most and so waits for its build (24 channels, 8 images of 9x17, forward: 19.7 against 18.8 us);
        // with more tiles they cost the epilogue beside them more than they give (16 channels, 14 images of 47x44: 21.6 against 22.6 us), and beside sixteen
        // epilogue warps there are no registers for them.
        s.NBT = s.EW == 8 && g.chunk <= 128 && !tight ? 320 : 192;
        g.RS = s.NBT / g.nit; g.step_r = g.RS / g.pitch; g.step_c = g.RS % g.pitch;
        g.piece = g.RS;
        while (!tight && 2 * g.piece * g.rowb * tensors <= 12800) g.piece *= 2;
        g.raw_bytes = round_up(g.piece * g.rowb, 128) * tensors;
        g.wtile_bytes = (g.BN * g.KC * 2 + 1023) & ~1023;
        const int T = (g.chunk + 127) / 128, fixed = 1024 + k * k * g.wtile_bytes + (int)sizeof(FusedShared) + 64;
        const int aux1 = aux ? s.EW * kAuxBytes : 0, sets = s.EW / 4 / g.groups, own_tiles = (T + sets - 1) / sets;
        // planes are skewed against each other so that the chunks of a pixel, written by adjacent threads, hit different banks
        auto plane_of = [&](int S) { return round_up(S * 128 + 2 * g.halo, 8) + (g.nch <= 2 ? 4 : (g.nch <= 4 ? 2 : 1)); };
        auto seg_of = [&](int S) { return round_up(nchp * plane_of(S) * 16, 128); };
        auto tab_of = [&](int S) { return k == 3 ? (((S * 128 < g.chunk ? S * 128 : g.chunk) + 2 * g.halo) * 4 + 127) & ~127 : 0; };
        auto pieces_of = [&](int S) { return ((S * 128 < g.chunk ? S * 128 : g.chunk) + 2 * g.halo + g.piece - 1) / g.piece; };
        const int room = 227 * 1024 - fixed, least = 20480;      // least: the last reduction borrows the operand region, (512 + 128) x 4 doubles
        // the whole range as one segment if it fits, else the longest segments of which two fit; beside them two pieces of the
        // input and, for each epilogue warp, one tile's partner rows at least
        auto tabs_of = [&](int nseg) { return nseg == 2 && 32 % g.nit != 0 ? 2 : 1; };
        auto fits = [&](int S, int nseg) {
            const int op = nseg * seg_of(S);
            return (op < least ? least : op) + (tight || (T <= S && pieces_of(S) < 2) ? 1 : 2) * g.raw_bytes + aux1 + tabs_of(nseg) * tab_of(S) <= room;
        };
        // (1x1: no halo to build twice, short segments leave the room to the rings)
        if (T <= (k == 1 ? 2 : kFullBars) && fits(T, 1)) { g.S = T; g.nseg = 1; }
        else {
            g.nseg = 2; g.S = k == 1 ? 2 : kFullBars / 2;
            while (g.S > 1 && !fits(g.S, 2)) g.S--;
            // One buffer of longer segments, where the 2 halo rows that every segment builds again cost more than the wait for the MMAs at each
            // end of a segment, about as long as two rounds of RS rows
            int S1 = kFullBars;
            while (S1 > 1 && !fits(S1, 1)) S1--;
            const int segs1 = (T + S1 - 1) / S1, segs2 = (T + g.S - 1) / g.S;
            if (!fits(g.S, 2) || (k == 3 && g.halo * (segs2 - segs1) >= g.RS * (segs1 - 1))) { g.nseg = 1; g.S = (T + segs1 - 1) / segs1; }
        }
        g.plane16 = plane_of(g.S);
        g.seg_bytes = seg_of(g.S);
        g.op_bytes = g.nseg * g.seg_bytes;
        if (g.op_bytes < least) g.op_bytes = least;
        g.tab_bytes = tab_of(g.S); g.tabs = tabs_of(g.nseg);
        const int tab = g.tabs * g.tab_bytes;
        g.pps = pieces_of(g.S); g.dpps = fast_div(g.pps);
        g.pieces = T <= g.S ? g.pps : 2 * kRawSlots;        // (more than the ring holds, or counted as if)
        // what is left goes to more pieces and more partner rows in flight, whichever has less
        // (a range that fits in two pieces beside two tiles of partner rows comes in two, the first with the first tile's rows at least:
        // every piece costs a build warp 0.3 us)
        if (T <= g.S && !tight) {
            const int rows = g.chunk + 2 * g.halo, first = 128 + 2 * g.halo, half = (rows + 1) / 2;
            const int R = round_up(half < first && first < rows ? first : half, g.RS), bytes = round_up(R * g.rowb, 128) * tensors;
            if (R > g.piece && g.op_bytes + tab + (R >= rows ? 1 : 2) * bytes + 2 * aux1 <= room) {
                g.piece = R; g.raw_bytes = bytes; g.pps = g.pieces = pieces_of(g.S); g.dpps = fast_div(g.pps);
            }
        }
        // several segments: pieces as long as two of them fit, at most two thirds of a segment (24 -> 48 KB: 64 channels at 32x32, batch 128, forward 174 -> 170 us)
        if (T > g.S && !tight) {
            while (g.op_bytes + tab + 2 * round_up(2 * g.piece * g.rowb, 128) * tensors + aux1 <= room && 3 * g.piece <= g.S * 128 + 2 * g.halo) {
                g.piece *= 2; g.raw_bytes = round_up(g.piece * g.rowb, 128) * tensors;
            }
            g.pps = pieces_of(g.S); g.dpps = fast_div(g.pps);
        }
        const int most_raw = T <= g.S ? (pieces_of(g.S) < kRawSlots ? pieces_of(g.S) : kRawSlots) : kRawSlots;
        const int most_aux = !aux ? 0 : (own_tiles < kAuxSlots ? own_tiles : kAuxSlots);
        g.raw_slots = most_raw < 2 || tight ? 1 : 2; g.aux_slots = aux ? 1 : 0;
        int left = room - g.op_bytes - tab - g.raw_slots * g.raw_bytes - g.aux_slots * aux1;
        s.smem = 227 * 1024 - left;
        if (left >= 0 && g.plane16 < (1 << 14)) {
            while (true) {
                const bool r = g.raw_slots < most_raw && left >= g.raw_bytes, x = g.aux_slots < most_aux && left >= aux1;
                if (!r && !x) break;
                if (r && (!x || g.raw_slots * g.raw_bytes <= g.aux_slots * aux1)) { g.raw_slots++; left -= g.raw_bytes; }
                else { g.aux_slots++; left -= aux1; }
            }
            s.smem = 227 * 1024 - left;
            return true;
        }
        if (g.BN < 32) { if (tight) return false; tight = true; }
    }
}

// Whether a data gradient takes its input through the BN backward of the layer behind (s: its shape as kInBwd).
// Only where a build thread has few rows: its pass costs 0.3 us per row and thread, twice that of a bf16 input with
// twice the threads per row, against 5 us for the launch that it saves.  Odd-sized block (24 channels, a tile per CTA, five and a half rows)
// 151 -> 144.5 us; 56 channels at 8x8 (eleven rows) and 16 at 32x32 (twenty-one): 38-layer step 1665 -> 1686.
static inline bool fused_folds(const FusedShape &s) { return (long long)(s.g.chunk + 2 * s.g.halo) * s.g.nit <= 6 * 192; }
