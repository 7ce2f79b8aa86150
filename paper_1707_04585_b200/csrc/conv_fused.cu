// BN -> ReLU -> conv as ONE kernel for layers with at most 64 input channels (stride 1, k = 1 or 3):
// the layers whose cost is memory traffic and latency, not arithmetic (Eq. 2: c_k(x) = Conv_kxk(ReLU(BN(x)))).
//
// What bounds it: on the CIFAR-sized networks a launch has one to eight 128-row tiles per SM, so its time is the chain of
// dependent steps from the predecessor's end to its own, not its bytes.  Everything here serves a short chain.
//
// Positions.  For a 3x3 layer the pixels are numbered with one padding column behind every image row and one padding row
// behind every image: position p = (n (H+1) + r)(W+1) + c.  The neighbour at tap (kh, kw) is then position
// p + (kh-1)(W+1) + (kw-1) whatever p is -- left of column 0 lies the padding column of the row above, above row 0 the
// padding row of the image before -- so a GEMM tile is ANY 128 consecutive positions, for any H and W, and a CTA takes one
// contiguous range of positions.  (1x1 layers: position = pixel.)
// Operand.  The activated bf16 rows of a range sit in shared memory in the unswizzled K-major layout, one plane of 16 bytes
// per row for every 8 channels: row l of plane j at j * plane + 16 l.  A tap's operand is the same planes from a row further
// on, so every pixel is loaded, normalised and written once per range (plus the halo of W + 2 rows on either side), not
// once per tap or per tile.
// Input and partner rows arrive through shared memory, not through registers: the pixels of consecutive positions lie side by side in memory,
// so the input of a range is a handful of bulk copies (pieces of about 12 KB), all of them under way as soon as the kernel before has ended,
// and the partner rows of an epilogue warp's part of a tile are one TMA box of 32 rows x 64 bytes, in a ring of its own.
// Roles (one CTA per SM):
//   EW warps    epilogue (8, or 16 for 64 output columns), one accumulator row and 16 columns per thread, straight
//               from tensor memory to global memory with 32-byte accesses: coupling on the float or fixed-point state, or plain
//               store; the per-channel sums (batch statistics of the stored result, or the two sums of the BN+ReLU backward)
//               stay in registers until the last tile.  Four warps make a group (128 rows x 16 columns); the groups split a
//               tile's columns between them, and what is left over takes alternate tiles.  Before the first tile eight of
//               them add the statistics records of the kernel before (BnRef::part).
//   1 warp      weights (TMA, resident), tensor memory, MMA issue; two or four accumulators
//   1 warp      the input's pieces and the first partner rows
//   6 warps     (or 10) build: a row's 8 channels from shared memory, scale*x + shift, ReLU, bf16 rounding, one 16-byte store to the operand
//               (and one to the activated tensor the weight gradient will read)
// The same kernel computes data gradients: its input is then the bf16 upstream gradient, taken as it is, or (kInBwd) the gradient and
// the BN input of the layer behind, whose BN + ReLU backward the build applies; the weights are the mirrored, transposed pack.
// Measured, from the end of the wait for the kernel before to the last CTA's end, against the form whose seven build warps and epilogue warps
// loaded from global memory into registers (four loads in flight per thread): data gradient of 16 channels at 32x32, batch 128, 12.3 -> 10.7 us,
// of 32 at 16x16 12.3 -> 10.3, forward 12.0 -> 11.5; 32 -> 128 channels of the CIFAR-sized bottleneck network at 32x32 (1x1) 57.7 us by
// events, 45 now.  Where a launch's time goes (16 channels, 32x32): first pieces there after 1.0 us, records added after 1.7, coefficients
// after 2.2, first tile built after 3.4, last after 7.2, last accumulator drained after 8.5, sums 1.1 more.  The build is a chain of
// latencies: 0.2 us per row and thread, 0.1 per tile signalled, 0.3 per piece.
// Every mbarrier wait is bounded; on expiry the kernel records a status word and leaves.
#include "common.cuh"
#include "tc_ptx.cuh"
#include "conv_epilogue.cuh"
#include "conv_fused_shape.cuh"
#include <cuda.h>
#include <string.h>

using namespace tc;

namespace {

// The epilogue of one layer (field names as epilogue_publish expects them)
struct FusedEpi {
    int mode, sign, n_cols;
    float *out;            // [P, n_cols]
    float q;               // format of out (and of the coupling partner), or of the BN input of a data gradient: 0 float, else fixed-point step
    float *part;           // per-CTA records of the column sums, or null
    unsigned int *counter; // a word per N tile; null: the records stay pending, their consumer adds them
    double inv_count;
    float eps;
    float *mean, *rstd;
    BnRef bn;              // EPI_BNBWD
    float *dgamma, *dbeta, *coef;
};
struct FusedLayer {
    int in_mode;
    int wide_out;          // 32-byte aligned rows: 32-byte accesses
    int w_early;           // the weights were packed before the predecessor kernel: they may be loaded while it runs
    const void *in;
    const float *in_t;     // kInBwd: the BN input (in: the gradient w.r.t. the activated tensor)
    float in_q;            // kInFixed: fixed-point step of the input
    BnRef bn;              // all but kInBf16.  kInBwd: part holds the records of the backward sums
    float *in_dgamma, *in_dbeta;          // kInBwd: where those sums go
    bf16 *a_out;           // all but kInBf16, optional: the operand tensor [P, cin] (for the weight gradient)
    FusedEpi epi;
};
struct FusedArgs {
    CUtensorMap map_w, map_x;     // weights; coupling partner, or the BN input of a data gradient
    FusedGeom g;
    FusedLayer ly;
    int *status;
    unsigned long long *stamp;    // timeline slot of this launch (nullptr: off)
};

// two floats -> (ReLU ->) bf16x2 (round to nearest even), one instruction
__device__ __forceinline__ uint32_t relu_pack2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// a bounded wait of a whole warp: lane 0 polls
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, int lane) {
    bool ok = true;
    if (lane == 0) ok = mbar_wait(bar, parity);
    return __shfl_sync(0xffffffffu, ok, 0);
}
// bytes (a multiple of 16, both addresses too) from global to shared memory
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// pixel at position q, -1 for padding and for positions outside the batch
__device__ __forceinline__ int pixel_at(const FusedGeom &g, int q) {
    if ((unsigned)q >= (unsigned)g.total) return -1;
    if (g.k == 1) return q;
    uint32_t row, c, n, r;
    g.dpitch.divmod((uint32_t)q, row, c);
    g.drows.divmod(row, n, r);
    return (int)c < g.W && (int)r < g.H ? (int)(n * g.H + r) * g.W + (int)c : -1;
}
// pixels before position q
__device__ __forceinline__ int pixels_before(const FusedGeom &g, int q) {
    if (q <= 0) return 0;
    if (q >= g.total) return g.P;
    if (g.k == 1) return q;
    uint32_t row, c, n, r;
    g.dpitch.divmod((uint32_t)q, row, c);
    g.drows.divmod(row, n, r);
    return (int)(n * g.H + r) * g.W + ((int)r < g.H ? ((int)c < g.W ? (int)c : g.W) : 0);
}
// image, row and column of position q (3x3 layers; q may lie before the first image: image -1)
__device__ __forceinline__ void place_at(const FusedGeom &g, int q, int &n, int &r, int &c) {
    const int img = g.pitch * (g.H + 1);
    uint32_t row, cc, nn, rr;
    g.dpitch.divmod((uint32_t)(q + img), row, cc);        // the halo reaches W + 2 positions back, never more than an image
    g.drows.divmod(row, nn, rr);
    n = (int)nn - 1; r = (int)rr; c = (int)cc;
}

// unswizzled K-major operand: rows 16 bytes apart (groups of eight 128 bytes apart), 8-channel planes plane16 16-byte units apart
__device__ __forceinline__ uint64_t plane_desc(uint32_t addr, int plane16) {
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(plane16 & 0x3FFF) << 16) | ((uint64_t)8 << 32) | ((uint64_t)1 << 46);
}

// All MMAs of one tile (one thread): taps in row-major order, KS steps of 16 channels each
template <int KS>
__device__ __forceinline__ void issue_tile(const FusedGeom &g, uint32_t acc, uint64_t a, uint64_t w, uint32_t idesc) {
    const uint32_t wtile16 = (uint32_t)g.wtile_bytes >> 4;
    uint32_t accum = 0;
    int kw = 0;
    for (int tap = 0; tap < g.k * g.k; tap++) {
#pragma unroll
        for (int kk = 0; kk < KS; kk++) {
            mma_bf16(acc, a + (uint32_t)(2 * kk * g.plane16), w + (uint32_t)(2 * kk), idesc, accum);
            accum = 1;
        }
        w += wtile16;
        a += 1;
        if (++kw == g.k) { kw = 0; a += (uint32_t)(g.pitch - g.k); }
    }
}

// The input of a CTA arrives in pieces, through a ring.  The pixels of consecutive positions lie side by side in memory: a piece is one bulk
// copy (kInBwd: two).  First and last pixel of piece n:
__device__ __forceinline__ void piece_at(const FusedGeom &g, int pos0, int pos1, int n, int &a, int &b) {
    uint32_t seg, j;
    g.dpps.divmod((uint32_t)n, seg, j);
    const int sb = pos0 + (int)seg * g.S * 128, own = pos1 - sb < g.S * 128 ? pos1 - sb : g.S * 128, rows = own + 2 * g.halo;
    const int r0 = (int)j * g.piece, r1 = r0 + g.piece < rows ? r0 + g.piece : rows;
    a = pixels_before(g, sb - g.halo + r0); b = pixels_before(g, sb - g.halo + r1);
}
__device__ __forceinline__ void load_piece(const FusedGeom &g, const FusedLayer &p, FusedShared *sh, uint8_t *raw, int slot, int a, int b) {      // one thread
    const bool two = p.in_mode == kInBwd;
    const uint32_t bytes = (uint32_t)((b - a) * g.rowb);
    uint8_t *dst = raw + slot * g.raw_bytes;
    sh->raw_px[slot] = a;
    mbar_expect_tx(&sh->raw_full[slot], two ? 2 * bytes : bytes);
    if (bytes) {
        bulk_load(dst, reinterpret_cast<const uint8_t *>(p.in) + (size_t)a * g.rowb, bytes, &sh->raw_full[slot]);
        if (two) bulk_load(dst + (g.raw_bytes >> 1), reinterpret_cast<const uint8_t *>(p.in_t) + (size_t)a * g.rowb, bytes, &sh->raw_full[slot]);
    }
}

// The build of a CTA's operand rows.  A thread keeps its channels (eight; kInBwd: four) and takes rows r0, r0 + RS, ... of each
// segment.  The pixels of its rows (-1: padding) stand in a table, for the first segment filled while the kernel before this one
// still runs: six build warps are one or two per scheduler, so every instruction between a row's load and its
// store costs its full latency.  One row per iteration: a loop that outgrows the scheduler's instruction buffer is slower than a
// short one with nothing in flight.
// The nit threads of a row write the same entry.  Where nit does not divide 32 they can sit in two warps, and one warp may be a segment
// ahead of the other: segments in two buffers then have a table each, filled behind the wait for the segment's buffer.  That wait
// ends when the MMAs have read the segment that had the buffer before, so every warp has built all its rows and left its table.
struct BuildPlace { int item, r0, low0; };
__device__ __forceinline__ BuildPlace build_place(const FusedGeom &g, int bt) {
    BuildPlace b;
    uint32_t q, r;
    g.dnit.divmod((uint32_t)bt, q, r);
    b.item = (int)r; b.r0 = (int)q; b.low0 = (int)g.dnit.div((uint32_t)(bt & ~31));
    return b;
}
__device__ __forceinline__ void build_table(const FusedGeom &g, int *tab, int r0, int first, int rows) {      // first: position of row 0
    if (g.k == 1 || r0 >= g.RS) return;
    int n, r, c;
    place_at(g, first + r0, n, r, c);
    for (int l = r0; l < rows; l += g.RS) {
        tab[l] = c < g.W && (unsigned)r < (unsigned)g.H && (unsigned)n < (unsigned)g.N ? (n * g.H + r) * g.W + c : -1;
        c += g.step_c; r += g.step_r;
        if (c >= g.pitch) { c -= g.pitch; r++; }
        while (r > g.H) { r -= g.H + 1; n++; }
    }
}
// K1: 1x1 layers, where position and pixel are the same and no row is padding.
template <int IN, int EW, int NBT, bool K1>
__device__ __forceinline__ bool build_rows(const FusedGeom &g, const FusedLayer &p, FusedShared *sh, const uint8_t *raw, uint8_t *abuf, int *tab, int pos0, int pos1,
                                           const BuildPlace bp, int lane) {
    constexpr int V = IN == kInBwd ? 4 : 8;               // channels of a thread
    const int RS = g.RS, it = bp.item;
    const int n_tiles = (pos1 - pos0 + 127) >> 7;
    float sc[V], sf[V], mu[V], rs[V], k0[V], k1[V], k2[V];       // (the last five: kInBwd)
    bool first = true;
    int slot = 0; uint32_t round = 0;
    for (int t0 = 0, seg = 0; t0 < n_tiles; t0 += g.S, seg++) {
        const int T = n_tiles - t0 < g.S ? n_tiles - t0 : g.S;
        const int sb = pos0 + t0 * 128, own = pos1 - sb < T * 128 ? pos1 - sb : T * 128, rows = own + 2 * g.halo;
        const int my_rows = bp.r0 < RS ? rows : 0;
        uint8_t *dst = abuf + (g.nseg == 2 ? (seg & 1) : 0) * g.seg_bytes + (IN == kInBwd ? (it >> 1) * g.plane16 * 16 + (it & 1) * 8 : it * g.plane16 * 16);
        if (seg >= g.nseg && !warp_wait(&sh->seg_empty[g.nseg == 2 ? (seg & 1) : 0], (uint32_t)((g.nseg == 2 ? seg >> 1 : seg) - 1) & 1u, lane)) return false;
        if (!K1 && seg > 0) {
            if (g.tabs == 2) tab += seg & 1 ? g.tab_bytes >> 2 : -(g.tab_bytes >> 2);
            build_table(g, tab, bp.r0, sb - g.halo, rows);
        }
        int l = bp.r0, low = bp.low0, j = 0, ready = 128 + 2 * g.halo;          // ready: rows that the tile to be signalled next needs
        auto signal = [&]() {
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->full[(t0 + j) & (kFullBars - 1)]);
            j++; ready += 128;
        };
        for (int pr = 0; pr < rows; pr += g.piece) {
            const bool here = mbar_wait(&sh->raw_full[slot], round & 1u);
            if (first) {                                     // (also when the wait ran out: the epilogue warps stand at this barrier)
                first = false;
                if (IN != kInBf16) {
                    named_barrier(3, EW * 32 + NBT + 32);         // the coefficients are there
#pragma unroll
                    for (int i = 0; i < V; i++) {
                        const int c = it * V + i;
                        sc[i] = sh->cf[0][c] * (IN == kInFixed ? p.in_q : 1.f); sf[i] = sh->cf[1][c];
                        if (IN == kInBwd) { mu[i] = sh->cf[2][c]; rs[i] = sh->cf[3][c]; k0[i] = sh->cf[4][c]; k1[i] = sh->cf[5][c]; k2[i] = sh->cf[6][c]; }
                    }
                }
            }
            if (!__all_sync(0xffffffffu, here)) return false;
            const int pxs = sh->raw_px[slot];
            const uint8_t *src = raw + slot * g.raw_bytes + it * (IN == kInFloat || IN == kInFixed ? 32 : 16);
#pragma unroll 1
            for (int i = 0; i < g.piece && low < rows; i += RS) {
                if (l < my_rows) {
                    const int px = K1 ? sb + l : tab[l];
                    const uint8_t *s = src + (px - pxs) * g.rowb;
                    const bool keep = p.a_out && (K1 || (unsigned)(l - g.halo) < (unsigned)own);
                    if constexpr (IN == kInBwd) {
                        uint2 v = make_uint2(0u, 0u);
                        if (K1 || px >= 0) {
                            const float4 d4 = *reinterpret_cast<const float4 *>(s), t4 = *reinterpret_cast<const float4 *>(s + (g.raw_bytes >> 1));
                            const float d[4] = {d4.x, d4.y, d4.z, d4.w}, t[4] = {t4.x, t4.y, t4.z, t4.w};
                            float o[4];
                            // (as bn_relu_bwd_apply_kernel has it)
#pragma unroll
                            for (int c = 0; c < 4; c++) o[c] = k0[c] * (fmaf(sc[c], t[c], sf[c]) > 0.f ? d[c] : 0.f) - k1[c] - k2[c] * ((t[c] - mu[c]) * rs[c]);
                            v = make_uint2(pack2(o[0], o[1]), pack2(o[2], o[3]));
                            if (keep) *reinterpret_cast<uint2 *>(p.a_out + (size_t)px * g.cin + it * 4) = v;
                        }
                        *reinterpret_cast<uint2 *>(dst + l * 16) = v;
                    } else {
                        uint4 v = make_uint4(0u, 0u, 0u, 0u);
                        if (K1 || px >= 0) {
                            v = *reinterpret_cast<const uint4 *>(s);
                            if constexpr (IN != kInBf16) {
                                const uint4 w = *reinterpret_cast<const uint4 *>(s + 16);
                                const uint32_t r[8] = {v.x, v.y, v.z, v.w, w.x, w.y, w.z, w.w};
                                float x[8];
#pragma unroll
                                for (int c = 0; c < 8; c++) x[c] = fmaf(sc[c], IN == kInFixed ? __int2float_rn((int)r[c]) : __uint_as_float(r[c]), sf[c]);
                                v = make_uint4(relu_pack2(x[0], x[1]), relu_pack2(x[2], x[3]), relu_pack2(x[4], x[5]), relu_pack2(x[6], x[7]));
                                if (keep) *reinterpret_cast<uint4 *>(p.a_out + (size_t)px * g.cin + it * 8) = v;
                            }
                        }
                        *reinterpret_cast<uint4 *>(dst + l * 16) = v;
                    }
                }
                l += RS; low += RS;
                while (j < T && low >= ready) signal();
            }
            if (g.pieces > g.raw_slots) {                    // (else nothing waits for the slot)
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh->raw_empty[slot]);
            }
            if (++slot == g.raw_slots) { slot = 0; round++; }
        }
        while (j < T) signal();
    }
    return true;
}

// An epilogue warp's own ring of partner rows (its 32 rows and 16 columns of a tile): the copy of its k-th tile
struct AuxRing { uint8_t *buf; uint64_t *bar; int col, on; };
__device__ __forceinline__ AuxRing aux_ring(const FusedArgs &A, FusedShared *sh, uint8_t *auxb, int warp) {
    const FusedGeom &g = A.g;
    AuxRing x;
    x.buf = auxb + warp * g.aux_slots * kAuxBytes; x.bar = sh->aux_full + warp * kAuxSlots;
    x.col = (int)blockIdx.y * g.BN + ((warp >> 2) & (g.groups - 1)) * NC;
    x.on = A.ly.epi.mode != EPI_PLAIN && x.col < A.ly.epi.n_cols;
    return x;
}
__device__ __forceinline__ void aux_load(const FusedArgs &A, const AuxRing &x, int slot, int row) {       // one thread; row: the first pixel
    mbar_expect_tx(&x.bar[slot], kAuxBytes);
    tma_load_2d(x.buf + slot * kAuxBytes, &A.map_x, &x.bar[slot], x.col, row);
}

// Epilogue of one warp's rows.  EK: 0 plain, 1 float coupling, 2 fixed-point coupling, 3 / 4 BN+ReLU backward with a float /
// fixed-point BN input.
template <int EW, int EK>
__device__ __forceinline__ bool epilogue_loop(const FusedArgs &A, FusedShared *sh, const AuxRing &ax, int pos0, int pos1, int warp, int lane, uint32_t tmem_d,
                                              float (&s)[NC], float (&ss)[NC]) {
    const FusedGeom &g = A.g;
    const FusedLayer &p = A.ly;
    const FusedEpi &e = p.epi;
    const int grp = warp >> 2, wrow = (warp & 3) * 32;
    const int sets = EW / 4 / g.groups, set = grp / g.groups;                     // tiles set, set + sets, ...
    const bool wide = p.wide_out != 0;
    const int lc = (grp & (g.groups - 1)) * NC, col = ax.col;                           // this thread's first column: in the CTA, in the tensor
    const float q = e.q, out_s = (EK <= 2 && q != 0.f) ? 1.f / q : 0.f, sgn = e.sign < 0 ? -1.f : 1.f;
    const int isgn = e.sign < 0 ? -1 : 1;
    const float4 *coef = sh->coef + lc;
    const int n_tiles = (pos1 - pos0 + 127) >> 7;
    const uint32_t tm = tmem_d + ((uint32_t)wrow << 16) + (uint32_t)lc;
    int slot = 0; uint32_t round = 0;
    for (int ti = set; ti < n_tiles; ti += sets) {
        const int qw = pos0 + ti * 128 + wrow, q0 = qw + lane, px = q0 < pos1 ? pixel_at(g, q0) : -1;
        const size_t off = (size_t)(px < 0 ? 0 : px) * e.n_cols + col;
        const uint32_t keep = px >= 0 ? 0xffffffffu : 0u;      // rows that hold no pixel add nothing (a select, not a branch per column)
        const int xr = px < 0 ? 0 : px - pixels_before(g, qw);
        const uint8_t *xrow = ax.buf + slot * kAuxBytes + xr * 64;
        const int swz = (xr >> 1) & 3, buf = ti & (g.nacc - 1);
        bool ok = true;
        if (lane == 0) {
            if (EK > 0 && ax.on) ok = mbar_wait(&ax.bar[slot], round & 1u);
            ok = ok && mbar_wait(&sh->acc_full[buf], (uint32_t)(ti >> g.acc_shift) & 1u);
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) return false;
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < NC; c += 8) {
            float v[8];
            uint32_t o[8], x[8];
            if (EK > 0) {
                const uint4 a = *reinterpret_cast<const uint4 *>(xrow + (((c >> 2) ^ swz) << 4)), b = *reinterpret_cast<const uint4 *>(xrow + ((((c >> 2) + 1) ^ swz) << 4));
                x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
            }
            tmem_ld8(tm + (uint32_t)(buf * g.BN + c), v);
#pragma unroll
            for (int i = 0; i < 8; i++) {
                float st = 0.f;               // what is summed
                if (EK == 0) {
                    if (q != 0.f) { const int iv = __float2int_rn(v[i] * out_s); o[i] = (uint32_t)iv; st = __int2float_rn(iv) * q; }
                    else { o[i] = __float_as_uint(v[i]); st = v[i]; }
                } else if (EK == 1) {
                    st = fmaf(sgn, v[i], __uint_as_float(x[i]));
                    o[i] = __float_as_uint(st);
                } else if (EK == 2) {
                    const int iv = (int)x[i] + isgn * __float2int_rn(v[i] * out_s);
                    o[i] = (uint32_t)iv; st = __int2float_rn(iv) * q;
                } else o[i] = __float_as_uint(v[i]);
                if (EK <= 2) {
                    st = __uint_as_float(__float_as_uint(st) & keep);
                    s[c + i] += st;
                    ss[c + i] = fmaf(st, st, ss[c + i]);
                } else {
                    const uint32_t xi = x[i] & keep;
                    const float t = EK == 4 ? __int2float_rn((int)xi) * q : __uint_as_float(xi);
                    const float4 k = coef[c + i];           // scale, shift, mean, rstd
                    const float d = fmaf(k.x, t, k.y) > 0.f ? __uint_as_float(__float_as_uint(v[i]) & keep) : 0.f;
                    s[c + i] += d;
                    ss[c + i] = fmaf(d, (t - k.z) * k.w, ss[c + i]);
                }
            }
            if (px >= 0) {
                float *dst = e.out + off + c;
                if (col + c + 8 <= e.n_cols) st8(dst, o, wide);
                else if (col + c < e.n_cols) *reinterpret_cast<uint4 *>(dst) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
            mbar_arrive(&sh->acc_empty[buf]);
            if (EK > 0 && ax.on && ti + g.aux_slots * sets < n_tiles) aux_load(A, ax, slot, pixels_before(g, qw + g.aux_slots * sets * 128));
        }
        if (++slot == g.aux_slots) { slot = 0; round++; }
    }
    return true;
}

// sums of each column over the 32 rows of a warp: after the call lane l holds column l & 15 in a[0]
__device__ __forceinline__ void column_sums(float (&a)[NC], int lane) {
#pragma unroll
    for (int o = NC / 2; o >= 1; o >>= 1) {
#pragma unroll
        for (int i = 0; i < o; i++) {
            const bool up = (lane & o) != 0;
            const float send = up ? a[i] : a[i + o], keep = up ? a[i + o] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 16);
}

// Registers: with eight epilogue warps 96, for 512 or 640 threads (80, for a bound of 672 threads, spill: 38-layer step 12 % slower).  No CTA of
// another stream shares the SM, the rings take what shared memory there is: weight gradients run on the SMs that a layer leaves empty.
template <int EW, int NBT>
__global__ void __launch_bounds__(EW == 8 ? 640 : fused_threads(EW, NBT), 1) conv_fused_kernel(const __grid_constant__ FusedArgs A) {
    extern __shared__ uint8_t smem_raw[];
    const FusedGeom &g = A.g;
    const FusedLayer &p = A.ly;
    const FusedEpi &e = p.epi;
    uint8_t *wres = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int taps = g.k * g.k;
    uint8_t *auxb = wres + taps * g.wtile_bytes;                            // partner rings (512-byte aligned for their swizzle)
    uint8_t *abuf = auxb + EW * g.aux_slots * kAuxBytes;
    uint8_t *raw = abuf + g.op_bytes;
    int *tab = (int *)(raw + g.raw_slots * g.raw_bytes);
    FusedShared *sh = (FusedShared *)((uint8_t *)tab + g.tabs * g.tab_bytes);

    constexpr int kMmaWarp = EW, kLoadWarp = EW + 1, kBuildWarp0 = EW + 2;
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const bool direct = p.in_mode == kInBf16;
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < g.nacc * g.BN) tmem_cols <<= 1;
    const int col0 = blockIdx.y * g.BN;
    const int pos0 = (int)blockIdx.x * g.chunk, pos1 = pos0 + g.chunk < g.total ? pos0 + g.chunk : g.total;
    auto load_weights = [&]() {
        mbar_expect_tx(&sh->w_full, (uint32_t)(taps * g.BN * g.KC * 2));
        for (int tap = 0; tap < taps; tap++) tma_load_2d(wres + tap * g.wtile_bytes, &A.map_w, &sh->w_full, tap * g.wpitch, col0);
    };

    BuildPlace bp{};
    AuxRing ax{};
    int piece_a = 0, piece_b = 0;        // loader: lane n's piece of the first ringful
    if (warp == kMmaWarp) {
        if (elect_one()) {
            tma_prefetch_desc(&A.map_w);
            for (int b = 0; b < kFullBars; b++) mbar_init(&sh->full[b], NBT / 32);
            for (int b = 0; b < 2; b++) mbar_init(&sh->seg_empty[b], 1);
            for (int b = 0; b < kAccBufs; b++) { mbar_init(&sh->acc_full[b], 1); mbar_init(&sh->acc_empty[b], 4 * g.groups); }
            mbar_init(&sh->w_full, 1);
            sh->failed = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            if (p.w_early) load_weights();
        }
        tmem_alloc(&sh->tmem_base, tmem_cols);
    } else if (warp == kLoadWarp) {
        if (lane < g.raw_slots) {
            mbar_init(&sh->raw_full[lane], 1); mbar_init(&sh->raw_empty[lane], NBT / 32);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            piece_at(g, pos0, pos1, lane, piece_a, piece_b);
        }
    } else if (warp >= kBuildWarp0) {
        bp = build_place(g, (int)threadIdx.x - kBuildWarp0 * 32);
        {
            const int own = pos1 - pos0 < g.S * 128 ? pos1 - pos0 : g.S * 128;
            build_table(g, tab, bp.r0, pos0 - g.halo, own + 2 * g.halo);
        }
        if (g.nch & 1) {
            // an odd number of 8-channel planes: the one that fills up the last MMA step holds zeros for good
            for (int b = 0; b < g.nseg; b++)
                for (int l = (int)threadIdx.x - kBuildWarp0 * 32; l < g.plane16; l += NBT)
                    *reinterpret_cast<uint4 *>(abuf + b * g.seg_bytes + (g.nch * g.plane16 + l) * 16) = make_uint4(0u, 0u, 0u, 0u);
            fence_proxy_async();
        }
    } else {
        ax = aux_ring(A, sh, auxb, warp);
        if (lane == 0 && ax.on) {
            tma_prefetch_desc(&A.map_x);
            for (int b = 0; b < g.aux_slots; b++) mbar_init(&ax.bar[b], 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_enter();             // the set-up above may overlap the kernel before; its outputs are read from here on
    stamp_begin(A.stamp);
    const uint32_t tmem_d = sh->tmem_base;
    bool ok = true;

    if (warp == kMmaWarp) {
        if (elect_one()) {
            if (!p.w_early) load_weights();
            const uint32_t idesc = instr_desc(g.BN);
            const uint64_t a0 = plane_desc(smem_u32(abuf), g.plane16), w0 = smem_desc(smem_u32(wres), g.KC * 2);
            const int n_tiles = (pos1 - pos0 + 127) >> 7;
            ok = mbar_wait(&sh->w_full, 0);
            int j = 0, sbuf = 0;                // tile within its segment, segment buffer
            for (int ti = 0; ti < n_tiles && ok; ti++) {
                const int buf = ti & (g.nacc - 1);
                if (!mbar_wait(&sh->full[ti & (kFullBars - 1)], (uint32_t)(ti / kFullBars) & 1u)) { ok = false; break; }
                if (ti >= g.nacc && !mbar_wait(&sh->acc_empty[buf], (uint32_t)((ti >> g.acc_shift) - 1) & 1u)) { ok = false; break; }
                tc_fence_after();
                const uint32_t acc = tmem_d + (uint32_t)(buf * g.BN);
                const uint64_t a = a0 + (uint32_t)((sbuf * g.seg_bytes >> 4) + j * 128);
                if (g.ksteps == 1) issue_tile<1>(g, acc, a, w0, idesc);
                else if (g.ksteps == 2) issue_tile<2>(g, acc, a, w0, idesc);
                else if (g.ksteps == 3) issue_tile<3>(g, acc, a, w0, idesc);
                else issue_tile<4>(g, acc, a, w0, idesc);
                mma_commit(&sh->acc_full[buf]);
                if (++j == g.S) { mma_commit(&sh->seg_empty[sbuf]); j = 0; if (g.nseg == 2) sbuf ^= 1; }
            }
        }
        __syncwarp();
    } else if (warp == kLoadWarp) {
        // the first ringful, a lane per piece; the partner rows of every epilogue warp's first tiles; then piece after piece
        const int n_tiles = (pos1 - pos0 + 127) >> 7, full = (pos1 - pos0) / (g.S * 128), rest = pos1 - pos0 - full * g.S * 128;
        const int n = full * g.pps + (rest > 0 ? (rest + 2 * g.halo + g.piece - 1) / g.piece : 0);
        if (lane < g.raw_slots && lane < n) load_piece(g, p, sh, raw, lane, piece_a, piece_b);
        // (the partner rows wait until the records of the statistics are in: those, and the first rows, are needed first)
        const int sets = EW / 4 / g.groups, w = lane & (EW - 1);          // lane: slots lane / EW, + 32 / EW, ... of warp w's ring
        const AuxRing x = aux_ring(A, sh, auxb, w);
        int slot = lane / EW, ti = (w >> 2) / g.groups + slot * sets;
        int row = pixels_before(g, pos0 + ti * 128 + (w & 3) * 32);
        if (!direct) named_barrier(3, EW * 32 + NBT + 32);
        if (x.on)
            while (slot < g.aux_slots && ti < n_tiles) {
                aux_load(A, x, slot, row);
                slot += 32 / EW; ti += 32 / EW * sets;
                row = pixels_before(g, pos0 + ti * 128 + (w & 3) * 32);
            }
        __syncwarp();
        if (elect_one()) {
            int slot = 0, round = 0;
            for (int i = g.raw_slots; i < n && ok; i++) {
                int a, b;
                piece_at(g, pos0, pos1, i, a, b);
                ok = mbar_wait(&sh->raw_empty[slot], (uint32_t)round & 1u);
                if (ok) load_piece(g, p, sh, raw, slot, a, b);
                if (++slot == g.raw_slots) { slot = 0; round++; }
            }
        }
        __syncwarp();
    } else if (warp < EW) {
        const int etid = (int)threadIdx.x;
        if (!direct && warp < 8) {
            // the statistics of the input (kInBwd: the sums of the BN backward) may still be per-CTA records of the kernel before: every
            // CTA adds them, the same way, while its first rows are on the way, and the first CTA stores the result for later readers
            const int c = etid;
            const bool mine = c < g.cin;
            float gam = 0.f, bet = 0.f, mean = 0.f, rstd = 0.f;
            if (mine) {
                gam = p.bn.gamma[c]; bet = p.bn.beta[c];
                if (!p.bn.part || p.in_mode == kInBwd) { mean = p.bn.mean[c]; rstd = p.bn.rstd[c]; }
            }
            if (p.bn.part) reduce_records<256, 10>(p.bn.part, p.bn.parts, g.cin, 0, g.cin >> 1, sh->red, sh->tot, etid);
            if (c < 64) {
                float sc = 0.f, sf = 0.f, k0 = 0.f, k1 = 0.f, k2 = 0.f;
                if (mine) {
                    const double sum = p.bn.part ? sh->tot[(2 * (c >> 2)) * 4 + (c & 3)] : 0., sum2 = p.bn.part ? sh->tot[(2 * (c >> 2) + 1) * 4 + (c & 3)] : 0.;
                    const bool store = blockIdx.x == 0 && blockIdx.y == 0;
                    if (p.in_mode == kInBwd) {
                        const double gr = (double)gam * (double)rstd;
                        k0 = (float)gr; k1 = (float)(gr * sum * p.bn.inv_count); k2 = (float)(gr * sum2 * p.bn.inv_count);
                        if (store) { p.in_dbeta[c] = (float)sum; p.in_dgamma[c] = (float)sum2; }
                    } else if (p.bn.part) {
                        moments_of(sum, sum2, p.bn.inv_count, p.bn.eps, mean, rstd);
                        if (store) { const_cast<float *>(p.bn.mean)[c] = mean; const_cast<float *>(p.bn.rstd)[c] = rstd; }
                    }
                    bn_sc_sh(gam, bet, mean, rstd, sc, sf);
                }
                sh->cf[0][c] = sc; sh->cf[1][c] = sf;
                if (p.in_mode == kInBwd) { sh->cf[2][c] = mean; sh->cf[3][c] = rstd; sh->cf[4][c] = k0; sh->cf[5][c] = k1; sh->cf[6][c] = k2; }
            }
        }
        if (!direct) named_barrier(3, EW * 32 + NBT + 32);
        float s[NC], ss[NC];
#pragma unroll
        for (int i = 0; i < NC; i++) s[i] = ss[i] = 0.f;
        if (e.mode == EPI_BNBWD) {
            if (etid < g.BN) {
                const int c = col0 + etid;
                float4 k = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c < e.n_cols) { k.z = e.bn.mean[c]; k.w = e.bn.rstd[c]; bn_sc_sh(e.bn.gamma[c], e.bn.beta[c], k.z, k.w, k.x, k.y); }
                sh->coef[etid] = k;
            }
            named_barrier(2, EW * 32);
            ok = e.q == 0.f ? epilogue_loop<EW, 3>(A, sh, ax, pos0, pos1, warp, lane, tmem_d, s, ss)
                            : epilogue_loop<EW, 4>(A, sh, ax, pos0, pos1, warp, lane, tmem_d, s, ss);
        } else if (e.mode == EPI_COUPLE) {
            ok = e.q == 0.f ? epilogue_loop<EW, 1>(A, sh, ax, pos0, pos1, warp, lane, tmem_d, s, ss)
                            : epilogue_loop<EW, 2>(A, sh, ax, pos0, pos1, warp, lane, tmem_d, s, ss);
        } else ok = epilogue_loop<EW, 0>(A, sh, ax, pos0, pos1, warp, lane, tmem_d, s, ss);
        if (e.part) {
            // per-CTA record: rows of a warp by shuffles, then the warps that share a column in order
            column_sums(s, lane); column_sums(ss, lane);
            if (lane < NC) { sh->sums[warp][lane] = s[0]; sh->sums[warp][NC + lane] = ss[0]; }
            ok = named_barrier_and(2, EW * 32, ok);
            if (ok && etid < g.BN && col0 + etid < e.n_cols) {
                const int lc = etid % NC;
                float a = 0.f, b = 0.f;
#pragma unroll
                for (int w = 0; w < EW; w++)
                    if (((w >> 2) & (g.groups - 1)) == etid / NC) { a += sh->sums[w][lc]; b += sh->sums[w][NC + lc]; }
                const int c = col0 + etid;
                float *mine = e.part + (size_t)blockIdx.x * 2 * e.n_cols + (c >> 2) * 8 + (c & 3);
                mine[0] = a; mine[4] = b;
            }
            // (Without a counter the consumer adds the records.)  Layers of at most 64 columns have a record per SM or nearly so, and
            // all sixteen warps add them (38-layer step 1899 -> 1875 us); of wider ones, split over fewer CTAs, eight warps are quicker
            // (all sixteen everywhere: 164-layer step 0.6 % slower)
            if (ok && e.counter) {
                named_barrier(2, EW * 32);
                if (EW == 16 && e.n_cols <= 64) epilogue_publish<512>(e, col0, g.BN, reinterpret_cast<float *>(abuf), etid);
                else if (warp < 8) epilogue_publish<256>(e, col0, g.BN, reinterpret_cast<float *>(abuf), etid);
            }
        }
    } else {
#define RV_BUILD(IN) ok = g.k == 1 ? build_rows<IN, EW, NBT, true>(g, p, sh, raw, abuf, tab, pos0, pos1, bp, lane) : build_rows<IN, EW, NBT, false>(g, p, sh, raw, abuf, tab, pos0, pos1, bp, lane)
        if (direct) RV_BUILD(kInBf16);
        else if (p.in_mode == kInFixed) RV_BUILD(kInFixed);
        else if (p.in_mode == kInFloat) RV_BUILD(kInFloat);
        else RV_BUILD(kInBwd);
#undef RV_BUILD
    }
    if (!ok) atomicExch(&sh->failed, 1u);
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && sh->failed) atomicExch(A.status, (int)REVNET_E_TIMEOUT);
    stamp_end(A.stamp);
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem_d, tmem_cols);
    }
}

// fused_shape, which a call asks for every layer several times over (sizing run, launch, whether a neighbour can leave its records): the last
// shapes of a thread are at hand.  (16 channels at 32x32: sizing a block backward 4.0 -> 2.4 us on the host)
const FusedShape *shape_of(Geom geo, int cin, int cout, int k, int sm_count, int in_mode, bool aux) {
    struct Entry { int key[8]; bool ok; FusedShape s; };
    constexpr int kEntries = 16;
    static thread_local Entry memo[kEntries];          // (an empty entry has k = 0)
    static thread_local int next = 0;
    if (in_mode == kInFixed) in_mode = kInFloat;       // the same rows
    const int key[8] = {geo.N, geo.H, geo.W, cin, cout, k, sm_count, in_mode * 2 + (aux ? 1 : 0)};
    for (const Entry &e : memo) if (!memcmp(e.key, key, sizeof key)) return e.ok ? &e.s : nullptr;
    Entry &e = memo[next];
    next = (next + 1) % kEntries;
    memcpy(e.key, key, sizeof key);
    e.ok = fused_shape(geo, cin, cout, k, sm_count, in_mode, aux, e.s);
    return e.ok ? &e.s : nullptr;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// in: [P, cin]; out, partner and the BN input of a data gradient must be plain (unsplit) tensors of cout channels
// behind: kInBwd, the BN whose backward the input still has to go through (bn names it too).  sums: where the records of the fused backward
// sums may stay for their consumer
bool run_fused(Exec &ex, const char *what, int in_mode, const void *in, float in_q, BnRef bn, Geom geo, int cin, int cout, int k,
               const float *Wsrc, const bf16 *prepacked, bool transposed, Pair out, Pair partner, int sign, EpiReq req, bf16 *a_out,
               const BnBwdReq *behind = nullptr, BwdSums *sums = nullptr) {
    if (out.c1 != 0 || (sign && partner.c1 != 0) || (req.bnbwd && req.bnbwd->t.c1 != 0)) return false;
    const bool aux = sign != 0 || req.bnbwd;
    const FusedShape *sp = shape_of(geo, cin, cout, k, ex.ctx->sm_count, in_mode, aux);
    if (!sp) return false;
    const FusedShape &s = *sp;
    EncodeTiledFn enc = nullptr;
    if (!ex.dry) { enc = (EncodeTiledFn)tc_encoder(ex.ctx); if (!enc) return false; }
    const int taps = k * k;
    ex.flops += 2ull * geo.P() * cout * cin * taps;
    const int ctas = s.ctas;
    size_t m = ex.ws.mark();
    const size_t pack_elems = tc_pack_elems(transposed ? cout : cin, transposed ? cin : cout, k, transposed);
    bf16 *wp = prepacked ? const_cast<bf16 *>(prepacked) : ex.ws.get<bf16>(pack_elems);
    const bool reduce = req.stats || req.bnbwd;
    // statistics whose owner has room for the records stay pending: the kernel that consumes them adds the records
    const bool defer = req.stats && !req.bnbwd && req.stats->part && (size_t)ctas * 2 * cout <= req.stats->part_cap;
    float *part = defer ? req.stats->part : (sums ? sums->part : (reduce ? ex.ws.get<float>((size_t)ctas * 2 * cout) : nullptr));
    if (sums) { sums->parts = ctas; sums->inv_count = 1.0 / (double)geo.P(); }
    if (req.stats) {
        req.stats->valid = true;
        req.stats->pending = defer; req.stats->parts = ctas; req.stats->inv_count = 1.0 / (double)geo.P();
    }
    if (!ex.dry) {
        if (!prepacked) tc_pack_now(ex, Wsrc, wp, transposed ? cout : cin, transposed ? cin : cout, k, transposed);
        const int rp16 = round_up(cout, 16), rows_pad = rp16 <= 128 ? rp16 : round_up(rp16, 128);
        FusedArgs A;
        memset(&A, 0, sizeof A);
        A.g = s.g;
        const CUtensorMapSwizzle sw = s.g.KC == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (s.g.KC == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
        // a box of KC channels may reach into the next tap (48 channels in 64-channel rows): the MMAs stop at wpitch
        cuuint64_t dims[2] = {(cuuint64_t)taps * s.g.wpitch, (cuuint64_t)rows_pad};
        cuuint64_t strides[1] = {(cuuint64_t)taps * s.g.wpitch * 2};
        cuuint32_t box[2] = {(cuuint32_t)s.g.KC, (cuuint32_t)s.g.BN};
        cuuint32_t es[2] = {1, 1};
        if (enc(&A.map_w, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)wp, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            ex.failed = true; ex.ctx->err = std::string(what) + ": tensor map rejected"; ex.ws.release(m); return true;
        }
        if (aux) {
            cuuint64_t xdims[2] = {(cuuint64_t)cout, (cuuint64_t)geo.P()}, xstrides[1] = {(cuuint64_t)cout * 4};
            cuuint32_t xbox[2] = {NC, 32};
            if (enc(&A.map_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void *)(req.bnbwd ? req.bnbwd->t.p0 : partner.p0), xdims, xstrides, xbox, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
                ex.failed = true; ex.ctx->err = std::string(what) + ": tensor map (partner) rejected"; ex.ws.release(m); return true;
            }
        }
        FusedLayer &p = A.ly;
        p.in_mode = in_mode; p.in = in; p.in_q = in_q; p.bn = bn; p.a_out = a_out;
        if (behind) { p.in_t = behind->t.p0; p.in_dgamma = behind->dgamma; p.in_dbeta = behind->dbeta; }
        p.wide_out = ((uintptr_t)out.p0 & 31) == 0 && cout % 8 == 0;
        p.w_early = prepacked ? 1 : 0;
        A.status = ex.ctx->dev_status; A.stamp = ex.stamp_slot();
        FusedEpi &e = p.epi;
        e.mode = req.bnbwd ? EPI_BNBWD : (sign ? EPI_COUPLE : EPI_PLAIN);
        e.out = out.p0; e.q = req.bnbwd ? req.bnbwd->t.q : out.q; e.sign = sign; e.n_cols = cout;
        e.part = part; e.counter = (reduce && !defer && !sums) ? ex.ctx->counter(s.n_tiles) : nullptr;
        e.inv_count = 1.0 / (double)geo.P(); e.eps = ex.eps;
        if (req.stats) { e.mean = req.stats->mean; e.rstd = req.stats->rstd; }
        if (req.bnbwd) { e.bn = req.bnbwd->bn; e.dgamma = req.bnbwd->dgamma; e.dbeta = req.bnbwd->dbeta; e.coef = req.bnbwd->coef; }
        static OncePerDevice once;
        if (once.first(ex.ctx->device)) {
            cudaFuncSetAttribute(conv_fused_kernel<16, 192>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
            cudaFuncSetAttribute(conv_fused_kernel<8, 192>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
            cudaFuncSetAttribute(conv_fused_kernel<8, 320>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        }
        dim3 grid((unsigned)ctas, (unsigned)s.n_tiles);
        launch(ex, s.EW == 16 ? conv_fused_kernel<16, 192> : (s.NBT == 320 ? conv_fused_kernel<8, 320> : conv_fused_kernel<8, 192>), grid, fused_threads(s.EW, s.NBT), s.smem, A);
        const double bytes = (double)geo.P() * cin * (in_mode == kInBf16 ? 2 : (in_mode == kInBwd ? 8 : 4)) + (double)geo.P() * cout * (sign || req.bnbwd ? 8 : 4) +
                             (double)cout * taps * cin * 2 + (a_out ? (double)geo.P() * cin * 2 : 0.0);
        ex.check(what, bytes, 2.0 * geo.P() * cout * cin * taps);
    }
    ex.ws.release(m);
    return true;
}

}  // namespace

// whether conv_fprop_fused takes layer L on images gi (and so adds pending statistics of its input itself)
bool conv_fused_takes(Exec &ex, Geom gi, const Layer &L) {
    return L.stride == 1 && shape_of(gi, L.cin, L.cout, L.k, ex.ctx->sm_count, kInFloat, true);
}

// out = partner + sign * conv(ReLU(BN(t)));  a_out (optional): the activated tensor, for the weight gradient
bool conv_fprop_fused(Exec &ex, Pair t, BnRef bn, Geom gi, const Layer &L, Pair out, Pair partner, int sign, Moments *stats, bf16 *a_out) {
    if (L.stride != 1 || t.c1 != 0) return false;
    EpiReq req; req.stats = stats;
    return run_fused(ex, "conv_fprop_fused", t.q != 0.f ? kInFixed : kInFloat, t.p0, t.q, bn, gi, L.cin, L.cout, L.k, L.W, L.Wp_fprop, false, out, partner, sign, req, a_out);
}

// da = conv^T(g) for a stride-1 layer, g bf16 [P, cout]
bool conv_dgrad_fused(Exec &ex, const void *g, Geom gi, const Layer &L, float *da, const BnBwdReq *bb, BwdSums *sums) {
    if (L.stride != 1) return false;
    EpiReq req; req.bnbwd = bb;
    return run_fused(ex, "conv_dgrad_fused", kInBf16, g, 0.f, BnRef{}, gi, L.cout, L.cin, L.k, L.W, L.Wp_dgrad, true, single(da, L.cin), Pair{}, 0, req, nullptr,
                     nullptr, sums);
}

// whether conv_dgrad_fused takes the data gradient of L, with a bf16 input or (behind) through the BN backward of the layer behind; parts: the
// records of 2 cin sums that it leaves
bool conv_dgrad_fused_takes(Exec &ex, Geom gi, const Layer &L, bool behind, int *parts) {
    const FusedShape *s = L.stride == 1 ? shape_of(gi, L.cout, L.cin, L.k, ex.ctx->sm_count, behind ? kInBwd : kInBf16, true) : nullptr;
    if (!s || !(ex.dry || tc_encoder(ex.ctx))) return false;
    *parts = s->ctas;
    return !behind || fused_folds(*s);
}

// The same where the gradient still has to go through the BN + ReLU backward of the layer behind L: g is da of that layer (float), `behind` its
// BN with a plain float input, `bsums` its pending sums.  dgamma and dbeta of that BN are stored, and the bf16 gradient (for the
// weight gradient) in g_out.
// The pass over the tensor between the two data gradients goes, and with it its launch and the last CTA's reduction in front of it.
bool conv_dgrad_fused_behind(Exec &ex, const float *g, const BnBwdReq &behind, const BwdSums &bsums, bf16 *g_out, Geom gi, const Layer &L, float *da, const BnBwdReq *bb,
                             BwdSums *sums) {
    EpiReq req; req.bnbwd = bb;
    BnRef bn = behind.bn;
    bn.part = bsums.part; bn.parts = bsums.parts; bn.inv_count = bsums.inv_count; bn.eps = ex.eps;
    return run_fused(ex, "conv_dgrad_fused", kInBwd, g, 0.f, bn, gi, L.cout, L.cin, L.k, L.W, L.Wp_dgrad, true, single(da, L.cin), Pair{}, 0, req, g_out, &behind, sums);
}
