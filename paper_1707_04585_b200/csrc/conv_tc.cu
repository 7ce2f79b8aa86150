// Tensor-core convolution for sm_100a: implicit GEMM with bf16 operands, fp32 accumulation in
// tensor memory (tcgen05.mma), operand tiles staged in shared memory by TMA.
//
//   out[p, co] = sum_{tap, ci} a[p (+) tap, ci] * Wp[co, tap, ci]        (Eq. 2, Conv_kxk; stride 1)
//
// GEMM view: M = 128 output pixels per CTA (whole image rows, so a tile is one TMA box of the NHWC
// tensor), N = output channels, K = taps x input channels.  For every tap the A tile is the same
// box shifted by (kh - pad, kw - pad); TMA zero-fills what falls outside the image, which is
// exactly the convolution's zero padding because the activated tensor is materialised.
// dgrad is the same kernel run on the upstream gradient with the tap-mirrored, transposed pack
// of the weights.  Each entry point returns false for shapes it does not take.
//
// Roles inside a CTA: warp 0 issues TMA loads, warp 1 allocates tensor memory and issues the MMAs,
// the remaining warps drain the accumulator (tcgen05.ld), apply the coupling epilogue (out = partner
// +/- acc on the float or fixed-point state) and store: two or four groups of four warps where the
// epilogue's tiles move through TMA, one group (192 threads) in the staged form.
// Every mbarrier wait is bounded; on expiry the kernel records a status word and leaves.
#include "common.cuh"
#include "tc_ptx.cuh"
#include "conv_epilogue.cuh"
#include <cuda.h>
#include <string.h>
#include <stdlib.h>

using namespace tc;

namespace {

constexpr int kStages = 6;       // most operand stages of the convolution kernel
constexpr int kWgStages = 4;     // ... of the weight-gradient kernel
constexpr int kThreads = 192;      // TMA warp, MMA warp, four epilogue warps
constexpr int kMaxGroups = 4;      // epilogue through TMA: two or four groups of four epilogue warps
constexpr int kThreadsTma = 64 + kMaxGroups * 128;
constexpr int kThreadsPair = 64 + 2 * 128;      // conv_tc2_kernel: two groups

struct TcParams {
    int taps;        // k*k
    int k;           // kernel size
    int chunks;      // channel chunks per tap
    int KC;          // channels per chunk (16, 32 or 64)
    int cin_pad;     // chunks * KC
    int BN;          // N tile
    int stride;      // 1 or 2: input pixel = output pixel * stride + tap - pad (TMA traversal stride)
    TileGeom g;      // output tiles
    EpiArgs epi;
    int *status;
    int stages;      // operand ring depth (<= kStages)
    // epilogue through TMA: the output tile leaves, and the tile read besides the accumulator (coupling
    // partner, or BN input of a data gradient) arrives, as column groups of GW floats per pixel row
    int GW;          // 32 or 16 floats: rows of 128 / 64 bytes, stored with the matching TMA swizzle
    int epi_bytes;   // partner rings, output slots and sums of the TMA epilogue
    int group_bytes; // one column group of a tile (128 pixel rows), a multiple of 1024
    int need_aux;
    int groups;      // epilogue warp groups
    int aux_slots;   // slots of each group's partner ring
    int inplace;     // coupling: the result is written over the partner group and stored from there (no output slots)
    int split_o, split_x;   // channels in the first tensor of a channel-split output / partner (0: one tensor)
    // the taps this launch sums: offset of the operand box in rows / columns of the operand tensor, and the tap's
    // place in the weight pack.  A plain convolution lists all k*k taps; one parity class of a stride-2 data
    // gradient lists the one, two or four taps that reach its output pixels.
    // A launch with n_cls classes walks n_cls * n_px_tiles tiles: tile t belongs to class t / n_px_tiles (a plain
    // convolution has one class).  CTAs stride over that list, so every CTA gets its share of the short and long classes.
    int n_cls;
    int ntap[4];
    signed char tdy[4][9], tdx[4][9], tid[4][9];
    int ostride, oy[4], ox[4];    // epilogue through TMA: output pixel = tile pixel * ostride + (oy, ox)
    // conv_tc2_kernel, 3x3 stride 1 ("halo" operand): one box per channel chunk holds the tile's pixels WITH their
    // halo, (BH + 2) rows of Wp = W + 2 pixels; tap (kh, kw) reads the 128 rows that start kh * Wp + kw rows further
    // on, so the activations cross L2 -> shared memory once per chunk instead of once per tap.  Accumulator row m is
    // then pixel (m / Wp, m % Wp) of the tile; rows with m % Wp >= W are padding.
    int halo, Wp;
    int a_slots, a_slot_bytes, a_box_bytes;
    unsigned long long *stamp;    // timeline slot of this launch (nullptr: off)
};

struct __align__(8) TcShared {
    uint64_t full[kStages];
    uint64_t empty[kStages];
    uint64_t acc_full[4];            // by tile & 3: with four epilogue groups on alternate tiles each of them sees every phase of its own
    
    uint64_t acc_empty[2];
    uint64_t aux_full[8];
    uint64_t afull[8], aempty[4];     // halo operand ring of conv_tc2_kernel, raw ring of conv1x1_bn_kernel
    uint32_t tmem_base;
    uint32_t failed;
    RowMap rows;
};

// ---- epilogue through TMA.  One column group (GW accumulator columns) at a time:
//   pass A  thread = accumulator row: tensor memory (+ partner row in shared memory) -> output group in shared memory
//   store   one TMA store of the group
//   pass B  thread = (channel quad, every rpp-th pixel): per-channel sums over the valid pixels of the group
// KA: 0 plain float, 1 plain onto the fixed-point grid, 2 / 3 float coupling + / -, 4 / 5 fixed-point coupling + / -.
// These two passes run once per column group between barriers, on two warps per scheduler: straight-line code that
// is executed once per visit is paid for in instruction fetches, not in issue slots.  So they are kept SMALL (rolled
// loops, the plain conversion instructions) rather than unrolled.
template <int KA>
__device__ __forceinline__ void tma_pass_a(uint32_t tm, int GW, int row, bool valid, const uint8_t *aux, uint8_t *outb, float out_s) {
    const int row_b = GW * 4;
    const int swz = GW == 32 ? (row & 7) : ((row >> 1) & 3);
#pragma unroll 1
    for (int c = 0; c < GW; c += 8) {
        float v[8];
        tmem_ld8(tm + (uint32_t)c, v);
        if (!valid) continue;
#pragma unroll
        for (int j = 0; j < 2; j++) {
            const int off = row * row_b + ((((c >> 2) + j) ^ swz) << 4);
            float4 r = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            if (KA == 2 || KA == 3) {
                const float4 pr = *reinterpret_cast<const float4 *>(aux + off);
                if (KA == 2) { r.x = pr.x + r.x; r.y = pr.y + r.y; r.z = pr.z + r.z; r.w = pr.w + r.w; }
                else { r.x = pr.x - r.x; r.y = pr.y - r.y; r.z = pr.z - r.z; r.w = pr.w - r.w; }
            } else if (KA != 0) {
                int4 iv = make_int4(__float2int_rn(r.x * out_s), __float2int_rn(r.y * out_s), __float2int_rn(r.z * out_s), __float2int_rn(r.w * out_s));
                if (KA >= 4) {
                    const int4 pi = *reinterpret_cast<const int4 *>(aux + off);
                    if (KA == 4) { iv.x = pi.x + iv.x; iv.y = pi.y + iv.y; iv.z = pi.z + iv.z; iv.w = pi.w + iv.w; }
                    else { iv.x = pi.x - iv.x; iv.y = pi.y - iv.y; iv.z = pi.z - iv.z; iv.w = pi.w - iv.w; }
                }
                r = make_float4(__int_as_float(iv.x), __int_as_float(iv.y), __int_as_float(iv.z), __int_as_float(iv.w));
            }
            *reinterpret_cast<float4 *>(outb + off) = r;
        }
    }
}
// KB 0 / 1: sums and second sums of the stored values (float / fixed point); 2 / 3: the two sums of the
// BN+ReLU backward with a float / fixed-point BN input group.  Rows are added in a fixed order.
template <int KB>
__device__ __forceinline__ void tma_pass_b(int GW, const uint8_t *ob, const uint8_t *aux, int jq, int r0, int rpp, int valid_px,
                                           float q, float4 sc4, float4 sh4, float4 mu4, float4 rs4, float (&acc)[8]) {
    const int row_b = GW * 4;
#pragma unroll 1
    for (int pl = r0; pl < valid_px; pl += rpp) {
        const int off = pl * row_b + ((jq ^ (GW == 32 ? (pl & 7) : ((pl >> 1) & 3))) << 4);
        float4 v = *reinterpret_cast<const float4 *>(ob + off);
        if (KB >= 2) {
            float4 tt = *reinterpret_cast<const float4 *>(aux + off);
            if (KB == 3) tt = make_float4(__int2float_rn(__float_as_int(tt.x)) * q, __int2float_rn(__float_as_int(tt.y)) * q,
                                          __int2float_rn(__float_as_int(tt.z)) * q, __int2float_rn(__float_as_int(tt.w)) * q);
            const float dx = fmaf(sc4.x, tt.x, sh4.x) > 0.f ? v.x : 0.f, dy = fmaf(sc4.y, tt.y, sh4.y) > 0.f ? v.y : 0.f;
            const float dz = fmaf(sc4.z, tt.z, sh4.z) > 0.f ? v.z : 0.f, dw = fmaf(sc4.w, tt.w, sh4.w) > 0.f ? v.w : 0.f;
            acc[0] += dx; acc[1] += dy; acc[2] += dz; acc[3] += dw;
            acc[4] += dx * ((tt.x - mu4.x) * rs4.x); acc[5] += dy * ((tt.y - mu4.y) * rs4.y);
            acc[6] += dz * ((tt.z - mu4.z) * rs4.z); acc[7] += dw * ((tt.w - mu4.w) * rs4.w);
        } else {
            if (KB == 1) v = make_float4(__int2float_rn(__float_as_int(v.x)) * q, __int2float_rn(__float_as_int(v.y)) * q,
                                         __int2float_rn(__float_as_int(v.z)) * q, __int2float_rn(__float_as_int(v.w)) * q);
            acc[0] += v.x; acc[1] += v.y; acc[2] += v.z; acc[3] += v.w;
            acc[4] += v.x * v.x; acc[5] += v.y * v.y; acc[6] += v.z * v.z; acc[7] += v.w * v.w;
        }
    }
}

// The epilogue of a CTA through TMA, by p.groups warp groups of four warps (wg; warps 2, 3, ... of the CTA).  A visit is one column
// group of one tile: a chain of four barriers and two passes over shared memory whose time is latency, 3000 to 4700 clocks for 128 x
// 32 floats, so its rate is set by how many groups work side by side.  With at least as many column groups as warp
// groups, warp group wg takes the column groups wg, wg + groups, ... of every tile; with fewer, the warp groups also alternate
// tiles (the host makes their number a multiple).  Partner groups arrive through a ring of aux_slots per warp group; a
// coupling writes its result over the partner group and stores it from there, other modes have an output slot per warp group.
// Four groups pay in the single-CTA kernel, whose tiles are short (large-image step: 16.1 -> 14.9 ms of its launches, 164-layer step
// 4.86 -> 3.82 ms together with the records left to the consumer); the pair kernel has two: its tiles are bound by the MMAs,
// and four would cost it operand stages (20.9 -> 22.3 ms).
// PAIR: the tile of a CTA pair's tile pair (see conv_tc2_kernel).
// warp groups that visit a tile, so the arrivals that free its accumulator
__device__ __forceinline__ int epilogue_arrivals(const TcParams &p) { const int ng = p.BN / p.GW; return ng < p.groups ? ng : p.groups; }
struct EpiMaps { const CUtensorMap *o0, *o1, *x0, *x1; };
template <bool PAIR>
__device__ __forceinline__ void tma_epilogue(const TcParams &p, TcShared *sh, const EpiMaps maps, uint8_t *auxr, uint32_t tmem_d, int col0, int warp, int lane,
                                             int rank, int first, int step, int n_v, int per_cls) {
    const int ng = p.BN / p.GW, NG = p.groups;
    const int wg = (warp - 2) >> 2;
    const int bar_a = 1 + 2 * wg, bar_b = 2 + 2 * wg, bar_all = 9;
    const int etid = ((warp & 3) << 5) | lane;
    const EpiArgs &e = p.epi;
    const int GW = p.GW, QW = GW >> 2, rpp = 128 / QW;
    const int jq = etid % QW, r0 = etid / QW;
    const int box_px_o = p.g.BIMG * p.g.BH * p.g.W;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const float out_q = e.out.q, out_s = out_q != 0.f ? 1.f / out_q : 0.f, t_q = e.t.q;
    const uint32_t aux_tx = (uint32_t)(box_px_o * GW * 4);
    const int SW = p.aux_slots;
    uint8_t *auxg = auxr + wg * SW * p.group_bytes;                                  // this group's ring
    uint8_t *outr = auxr + (p.need_aux ? NG * SW * p.group_bytes : 0);
    uint8_t *out_slot = outr + wg * p.group_bytes;
    float *gsums = (float *)(outr + (p.inplace ? 0 : NG * p.group_bytes));           // [ng][128][8], only if ng > groups
    // this group's visits: column groups gi0, gi0 + gstep, ... < ng of the tiles first + step * (it0, it0 + itstep, ...)
    const bool many = ng > NG;
    const int gi0 = many || ng == NG ? wg : wg % ng, gstep = many ? NG : ng;
    const int it0 = ng < NG ? wg / ng : 0, itstep = ng < NG ? NG / ng : 1;
    // pixel of the tile's box (rows of W pixels) this thread's accumulator row holds; -1: padding
    int srow = etid;
    if (p.halo) { const int hh = etid / p.Wp, ww = etid - hh * p.Wp; srow = (hh < p.g.BH && ww < p.g.W) ? hh * p.g.W + ww : -1; }
    const int prow = srow < 0 ? 0 : srow;
    // class and pixel tile at place v of the tile list; false: the second tile of the last pair of an odd number
    auto tile_of = [&](int v, int &cls, int &t) {
        cls = v / per_cls;
        t = PAIR ? 2 * (v - cls * per_cls) + rank : v - cls * per_cls;
        return !PAIR || t < p.g.n_px_tiles;
    };
    // the partner groups in the order of the visits; visits beyond the valid channels and tiles have none
    int l_v = first + it0 * step, l_gi = gi0, l_slot = 0;
    auto load_next_aux = [&]() {                         // one thread; returns without loading once the visits are used up
        while (l_v < n_v) {
            int cls, t, n0, h0;
            const int col = col0 + l_gi * GW;
            const bool live = tile_of(l_v, cls, t) && col < e.n_cols;
            l_gi += gstep;
            const bool last_of_tile = l_gi >= ng;
            if (live) {
                tile_origin(p.g, t, n0, h0);
                const bool second = p.split_x && col >= p.split_x;
                uint64_t *bar = &sh->aux_full[wg * SW + l_slot];
                mbar_expect_tx(bar, aux_tx);
                tma_load_4d(auxg + l_slot * p.group_bytes, second ? maps.x1 : maps.x0, bar, second ? col - p.split_x : col, p.ox[cls], h0 * p.ostride + p.oy[cls], n0);
                if (++l_slot == SW) l_slot = 0;
            }
            if (last_of_tile) { l_gi = gi0; l_v += itstep * step; }
            if (live) return;
        }
    };
    if (etid == 0 && p.need_aux)
        for (int i = 0; i < SW; i++) load_next_aux();
    if (many) {
        for (int i = wg * 128 + etid; i < ng * 128 * 8; i += NG * 128) gsums[i] = 0.f;
        named_barrier(bar_all, NG * 128);
    }
    float acc[8];
#pragma unroll
    for (int j = 0; j < 8; j++) acc[j] = 0.f;
    bool ok = true, refill = false;
    int c_slot = 0; uint32_t c_par = 0;
    int it = it0;
#pragma unroll 1
    for (int v = first + it0 * step; v < n_v; v += itstep * step, it += itstep) {
        const int buf = it & 1;
        int cls, t, n0, h0, valid_px = 0;
        const bool in_range = tile_of(v, cls, t);
        tile_origin(p.g, t, n0, h0);
        if (in_range)
            valid_px = p.g.BIMG > 1 ? (p.g.N - n0 < p.g.BIMG ? p.g.N - n0 : p.g.BIMG) * p.g.BH * p.g.W
                                    : (p.g.H - h0 < p.g.BH ? p.g.H - h0 : p.g.BH) * p.g.W;
        const uint32_t tm = tmem_d + lane_base + (uint32_t)(buf * p.BN);
#pragma unroll 1
        for (int gi = gi0; gi < ng; gi += gstep) {
            const int col = col0 + gi * GW;
            const bool live = in_range && col < e.n_cols;          // groups beyond the valid channels only drain their columns
            const bool visit = p.need_aux && live;                 // the partner group sits in ring slot c_slot
            const bool last_of_tile = gi + gstep >= ng;            // this warp group's last visit to the tile
            const uint8_t *ax = auxg + c_slot * p.group_bytes;
            uint8_t *ob = p.inplace ? auxg + c_slot * p.group_bytes : out_slot;
            if (etid == 0) {
                tma_store_wait_read();                             // this group's last store is done with its slot
                if (refill) load_next_aux();                       // (in place: which can take the next partner group now)
                if (gi == gi0)                                     // (the accumulator is complete for the tile's later visits as well)
                    ok = (PAIR ? mbar_wait_cluster(&sh->acc_full[it & 3], (it >> 2) & 1) : mbar_wait(&sh->acc_full[it & 3], (it >> 2) & 1)) && sh->failed == 0;
                if (ok && visit) ok = mbar_wait(&sh->aux_full[wg * SW + c_slot], c_par);
            }
            refill = p.inplace && visit;
            if (visit && ++c_slot == SW) { c_slot = 0; c_par ^= 1u; }
            ok = named_barrier_and(bar_b, 128, ok);
            if (!ok) break;
            if (gi == gi0) tc_fence_after();
            const bool rowv = live && srow >= 0 && srow < valid_px;
            const uint32_t tg = tm + (uint32_t)(gi * GW);
            if (e.mode != EPI_COUPLE) {
                if (out_q == 0.f) tma_pass_a<0>(tg, GW, prow, rowv, ax, ob, out_s); else tma_pass_a<1>(tg, GW, prow, rowv, ax, ob, out_s);
            } else if (out_q == 0.f) {
                if (e.sign > 0) tma_pass_a<2>(tg, GW, prow, rowv, ax, ob, out_s); else tma_pass_a<3>(tg, GW, prow, rowv, ax, ob, out_s);
            } else {
                if (e.sign > 0) tma_pass_a<4>(tg, GW, prow, rowv, ax, ob, out_s); else tma_pass_a<5>(tg, GW, prow, rowv, ax, ob, out_s);
            }
            if (last_of_tile) tc_fence_before();
            fence_proxy_async();
            named_barrier(bar_a, 128);
            if (etid == 0) {
                if (live) {
                    const bool second = p.split_o && col >= p.split_o;
                    tma_store_4d(second ? maps.o1 : maps.o0, ob, second ? col - p.split_o : col, p.ox[cls], h0 * p.ostride + p.oy[cls], n0);
                    tma_store_commit();
                }
                // this warp group has drained its columns of the tile.  Once per tile and behind the store: on a pair the arrival
                // is a release at cluster scope, and one per column group in front of the store cost 300 to 600 clocks each
                // (32 -> 1248 channels, 12800 pixels, 16-column groups: 53 us, now 42)
                if (last_of_tile) {
                    if (PAIR) mbar_arrive_cluster(mapa_shared(smem_u32(&sh->acc_empty[buf]), 0));
                    else mbar_arrive(&sh->acc_empty[buf]);
                }
            }
            if (e.part && live && col + jq * 4 < e.n_cols) {
                float4 sc4 = make_float4(0, 0, 0, 0), sh4 = sc4, mu4 = sc4, rs4 = sc4;
                if (e.mode == EPI_BNBWD) bn_coef4(e.bn, col + jq * 4, sc4, sh4, mu4, rs4);
                float4 *slot = reinterpret_cast<float4 *>(gsums + (gi * 128 + etid) * 8);
                if (many) {
                    const float4 a0 = slot[0], a1 = slot[1];
                    acc[0] = a0.x; acc[1] = a0.y; acc[2] = a0.z; acc[3] = a0.w; acc[4] = a1.x; acc[5] = a1.y; acc[6] = a1.z; acc[7] = a1.w;
                }
                if (e.mode == EPI_BNBWD) {
                    if (t_q == 0.f) tma_pass_b<2>(GW, ob, ax, jq, r0, rpp, valid_px, 0.f, sc4, sh4, mu4, rs4, acc);
                    else tma_pass_b<3>(GW, ob, ax, jq, r0, rpp, valid_px, t_q, sc4, sh4, mu4, rs4, acc);
                } else if (out_q == 0.f) tma_pass_b<0>(GW, ob, ax, jq, r0, rpp, valid_px, 0.f, sc4, sh4, mu4, rs4, acc);
                else tma_pass_b<1>(GW, ob, ax, jq, r0, rpp, valid_px, out_q, sc4, sh4, mu4, rs4, acc);
                if (many) { slot[0] = make_float4(acc[0], acc[1], acc[2], acc[3]); slot[1] = make_float4(acc[4], acc[5], acc[6], acc[7]); }
            }
            named_barrier(bar_a, 128);                             // the partner group and the output slot have been read
            if (etid == 0 && visit && !p.inplace) load_next_aux();
        }
        if (!ok) break;
    }
    if (etid == 0) tma_store_wait_read();
    if (!ok && lane == 0) atomicExch(&sh->failed, 1u);
    __threadfence_block();
    named_barrier(bar_all, NG * 128);
    if (!e.part) {
        if (etid == 0) tma_store_wait_all();
        return;
    }
    float *sums = many ? gsums : (float *)auxr;                    // (every load and store of the slots has completed)
    if (!many) {
        float4 *slot = reinterpret_cast<float4 *>(sums + (wg * 128 + etid) * 8);
        slot[0] = make_float4(acc[0], acc[1], acc[2], acc[3]); slot[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
        named_barrier(bar_all, NG * 128);
    }
    ok = named_barrier_and(bar_all, NG * 128, *(volatile uint32_t *)&sh->failed == 0);
    if (ok) {
        // per-CTA record: the warp groups, then the threads, that share a channel quad are added in order; a thread per value (the
        // eight sums of a quad lie side by side, in the slots as in the record)
        float *mine = e.part + (size_t)blockIdx.x * 2 * e.n_cols;
        const int per = QW * 8;
        for (int o = wg * 128 + etid; o < ng * per; o += NG * 128) {
            const int gi = o / per, w = o - gi * per, col = col0 + gi * GW + (w >> 3) * 4;
            if (col >= e.n_cols) continue;
            float r = 0.f;
            for (int q = gi; q < (many ? gi + 1 : NG); q += many ? 1 : ng)
#pragma unroll 8
                for (int y = 0; y < rpp; y++) r += sums[q * 128 * 8 + y * per + w];
            mine[2 * col + (w & 7)] = r;
        }
    }
    // the last CTA adds the records with all its epilogue threads (128 of them took four rounds of dependent reads for 148
    // records); without a counter the records stay pending and their consumer adds them
    if (ok && e.counter) {
        float *scratch = reinterpret_cast<float *>(auxr + (many ? 0 : NG * 4096));
        if (NG == 4) epilogue_publish<512>(e, col0, p.BN, scratch, wg * 128 + etid);
        else if (NG == 2) epilogue_publish<256>(e, col0, p.BN, scratch, wg * 128 + etid);
        else if (wg == 0) epilogue_publish<128>(e, col0, p.BN, scratch, etid);
    }
    if (etid == 0) tma_store_wait_all();
}

// Persistent CTA: walks the pixel tiles blockIdx.x, blockIdx.x + gridDim.x, ... of N tile blockIdx.y.
// The operand ring runs on across tiles; the accumulator alternates between two tensor-memory
// buffers so that the epilogue of one tile overlaps the MMAs of the next.
// EPI_TMA: the epilogue through TMA; else the staged one, for channel-split tensors whose halves are no multiple of 16.  Two kernels,
// so that each has the registers of its own block size: under the 576 threads of the other the staged one had 96 and
// spilled, and its launches took 6 to 10 % longer than with the 133 that it has for its 192 (48 -> 1744 channels,
// stride 2, 81 images of 28x28: 117 and 107 us forward).
template <bool EPI_TMA>
__global__ void __launch_bounds__(EPI_TMA ? kThreadsTma : kThreads, 1)
conv_tc_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const __grid_constant__ CUtensorMap map_o0, const __grid_constant__ CUtensorMap map_o1,
               const __grid_constant__ CUtensorMap map_x0, const __grid_constant__ CUtensorMap map_x1, const TcParams p) {
    extern __shared__ uint8_t smem_raw[];
    // operand stages first (1024-byte aligned for the 128-byte swizzle), epilogue stage and bookkeeping behind them
    uint8_t *tiles = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int box_px = p.g.BIMG * p.g.BH * p.g.W;
    const int a_bytes = box_px * p.KC * 2, b_bytes = p.BN * p.KC * 2;
    const int b_off = (128 * p.KC * 2 + 1023) & ~1023;
    const int stage_bytes = b_off + ((b_bytes + 1023) & ~1023);
    // behind the operand ring: the staged epilogue's row stage and running sums, or (EPI_TMA) the partner ring,
    // two output groups and the running sums per column group
    float *estage = (float *)(tiles + p.stages * stage_bytes);
    const int ng = EPI_TMA ? p.BN / p.GW : 0;
    uint8_t *auxr = (uint8_t *)estage;
    TcShared *sh = EPI_TMA ? (TcShared *)(auxr + p.epi_bytes) : (TcShared *)((uint8_t *)estage + kEpiStageBytes + kEpiSumFloats * 4);

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int n_vt = p.n_cls * p.g.n_px_tiles;     // tiles of all classes
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < 2 * p.BN) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; s++) { mbar_init(&sh->full[s], 1); mbar_init(&sh->empty[s], 1); }
        for (int b = 0; b < 2; b++) mbar_init(&sh->acc_empty[b], EPI_TMA ? epilogue_arrivals(p) : 128);
        for (int b = 0; b < 4; b++) mbar_init(&sh->acc_full[b], 1);
        for (int b = 0; b < 8; b++) mbar_init(&sh->aux_full[b], 1);
        sh->failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_prefetch_desc(&map_a); tma_prefetch_desc(&map_b);
        if (EPI_TMA) { tma_prefetch_desc(&map_o0); tma_prefetch_desc(&map_o1); tma_prefetch_desc(&map_x0); tma_prefetch_desc(&map_x1); }
    }
    if (warp == 1) tmem_alloc(&sh->tmem_base, tmem_cols);
    if (warp >= 2) build_row_map(p.g, &sh->rows, ((warp & 3) << 5) | lane);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_enter();             // the set-up above may overlap the kernel before; its outputs are read from here on
    stamp_begin(p.stamp);
    const uint32_t tmem_d = sh->tmem_base;
    const int col0 = blockIdx.y * p.BN;

    // The two single-thread loops below (TMA producer, MMA issuer) set the pace of the whole CTA: a lone thread gets no
    // latency hiding, every instruction costs its full pipeline latency, and a stage's four MMAs take only 256-512
    // clocks.  So no divisions, no table look-ups and no descriptor construction inside them: the ring position is
    // stepped, tap data is read once per tap, descriptors are a base plus increments of the address field.
    if (warp == 0) {
        if (elect_one()) {
            int s = 0; uint32_t round = 0;
            bool ok = true;
            const uint32_t tx = (uint32_t)(a_bytes + b_bytes);
            for (int t = blockIdx.x; t < n_vt && ok; t += gridDim.x) {
                int n0, h0;
                const int cls = t / p.g.n_px_tiles;
                tile_origin(p.g, t - cls * p.g.n_px_tiles, n0, h0);
                const int ntap = p.ntap[cls], hs = h0 * p.stride;
                for (int ti = 0; ti < ntap && ok; ti++) {
                    const int dx = p.tdx[cls][ti], yy = hs + p.tdy[cls][ti];
                    int wc = p.tid[cls][ti] * p.cin_pad;
                    for (int cc = 0; cc < p.cin_pad; cc += p.KC, wc += p.KC) {
                        if (round > 0 && !mbar_wait(&sh->empty[s], (round - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                        uint8_t *sa = tiles + s * stage_bytes;
                        mbar_expect_tx(&sh->full[s], tx);
                        tma_load_4d(sa, &map_a, &sh->full[s], cc, dx, yy, n0);
                        tma_load_2d(sa + b_off, &map_b, &sh->full[s], wc, col0);
                        if (++s == p.stages) { s = 0; round++; }
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = instr_desc(p.BN);
            const int row_bytes = p.KC * 2, nk = p.KC >> 4;
            const uint64_t da0 = smem_desc(smem_u32(tiles), row_bytes), db0 = smem_desc(smem_u32(tiles) + b_off, row_bytes);
            const uint32_t stage16 = (uint32_t)stage_bytes >> 4;      // the descriptors' address field counts 16-byte units
            int s = 0; uint32_t round = 0, soff = 0;
            bool ok = true;
            int ti = 0;
            for (int t = blockIdx.x; t < n_vt && ok; t += gridDim.x, ti++) {
                const int buf = ti & 1; const uint32_t use = ti >> 1;
                const int iters = p.ntap[t / p.g.n_px_tiles] * p.chunks;
                if (use > 0 && !mbar_wait(&sh->acc_empty[buf], (use - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                tc_fence_after();
                const uint32_t acc = tmem_d + (uint32_t)(buf * p.BN);
                uint32_t accum = 0;
                for (int it = 0; it < iters; it++) {
                    if (!mbar_wait(&sh->full[s], round & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                    tc_fence_after();
                    const uint64_t da = da0 + soff, db = db0 + soff;
                    mma_bf16(acc, da, db, idesc, accum);
                    accum = 1;
                    for (int kk = 1; kk < nk; kk++) mma_bf16(acc, da + 2 * kk, db + 2 * kk, idesc, 1u);
                    mma_commit(&sh->empty[s]);          // frees the stage once these MMAs have read it
                    soff += stage16;
                    if (++s == p.stages) { s = 0; soff = 0; round++; }
                }
                if (ok) mma_commit(&sh->acc_full[ti & 3]);
            }
        }
    } else if constexpr (!EPI_TMA) {
        // epilogue: this warp may touch accumulator lanes 32*(warp%4) .. +31
        const int etid = ((warp & 3) << 5) | lane;
        float *esums = estage + 128 * kEpiPitch;
        epilogue_init(esums, etid);
        named_barrier(1, 128);
        bool ok = true;
        int ti = 0;
        for (int t = blockIdx.x; t < p.g.n_px_tiles; t += gridDim.x, ti++) {
            const int buf = ti & 1;
            int n0, h0;
            tile_origin(p.g, t, n0, h0);
            EpiPrefetch pre;
            epilogue_prefetch(p.epi, p.BN, col0, &sh->rows, p.g, n0, h0, etid, pre);     // before the accumulator is ready
            if (etid == 0) ok = mbar_wait(&sh->acc_full[ti & 3], (ti >> 2) & 1) && sh->failed == 0;     // one thread polls, the rest block
            ok = named_barrier_and(2, 128, ok);
            if (!ok) break;
            tc_fence_after();
            epilogue_tile(p.epi, tmem_d + (uint32_t)(buf * p.BN), p.BN, col0, &sh->rows, p.g, n0, h0, estage, esums, etid, &sh->acc_empty[buf], pre);
        }
        if (ok) epilogue_finish(p.epi, p.BN, col0, estage, esums, etid);
        else if (lane == 0) atomicExch(&sh->failed, 1u);
    } else {
        tma_epilogue<false>(p, sh, EpiMaps{&map_o0, &map_o1, &map_x0, &map_x1}, auxr, tmem_d, col0, warp, lane, 0, (int)blockIdx.x, (int)gridDim.x, n_vt, p.g.n_px_tiles);
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && sh->failed) atomicExch(p.status, (int)REVNET_E_TIMEOUT);
    stamp_end(p.stamp);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_d, tmem_cols);
    }
}

// BN -> ReLU -> 1x1 convolution as one kernel, for layers of 128 input channels and more onto at most 128 (the first layer of a
// bottleneck function): out[p, co] = sum_ci bf16(ReLU(BN(t[p, ci]))) W[co, ci].
// The separate kernels write the activated tensor and read it back; here TMA brings the raw tensor, 64 channels of 128 pixels at
// a time, into a ring of shared memory, eight warps normalise it into the swizzled operand (and, where the weight gradient will
// want it, write it out), and the weights arrive beside it.  Everything else is conv_tc_kernel with flattened pixels.
// Warps: 0 raw tiles, 1 tensor memory and MMAs, 2-9 epilogue, 10-17 build, 18 weights.
// Bound by HBM (large tensors) or by the launch's fixed steps (CIFAR-sized ones).  Measured, 512 -> 128 channels, 200704 pixels:
// BN-ReLU 87 us and convolution 62 us before, now 102 us (514 MB, 5.0 TB/s); with the eight build warps as one team 111 us.
constexpr int kBnBuildWarps = 8, kBnThreads = (2 + 8 + kBnBuildWarps + 1) * 32, kRawBytes = 128 * 64 * 4;
struct BnConvParams {
    TcParams p;
    BnRef bn;
    float in_q;            // fixed-point step of the input, 0: float
    bf16 *a_out;           // the activated tensor [P, cin], or null
    int P, raw_stages;
};
__global__ void __launch_bounds__(kBnThreads, 1)
conv1x1_bn_kernel(const __grid_constant__ CUtensorMap map_raw, const __grid_constant__ CUtensorMap map_b, const __grid_constant__ CUtensorMap map_o,
                  const __grid_constant__ BnConvParams q) {
    extern __shared__ uint8_t smem_raw[];
    const TcParams &p = q.p;
    uint8_t *tiles = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int b_bytes = p.BN * 128, stage_bytes = 16384 + ((b_bytes + 1023) & ~1023), cin = p.cin_pad;
    uint8_t *raw = tiles + p.stages * stage_bytes;
    uint8_t *auxr = raw + q.raw_stages * kRawBytes;
    float *sc = (float *)(auxr + p.epi_bytes), *sf = sc + cin;
    TcShared *sh = (TcShared *)(sf + cin);
    const int warp = warp_index(), lane = threadIdx.x & 31, ng = p.BN / p.GW;
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < 2 * p.BN) tmem_cols <<= 1;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; s++) { mbar_init(&sh->full[s], 1 + kBnBuildWarps / 2); mbar_init(&sh->empty[s], 1); }
        for (int b = 0; b < 8; b++) mbar_init(&sh->afull[b], 1);
        for (int b = 0; b < 4; b++) { mbar_init(&sh->aempty[b], kBnBuildWarps / 2); mbar_init(&sh->acc_full[b], 1); }
        for (int b = 0; b < 2; b++) mbar_init(&sh->acc_empty[b], epilogue_arrivals(p));
        for (int b = 0; b < 8; b++) mbar_init(&sh->aux_full[b], 1);
        sh->failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_prefetch_desc(&map_raw); tma_prefetch_desc(&map_b); tma_prefetch_desc(&map_o);
    }
    if (warp == 1) tmem_alloc(&sh->tmem_base, tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_enter();
    stamp_begin(p.stamp);
    const uint32_t tmem_d = sh->tmem_base;
    const int n_tiles = p.g.n_px_tiles;

    if (warp == 0) {
        if (elect_one()) {
            // the full barrier of chunk n is n mod twice the slots: a build team takes every second chunk, and so sees every phase of
            // the barriers that it waits on
            int s = 0, f = 0; uint32_t round = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x)
                for (int cc = 0; cc < cin; cc += 64) {
                    if (round > 0 && !mbar_wait(&sh->aempty[s], (round - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                    mbar_expect_tx(&sh->afull[f], kRawBytes);
                    tma_load_2d(raw + s * kRawBytes, &map_raw, &sh->afull[f], cc, t * 128);
                    tma_load_2d(raw + s * kRawBytes + kRawBytes / 2, &map_raw, &sh->afull[f], cc + 32, t * 128);
                    if (++f == 2 * q.raw_stages) f = 0;
                    if (++s == q.raw_stages) { s = 0; round++; }
                }
        }
    } else if (warp == 10 + kBnBuildWarps) {
        if (elect_one()) {
            int s = 0; uint32_t round = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x)
                for (int cc = 0; cc < cin; cc += 64) {
                    if (round > 0 && !mbar_wait(&sh->empty[s], (round - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                    mbar_expect_tx(&sh->full[s], (uint32_t)b_bytes);
                    tma_load_2d(tiles + s * stage_bytes + 16384, &map_b, &sh->full[s], cc, 0);
                    if (++s == p.stages) { s = 0; round++; }
                }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = instr_desc(p.BN);
            const uint64_t da0 = smem_desc(smem_u32(tiles), 128), db0 = smem_desc(smem_u32(tiles) + 16384, 128);
            const uint32_t stage16 = (uint32_t)stage_bytes >> 4;
            int s = 0, ti = 0; uint32_t round = 0, soff = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ti++) {
                const int buf = ti & 1; const uint32_t use = ti >> 1;
                if (use > 0 && !mbar_wait(&sh->acc_empty[buf], (use - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                tc_fence_after();
                const uint32_t acc = tmem_d + (uint32_t)(buf * p.BN);
                uint32_t accum = 0;
                for (int it = 0; it < p.chunks; it++) {
                    if (!mbar_wait(&sh->full[s], round & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                    tc_fence_after();
                    const uint64_t da = da0 + soff, db = db0 + soff;
                    mma_bf16(acc, da, db, idesc, accum);
                    accum = 1;
                    for (int kk = 1; kk < 4; kk++) mma_bf16(acc, da + 2 * kk, db + 2 * kk, idesc, 1u);
                    mma_commit(&sh->empty[s]);
                    soff += stage16;
                    if (++s == p.stages) { s = 0; soff = 0; round++; }
                }
                if (ok) mma_commit(&sh->acc_full[ti & 3]);
            }
        }
    } else if (warp < 10) {
        tma_epilogue<false>(p, sh, EpiMaps{&map_o, &map_o, &map_o, &map_o}, auxr, tmem_d, 0, warp, lane, 0, (int)blockIdx.x, (int)gridDim.x, n_tiles, n_tiles);
    } else {
        // build: two teams of warps on alternate chunks, so that one's waits lie behind the other's work; thread = (8-channel
        // group of the chunk, row), eight rows 16 apart in two batches
        const int bt = (int)threadIdx.x - 320, team = bt >> 7, ck = bt & 7, r0 = (bt & 127) >> 3;
        for (int c = bt; c < cin; c += kBnBuildWarps * 32) {
            float a, b;
            bn_sc_sh(q.bn.gamma[c], q.bn.beta[c], q.bn.mean[c], q.bn.rstd[c], a, b);
            sc[c] = q.in_q != 0.f ? a * q.in_q : a; sf[c] = b;
        }
        named_barrier(10, kBnBuildWarps * 32);
        int rs = team, f = team, s = team, t = blockIdx.x, it = team; uint32_t fround = 0, round = 0;
        const bool fixed = q.in_q != 0.f;
        bool ok = true;
        while (true) {
            if (it >= p.chunks) { it -= p.chunks; t += gridDim.x; }          // (two chunks at least: one step back is enough)
            if (t >= n_tiles) break;
            if (lane == 0) {
                ok = mbar_wait(&sh->afull[f], fround & 1);
                if (ok && round > 0) ok = mbar_wait(&sh->empty[s], (round - 1) & 1);
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            const int cc = it * 64;
            const uint8_t *src = raw + rs * kRawBytes + (ck >> 2) * (kRawBytes / 2);
            uint8_t *dst = tiles + s * stage_bytes;
            float a[8], b[8];
#pragma unroll
            for (int i = 0; i < 8; i += 4) {
                const float4 u = *reinterpret_cast<const float4 *>(sc + cc + ck * 8 + i), w = *reinterpret_cast<const float4 *>(sf + cc + ck * 8 + i);
                a[i] = u.x; a[i + 1] = u.y; a[i + 2] = u.z; a[i + 3] = u.w; b[i] = w.x; b[i + 1] = w.y; b[i + 2] = w.z; b[i + 3] = w.w;
            }
#pragma unroll 1
            for (int half = 0; half < 2; half++) {
                float4 v[4][2];
                // (the two boxes of a chunk share banks: the lanes of the second read their halves in the other order)
#pragma unroll
                for (int i = 0; i < 4; i++)
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const int row = r0 + 16 * (4 * half + i);
                        v[i][h] = *reinterpret_cast<const float4 *>(src + row * 128 + ((((ck & 3) * 2 + (h ^ (ck >> 2))) ^ (row & 7)) << 4));
                    }
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int row = r0 + 16 * (4 * half + i), px = t * 128 + row;
                    const bool sw = ck >= 4;
                    const float4 lo = sw ? v[i][1] : v[i][0], hi = sw ? v[i][0] : v[i][1];
                    const float x[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                    uint32_t o[4];
#pragma unroll
                    for (int j = 0; j < 8; j += 2) {
                        const float x0 = fmaf(a[j], fixed ? __int2float_rn(__float_as_int(x[j])) : x[j], b[j]);
                        const float x1 = fmaf(a[j + 1], fixed ? __int2float_rn(__float_as_int(x[j + 1])) : x[j + 1], b[j + 1]);
                        asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(o[j >> 1]) : "f"(x1), "f"(x0));
                    }
                    *reinterpret_cast<uint4 *>(dst + row * 128 + ((ck ^ (row & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
                    if (q.a_out && px < q.P) *reinterpret_cast<uint4 *>(q.a_out + (size_t)px * cin + cc + ck * 8) = make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) { mbar_arrive(&sh->full[s]); mbar_arrive(&sh->aempty[rs]); }
            rs += 2; if (rs >= q.raw_stages) rs -= q.raw_stages;
            f += 2; if (f >= 2 * q.raw_stages) { f -= 2 * q.raw_stages; fround++; }
            s += 2; if (s >= p.stages) { s -= p.stages; round++; }
            it += 2;
        }
        if (!ok) atomicExch(&sh->failed, 1u);
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && sh->failed) atomicExch(p.status, (int)REVNET_E_TIMEOUT);
    stamp_end(p.stamp);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_d, tmem_cols);
    }
}

// The same convolution on a CTA PAIR (a cluster of two CTAs on the two SMs of a TPC, tcgen05 cta_group::2): one
// MMA of M = 256 covers two adjacent pixel tiles, CTA `rank` holding the operand rows of its own 128 pixels and its
// half of the N tile's weight rows, and receiving its 128 accumulator rows in its own tensor memory.  Per MMA an SM
// then reads 128 x 16 activations and only N/2 x 16 weights from shared memory (and fetches only half of the weight
// tile from L2), which is what lets 256-wide tiles run at the tensor cores' rate instead of the shared-memory port's.
// The leader (rank 0) issues the MMAs for both; each CTA loads its own operands (plain tile loads, no multicast)
// and signals the leader's barrier; commits arrive on the barriers of both CTAs.  Each CTA runs the epilogue of its
// own tile exactly as the single-CTA kernel does (epilogue through TMA only).
// Tile pairs: class c, pair j holds the pixel tiles 2j and 2j + 1 of the class; with an odd tile count the last pair's
// second tile lies outside the tensor (TMA delivers zeros, nothing is stored).
__global__ void __launch_bounds__(kThreadsPair, 1)
conv_tc2_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                const __grid_constant__ CUtensorMap map_o0, const __grid_constant__ CUtensorMap map_o1,
                const __grid_constant__ CUtensorMap map_x0, const __grid_constant__ CUtensorMap map_x1, const TcParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *tiles = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int box_px = p.g.BIMG * p.g.BH * p.g.W;
    const int BNH = p.BN >> 1;                                   // weight rows this CTA holds
    const int a_bytes = box_px * p.KC * 2, b_bytes = BNH * p.KC * 2;
    const int b_off = (128 * p.KC * 2 + 1023) & ~1023;
    const int stage_bytes = b_off + ((b_bytes + 1023) & ~1023);
    // halo mode: the ring holds weight tiles only, the activation boxes have a ring of their own in front of it
    uint8_t *abuf = tiles;
    const int wstage_bytes = (b_bytes + 1023) & ~1023;
    uint8_t *wring = tiles + (p.halo ? p.a_slots * p.a_slot_bytes : 0);
    uint8_t *auxr = p.halo ? wring + p.stages * wstage_bytes : tiles + p.stages * stage_bytes;
    TcShared *sh = (TcShared *)(auxr + p.epi_bytes);

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = (int)blockIdx.x >> 1, n_pairs = (int)gridDim.x >> 1;
    const int n_pp = (p.g.n_px_tiles + 1) >> 1;                  // tile pairs per class
    const int n_vp = p.n_cls * n_pp;
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < 2 * p.BN) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; s++) { mbar_init(&sh->full[s], 1); mbar_init(&sh->empty[s], 1); }
        for (int b = 0; b < 2; b++) mbar_init(&sh->acc_empty[b], 2 * epilogue_arrivals(p));     // (used in the leader) those of either CTA
        for (int b = 0; b < 4; b++) mbar_init(&sh->acc_full[b], 1);
        for (int b = 0; b < 8; b++) mbar_init(&sh->aux_full[b], 1);
        for (int b = 0; b < 4; b++) { mbar_init(&sh->afull[b], 1); mbar_init(&sh->aempty[b], 1); }
        sh->failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_prefetch_desc(&map_a); tma_prefetch_desc(&map_b);
        tma_prefetch_desc(&map_o0); tma_prefetch_desc(&map_o1); tma_prefetch_desc(&map_x0); tma_prefetch_desc(&map_x1);
    }
    if (warp == 1) tmem2_alloc(&sh->tmem_base, tmem_cols);       // the same warp of both CTAs
    if (warp >= 2) build_row_map(p.g, &sh->rows, ((warp & 3) << 5) | lane);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();      // the peer's barriers are initialised and its tensor memory allocated before anything crosses over
    tc_fence_after();
    pdl_enter();
    stamp_begin(p.stamp);
    const uint32_t tmem_d = sh->tmem_base;
    const int col0 = blockIdx.y * p.BN;
    // this CTA's tile of tile pair vp
    auto my_tile = [&](int vp, int &cls, int &t) { cls = vp / n_pp; t = 2 * (vp - cls * n_pp) + (int)rank; };

    // (single-thread loops kept lean, as in conv_tc_kernel)
    if (warp == 0) {
        if (elect_one()) {
            int s = 0, as = 0; uint32_t round = 0, ar = 0;
            bool ok = true;
            const uint32_t full0 = mapa_shared(smem_u32(&sh->full[0]), 0), afull0 = mapa_shared(smem_u32(&sh->afull[0]), 0);   // the leader's barriers
            const uint32_t tx = (uint32_t)(2 * (a_bytes + b_bytes)), txw = (uint32_t)(2 * b_bytes), txa = (uint32_t)(2 * p.a_box_bytes);
            const int wcol = col0 + (int)rank * BNH;
            for (int vp = pair; vp < n_vp && ok; vp += n_pairs) {
                int cls, t, n0, h0;
                my_tile(vp, cls, t);
                tile_origin(p.g, t, n0, h0);         // beyond the last tile the origin lies outside the tensor: zeros arrive
                if (p.halo) {
                    // per channel chunk: one activation box with its halo, then the nine weight tiles
                    for (int cc = 0; cc < p.cin_pad && ok; cc += p.KC) {
                        if (ar > 0 && !mbar_wait(&sh->aempty[as], (ar - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                        if (rank == 0) mbar_expect_tx(&sh->afull[as], txa);
                        tma2_load_4d(abuf + as * p.a_slot_bytes, &map_a, afull0 + 8u * as, cc, -1, h0 - 1, n0);
                        if (++as == p.a_slots) { as = 0; ar++; }
                        int wc = cc;
                        for (int ti = 0; ti < 9; ti++, wc += p.cin_pad) {      // tap ti of a plain 3x3 layer sits at ti * cin_pad in the pack
                            if (round > 0 && !mbar_wait(&sh->empty[s], (round - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                            if (rank == 0) mbar_expect_tx(&sh->full[s], txw);
                            tma2_load_2d(wring + s * wstage_bytes, &map_b, full0 + 8u * s, wc, wcol);
                            if (++s == p.stages) { s = 0; round++; }
                        }
                    }
                    continue;
                }
                const int ntap = p.ntap[cls], hs = h0 * p.stride;
                for (int ti = 0; ti < ntap && ok; ti++) {
                    const int dx = p.tdx[cls][ti], yy = hs + p.tdy[cls][ti];
                    int wc = p.tid[cls][ti] * p.cin_pad;
                    for (int cc = 0; cc < p.cin_pad; cc += p.KC, wc += p.KC) {
                        if (round > 0 && !mbar_wait(&sh->empty[s], (round - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                        uint8_t *sa = tiles + s * stage_bytes;
                        if (rank == 0) mbar_expect_tx(&sh->full[s], tx);      // the leader's barrier collects the bytes of both CTAs
                        tma2_load_4d(sa, &map_a, full0 + 8u * s, cc, dx, yy, n0);
                        tma2_load_2d(sa + b_off, &map_b, full0 + 8u * s, wc, wcol);
                        if (++s == p.stages) { s = 0; round++; }
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0 && elect_one()) {
            const uint32_t idesc = instr_desc_m256(p.BN);
            const int row_bytes = p.KC * 2, nk = p.KC >> 4;
            const uint64_t da0 = smem_desc(smem_u32(tiles), row_bytes), db0 = smem_desc(smem_u32(tiles) + b_off, row_bytes);
            const uint64_t ha0 = smem_desc(smem_u32(abuf), 128), hb0 = smem_desc(smem_u32(wring), 128);      // halo mode: boxes, weight ring
            const uint32_t stage16 = (uint32_t)stage_bytes >> 4, wstage16 = (uint32_t)wstage_bytes >> 4, aslot16 = (uint32_t)p.a_slot_bytes >> 4;
            const uint32_t wp8 = (uint32_t)p.Wp * 8u;      // one halo row of pixels, in 16-byte units (128-byte operand rows)
            int s = 0, as = 0; uint32_t round = 0, ar = 0, soff = 0, aoff = 0;
            bool ok = true;
            int ti = 0;
            for (int vp = pair; vp < n_vp && ok; vp += n_pairs, ti++) {
                const int buf = ti & 1; const uint32_t use = ti >> 1;
                if (use > 0 && !mbar_wait_cluster(&sh->acc_empty[buf], (use - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                tc_fence_after();
                const uint32_t acc = tmem_d + (uint32_t)(buf * p.BN);
                uint32_t accum = 0;
                if (p.halo) {
                    for (int ch = 0; ch < p.chunks && ok; ch++) {
                        if (!mbar_wait_cluster(&sh->afull[as], ar & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                        // tap (kh, kw): the operand starts kh * Wp + kw rows (of 128 bytes) into the box.  The 128-byte
                        // swizzle is a function of the shared-memory ADDRESS (bits 4..6 xor bits 7..9), for the TMA
                        // write as for the MMA read, so a start on any row reads the rows as they were written
                        uint64_t da_row = ha0 + aoff;
                        for (int kh = 0; kh < 3 && ok; kh++, da_row += wp8) {
                            uint64_t da = da_row;
                            for (int kw = 0; kw < 3; kw++, da += 8) {
                                if (!mbar_wait_cluster(&sh->full[s], round & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                                tc_fence_after();
                                const uint64_t db = hb0 + soff;
                                mma2_bf16(acc, da, db, idesc, accum);
                                accum = 1;
                                mma2_bf16(acc, da + 2, db + 2, idesc, 1u);
                                mma2_bf16(acc, da + 4, db + 4, idesc, 1u);
                                mma2_bf16(acc, da + 6, db + 6, idesc, 1u);
                                mma2_commit_both(&sh->empty[s]);
                                soff += wstage16;
                                if (++s == p.stages) { s = 0; soff = 0; round++; }
                            }
                        }
                        if (ok) mma2_commit_both(&sh->aempty[as]);      // the box is free once the MMAs of its nine taps have read it
                        aoff += aslot16;
                        if (++as == p.a_slots) { as = 0; aoff = 0; ar++; }
                    }
                    if (ok) mma2_commit_both(&sh->acc_full[ti & 3]);
                    continue;
                }
                const int iters = p.ntap[vp / n_pp] * p.chunks;
                for (int it = 0; it < iters; it++) {
                    if (!mbar_wait_cluster(&sh->full[s], round & 1)) { atomicExch(&sh->failed, 1u); ok = false; break; }
                    tc_fence_after();
                    const uint64_t da = da0 + soff, db = db0 + soff;
                    mma2_bf16(acc, da, db, idesc, accum);
                    accum = 1;
                    for (int kk = 1; kk < nk; kk++) mma2_bf16(acc, da + 2 * kk, db + 2 * kk, idesc, 1u);
                    mma2_commit_both(&sh->empty[s]);         // frees the stage in both CTAs once these MMAs have read it
                    soff += stage16;
                    if (++s == p.stages) { s = 0; soff = 0; round++; }
                }
                if (ok) mma2_commit_both(&sh->acc_full[ti & 3]);
            }
        }
    } else {
        // epilogue of this CTA's own tile, as in conv_tc_kernel
        tma_epilogue<true>(p, sh, EpiMaps{&map_o0, &map_o1, &map_x0, &map_x1}, auxr, tmem_d, col0, warp, lane, (int)rank, pair, n_pairs, n_vp, n_pp);
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && sh->failed) atomicExch(p.status, (int)REVNET_E_TIMEOUT);
    stamp_end(p.stamp);
    // neither CTA leaves, or frees tensor memory, while the other may still read its operands or signal its barriers
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem2_dealloc(tmem_d, tmem_cols);
    }
}

// ---- weight packs (see PackJob).  Bound by HBM: each weight is read once and written to both packs.  A block of 256
// threads takes tiles of 64 output x 64 input channels of one tap: 256-byte reads, 128-byte writes to either pack, the
// transposed one through shared memory; consecutive tiles walk the weights in memory order.
// Measured: a 75 M weight layer 638 -> 87 us per pack (one element per thread and uncoalesced reads of the transposed pack
// before); a block's eight launches are one; all packs of a step, each weight read once instead of twice: large-image step 68.9 -> 67.9 ms.
constexpr int kPackTile = 64;
__device__ __forceinline__ uint2 pack_bf16x4(float a, float b, float c, float d) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    return make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
}
__host__ __device__ __forceinline__ int pack_ct(const PackJob &j) { const int n = j.ci_f > j.ci_d ? j.ci_f : j.ci_d; return (n + kPackTile - 1) / kPackTile; }
__host__ __device__ __forceinline__ int pack_rt(const PackJob &j) { const int n = j.co_f > j.co_d ? j.co_f : j.co_d; return (n + kPackTile - 1) / kPackTile; }
__device__ __forceinline__ void pack_layer(const PackJob &j, int first, int end, int step) {
    __shared__ float tile[kPackTile][kPackTile + 1];
    const int taps = j.k * j.k, ct = pack_ct(j);
    const int lx = threadIdx.x & 15, ly = threadIdx.x >> 4;
    for (int t = first; t < end; t += step) {
        const int ci0 = (t % ct) * kPackTile, tap = (t / ct) % taps, co0 = t / (ct * taps) * kPackTile;
        const int ci = ci0 + 4 * lx;
        float4 v[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int co = co0 + ly + 16 * i;
            v[i] = (co < j.Co && ci < j.Ci) ? *reinterpret_cast<const float4 *>(j.W + ((size_t)co * taps + tap) * j.Ci + ci) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int co = co0 + ly + 16 * i;
            if (j.f && co < j.co_f && ci < j.ci_f)
                *reinterpret_cast<uint2 *>(j.f + ((size_t)co * taps + tap) * j.ci_f + ci) = pack_bf16x4(v[i].x, v[i].y, v[i].z, v[i].w);
            if (j.d) { float *r = tile[ly + 16 * i] + 4 * lx; r[0] = v[i].x; r[1] = v[i].y; r[2] = v[i].z; r[3] = v[i].w; }
        }
        if (!j.d) continue;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; i++) {
            // rows of this pack are input channels, columns output channels, taps mirrored
            const int r = ly + 16 * i, c = co0 + 4 * lx;
            if (ci0 + r < j.ci_d && c < j.co_d)
                *reinterpret_cast<uint2 *>(j.d + ((size_t)(ci0 + r) * taps + (taps - 1 - tap)) * j.co_d + c) =
                    pack_bf16x4(tile[4 * lx][r], tile[4 * lx + 1][r], tile[4 * lx + 2][r], tile[4 * lx + 3][r]);
        }
        __syncthreads();
    }
}
// Every layer of a step (table in device memory): a CTA takes `run` consecutive tiles of all of them and finds its first layer
// with a 32-way search.  (With one row of CTAs per layer, as many as the largest layer has tiles, the launch of nearly two
// hundred thousand mostly empty CTAs took 202 us in the step of the 164-layer network; now 23 us.)
__global__ void __launch_bounds__(256) pack_weights_batch_kernel(const PackJob *__restrict__ jobs, int n_jobs, int tiles, int run) {
    pdl_enter();
    int t = blockIdx.x * run;
    const int end = t + run < tiles ? t + run : tiles, lane = threadIdx.x & 31;
    int lo = 0, len = n_jobs;
    while (true) {                               // the last job with tile0 <= t
        const int step = (len + 31) >> 5;
        const int n = __popc(__ballot_sync(0xffffffffu, lane * step < len && jobs[lo + lane * step].tile0 <= t)) - 1;
        lo += n * step;
        if (step <= 1) break;
        len = len - n * step < step ? len - n * step : step;
    }
    while (t < end) {
        const PackJob j = jobs[lo++];
        const int job_end = j.tile0 + pack_ct(j) * pack_rt(j) * j.k * j.k, stop = job_end < end ? job_end : end;
        pack_layer(j, t - j.tile0, stop - j.tile0, 1);
        t = stop;
    }
}
// the layers of a block, or a single one (table by value); blockIdx.y picks the layer
__global__ void __launch_bounds__(256) pack_weights_kernel(const __grid_constant__ PackJobs jobs) {
    pdl_enter();
    const PackJob &j = jobs.job[blockIdx.y];
    pack_layer(j, blockIdx.x, pack_ct(j) * pack_rt(j) * j.k * j.k, gridDim.x);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encoder(revnet_ctx *ctx) {
    if (!ctx->encode_tiled) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || qres != cudaDriverEntryPointSuccess)
            fn = nullptr;
        ctx->encode_tiled = fn;
    }
    return (EncodeTiledFn)ctx->encode_tiled;
}

int round_up(int x, int m) { return (x + m - 1) / m * m; }

// 128-row tiles over an output of N x H x W pixels: whole rows of one image (the last tile of an
// image may be ragged), or whole images when an image has at most 64 pixels.  Rows of the tile
// that fall outside are padding: TMA fills their operand rows with zeros and the epilogue skips them.
bool tile_geom(Geom g, TileGeom &t) {
    if (g.W > 128 || g.W < 1) return false;
    t.N = g.N; t.H = g.H; t.W = g.W;
    t.BH = 128 / g.W; if (t.BH > g.H) t.BH = g.H;
    t.BIMG = 1;
    if (t.BH == g.H) { t.BIMG = 128 / (g.H * g.W); if (t.BIMG > g.N) t.BIMG = g.N; if (t.BIMG < 1) t.BIMG = 1; }
    t.tiles_per_img = (g.H + t.BH - 1) / t.BH;
    t.n_px_tiles = t.BIMG > 1 ? (g.N + t.BIMG - 1) / t.BIMG : g.N * t.tiles_per_img;
    return true;
}

struct TcShape { int KC, cin_pad, chunks, BN, n_tiles, smem; TileGeom g; };

// Which shapes the kernel takes: stride 1 or 2, k in {1,3}, channel rows 16-byte aligned for TMA.
bool tc_shape(Geom g, int cin, int cout, int k, int stride, TcShape &s, bool wide = false) {   // g: output geometry
    if ((stride != 1 && stride != 2) || (k != 1 && k != 3) || cin % 8 || cout % 4) return false;
    if (!tile_geom(g, s.g)) return false;
    if (s.g.W * stride > 256 || s.g.BH * stride > 256) return false;
    s.cin_pad = round_up(cin, 16);
    s.KC = s.cin_pad % 64 == 0 ? 64 : (s.cin_pad % 32 == 0 ? 32 : 16);
    s.chunks = s.cin_pad / s.KC;
    const int cout_pad = round_up(cout, 16);
    s.BN = cout_pad <= 128 ? cout_pad : 128;
    if (wide && cout_pad >= 256) s.BN = 256;        // 128 x 256 tiles: fewer operand bytes per flop
    s.n_tiles = (cout_pad + s.BN - 1) / s.BN;
    const int a_bytes = 128 * s.KC * 2, b_bytes = s.BN * s.KC * 2;
    s.smem = 1024 + 4 * (((a_bytes + 1023) & ~1023) + ((b_bytes + 1023) & ~1023)) + kEpiStageBytes + kEpiSumFloats * 4 + (int)sizeof(TcShared) + 64;
    return true;
}

// act: bf16 [N,H,W,cin]; Wsrc: fp32 weights; transposed selects the dgrad pack
// s2: the data gradient of a 3x3 stride-2 layer.  `act` is then the upstream gradient on the layer's output grid
// (gin), `out` the gradient on the input grid (twice as fine), and the launch's tile list runs over the four parity classes of the
// input pixels: class (py, px) fills the pixels (2i + py, 2j + px) from the taps that reach them,
//   da[2i+py, 2j+px] = sum over th in T(py), tw in T(px) of g[i + th/2, j + tw/2] Wd[th, tw],  T(0) = {1}, T(1) = {0, 2}
// (Wd the mirrored, transposed pack), so the four classes together cost the nine taps once per four pixels.
bool run_conv_tc(Exec &ex, const char *what, const void *act, Geom gin, int cin, int cout, int k, int stride,
                 const float *Wsrc, const bf16 *prepacked, bool transposed, Pair out, Pair partner, int sign, EpiReq req,
                 bool s2 = false) {
    TcShape s;
    // a 1x1 layer has no neighbours: its pixels as one column, 128 of them per tile (by image rows a tile holds 112 of 56x56 or
    // 28x28 images, 98 of 7x7)
    if (k == 1 && stride == 1 && !s2 && gin.P() < (1u << 30)) gin = Geom{1, (int)gin.P(), 1};
    if (stride == 2 && (gin.H % 2 || gin.W % 2)) return false;
    if (s2 && (stride != 1 || k != 3 || !transposed || sign || req.stats || out.c1)) return false;
    const Geom g{gin.N, conv_out(gin.H, k, stride), conv_out(gin.W, k, stride)};   // geometry of the tiles
    if (!tc_shape(g, cin, cout, k, stride, s)) return false;
    const int taps = k * k;
    if (!ex.dry && !encoder(ex.ctx)) return false;
    // the taps of every class of this launch
    const int n_cls = s2 ? 4 : 1;
    int ntap[4] = {0, 0, 0, 0}, ntap_all = 0;
    signed char tdy[4][9], tdx[4][9], tid[4][9];
    memset(tdy, 0, sizeof tdy); memset(tdx, 0, sizeof tdx); memset(tid, 0, sizeof tid);
    for (int c = 0; c < n_cls; c++) {
        const int py = c >> 1, px = c & 1;
        for (int th = 0; th < k; th++)
            for (int tw = 0; tw < k; tw++) {
                if (s2 && ((th & 1) == py || (tw & 1) == px)) continue;
                const int i = ntap[c]++;
                tdy[c][i] = (signed char)(s2 ? th / 2 : th - k / 2); tdx[c][i] = (signed char)(s2 ? tw / 2 : tw - k / 2);
                tid[c][i] = (signed char)(th * k + tw);
            }
        ntap_all += ntap[c];
    }
    // epilogue through TMA where a column group never straddles the halves of a channel-split tensor
    const bool need_aux = sign != 0 || req.bnbwd != nullptr;
    const Pair auxp = req.bnbwd ? req.bnbwd->t : partner;
    const int ntap_max = s2 ? 4 : taps;
    // arithmetic-bound layers without a partner tile (transitions, their data gradients): 128 x 256 tiles
    if (!need_aux && !(out.c1 && out.c0 % 32) && (long long)ntap_max * cin >= 1024 && cout >= 256 && cout % 32 == 0) tc_shape(g, cin, cout, k, stride, s, true);
    // 1x1 layers onto 256 channels and more on a CTA pair with 256 x 256 tiles: half the operand traffic from L2 per flop.
    // Measured on the large-image network: layers WITHOUT a partner tile (2048 -> 512 and the like, many channel chunks
    // per tile) 8-12 % faster; layers WITH one (the last layer of a bottleneck function, epilogue-bound, and a partner
    // ring that the wide tile leaves only two slots per warp group) 7-12 % slower.  REVNET_CONV_PAIR1X1 overrides:
    // bit 0 layers with a partner tile, bit 1 layers without (default 2)
    static const bool pair_enabled = [] { const char *v = getenv("REVNET_CONV_PAIR"); return !(v && v[0] == '0'); }();
    static const int pair1x1 = [] { const char *v = getenv("REVNET_CONV_PAIR1X1"); return v ? atoi(v) : 2; }();
    const bool wide1 = k == 1 && stride == 1 && !s2 && cout >= 256 && cout % 32 == 0 && !(out.c1 && out.c0 % 32) &&
                       !(need_aux && auxp.c1 && auxp.c0 % 32) && s.KC == 64 &&
                       pair_enabled && ex.ctx->sm_count % 2 == 0 && s.g.n_px_tiles >= 2 && ((need_aux && (pair1x1 & 1)) || (!need_aux && (pair1x1 & 2)));
    if (wide1) tc_shape(g, cin, cout, k, stride, s, true);
    // 3x3 stride-1 layers with a partner tile (data gradients with the BN-backward sums fused) on a pair: 256-wide tiles
    // too, the partner groups through a ring of two slots per warp group (REVNET_CONV_WIDE3X3=0: 128-wide, as before)
    static const bool wide3_enabled = [] { const char *v = getenv("REVNET_CONV_WIDE3X3"); return !(v && v[0] == '0'); }();
    const bool wide3 = wide3_enabled && k == 3 && stride == 1 && !s2 && need_aux && cout >= 256 && cout % 32 == 0 && !(out.c1 && out.c0 % 32) &&
                       !(auxp.c1 && auxp.c0 % 32) && s.KC == 64 && pair_enabled && ex.ctx->sm_count % 2 == 0 && s.g.n_px_tiles >= 2;
    if (wide3) tc_shape(g, cin, cout, k, stride, s, true);
    // rows of the weight pack (a multiple of its 128-row blocks, whatever the N tile); TMA fills rows beyond with zeros
    const int rp16 = round_up(cout, 16), rows_pad = rp16 <= 128 ? rp16 : round_up(rp16, 128);
    // column groups of 32 floats, or of 16 where the N tile or the halves of a channel-split tensor ask for it
    int GW = s.BN % 32 == 0 ? 32 : 16;
    if (GW == 32 && s.BN <= 128 && ((out.c1 && out.c0 % 32) || (need_aux && auxp.c1 && auxp.c0 % 32))) GW = 16;
    const int ng = s.BN / GW, group_bytes = (128 * GW * 4 + 1023) & ~1023;
    bool epi_tma = !(out.c1 && out.c0 % GW) && !(need_aux && auxp.c1 && auxp.c0 % GW) && ng <= 8;
    const int ostride = s2 ? 2 : 1;
    if (s2 && (!epi_tma || g.W * 2 > 256 || s.g.BH * 2 > 256)) return false;
    int stages = 4;
    // CTA pairs (conv_tc2_kernel) wherever the epilogue runs through TMA, the N tile splits into two halves of whole
    // 16-row groups and there are at least two pixel tiles; REVNET_CONV_PAIR=0 keeps the single-CTA kernel (for comparison)
    // (1x1 layers are bound by the activations' way from HBM, which a pair does not shorten: measured 3-10 % slower there)
    bool pair = pair_enabled && epi_tma && (k == 3 || wide1) && s.BN % 32 == 0 && s.BN >= 64 && s.g.n_px_tiles >= 2 && ex.ctx->sm_count % 2 == 0;
    // 3x3 stride-1 layers on a pair: the activations of a tile arrive once per channel chunk as one box with its halo
    // (see TcParams::halo); needs 64-channel chunks (128-byte operand rows) and tiles of whole image rows
    static const bool halo_enabled = [] { const char *v = getenv("REVNET_CONV_HALO"); return !(v && v[0] == '0'); }();
    bool halo = halo_enabled && pair && k == 3 && stride == 1 && !s2 && s.KC == 64 && s.g.BIMG == 1 && g.W + 2 <= 128;
    int a_slot_bytes = 0, a_box_bytes = 0;
    const int a_slots = 2;
    if (halo) {
        const int Wp = g.W + 2;
        int bh = 128 / Wp; if (bh > g.H) bh = g.H;
        s.g.BH = bh;
        s.g.tiles_per_img = (g.H + bh - 1) / bh;
        s.g.n_px_tiles = g.N * s.g.tiles_per_img;
        const int box_rows = (bh + 2) * Wp, read_rows = 2 * Wp + 2 + 128;       // rows the box holds / rows the last tap reads up to
        a_box_bytes = box_rows * 128;
        a_slot_bytes = ((box_rows > read_rows ? box_rows : read_rows) * 128 + 1023) & ~1023;
    }
    int groups = 2, aux_slots = 0, epi_bytes = 0;
    bool inplace = false;
    if (epi_tma) {
        auto stage_bytes_of = [&](bool pr) {
            if (halo) return ((s.BN / 2) * s.KC * 2 + 1023) & ~1023;           // weight tiles only; the boxes are counted below
            return ((128 * s.KC * 2 + 1023) & ~1023) + (((pr ? s.BN / 2 : s.BN) * s.KC * 2 + 1023) & ~1023);
        };
        // Warp groups, partner slots per group and operand stages: the first of these that fits.  Single-CTA kernel: four groups (a
        // divisor or a multiple of the column groups: three for three) as long as three operand stages remain (two if a tile has no more
        // chunks); a coupling works in place in two slots per group.
        const int iters = ntap_max * s.chunks, few = iters < 3 ? 2 : 3, want = pair ? 2 : (ng == 3 ? 3 : 4);
        const struct { int groups, slots, stages; } tries[] = {{want, 2, few}, {want, 1, few}, {2, 2, few}, {2, 1, few}, {2, 2, 2}, {2, 1, 2}, {1, 1, 2}};
        inplace = sign != 0;
        bool fits = false;
        for (const auto &y : tries) {
            if (inplace && y.slots < 2) continue;
            if (ng < y.groups && y.groups % ng) continue;
            groups = y.groups; aux_slots = y.slots;
            epi_bytes = ((need_aux ? groups * aux_slots : 0) + (inplace ? 0 : groups)) * group_bytes + (ng > groups ? ng * 4096 : 0);
            const int least = groups * 4096 + (groups * 128 + 128) * 32;        // the sums at the end, and the last reduction
            if (epi_bytes < least) epi_bytes = least;
            auto smem_of = [&](int st) { return 1024 + (halo ? a_slots * a_slot_bytes : 0) + st * stage_bytes_of(pair) + epi_bytes + (int)sizeof(TcShared) + 64; };
            stages = kStages;
            while (stages > y.stages && smem_of(stages) > 227 * 1024) stages--;
            if (smem_of(stages) <= 227 * 1024) { fits = true; s.smem = smem_of(stages); break; }
        }
        // On a pair (two groups, eight partner barriers) room that the operand ring leaves goes to more partner slots, up to the four
        // column groups that a warp group has in a tile: with two, narrow column groups or a result stored from its slot leave
        // the next partner group too little time to arrive
        for (int more = aux_slots + 1; fits && pair && need_aux && more <= 4 && more <= (ng + groups - 1) / groups + (inplace ? 1 : 0); more++) {
            const int bytes = ((groups * more) + (inplace ? 0 : groups)) * group_bytes + (ng > groups ? ng * 4096 : 0), extra = bytes > epi_bytes ? bytes - epi_bytes : 0;
            if (s.smem + extra > 227 * 1024) break;
            aux_slots = more; epi_bytes += extra; s.smem += extra;
        }
        if (!fits) {
            if (s.BN == 256) return false;      // (does not happen)
            epi_tma = false; pair = false; stages = 4;
            if (halo) { halo = false; tile_geom(g, s.g); }
        }
    }
    if ((s2 || s.BN == 256) && !epi_tma) return false;
    ex.flops += 2ull * g.P() * cout * cin * ntap_all;
    int occ = (227 * 1024) / s.smem; if (occ > 2) occ = 2; if (occ < 1 || groups > 2) occ = 1;      // (registers: 18 warps leave no room for a second CTA)
    int ctas = ex.ctx->sm_count * occ / s.n_tiles; if (ctas < 1) ctas = 1;
    if (ctas > s.g.n_px_tiles * n_cls) ctas = s.g.n_px_tiles * n_cls;
    if (pair) {
        // one pair per TPC and N tile; a pair walks tile pairs
        const int n_vp = n_cls * ((s.g.n_px_tiles + 1) / 2);
        int pairs = (ex.ctx->sm_count / 2) / s.n_tiles; if (pairs < 1) pairs = 1;
        if (pairs > n_vp) pairs = n_vp;
        ctas = 2 * pairs;
    }
    size_t m = ex.ws.mark();
    bf16 *wp = prepacked ? const_cast<bf16 *>(prepacked) : ex.ws.get<bf16>((size_t)rows_pad * taps * s.cin_pad);
    const bool reduce = req.stats || req.bnbwd;
    // statistics that the next layer's kernel adds up itself stay pending
    const bool defer = req.stats && !req.bnbwd && epi_tma && req.stats->defer && req.stats->part && (size_t)ctas * 2 * cout <= req.stats->part_cap;
    float *part = defer ? req.stats->part : (reduce ? ex.ws.get<float>((size_t)ctas * 2 * cout) : nullptr);
    if (req.stats) {
        req.stats->valid = true;
        req.stats->pending = defer; req.stats->parts = ctas; req.stats->inv_count = 1.0 / ((double)g.P() * ostride * ostride);
    }
    if (!ex.dry) {
        EncodeTiledFn enc = encoder(ex.ctx);
        // without a pack made earlier in the step, build it from the fp32 master weights now
        if (!prepacked) {
            // (the pack's own sizes are those of tc_pack_elems: rows rounded up to its 128-row blocks, columns to 16)
            tc_pack_now(ex, Wsrc, wp, transposed ? cout : cin, transposed ? cin : cout, k, transposed);
        }
        CUtensorMap map_a, map_b;
        const CUtensorMapSwizzle sw = s.KC == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (s.KC == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
        {
            // the box spans stride x the tile in the input image and is walked with that stride
            cuuint64_t dims[4] = {(cuuint64_t)cin, (cuuint64_t)gin.W, (cuuint64_t)gin.H, (cuuint64_t)gin.N};
            cuuint64_t strides[3] = {(cuuint64_t)cin * 2, (cuuint64_t)gin.W * cin * 2, (cuuint64_t)gin.H * gin.W * cin * 2};
            cuuint32_t box[4] = {(cuuint32_t)s.KC, (cuuint32_t)(g.W * stride), (cuuint32_t)(s.g.BH * stride), (cuuint32_t)s.g.BIMG};
            if (halo) { box[1] = (cuuint32_t)(g.W + 2); box[2] = (cuuint32_t)(s.g.BH + 2); }
            cuuint32_t es[4] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1};
            CUresult r = enc(&map_a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)act, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                             sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) { ex.failed = true; ex.ctx->err = std::string(what) + ": tensor map (activations) rejected"; ex.ws.release(m); return true; }
        }
        {
            cuuint64_t dims[2] = {(cuuint64_t)taps * s.cin_pad, (cuuint64_t)rows_pad};
            cuuint64_t strides[1] = {(cuuint64_t)taps * s.cin_pad * 2};
            cuuint32_t box[2] = {(cuuint32_t)s.KC, (cuuint32_t)(pair ? s.BN / 2 : s.BN)};     // a CTA of a pair loads its half of the N tile
            cuuint32_t es[2] = {1, 1};
            CUresult r = enc(&map_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)wp, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                             sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) { ex.failed = true; ex.ctx->err = std::string(what) + ": tensor map (weights) rejected"; ex.ws.release(m); return true; }
        }
        CUtensorMap map_o[2], map_x[2];
        memset(map_o, 0, sizeof map_o); memset(map_x, 0, sizeof map_x);
        if (epi_tma) {
            const CUtensorMapSwizzle gsw = GW == 32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
            auto enc_f32 = [&](CUtensorMap *map, const float *base, int C) {
                // the epilogue's tensors live on the output grid: the tile's grid, or (parity class) the twice finer
                // one walked with stride 2
                const cuuint64_t Wo = (cuuint64_t)g.W * ostride, Ho = (cuuint64_t)g.H * ostride;
                cuuint64_t dims[4] = {(cuuint64_t)C, Wo, Ho, (cuuint64_t)g.N};
                cuuint64_t strides[3] = {(cuuint64_t)C * 4, Wo * C * 4, Ho * Wo * C * 4};
                cuuint32_t box[4] = {(cuuint32_t)GW, (cuuint32_t)(g.W * ostride), (cuuint32_t)(s.g.BH * ostride), (cuuint32_t)s.g.BIMG};
                cuuint32_t es[4] = {1, (cuuint32_t)ostride, (cuuint32_t)ostride, 1};
                return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void *)base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           gsw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
            };
            bool ok = enc_f32(&map_o[0], out.p0, out.c0);
            if (out.c1) ok = ok && enc_f32(&map_o[1], out.p1, out.c1); else map_o[1] = map_o[0];
            if (need_aux) {
                ok = ok && enc_f32(&map_x[0], auxp.p0, auxp.c0);
                if (auxp.c1) ok = ok && enc_f32(&map_x[1], auxp.p1, auxp.c1); else map_x[1] = map_x[0];
            } else { map_x[0] = map_x[1] = map_o[0]; }
            if (!ok) { ex.failed = true; ex.ctx->err = std::string(what) + ": tensor map (epilogue) rejected"; ex.ws.release(m); return true; }
        }
        TcParams p;
        p.stages = stages; p.GW = GW; p.group_bytes = group_bytes; p.need_aux = need_aux ? 1 : 0;
        p.groups = groups; p.aux_slots = need_aux ? aux_slots : 0; p.inplace = inplace ? 1 : 0; p.epi_bytes = epi_bytes;
        p.split_o = out.c1 ? out.c0 : 0; p.split_x = (need_aux && auxp.c1) ? auxp.c0 : 0;
        memcpy(p.ntap, ntap, sizeof ntap); memcpy(p.tdy, tdy, sizeof tdy); memcpy(p.tdx, tdx, sizeof tdx); memcpy(p.tid, tid, sizeof tid);
        p.ostride = ostride; p.n_cls = n_cls;
        p.halo = halo ? 1 : 0; p.Wp = g.W + 2; p.a_slots = a_slots; p.a_slot_bytes = a_slot_bytes; p.a_box_bytes = a_box_bytes;
        for (int c = 0; c < 4; c++) { p.oy[c] = s2 ? c >> 1 : 0; p.ox[c] = s2 ? c & 1 : 0; }
        p.taps = taps; p.k = k; p.chunks = s.chunks; p.KC = s.KC; p.cin_pad = s.cin_pad; p.BN = s.BN; p.stride = stride; p.g = s.g;
        p.status = ex.ctx->dev_status;
        p.stamp = ex.stamp_slot();
        EpiArgs &e = p.epi;
        memset(&e, 0, sizeof e);
        e.mode = req.bnbwd ? EPI_BNBWD : (sign ? EPI_COUPLE : EPI_PLAIN);
        e.out = out; e.partner = partner; e.sign = sign; e.n_cols = cout; e.pitch = kEpiPitch;
        e.part = part; e.counter = reduce && !defer ? ex.ctx->counter(s.n_tiles) : nullptr;
        e.inv_count = 1.0 / ((double)g.P() * ostride * ostride); e.eps = ex.eps;     // pixels of the output grid
        if (req.stats) { e.mean = req.stats->mean; e.rstd = req.stats->rstd; }
        if (req.bnbwd) { e.t = req.bnbwd->t; e.bn = req.bnbwd->bn; e.dgamma = req.bnbwd->dgamma; e.dbeta = req.bnbwd->dbeta; e.coef = req.bnbwd->coef; }
        static OncePerDevice once;
        if (once.first(ex.ctx->device)) {
            cudaFuncSetAttribute(conv_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
            cudaFuncSetAttribute(conv_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
            cudaFuncSetAttribute(conv_tc2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        }
        dim3 grid((unsigned)ctas, (unsigned)s.n_tiles);
        if (pair) launch_cluster(ex, conv_tc2_kernel, grid, 64 + groups * 128, s.smem, 2, map_a, map_b, map_o[0], map_o[1], map_x[0], map_x[1], p);
        else launch(ex, epi_tma ? conv_tc_kernel<true> : conv_tc_kernel<false>, grid, epi_tma ? 64 + groups * 128 : kThreads, s.smem, map_a, map_b, map_o[0], map_o[1], map_x[0], map_x[1], p);
        const double bytes = (double)gin.P() * cin * 2 + (double)g.P() * cout * (sign || req.bnbwd ? 8 : 4) + (double)cout * taps * cin * 2;
        // (records of launches on a CTA pair carry the pair kernel's name)
        ex.check(!pair ? what : (transposed ? "conv_dgrad_tc2" : "conv_fprop_tc2"), bytes, 2.0 * g.P() * cout * cin * ntap_all);
    }
    ex.ws.release(m);
    return true;
}

bool run_bn_conv(Exec &ex, Pair t, BnRef bn, Geom gi, const Layer &L, Pair out, Moments *stats, bf16 *a_out) {
    const int cin = L.cin, cout = L.cout;
    if (L.k != 1 || L.stride != 1 || cin < 128 || cin % 64 || cin > 1024 || cout % 8 || cout > 128 || t.c1 || out.c1 || out.q != 0.f || bn.part || gi.P() >= (1u << 30)) return false;
    if (!ex.dry && !encoder(ex.ctx)) return false;
    const int P = (int)gi.P(), BN = round_up(cout, 16), GW = BN % 32 == 0 ? 32 : 16, ng = BN / GW, group_bytes = 128 * GW * 4;
    const int stage_bytes = 16384 + ((BN * 128 + 1023) & ~1023);
    const int groups = 2;
    int epi_bytes = groups * group_bytes + (ng > groups ? ng * 4096 : 0);
    const int least = groups * 4096 + (groups * 128 + 128) * 32;
    if (epi_bytes < least) epi_bytes = least;
    const int fixed = 1024 + epi_bytes + 8 * cin + (int)sizeof(TcShared) + 64;
    // operand stages: an even number (a build team keeps to its own: it sees every phase of their empty barriers)
    int stages = 4, raws = 4;
    if (fixed + stages * stage_bytes + 3 * kRawBytes > 227 * 1024) stages = 2;
    while (raws > 2 && fixed + stages * stage_bytes + raws * kRawBytes > 227 * 1024) raws--;
    const int smem = fixed + stages * stage_bytes + raws * kRawBytes;
    if (smem > 227 * 1024) return false;
    TileGeom tg;
    if (!tile_geom(Geom{1, P, 1}, tg)) return false;
    ex.flops += 2ull * P * cout * cin;
    int ctas = ex.ctx->sm_count; if (ctas > tg.n_px_tiles) ctas = tg.n_px_tiles;
    size_t m = ex.ws.mark();
    const size_t pack_elems = tc_pack_elems(cin, cout, 1, false);
    bf16 *wp = L.Wp_fprop ? const_cast<bf16 *>((const bf16 *)L.Wp_fprop) : ex.ws.get<bf16>(pack_elems);
    const bool defer = stats && stats->defer && stats->part && (size_t)ctas * 2 * cout <= stats->part_cap;
    float *part = defer ? stats->part : (stats ? ex.ws.get<float>((size_t)ctas * 2 * cout) : nullptr);
    if (stats) { stats->valid = true; stats->pending = defer; stats->parts = ctas; stats->inv_count = 1.0 / (double)P; }
    if (!ex.dry) {
        EncodeTiledFn enc = encoder(ex.ctx);
        if (!L.Wp_fprop) tc_pack_now(ex, L.W, wp, cin, cout, 1, false);
        BnConvParams q;
        memset(&q, 0, sizeof q);
        TcParams &p = q.p;
        CUtensorMap map_raw, map_b, map_o;
        auto enc2 = [&](CUtensorMap *map, CUtensorMapDataType dt, const void *base, int esz, int cols, int rows, int bc, int br) {
            cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)cols * esz};
            cuuint32_t box[2] = {(cuuint32_t)bc, (cuuint32_t)br}, es[2] = {1, 1};
            return enc(map, dt, 2, (void *)base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        };
        bool ok = enc2(&map_raw, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, t.p0, 4, cin, P, 32, 128) &&
                  enc2(&map_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, wp, 2, cin, round_up(cout, 16), 64, BN);
        {
            cuuint64_t dims[4] = {(cuuint64_t)cout, 1, (cuuint64_t)P, 1}, strides[3] = {(cuuint64_t)cout * 4, (cuuint64_t)cout * 4, (cuuint64_t)P * cout * 4};
            cuuint32_t box[4] = {(cuuint32_t)GW, 1, (cuuint32_t)tg.BH, 1}, es[4] = {1, 1, 1, 1};
            ok = ok && enc(&map_o, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void *)out.p0, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           GW == 32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
        }
        if (!ok) { ex.failed = true; ex.ctx->err = "conv1x1_bn: tensor map rejected"; ex.ws.release(m); return true; }
        p.taps = 1; p.k = 1; p.chunks = cin / 64; p.KC = 64; p.cin_pad = cin; p.BN = BN; p.stride = 1; p.g = tg;
        p.status = ex.ctx->dev_status; p.stamp = ex.stamp_slot(); p.stages = stages; p.groups = groups; p.epi_bytes = epi_bytes;
        p.GW = GW; p.group_bytes = group_bytes; p.n_cls = 1; p.ntap[0] = 1; p.ostride = 1;
        EpiArgs &e = p.epi;
        e.mode = EPI_PLAIN; e.out = out; e.n_cols = cout; e.part = part; e.counter = stats && !defer ? ex.ctx->counter() : nullptr;
        e.inv_count = 1.0 / (double)P; e.eps = ex.eps;
        if (stats) { e.mean = stats->mean; e.rstd = stats->rstd; }
        q.bn = bn; q.in_q = t.q; q.a_out = a_out; q.P = P; q.raw_stages = raws;
        static OncePerDevice once;
        if (once.first(ex.ctx->device)) cudaFuncSetAttribute(conv1x1_bn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        launch(ex, conv1x1_bn_kernel, ctas, kBnThreads, smem, map_raw, map_b, map_o, q);
        ex.check("conv_fprop_bn", (double)P * cin * (a_out ? 6 : 4) + (double)P * cout * 4 + (double)cout * cin * 2, 2.0 * P * cout * cin);
    }
    ex.ws.release(m);
    return true;
}

// ------------------------------------------------------------------------------------------------
// Weight gradient:  dW[co, tap, ci] = sum_p g[p, co] * a[p (+) tap, ci]
// GEMM view: the reduction runs over pixels.  Both operands are pixel-major in memory, so the tiles
// TMA delivers ([128 pixels][channel block]) are MN-major operands as they stand.  The M side
// stacks (tap, input-channel block) tiles -- one shifted TMA box each -- 128 rows per MMA group;
// the N side is a block of output channels.  A CTA owns up to two M groups and one N tile, walks
// its share of the pixel tiles (split-K) accumulating in tensor memory, and writes an fp32
// partial; the partials are summed in fixed order by splitk_sum_batch_kernel.
// For 3x3 layers of few channels the taps are split between the operands instead (sep):
//   dW[co, (kh, kw), ci] = sum_p a[p + (kh, 0), ci] * g[p - (0, kw), co]
// so the M side stacks the three vertical shifts of the activations, the N side the three horizontal
// shifts of the gradient: six boxes and one MMA group per pixel tile where the stacked form takes ten
// boxes and two groups.  (Activations outside the image are zero, so pixels p outside it add nothing.)
struct WgParams {
    int taps, k;
    int blockC, cblks, cin;      // input-channel block (16/32/64), blocks per tap, valid channels
    int total_blocks;            // taps * cblks
    int blockN, BN, cout;        // output-channel block, N tile, valid channels
    int GM;                      // M groups per CTA (1 or 2)
    int H, W, BH, BIMG;          // output geometry and tile
    int tiles_per_img, box_px;   // tiles per image (BIMG == 1); pixels a tile really holds (<= 128, the rest of its rows stay zero)
    int stride;
    int n_tiles_px;              // pixel tiles in all
    int stages;
    float *partial;              // splits > 1: [splits][taps][cin][cout], summed and transposed afterwards; else the gradient itself
    size_t slice;                // cout*taps*cin
    int *status;
    int a_region;                // bytes of a stage that hold activation blocks (the gradient blocks follow)
    int sep, cout_pad;           // sep: taps split between the operands (see the kernel); cout rounded up to 16
    int splits, m_chunks;        // this job's CTAs: split x M chunk x N tile, split fastest
    int cta0;                    // first CTA of the job in the launch
    int pair;                    // wgrad_tc2_kernel: BN is what ONE CTA of a pair holds of the pair's 2 * BN output channels,
                                 // GM the pair's M groups of 256 rows (CTA r takes the 128-row groups 2j + r of the chunk)
};

// One launch computes the weight gradients of up to kWgMaxJobs layers: each CTA finds its job from
// its index and then works on that layer alone.
constexpr int kWgMaxJobs = 4;
struct alignas(64) WgJob { CUtensorMap map_a, map_g; WgParams p; };
struct WgBatch { WgJob job[kWgMaxJobs]; int n; unsigned long long *stamp; };

__global__ void __launch_bounds__(kThreads, 1)
wgrad_tc_kernel(const __grid_constant__ WgBatch batch) {
    int jb = 0;
    while (jb + 1 < batch.n && (int)blockIdx.x >= batch.job[jb + 1].p.cta0) jb++;
    const WgParams &p = batch.job[jb].p;
    const CUtensorMap &map_a = batch.job[jb].map_a, &map_g = batch.job[jb].map_g;
    const int local = (int)blockIdx.x - p.cta0;
    const int split = local % p.splits, chunk = (local / p.splits) % p.m_chunks, ntile = local / (p.splits * p.m_chunks);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *tiles = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int blk_bytes_a = 256 * p.blockC, blk_bytes_b = 256 * p.blockN;   // [128 pixels][block] bf16
    // a stage holds only the blocks a CTA really loads.  An M group is 128 rows = 32 KB from its first block:
    // the MMAs of a group that is not full read on into what follows (their rows of the result are never
    // stored), so the launch reserves room behind the last stage for that.
    const int a_region = p.a_region;
    const int stage_bytes = a_region + ((256 * p.BN + 1023) & ~1023);
    TcShared *sh = (TcShared *)(tiles + p.stages * stage_bytes);

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int bpg = 128 / p.blockC;                          // blocks per M group
    const int first_block = chunk * p.GM * bpg;
    int n_blocks = p.total_blocks - first_block; if (n_blocks > p.GM * bpg) n_blocks = p.GM * bpg;
    const int groups = (n_blocks + bpg - 1) / bpg;
    const int col0 = ntile * p.BN;
    int nb_n = (p.cout - col0 + p.blockN - 1) / p.blockN; if (nb_n > p.BN / p.blockN) nb_n = p.BN / p.blockN;   // N blocks holding valid channels
    const int npk = p.cout_pad / p.blockN;                   // sep: N blocks per horizontal shift
    if (p.sep) nb_n = p.k * npk;
    const int my_tiles = (p.n_tiles_px - split + p.splits - 1) / p.splits;
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < p.GM * p.BN) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; s++) { mbar_init(&sh->full[s], 1); mbar_init(&sh->empty[s], 1); }
        mbar_init(&sh->acc_full[0], 1);
        sh->failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&sh->tmem_base, tmem_cols);
    if (p.box_px < 128) {
        // a tile holds fewer than 128 pixels: the rows TMA never writes must not add to the pixel sum
        uint4 *z = reinterpret_cast<uint4 *>(tiles);
        const int n16 = p.stages * stage_bytes / 16;
        for (int i = threadIdx.x; i < n16; i += kThreads) z[i] = make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    pdl_enter();             // the set-up above may overlap the kernel before; its outputs are read from here on
    stamp_begin(batch.stamp);
    const uint32_t tmem_d = sh->tmem_base;
    const int pad = p.k / 2;
    const int tiles_per_img = p.tiles_per_img;

    if (warp == 0) {
        // producer warp: lane 0 waits for the slot and arms the barrier, then every lane issues one box
        // (lane b < n_blocks: shifted activation block b; the next nb_n lanes: gradient blocks), so that
        // the loads of a tile leave in one instruction instead of one after the other
        const uint32_t tx = (uint32_t)(p.box_px * 2 * (n_blocks * p.blockC + nb_n * p.blockN));
        const bool a_lane = lane < n_blocks, g_lane = !a_lane && lane < n_blocks + nb_n;
        const int gb = first_block + lane, tap = gb / p.cblks, cb = gb - tap * p.cblks;
        const int kh = p.sep ? tap : tap / p.k, kw = p.sep ? p.k / 2 : tap - (tap / p.k) * p.k;
        const int bg = lane - n_blocks;
        const int g_c = p.sep ? (bg % npk) * p.blockN : col0 + bg * p.blockN;      // gradient box: first channel, first column
        const int g_x = p.sep ? p.k / 2 - bg / npk : 0;
        int s = 0; uint32_t round = 0;
        for (int it = 0; it < my_tiles; it++) {
            bool ok = true;
            if (lane == 0) {
                if (round > 0 && !mbar_wait(&sh->empty[s], (round - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; }
                if (ok) mbar_expect_tx(&sh->full[s], tx);
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            const int t = split + it * p.splits;
            const int n0 = p.BIMG > 1 ? t * p.BIMG : t / tiles_per_img;
            const int h0 = p.BIMG > 1 ? 0 : (t - n0 * tiles_per_img) * p.BH;
            uint8_t *sa = tiles + s * stage_bytes;
            if (a_lane) tma_load_4d(sa + lane * blk_bytes_a, &map_a, &sh->full[s], cb * p.blockC, kw - pad, h0 * p.stride + kh - pad, n0);
            else if (g_lane) tma_load_4d(sa + a_region + bg * blk_bytes_b, &map_g, &sh->full[s], g_c, g_x, h0, n0);
            if (++s == p.stages) { s = 0; round++; }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = instr_desc(p.BN, true);
            const int rba = p.blockC * 2, rbb = p.blockN * 2;
            // one thread issues everything: descriptors are a base plus increments of the address field (16-byte units),
            // the ring position is stepped (no divisions in the loop)
            const uint64_t da0 = smem_desc_mn(smem_u32(tiles), rba, blk_bytes_a), db0 = smem_desc_mn(smem_u32(tiles) + a_region, rbb, blk_bytes_b);
            const uint32_t stage16 = (uint32_t)stage_bytes >> 4;
            int s = 0; uint32_t round = 0, soff = 0;
            for (int it = 0; it < my_tiles; it++) {
                if (!mbar_wait(&sh->full[s], round & 1)) { atomicExch(&sh->failed, 1u); break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t accum = it > 0 ? 1u : 0u;
                for (int g = 0; g < groups; g++) {
                    uint64_t da = da0 + soff + (uint32_t)(g * 2048), db = db0 + soff;      // an M group is 32 KB from its first block
                    const uint32_t acc = tmem_d + (uint32_t)(g * p.BN);
                    mma_bf16(acc, da, db, idesc, accum);
                    for (int ks = 1; ks < 8; ks++) {         // 16 pixels per MMA
                        da += (uint32_t)rba; db += (uint32_t)rbb;
                        mma_bf16(acc, da, db, idesc, 1u);
                    }
                }
                mma_commit(&sh->empty[s]);
                soff += stage16;
                if (++s == p.stages) { s = 0; soff = 0; round++; }
            }
            mma_commit(&sh->acc_full[0]);
        }
    } else {
        const int quarter = warp & 3;
        bool ok = true;
        if (quarter == 0 && lane == 0) ok = mbar_wait(&sh->acc_full[0], 0);     // one thread polls, the rest block
        ok = named_barrier_and(2, 128, ok);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok && sh->failed == 0) {
            const int m = quarter * 32 + lane;
            float *dst = p.partial + (size_t)split * p.slice;
            for (int g = 0; g < groups; g++) {
                const int gb = first_block + g * bpg + m / p.blockC;
                const int tap_m = gb / p.cblks, ci = (gb - tap_m * p.cblks) * p.blockC + m % p.blockC;     // sep: tap_m is kh
                const bool row_ok = gb < p.total_blocks && ci < p.cin;
                for (int c = 0; c < p.BN; c += 16) {
                    float v[16];
                    tmem_ld16(tmem_d + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(g * p.BN + c), v);   // whole warp takes part
                    if (!row_ok) continue;
                    if (my_tiles == 0) {
#pragma unroll
                        for (int j = 0; j < 16; j++) v[j] = 0.f;
                    }
                    // column c of the accumulator: output channel cb0 + ..., and with sep the horizontal shift too
                    const int kw = p.sep ? c / p.cout_pad : 0;
                    const int cb0 = p.sep ? c - kw * p.cout_pad : col0 + c;
                    const int tap = p.sep ? tap_m * p.k + kw : tap_m;
                    if (p.splits > 1) {
                        // split partials are [tap][ci][co]: this row's output channels are contiguous (cout is a multiple of 8)
                        float *row = dst + ((size_t)tap * p.cin + ci) * p.cout + cb0;
#pragma unroll
                        for (int j = 0; j < 16; j += 4)
                            if (cb0 + j < p.cout) *reinterpret_cast<float4 *>(row + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j++) {
                            const int co = cb0 + j;
                            if (co < p.cout) dst[((size_t)co * p.taps + tap) * p.cin + ci] = v[j];
                        }
                    }
                }
            }
        } else if (lane == 0) {
            atomicExch(&sh->failed, 1u);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && sh->failed) atomicExch(p.status, (int)REVNET_E_TIMEOUT);
    stamp_end(batch.stamp);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_d, tmem_cols);
    }
}

// The same on a CTA pair (tcgen05 cta_group::2): an MMA of M = 256 covers two 128-row groups of (tap, input channel) rows,
// CTA `rank` holding the activation blocks of the groups 2j + rank and HALF of the pair's gradient channels; N = 2 * BN.
// Per pixel tile a CTA then loads GM x 32 KB of activations and BN x 256 B of gradients for GM x 8 MMAs of 256 x 2BN:
// half the operand bytes per flop of the single-CTA form, whose 94 bytes per MMA clock are more than an SM can take in.
// Not for the tap-split (sep) form.  Launched as clusters of two; every job of a launch is of this kind.
__global__ void __launch_bounds__(kThreads, 1)
wgrad_tc2_kernel(const __grid_constant__ WgBatch batch) {
    int jb = 0;
    while (jb + 1 < batch.n && (int)blockIdx.x >= batch.job[jb + 1].p.cta0) jb++;
    const WgParams &p = batch.job[jb].p;
    const CUtensorMap &map_a = batch.job[jb].map_a, &map_g = batch.job[jb].map_g;
    const uint32_t rank = cluster_ctarank();
    const int local = ((int)blockIdx.x - p.cta0) >> 1;         // pair index inside the job (cta0 is even)
    const int split = local % p.splits, chunk = (local / p.splits) % p.m_chunks, ntile = local / (p.splits * p.m_chunks);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *tiles = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int blk_bytes_a = 256 * p.blockC, blk_bytes_b = 256 * p.blockN;   // [128 pixels][block] bf16
    const int a_region = p.GM * 32768;                         // whole groups: 32 KB each
    const int stage_bytes = a_region + ((256 * p.BN + 1023) & ~1023);
    TcShared *sh = (TcShared *)(tiles + p.stages * stage_bytes);

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int bpg = 128 / p.blockC;                          // blocks per 128-row group
    const int first_block = chunk * 2 * p.GM * bpg;          // the pair's chunk: 2 * GM groups
    // blocks this CTA / the other CTA loads per pixel tile: group 2j + r holds the blocks first_block + (2j + r) * bpg ...
    auto blocks_of = [&](int r) { int n = 0; for (int j = 0; j < p.GM; j++) { int b = p.total_blocks - (first_block + (2 * j + r) * bpg); n += b < 0 ? 0 : (b > bpg ? bpg : b); } return n; };
    const int col0 = ntile * 2 * p.BN;                       // first output channel of the pair's N tile
    auto nblocks_of = [&](int r) { int n = (p.cout - (col0 + r * p.BN) + p.blockN - 1) / p.blockN; return n < 0 ? 0 : (n > p.BN / p.blockN ? p.BN / p.blockN : n); };
    const int my_tiles = (p.n_tiles_px - split + p.splits - 1) / p.splits;
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < p.GM * 2 * p.BN) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; s++) { mbar_init(&sh->full[s], 1); mbar_init(&sh->empty[s], 1); }
        mbar_init(&sh->acc_full[0], 1);
        sh->failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem2_alloc(&sh->tmem_base, tmem_cols);
    {
        // rows and blocks TMA never writes (short tiles, groups beyond the last block) must hold zeros, not stale bits:
        // their products land in rows that are never stored, but a NaN pattern would still be a NaN
        uint4 *z = reinterpret_cast<uint4 *>(tiles);
        const int n16 = p.stages * stage_bytes / 16;
        for (int i = threadIdx.x; i < n16; i += kThreads) z[i] = make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    pdl_enter();
    stamp_begin(batch.stamp);
    const uint32_t tmem_d = sh->tmem_base;
    const int pad = p.k / 2;
    const int tiles_per_img = p.tiles_per_img;

    if (warp == 0) {
        // lane (j, i) with j < GM, i < bpg: activation block i of this CTA's group 2j + rank; the next lanes: gradient blocks
        const uint32_t tx = (uint32_t)(p.box_px * 2 * ((blocks_of(0) + blocks_of(1)) * p.blockC + (nblocks_of(0) + nblocks_of(1)) * p.blockN));
        const int nb_n = nblocks_of((int)rank);
        const int ja = lane / bpg, ia = lane - ja * bpg;
        const int gb = first_block + (2 * ja + (int)rank) * bpg + ia;
        const bool a_lane = lane < p.GM * bpg && gb < p.total_blocks;
        const int tap = gb / p.cblks, cb = gb - tap * p.cblks;
        const int kh = tap / p.k, kw = tap - kh * p.k;
        const int bg = lane - p.GM * bpg;
        const bool g_lane = bg >= 0 && bg < nb_n;
        const int g_c = col0 + (int)rank * p.BN + bg * p.blockN;
        const uint32_t full0 = mapa_shared(smem_u32(&sh->full[0]), 0);
        int s = 0; uint32_t round = 0;
        for (int it = 0; it < my_tiles; it++) {
            bool ok = true;
            if (lane == 0) {
                if (round > 0 && !mbar_wait(&sh->empty[s], (round - 1) & 1)) { atomicExch(&sh->failed, 1u); ok = false; }
                if (ok && rank == 0) mbar_expect_tx(&sh->full[s], tx);       // the leader's barrier collects the bytes of both CTAs
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            const int t = split + it * p.splits;
            const int n0 = p.BIMG > 1 ? t * p.BIMG : t / tiles_per_img;
            const int h0 = p.BIMG > 1 ? 0 : (t - n0 * tiles_per_img) * p.BH;
            uint8_t *sa = tiles + s * stage_bytes;
            if (a_lane) tma2_load_4d(sa + ja * 32768 + ia * blk_bytes_a, &map_a, full0 + 8u * s, cb * p.blockC, kw - pad, h0 * p.stride + kh - pad, n0);
            else if (g_lane) tma2_load_4d(sa + a_region + bg * blk_bytes_b, &map_g, full0 + 8u * s, g_c, 0, h0, n0);
            if (++s == p.stages) { s = 0; round++; }
        }
    } else if (warp == 1) {
        if (rank == 0 && elect_one()) {
            const uint32_t idesc = instr_desc_m256(2 * p.BN) | (3u << 15);     // both operands M / N-major
            const int rba = p.blockC * 2, rbb = p.blockN * 2;
            const uint64_t da0 = smem_desc_mn(smem_u32(tiles), rba, blk_bytes_a), db0 = smem_desc_mn(smem_u32(tiles) + a_region, rbb, blk_bytes_b);
            const uint32_t stage16 = (uint32_t)stage_bytes >> 4;
            int s = 0; uint32_t round = 0, soff = 0;
            for (int it = 0; it < my_tiles; it++) {
                if (!mbar_wait_cluster(&sh->full[s], round & 1)) { atomicExch(&sh->failed, 1u); break; }
                tc_fence_after();
                const uint32_t accum = it > 0 ? 1u : 0u;
                for (int g = 0; g < p.GM; g++) {
                    uint64_t da = da0 + soff + (uint32_t)(g * 2048), db = db0 + soff;
                    const uint32_t acc = tmem_d + (uint32_t)(g * 2 * p.BN);
                    mma2_bf16(acc, da, db, idesc, accum);
                    for (int ks = 1; ks < 8; ks++) {         // 16 pixels per MMA
                        da += (uint32_t)rba; db += (uint32_t)rbb;
                        mma2_bf16(acc, da, db, idesc, 1u);
                    }
                }
                mma2_commit_both(&sh->empty[s]);
                soff += stage16;
                if (++s == p.stages) { s = 0; soff = 0; round++; }
            }
            mma2_commit_both(&sh->acc_full[0]);
        }
    } else {
        const int quarter = warp & 3;
        bool ok = true;
        if (quarter == 0 && lane == 0) ok = mbar_wait_cluster(&sh->acc_full[0], 0);
        ok = named_barrier_and(2, 128, ok);
        tc_fence_after();
        if (ok && sh->failed == 0) {
            const int m = quarter * 32 + lane;
            float *dst = p.partial + (size_t)split * p.slice;
            for (int g = 0; g < p.GM; g++) {
                const int gb = first_block + (2 * g + (int)rank) * bpg + m / p.blockC;
                const int tap = gb / p.cblks, ci = (gb - tap * p.cblks) * p.blockC + m % p.blockC;
                const bool row_ok = gb < p.total_blocks && ci < p.cin;
                for (int c = 0; c < 2 * p.BN; c += 16) {
                    float v[16];
                    tmem_ld16(tmem_d + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(g * 2 * p.BN + c), v);   // whole warp takes part
                    if (!row_ok) continue;
                    if (my_tiles == 0) {
#pragma unroll
                        for (int j = 0; j < 16; j++) v[j] = 0.f;
                    }
                    const int cb0 = col0 + c;
                    if (p.splits > 1) {
                        float *row = dst + ((size_t)tap * p.cin + ci) * p.cout + cb0;
#pragma unroll
                        for (int j = 0; j < 16; j += 4)
                            if (cb0 + j < p.cout) *reinterpret_cast<float4 *>(row + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j++) {
                            const int co = cb0 + j;
                            if (co < p.cout) dst[((size_t)co * p.taps + tap) * p.cin + ci] = v[j];
                        }
                    }
                }
            }
        } else if (lane == 0) {
            atomicExch(&sh->failed, 1u);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && sh->failed) atomicExch(p.status, (int)REVNET_E_TIMEOUT);
    stamp_end(batch.stamp);
    cluster_sync_all();      // neither CTA leaves, or frees tensor memory, while the other may still read its operands
    if (warp == 1) {
        tc_fence_after();
        tmem2_dealloc(tmem_d, tmem_cols);
    }
}

// dW[co][tap][ci] = sum over splits of part[z][tap][ci][co], in a fixed order: 8 interleaved groups of
// splits per element, combined through shared memory (256 threads = 32 elements x 8 groups); several
// (partials, destination) pairs in one launch, blockIdx.y picks the pair
struct SumBatch { const float *part[kWgMaxJobs]; float *out[kWgMaxJobs]; size_t n[kWgMaxJobs]; int splits[kWgMaxJobs], cout[kWgMaxJobs], rows[kWgMaxJobs]; };
__global__ void splitk_sum_batch_kernel(const SumBatch b) {
    pdl_enter();
    __shared__ float sm[8][33];
    const int j = blockIdx.y;
    const float *__restrict__ part = b.part[j];
    const size_t n = b.n[j];
    const int splits = b.splits[j];
    const int e = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const size_t i = (size_t)blockIdx.x * 32 + e;
    float s = 0.f;
    if (i < n)
        for (int z = grp; z < splits; z += 8) s += part[(size_t)z * n + i];
    sm[grp][e] = s;
    __syncthreads();
    if (grp == 0 && i < n) {
        for (int g = 1; g < 8; g++) s += sm[g][e];
        const size_t row = i / (size_t)b.cout[j];              // (tap, ci)
        const int co = (int)(i - row * (size_t)b.cout[j]);
        b.out[j][(size_t)co * b.rows[j] + row] = s;
    }
}

// The same sum for large gradients: 32 x 32 tiles ((tap, ci) rows x output channels) through shared memory, so that
// the reads of the partials (output channels contiguous) and the writes of dW ((tap, ci) contiguous) are both whole
// lines; a thread adds the splits of its four elements in ascending order, four loads in flight per element.
__global__ void __launch_bounds__(256) splitk_sum_tiled_kernel(const SumBatch b) {
    pdl_enter();
    __shared__ float tile[32][33];
    const int j = blockIdx.y;
    const float *__restrict__ part = b.part[j];
    const size_t n = b.n[j];
    const int splits = b.splits[j], C = b.cout[j], R = b.rows[j];
    const int tc_n = (C + 31) >> 5, tr_n = (R + 31) >> 5;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int t = blockIdx.x; t < tc_n * tr_n; t += gridDim.x) {
        const int c0 = (t % tc_n) << 5, r0 = (t / tc_n) << 5;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int row = r0 + ty + 8 * k, co = c0 + tx;
            float s = 0.f;
            if (row < R && co < C) {
                const float *src = part + (size_t)row * C + co;
                int z = 0;
                for (; z + 4 <= splits; z += 4) {
                    const float v0 = src[(size_t)z * n], v1 = src[(size_t)(z + 1) * n], v2 = src[(size_t)(z + 2) * n], v3 = src[(size_t)(z + 3) * n];
                    s += v0; s += v1; s += v2; s += v3;
                }
                for (; z < splits; z++) s += src[(size_t)z * n];
            }
            tile[ty + 8 * k][tx] = s;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int co = c0 + ty + 8 * k, row = r0 + tx;
            if (row < R && co < C) b.out[j][(size_t)co * R + row] = tile[tx][ty + 8 * k];
        }
        __syncthreads();
    }
}

int pick_block(int c_pad) { return c_pad % 64 == 0 ? 64 : (c_pad % 32 == 0 ? 32 : 16); }

// g: geometry of the tensor; (tile_w, BH, BIMG): the 128-pixel tile in units of the traversal stride
bool encode_act_map(Exec &ex, CUtensorMap *map, const void *base, Geom g, int C, int box_c, int tile_w, int BH, int BIMG, int stride) {
    const CUtensorMapSwizzle sw = box_c == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (box_c == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)g.W, (cuuint64_t)g.H, (cuuint64_t)g.N};
    cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)g.W * C * 2, (cuuint64_t)g.H * g.W * C * 2};
    cuuint32_t box[4] = {(cuuint32_t)box_c, (cuuint32_t)(tile_w * stride), (cuuint32_t)(BH * stride), (cuuint32_t)BIMG};
    cuuint32_t es[4] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1};
    return encoder(ex.ctx)(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// out = conv(ReLU(BN(t))) for wide 1x1 layers; a_out (optional): the activated tensor.  mean and rstd of bn must be there.
bool conv_fprop_bn(Exec &ex, Pair t, BnRef bn, Geom gi, const Layer &L, Pair out, Moments *stats, bf16 *a_out) {
    return run_bn_conv(ex, t, bn, gi, L, out, stats, a_out);
}
bool conv_fprop_tc(Exec &ex, const void *a, Geom gi, const Layer &L, Pair out, Pair partner, int sign, Moments *stats) {
    EpiReq req; req.stats = stats;
    return run_conv_tc(ex, "conv_fprop_tc", a, gi, L.cin, L.cout, L.k, L.stride, L.W, L.Wp_fprop, false, out, partner, sign, req);
}

// da[q,ci] = sum_{tap,co} g[q (-) tap, co] W[co,tap,ci]: a stride-1 convolution of g with the mirrored, transposed weights
bool conv_dgrad_tc(Exec &ex, const void *g, Geom gi, const Layer &L, float *da, const BnBwdReq *bb) {
    if (L.stride != 1) return false;
    EpiReq req; req.bnbwd = bb;
    return run_conv_tc(ex, "conv_dgrad_tc", g, gi, L.cout, L.cin, L.k, L.stride, L.W, L.Wp_dgrad, true, single(da, L.cin), Pair{}, 0, req);
}


// Data gradient of a 3x3 stride-2 layer: one launch whose tile list runs over the four parity classes of the input
// pixels (see run_conv_tc).  g: bf16 [N, H/2, W/2, cout]; da: fp32 [N, H, W, cin]; bb: BN-backward sums to fuse.
// Large layers (those that get 128 x 256 tiles when no partner tile has to fit beside the operand ring) leave the
// sums to their own pass instead: *fused tells which.
bool conv_dgrad_tc_s2(Exec &ex, const void *g, Geom gi, const Layer &L, float *da, const BnBwdReq *bb, bool *fused) {
    if (L.stride != 2 || L.k != 3 || gi.H % 2 || gi.W % 2) return false;
    const Geom go{gi.N, gi.H / 2, gi.W / 2};
    const bool wide = 4ll * L.cout >= 1024 && L.cin >= 256 && L.cin % 32 == 0;
    EpiReq req; req.bnbwd = wide ? nullptr : bb;
    *fused = req.bnbwd != nullptr;
    return run_conv_tc(ex, "conv_dgrad_tc", g, go, L.cout, L.cin, 3, 1, L.W, L.Wp_dgrad, true, single(da, L.cin), Pair{}, 0, req, true);
}

constexpr int kWgSmemMax = 224 * 1024;

// Shape decisions of one layer's weight gradient; cta_budget: the CTAs the job may take
struct WgPlan { WgParams p; Geom go; int n_tiles, stage_bytes, tail_bytes; };
// pair: plan for wgrad_tc2_kernel (cta_budget then counts CTAs too; the job takes an even number)
static bool wgrad_plan(Geom gi, const Layer &L, int cta_budget, WgPlan &w, bool allow_sep = true, bool pair = false) {
    if ((L.stride != 1 && L.stride != 2) || (L.k != 1 && L.k != 3) || L.cin % 8 || L.cout % 8) return false;
    if (L.stride == 2 && (gi.H % 2 || gi.W % 2)) return false;
    WgParams &p = w.p;
    w.go = Geom{gi.N, conv_out(gi.H, L.k, L.stride), conv_out(gi.W, L.k, L.stride)};   // tiles walk the output pixels
    TileGeom tg;
    if (!tile_geom(w.go, tg) || tg.W * L.stride > 256 || tg.BH * L.stride > 256) return false;
    p.BH = tg.BH; p.BIMG = tg.BIMG; p.tiles_per_img = tg.tiles_per_img; p.box_px = tg.BIMG * tg.BH * tg.W;
    const int taps = L.k * L.k, cin_pad = round_up(L.cin, 16), cout_pad = round_up(L.cout, 16);
    p.taps = taps; p.k = L.k; p.cin = L.cin; p.cout = L.cout;
    p.blockC = pick_block(cin_pad); p.cblks = cin_pad / p.blockC;
    p.blockN = pick_block(cout_pad);
    p.cout_pad = cout_pad;
    const int bpg = 128 / p.blockC;
    // taps split between the operands when the three shifted activation blocks fit one M group, the three
    // shifted gradient blocks one N tile, and the boxes of a pixel tile the lanes of the producer warp
    p.sep = (allow_sep && !pair && L.k == 3 && L.stride == 1 && 3 * cin_pad <= 128 && 3 * cout_pad <= 256 && 2 * bpg + 3 * (cout_pad / p.blockN) <= 32) ? 1 : 0;
    p.pair = pair ? 1 : 0;
    if (pair) {
        // a pair's N tile is 2 * BN wide (BN per CTA, a whole number of gradient blocks), its M chunk 2 * GM groups
        // (N tiles of less than 256 columns measured slower on a pair than 128-column tiles on one CTA: 89 against 72 us
        // for the 3x3 layer of 128 channels at 56 x 56, batch 64)
        if (cout_pad < 256 || cout_pad % 32) return false;
        p.total_blocks = taps * p.cblks;
        p.BN = 128;
        if (p.BN % p.blockN) { p.blockN = pick_block(p.BN); if (p.BN % p.blockN) return false; }
        const int groups_all = (p.total_blocks + bpg - 1) / bpg;
        if (groups_all < 2) return false;
        p.GM = groups_all >= 4 ? 2 : 1;
        p.m_chunks = (groups_all + 2 * p.GM - 1) / (2 * p.GM);
        w.n_tiles = (cout_pad + 2 * p.BN - 1) / (2 * p.BN);
        p.H = w.go.H; p.W = w.go.W; p.stride = L.stride;
        p.n_tiles_px = tg.n_px_tiles;
        p.a_region = p.GM * 32768;
        w.stage_bytes = p.a_region + ((256 * p.BN + 1023) & ~1023);
        w.tail_bytes = 0;
        p.stages = (kWgSmemMax - 2048) / w.stage_bytes; if (p.stages > kWgStages) p.stages = kWgStages;
        if (p.stages < 2) return false;
        const int units = p.m_chunks * w.n_tiles, budget = cta_budget / 2 < 1 ? 1 : cta_budget / 2;     // in pairs
        auto clampi = [&](int v) { return v < 1 ? 1 : (v > p.n_tiles_px ? p.n_tiles_px : v); };
        const int s_hi = clampi((budget + units - 1) / units), s_lo = clampi(budget / units);
        auto serial_tiles = [&](int sp) { return ((units * sp + budget - 1) / budget) * ((p.n_tiles_px + sp - 1) / sp); };
        p.splits = serial_tiles(s_lo) < serial_tiles(s_hi) ? s_lo : s_hi;
        p.slice = (size_t)L.cout * taps * L.cin;
        return true;
    }
    if (p.sep) {
        p.total_blocks = L.k * p.cblks;
        p.BN = L.k * cout_pad;
    } else {
        p.total_blocks = taps * p.cblks;
        p.BN = cout_pad <= 128 ? cout_pad : 128;
        if (p.BN % p.blockN) p.BN = p.blockN;
    }
    const int groups_all = (p.total_blocks + bpg - 1) / bpg;
    p.GM = groups_all >= 2 ? 2 : 1;
    p.m_chunks = (groups_all + p.GM - 1) / p.GM;
    w.n_tiles = p.sep ? 1 : (cout_pad + p.BN - 1) / p.BN;
    p.H = w.go.H; p.W = w.go.W; p.stride = L.stride;
    p.n_tiles_px = tg.n_px_tiles;
    const int blocks_max = p.total_blocks < p.GM * bpg ? p.total_blocks : p.GM * bpg;
    p.a_region = (blocks_max * 256 * p.blockC + 1023) & ~1023;
    w.stage_bytes = p.a_region + ((256 * p.BN + 1023) & ~1023);
    w.tail_bytes = p.GM * 32768 - p.a_region;        // what the MMAs of a partly filled group read past the last stage
    p.stages = (kWgSmemMax - 2048 - w.tail_bytes) / w.stage_bytes; if (p.stages > kWgStages) p.stages = kWgStages;
    if (p.stages < 2) return p.sep ? wgrad_plan(gi, L, cta_budget, w, false) : false;
    // split the pixel reduction so that the job's CTAs cover its share of the machine once: rounding the split
    // count up may spill a few CTAs into a second wave (these CTAs fill an SM each), rounding down leaves SMs idle;
    // take whichever walks fewer pixel tiles one after the other
    const int pairs = p.m_chunks * w.n_tiles;
    auto clampi = [&](int v) { return v < 1 ? 1 : (v > p.n_tiles_px ? p.n_tiles_px : v); };
    const int s_hi = clampi((cta_budget + pairs - 1) / pairs), s_lo = clampi(cta_budget / pairs);
    auto serial_tiles = [&](int sp) { return ((pairs * sp + cta_budget - 1) / cta_budget) * ((p.n_tiles_px + sp - 1) / sp); };
    int splits = serial_tiles(s_lo) < serial_tiles(s_hi) ? s_lo : s_hi;
    p.splits = splits;
    p.slice = (size_t)L.cout * taps * L.cin;
    return true;
}

// Weight gradients of n layers (n <= 4) in one launch, and one more launch that sums their split partials.
// scratch: room for the split partials if the caller provides it (else it comes from the arena);
// need: if non-null the call only reports whether it takes the shapes and how many floats of scratch it wants
bool conv_wgrad_tc_batch(Exec &ex, int n, const void *const *gq, const void *const *a, const Geom *gi, const Layer *const *L,
                         float *scratch, size_t *need) {
    if (n < 1 || n > kWgMaxJobs) return false;
    WgPlan w[kWgMaxJobs];
    const int budget = ex.ctx->sm_count / n;
    size_t total = 0;
    // CTA pairs (wgrad_tc2_kernel) when every layer of the launch takes them: a launch is made of clusters or it is not
    static const bool pair_enabled = [] { const char *v = getenv("REVNET_WGRAD_PAIR"); return !(v && v[0] == '0'); }();
    bool pair = pair_enabled && ex.ctx->sm_count % 2 == 0;
    for (int j = 0; j < n && pair; j++) pair = wgrad_plan(gi[j], *L[j], budget & ~1, w[j], false, true);
    for (int j = 0; j < n; j++) {
        if (!pair && !wgrad_plan(gi[j], *L[j], budget, w[j])) return false;
        if (w[j].p.splits > 1) total += (size_t)w[j].p.splits * w[j].p.slice;
    }
    if (need) { *need = total; return true; }
    if (!ex.dry && !encoder(ex.ctx)) return false;
    size_t m = ex.ws.mark();
    float *part = total ? (scratch ? scratch : ex.ws.get<float>(total)) : nullptr;
    for (int j = 0; j < n; j++) ex.flops += 2ull * w[j].go.P() * L[j]->cout * L[j]->cin * w[j].p.taps;
    if (!ex.dry) {
        WgBatch batch;
        SumBatch sums;
        batch.n = n;
        batch.stamp = ex.stamp_slot();
        int cta = 0, smem = 0, n_sums = 0;
        size_t off = 0, max_slice = 0;
        double bytes = 0, flops = 0, sum_bytes = 0;
        for (int j = 0; j < n; j++) {
            WgParams &p = w[j].p;
            if (!encode_act_map(ex, &batch.job[j].map_a, a[j], gi[j], L[j]->cin, p.blockC, w[j].go.W, p.BH, p.BIMG, L[j]->stride) ||
                !encode_act_map(ex, &batch.job[j].map_g, gq[j], w[j].go, L[j]->cout, p.blockN, w[j].go.W, p.BH, p.BIMG, 1)) {
                ex.failed = true; ex.ctx->err = "conv_wgrad_tc: tensor map rejected"; ex.ws.release(m); return true;
            }
            p.status = ex.ctx->dev_status;
            p.cta0 = cta;
            cta += p.splits * p.m_chunks * w[j].n_tiles * (pair ? 2 : 1);
            if (p.splits > 1) {
                p.partial = part + off;
                sums.part[n_sums] = p.partial; sums.out[n_sums] = L[j]->dW; sums.n[n_sums] = p.slice; sums.splits[n_sums] = p.splits;
                sums.cout[n_sums] = L[j]->cout; sums.rows[n_sums] = p.taps * L[j]->cin;
                n_sums++;
                off += (size_t)p.splits * p.slice;
                if (p.slice > max_slice) max_slice = p.slice;
                sum_bytes += (double)p.slice * 4 * (p.splits + 1);
            } else {
                p.partial = L[j]->dW;
            }
            batch.job[j].p = p;
            const int sm = 1024 + p.stages * w[j].stage_bytes + w[j].tail_bytes + (int)sizeof(TcShared) + 64;
            if (sm > smem) smem = sm;
            bytes += (double)gi[j].P() * L[j]->cin * 2 + (double)w[j].go.P() * L[j]->cout * 2 + (double)p.slice * 4 * p.splits;
            flops += 2.0 * w[j].go.P() * L[j]->cout * L[j]->cin * p.taps;
        }
        static OncePerDevice once;
        if (once.first(ex.ctx->device)) {
            cudaFuncSetAttribute(wgrad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmemMax);
            cudaFuncSetAttribute(wgrad_tc2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmemMax);
        }
        if (pair) launch_cluster(ex, wgrad_tc2_kernel, (unsigned)cta, kThreads, smem, 2, batch);
        else launch(ex, wgrad_tc_kernel, (unsigned)cta, kThreads, smem, batch);
        ex.check(pair ? "conv_wgrad_tc2" : "conv_wgrad_tc", bytes, flops);
        if (n_sums) {
            if (max_slice >= 524288) {
                size_t tiles = (max_slice + 1023) / 1024; if (tiles > (size_t)ex.ctx->sm_count * 8) tiles = (size_t)ex.ctx->sm_count * 8;
                dim3 grid((unsigned)tiles, (unsigned)n_sums);
                launch_stream(ex, sum_bytes, 20, splitk_sum_tiled_kernel, grid, 256, 0, sums);
            } else {
                dim3 grid((unsigned)((max_slice + 31) / 32), (unsigned)n_sums);
                launch_stream(ex, sum_bytes, 6, splitk_sum_batch_kernel, grid, 256, 0, sums);
            }
            ex.check("splitk_sum", sum_bytes);
        }
    }
    ex.ws.release(m);
    return true;
}

bool conv_wgrad_tc(Exec &ex, const void *gq, const void *a, Geom gi, const Layer &L, float *dW, float *scratch, size_t *need) {
    Layer one = L;
    one.dW = dW;
    const Layer *lp = &one;
    return conv_wgrad_tc_batch(ex, 1, &gq, &a, &gi, &lp, scratch, need);
}

void *tc_encoder(revnet_ctx *ctx) { return (void *)encoder(ctx); }

// pack of one layer built on the spot (calls that have no step-level pack)
void tc_pack_now(Exec &ex, const float *W, bf16 *out, int cin, int cout, int k, bool transposed) {
    PackJobs list;
    list.job[0] = tc_pack_job(W, transposed ? nullptr : out, transposed ? out : nullptr, cin, cout, k);
    tc_pack_list(ex, list, 1);
}

// ---- packs made once per step (the train step calls these before the forward pass)
static void pack_dims(int rows, int cols, int &rows_pad, int &cols_pad) {
    const int rp = round_up(rows, 16), BN = rp <= 128 ? rp : 128;
    rows_pad = (rp + BN - 1) / BN * BN;
    cols_pad = round_up(cols, 16);
}
size_t tc_pack_elems(int cin, int cout, int k, bool transposed) {
    int rp, cp;
    if (!transposed) pack_dims(cout, cin, rp, cp); else pack_dims(cin, cout, rp, cp);
    return (size_t)rp * k * k * cp;
}
PackJob tc_pack_job(const float *W, bf16 *f, bf16 *d, int cin, int cout, int k) {
    PackJob j{W, f, d, cout, cin, k, 0, 0, 0, 0, 0};
    if (f) pack_dims(cout, cin, j.co_f, j.ci_f);
    if (d) pack_dims(cin, cout, j.ci_d, j.co_d);
    return j;
}
int tc_pack_tiles(const PackJob &j) { return pack_ct(j) * pack_rt(j) * j.k * j.k; }
static double pack_job_bytes(const PackJob &j) {
    return (double)j.Co * j.Ci * j.k * j.k * 4 + 2.0 * j.k * j.k * ((double)j.co_f * j.ci_f + (double)j.ci_d * j.co_d);
}
// one tile per CTA while that leaves at most 32 CTAs per SM, else four
void tc_pack_batch(Exec &ex, const PackJob *jobs_dev, int n_jobs, double bytes, int tiles) {
    if (ex.dry || n_jobs == 0) return;
    const int run = tiles > ex.ctx->sm_count * 32 ? 4 : 1;
    launch(ex, pack_weights_batch_kernel, (tiles + run - 1) / run, 256, 0, jobs_dev, n_jobs, tiles, run);
    ex.check("pack_weights_batch", bytes);
}
// blocks per layer sized for the largest one, at most eight per SM
void tc_pack_list(Exec &ex, const PackJobs &jobs, int n_jobs) {
    if (ex.dry || n_jobs == 0) return;
    int tiles = 1; double bytes = 0;
    for (int i = 0; i < n_jobs; i++) { const int t = tc_pack_tiles(jobs.job[i]); if (t > tiles) tiles = t; bytes += pack_job_bytes(jobs.job[i]); }
    const int cap = ex.ctx->sm_count * 8;
    launch(ex, pack_weights_kernel, dim3((unsigned)(tiles < cap ? tiles : cap), (unsigned)n_jobs), 256, 0, jobs);
    ex.check("pack_weights", bytes);
}
