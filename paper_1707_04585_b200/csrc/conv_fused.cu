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
// Roles (one CTA per SM):
//   EW warps    epilogue (8, or 16 for more than 16 output columns), one accumulator row and 16 columns per thread, straight
//               from tensor memory to global memory with 32-byte accesses: coupling on the float or fixed-point state, or plain
//               store; the per-channel sums (batch statistics of the stored result, or the two sums of the BN+ReLU backward)
//               stay in registers until the last tile.  Four warps make a group (128 rows x 16 columns); the groups split a
//               tile's columns between them, and what is left over takes alternate tiles.  Before the first tile eight of
//               them add the statistics records of the kernel before (BnRef::part).
//   1 warp      weights (TMA, resident), tensor memory, MMA issue; two accumulators
//   7 warps     build: 32-byte loads (8 channels of a pixel), four in flight per thread, scale*x + shift, ReLU, bf16 rounding,
//               one 16-byte store to shared memory (and one to the activated tensor the weight gradient will read)
// The same kernel computes data gradients: its input is then the bf16 upstream gradient, taken as it is, and the weights
// are the mirrored, transposed pack.
// Measured against the kernel with two CTAs of 256 threads that took turns at every step and built three shifted copies:
// 16 channels at 32x32, batch 128: 19 -> 14 us per launch (nine MMAs of a tile issue in 500 clocks instead of 2200, a tile
// every 1200 clocks and SM); basic block forward + backward there 307 -> 263 us, 16/32/56-channel step 2.13 -> 1.94 ms.
// Every mbarrier wait is bounded; on expiry the kernel records a status word and leaves.
#include "common.cuh"
#include "tc_ptx.cuh"
#include "conv_epilogue.cuh"
#include <cuda.h>
#include <string.h>

using namespace tc;

namespace {

constexpr int kFullBars = 16;             // tiles the build may run ahead of the MMAs
constexpr int NC = 16;                    // columns per epilogue thread
constexpr int NBT = 224;                  // build threads: with the MMA warp a multiple of four warps, which keeps the most registers
__host__ __device__ constexpr int fused_threads(int EW) { return EW * 32 + 32 + NBT; }

// What all layers of a launch share
struct FusedGeom {
    int k;                 // 1 or 3
    int cin, nch;          // valid input channels, their 8-channel chunks
    int KC;                // channels of a weight row in shared memory: 16, 32 or 64 (rows of 32 / 64 / 128 bytes, swizzled by TMA)
    int ksteps;            // MMA steps of 16 channels per tap
    int wpitch;            // channels per tap in the weight pack (cin rounded up to 16)
    int BN, groups;        // output columns per CTA; groups = BN / NC: warp groups that share a tile (1, 2 or 4)
    int wtile_bytes;       // one tap of the weights: BN rows of KC bf16, rounded up to 1024
    int N, H, W, pitch;    // pitch: positions per image row (W + 1; 1x1: unused)
    int step_r, step_c;    // 3x3: the build's row stride in positions as whole image rows and columns
    int halo;              // operand rows before a tile's first position (3x3: W + 2, else 0)
    int total;             // positions in all
    int chunk;             // positions per CTA
    int S, nseg;           // tiles per operand segment, segment buffers (1 or 2)
    int plane16, seg_bytes, op_bytes;     // plane stride in 16-byte units; bytes of a segment buffer, of the whole operand region
    FastDiv dpitch, drows; // by positions per image row, by rows per image (H + 1)
};
// The epilogue of one layer (field names as epilogue_publish expects them)
struct FusedEpi {
    int mode, sign, n_cols;
    float *out;            // [P, n_cols]
    float q;               // format of out (and of the coupling partner), or of the BN input of a data gradient: 0 float, else fixed-point step
    float *part;           // per-CTA records of the column sums, or null
    unsigned int *counter; // null: the records stay pending, their consumer adds them
    double inv_count;
    float eps;
    float *mean, *rstd;
    BnRef bn;              // EPI_BNBWD
    float *dgamma, *dbeta, *coef;
};
struct FusedLayer {
    int in_mode;           // 0: float tensor through BN + ReLU; 2: fixed-point tensor likewise; 1: bf16 tensor as it is
    int wide_in, wide_out; // 32-byte aligned rows: 32-byte accesses
    int w_early;           // the weights were packed before the predecessor kernel: they may be loaded while it runs
    const void *in;
    float in_q;            // in_mode 2: fixed-point step of the input
    BnRef bn;              // in_mode 0, 2
    bf16 *a_out;           // in_mode 0, 2, optional: the activated tensor [P, cin] (operand of the weight gradient)
    const float *aux;      // coupling partner, or the BN input of a data gradient
    FusedEpi epi;
};
struct FusedArgs {
    CUtensorMap map_w;
    FusedGeom g;
    FusedLayer ly;
    int *status;
    unsigned long long *stamp;    // timeline slot of this launch (nullptr: off)
};

struct __align__(16) FusedShared {
    uint64_t full[kFullBars], seg_empty[2], acc_full[2], acc_empty[2], w_full;
    uint32_t tmem_base, failed;
    __align__(16) float sc[64];      // BN scale and shift per input channel
    __align__(16) float sf[64];
    __align__(16) float4 coef[64];   // BN+ReLU backward: (scale, shift, mean, rstd) of each output column
    __align__(16) float sums[16][2 * NC];     // per epilogue warp: NC sums, then NC second sums
    __align__(16) double red[256 * 4], tot[32 * 4];    // statistics records
};

// two floats -> ReLU -> bf16x2 (round to nearest even), one instruction
__device__ __forceinline__ uint32_t relu_pack2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// a bounded wait of a whole warp: lane 0 polls
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, int lane) {
    bool ok = true;
    if (lane == 0) ok = mbar_wait(bar, parity);
    return __shfl_sync(0xffffffffu, ok, 0);
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

// The build of a CTA's operand rows.  A thread keeps its channel chunk ck and takes rows r0, r0 + RS, ... of each segment;
// D loads are in flight while older rows are normalised and written.  IN: see FusedLayer::in_mode.
template <int IN, int EW>
__device__ __forceinline__ bool build_rows(const FusedGeom &g, const FusedLayer &p, FusedShared *sh, uint8_t *abuf, int pos0, int pos1, int bt, int lane) {
    constexpr int NW = IN == 1 ? 4 : 8;                  // 32-bit words of an item
    constexpr int D = 4;
    const int nch = g.nch, RS = NBT / nch, ck = bt % nch, r0 = bt / nch, low0 = (bt & ~31) / nch;
    const bool active = r0 < RS;
    const int n_tiles = (pos1 - pos0 + 127) >> 7;
    const bool wide = p.wide_in != 0;
    float sc[8], sf[8];
    bool first = true;
    for (int t0 = 0, seg = 0; t0 < n_tiles; t0 += g.S, seg++) {
        const int T = n_tiles - t0 < g.S ? n_tiles - t0 : g.S;
        const int sb = pos0 + t0 * 128, own = pos1 - sb < T * 128 ? pos1 - sb : T * 128, rows = own + 2 * g.halo;
        uint8_t *dst = abuf + (g.nseg == 2 ? (seg & 1) : 0) * g.seg_bytes + ck * g.plane16 * 16;
        uint32_t raw[D][NW];
        int pix[D];
        // the place of the next row to load, stepped by RS positions without divisions
        int lc = 0, lr = 0, ln = 0;
        if (g.k == 3) place_at(g, sb - g.halo + r0, ln, lr, lc);
        auto load = [&](int l, uint32_t (&v)[NW], int &px) {
            px = -1;
            if (g.k == 1) { if (active && l < rows && sb + l < g.total) px = sb + l; }
            else {
                if (active && l < rows && lc < g.W && (unsigned)lr < (unsigned)g.H && (unsigned)ln < (unsigned)g.N) px = (ln * g.H + lr) * g.W + lc;
                lc += g.step_c; lr += g.step_r;
                if (lc >= g.pitch) { lc -= g.pitch; lr++; }
                while (lr > g.H) { lr -= g.H + 1; ln++; }
            }
            if (px >= 0) {
                const size_t off = ((size_t)px * nch + ck) * (IN == 1 ? 16 : 32);
                if constexpr (IN == 1) {
                    const uint4 u = *reinterpret_cast<const uint4 *>(reinterpret_cast<const uint8_t *>(p.in) + off);
                    v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
                } else ld8(reinterpret_cast<const uint8_t *>(p.in) + off, v, wide);
            }
        };
        int ll = r0, l = r0, low = low0, j = 0;
#pragma unroll
        for (int u = 0; u < D; u++) { load(ll, raw[u], pix[u]); ll += RS; }
        if (first) {
            first = false;
            if (IN != 1) {
                named_barrier(3, EW * 32 + NBT);         // scale and shift are there
#pragma unroll
                for (int i = 0; i < 8; i++) { sc[i] = sh->sc[ck * 8 + i] * (IN == 2 ? p.in_q : 1.f); sf[i] = sh->sf[ck * 8 + i]; }
            }
        }
        if (seg >= g.nseg && !warp_wait(&sh->seg_empty[g.nseg == 2 ? (seg & 1) : 0], (uint32_t)((g.nseg == 2 ? seg >> 1 : seg) - 1) & 1u, lane)) return false;
        auto signal = [&](int tile) {
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->full[(t0 + tile) & (kFullBars - 1)]);
        };
        while (low < rows) {
#pragma unroll
            for (int u = 0; u < D; u++) {
                if (low >= rows) break;
                while (j < T && low >= (j + 1) * 128 + 2 * g.halo) signal(j++);
                if (active && l < rows) {
                    uint4 v = make_uint4(0u, 0u, 0u, 0u);
                    if (pix[u] >= 0) {
                        if constexpr (IN == 1) v = make_uint4(raw[u][0], raw[u][1], raw[u][2], raw[u][3]);
                        else {
                            float x[8];
#pragma unroll
                            for (int i = 0; i < 8; i++) x[i] = fmaf(sc[i], IN == 2 ? __int2float_rn((int)raw[u][i]) : __uint_as_float(raw[u][i]), sf[i]);
                            v = make_uint4(relu_pack2(x[0], x[1]), relu_pack2(x[2], x[3]), relu_pack2(x[4], x[5]), relu_pack2(x[6], x[7]));
                            if (p.a_out && l >= g.halo && l < g.halo + own)
                                *reinterpret_cast<uint4 *>(p.a_out + ((size_t)pix[u] * nch + ck) * 8) = v;
                        }
                    }
                    *reinterpret_cast<uint4 *>(dst + l * 16) = v;
                }
                l += RS; low += RS;
                load(ll, raw[u], pix[u]);
                ll += RS;
            }
        }
        while (j < T) signal(j++);
    }
    return true;
}

// Epilogue of one warp's rows.  EK: 0 plain, 1 float coupling, 2 fixed-point coupling, 3 / 4 BN+ReLU backward with a float /
// fixed-point BN input.
template <int EW, int EK>
__device__ __forceinline__ bool epilogue_loop(const FusedGeom &g, const FusedLayer &p, FusedShared *sh, int pos0, int pos1, int warp, int lane, uint32_t tmem_d,
                                              float (&s)[NC], float (&ss)[NC]) {
    const FusedEpi &e = p.epi;
    const int grp = warp >> 2, row = (warp & 3) * 32 + lane;
    const int sets = EW / 4 / g.groups, set = grp / g.groups;                     // tiles set, set + sets, ...
    const bool wide = p.wide_out != 0;
    const int lc = (grp % g.groups) * NC, col = (int)blockIdx.y * g.BN + lc;      // this thread's first column: in the CTA, in the tensor
    const float q = e.q, out_s = (EK <= 2 && q != 0.f) ? 1.f / q : 0.f, sgn = e.sign < 0 ? -1.f : 1.f;
    const int isgn = e.sign < 0 ? -1 : 1;
    const float4 *coef = sh->coef + lc;
    const int n_tiles = (pos1 - pos0 + 127) >> 7;
    const uint32_t tm = tmem_d + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)lc;
    for (int ti = set; ti < n_tiles; ti += sets) {
        const int q0 = pos0 + ti * 128 + row, px = q0 < pos1 ? pixel_at(g, q0) : -1;
        const size_t off = (size_t)(px < 0 ? 0 : px) * e.n_cols + col;
        // what the row needs besides the accumulator is on its way before the accumulator is complete
        uint32_t x[NC];
        if (EK > 0) {
#pragma unroll
            for (int c = 0; c < NC; c += 8) {
                uint32_t v[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
                if (px >= 0) {
                    if (col + c + 8 <= e.n_cols) ld8(p.aux + off + c, v, wide);
                    else if (col + c < e.n_cols) { const uint4 a = *reinterpret_cast<const uint4 *>(p.aux + off + c); v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; }
                }
#pragma unroll
                for (int i = 0; i < 8; i++) x[c + i] = v[i];
            }
        }
        const uint32_t keep = px >= 0 ? 0xffffffffu : 0u;      // rows that hold no pixel add nothing (a select, not a branch per column)
        const int buf = ti & 1;
        if (!warp_wait(&sh->acc_full[buf], (uint32_t)(ti >> 1) & 1u, lane)) return false;
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < NC; c += 8) {
            float v[8];
            uint32_t o[8];
            tmem_ld8(tm + (uint32_t)(buf * g.BN + c), v);
#pragma unroll
            for (int i = 0; i < 8; i++) {
                float st = 0.f;               // what is summed
                if (EK == 0) {
                    if (q != 0.f) { const int iv = __float2int_rn(v[i] * out_s); o[i] = (uint32_t)iv; st = __int2float_rn(iv) * q; }
                    else { o[i] = __float_as_uint(v[i]); st = v[i]; }
                } else if (EK == 1) {
                    st = fmaf(sgn, v[i], __uint_as_float(x[c + i]));
                    o[i] = __float_as_uint(st);
                } else if (EK == 2) {
                    const int iv = (int)x[c + i] + isgn * __float2int_rn(v[i] * out_s);
                    o[i] = (uint32_t)iv; st = __int2float_rn(iv) * q;
                } else o[i] = __float_as_uint(v[i]);
                if (EK <= 2) {
                    st = __uint_as_float(__float_as_uint(st) & keep);
                    s[c + i] += st;
                    ss[c + i] = fmaf(st, st, ss[c + i]);
                } else {
                    const float t = EK == 4 ? __int2float_rn((int)x[c + i]) * q : __uint_as_float(x[c + i]);
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
        if (lane == 0) mbar_arrive(&sh->acc_empty[buf]);
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

// Registers: 123 with eight epilogue warps; with sixteen the block of 768 threads leaves 80, and the epilogue, which holds 32 running sums,
// 16 partner words and 8 values, spills 304 bytes.
template <int EW>
__global__ void __launch_bounds__(fused_threads(EW), 1) conv_fused_kernel(const __grid_constant__ FusedArgs A) {
    extern __shared__ uint8_t smem_raw[];
    const FusedGeom &g = A.g;
    const FusedLayer &p = A.ly;
    const FusedEpi &e = p.epi;
    uint8_t *wres = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int taps = g.k * g.k;
    uint8_t *abuf = wres + taps * g.wtile_bytes;
    FusedShared *sh = (FusedShared *)(abuf + g.op_bytes);

    constexpr int kMmaWarp = EW, kBuildWarp0 = EW + 1;
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const bool direct = p.in_mode == 1;
    uint32_t tmem_cols = 32;
    while ((int)tmem_cols < 2 * g.BN) tmem_cols <<= 1;
    const int col0 = blockIdx.y * g.BN;
    const int pos0 = (int)blockIdx.x * g.chunk, pos1 = pos0 + g.chunk < g.total ? pos0 + g.chunk : g.total;
    auto load_weights = [&]() {
        mbar_expect_tx(&sh->w_full, (uint32_t)(taps * g.BN * g.KC * 2));
        for (int tap = 0; tap < taps; tap++) tma_load_2d(wres + tap * g.wtile_bytes, &A.map_w, &sh->w_full, tap * g.wpitch, col0);
    };

    if (warp == kMmaWarp) {
        if (elect_one()) {
            tma_prefetch_desc(&A.map_w);
            for (int b = 0; b < kFullBars; b++) mbar_init(&sh->full[b], NBT / 32);
            for (int b = 0; b < 2; b++) { mbar_init(&sh->seg_empty[b], 1); mbar_init(&sh->acc_full[b], 1); mbar_init(&sh->acc_empty[b], 4 * g.groups); }
            mbar_init(&sh->w_full, 1);
            sh->failed = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            if (p.w_early) load_weights();
        }
        tmem_alloc(&sh->tmem_base, tmem_cols);
    } else if (warp >= kBuildWarp0 && (g.nch & 1)) {
        // an odd number of 8-channel planes: the one that fills up the last MMA step holds zeros for good
        for (int b = 0; b < g.nseg; b++)
            for (int l = (int)threadIdx.x - kBuildWarp0 * 32; l < g.plane16; l += NBT)
                *reinterpret_cast<uint4 *>(abuf + b * g.seg_bytes + (g.nch * g.plane16 + l) * 16) = make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async();
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
                const int buf = ti & 1;
                if (!mbar_wait(&sh->full[ti & (kFullBars - 1)], (uint32_t)(ti / kFullBars) & 1u)) { ok = false; break; }
                if (ti > 1 && !mbar_wait(&sh->acc_empty[buf], (uint32_t)((ti >> 1) - 1) & 1u)) { ok = false; break; }
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
    } else if (warp < EW) {
        const int etid = (int)threadIdx.x;
        if (!direct && warp < 8) {
            if (p.bn.part) reduce_records<256>(p.bn.part, p.bn.parts, g.cin, 0, g.cin >> 1, sh->red, sh->tot, etid);
            if (etid < 64) {
                // the statistics of the input may still be per-CTA records of the kernel before: added above (every CTA the
                // same way, while its first rows are on the way), and the first CTA stores mean and rstd for later readers
                const int c = etid;
                float sc = 0.f, sf = 0.f;
                if (c < g.cin) {
                    float mean, rstd;
                    if (p.bn.part) {
                        moments_of(sh->tot[(2 * (c >> 2)) * 4 + (c & 3)], sh->tot[(2 * (c >> 2) + 1) * 4 + (c & 3)], p.bn.inv_count, p.bn.eps, mean, rstd);
                        if (blockIdx.x == 0 && blockIdx.y == 0) { const_cast<float *>(p.bn.mean)[c] = mean; const_cast<float *>(p.bn.rstd)[c] = rstd; }
                    } else { mean = p.bn.mean[c]; rstd = p.bn.rstd[c]; }
                    bn_sc_sh(p.bn.gamma[c], p.bn.beta[c], mean, rstd, sc, sf);
                }
                sh->sc[c] = sc; sh->sf[c] = sf;
            }
        }
        if (!direct) named_barrier(3, EW * 32 + NBT);
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
            ok = e.q == 0.f ? epilogue_loop<EW, 3>(g, p, sh, pos0, pos1, warp, lane, tmem_d, s, ss)
                            : epilogue_loop<EW, 4>(g, p, sh, pos0, pos1, warp, lane, tmem_d, s, ss);
        } else if (e.mode == EPI_COUPLE) {
            ok = e.q == 0.f ? epilogue_loop<EW, 1>(g, p, sh, pos0, pos1, warp, lane, tmem_d, s, ss)
                            : epilogue_loop<EW, 2>(g, p, sh, pos0, pos1, warp, lane, tmem_d, s, ss);
        } else ok = epilogue_loop<EW, 0>(g, p, sh, pos0, pos1, warp, lane, tmem_d, s, ss);
        if (e.part) {
            // per-CTA record: rows of a warp by shuffles, then the warps that share a column in order
            column_sums(s, lane); column_sums(ss, lane);
            if (lane < NC) { sh->sums[warp][lane] = s[0]; sh->sums[warp][NC + lane] = ss[0]; }
            ok = named_barrier_and(2, EW * 32, ok);
            if (ok && etid < g.BN && col0 + etid < e.n_cols) {
                const int lc = etid % NC;
                float a = 0.f, b = 0.f;
                for (int gr = etid / NC; gr < EW / 4; gr += g.groups)
                    for (int w = 4 * gr; w < 4 * gr + 4; w++) { a += sh->sums[w][lc]; b += sh->sums[w][NC + lc]; }
                const int c = col0 + etid;
                float *mine = e.part + (size_t)blockIdx.x * 2 * e.n_cols + (c >> 2) * 8 + (c & 3);
                mine[0] = a; mine[4] = b;
            }
            // (Without a counter the consumer adds the records.)  Layers of at most 64 columns have a record per SM or nearly so, and
            // all sixteen warps add them (38-layer step 1899 -> 1875 us); of wider ones, split over fewer CTAs, eight warps are quicker
            // (all sixteen everywhere: 164-layer step 0.6 % slower)
            if (ok && e.counter) {
                named_barrier(2, EW * 32);
                if (EW == 16 && e.n_cols <= 64) epilogue_publish<512>(e, reinterpret_cast<float *>(abuf), etid);
                else if (warp < 8) epilogue_publish<256>(e, reinterpret_cast<float *>(abuf), etid);
            }
        }
    } else {
        const int bt = (int)threadIdx.x - kBuildWarp0 * 32;
        if (direct) ok = build_rows<1, EW>(g, p, sh, abuf, pos0, pos1, bt, lane);
        else if (p.in_mode == 2) ok = build_rows<2, EW>(g, p, sh, abuf, pos0, pos1, bt, lane);
        else ok = build_rows<0, EW>(g, p, sh, abuf, pos0, pos1, bt, lane);
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

int round_up(int x, int m) { return (x + m - 1) / m * m; }

struct FusedShape { int n_tiles, ctas, smem; FusedGeom g; };

bool fused_shape(Geom geo, int cin, int cout, int k, int sm_count, FusedShape &s) {
    if ((k != 1 && k != 3) || cin % 8 || cout % 4 || cin < 8 || cin > 64) return false;
    FusedGeom &g = s.g;
    memset(&g, 0, sizeof g);
    g.k = k; g.cin = cin; g.nch = cin / 8; g.wpitch = round_up(cin, 16); g.ksteps = g.wpitch / 16;
    g.KC = cin <= 16 ? 16 : (cin <= 32 ? 32 : 64);
    g.N = geo.N; g.H = geo.H; g.W = geo.W; g.pitch = geo.W + 1;
    g.dpitch = fast_div(geo.W + 1); g.drows = fast_div(geo.H + 1);
    g.step_r = (NBT / g.nch) / g.pitch; g.step_c = (NBT / g.nch) % g.pitch;
    g.halo = k == 3 ? geo.W + 2 : 0;
    const size_t total = k == 3 ? (size_t)geo.N * (geo.H + 1) * (geo.W + 1) : geo.P();
    if (total >= (1u << 30)) return false;
    g.total = (int)total;
    const int cout_pad = round_up(cout, 16), tiles = (g.total + 127) / 128, nchp = (g.nch + 1) & ~1;
    g.BN = cout_pad <= 16 ? 16 : (cout_pad <= 32 ? 32 : 64);
    // few tiles (late stages): split the output channels so that more SMs take part
    while (g.BN > 16 && tiles * ((cout_pad + g.BN - 1) / g.BN) * 2 <= sm_count) g.BN /= 2;
    for (;; g.BN /= 2) {
        s.n_tiles = (cout_pad + g.BN - 1) / g.BN;
        g.groups = g.BN / NC;
        int ctas = sm_count / s.n_tiles; if (ctas < 1) ctas = 1;
        // a contiguous range of positions per CTA, a tile at least.  (Half tiles would put a small layer on every SM, but take as long and
        // leave none to the launches beside it: 110-layer step 4964 -> 4877 us, odd-sized basic block 167 -> 164 with whole ones.)
        g.chunk = round_up((g.total + ctas - 1) / ctas, 8); if (g.chunk < 128) g.chunk = 128;
        s.ctas = (g.total + g.chunk - 1) / g.chunk;
        g.wtile_bytes = (g.BN * g.KC * 2 + 1023) & ~1023;
        const int T = (g.chunk + 127) / 128, fixed = 1024 + k * k * g.wtile_bytes + (int)sizeof(FusedShared) + 64;
        // planes are skewed against each other so that the chunks of a pixel, written by adjacent threads, hit different banks
        auto seg_of = [&](int S) { g.plane16 = round_up(S * 128 + 2 * g.halo, 8) + (g.nch <= 2 ? 4 : (g.nch <= 4 ? 2 : 1)); return nchp * g.plane16 * 16; };
        const int room = 227 * 1024 - fixed;
        // the whole range as one segment if it fits, else the longest segments of which two fit
        if (T <= kFullBars && seg_of(T) <= room) { g.S = T; g.nseg = 1; }
        else {
            g.nseg = 2; g.S = kFullBars / 2;
            while (g.S > 1 && 2 * seg_of(g.S) > room) g.S--;
            if (2 * seg_of(g.S) > room) g.nseg = 1;
        }
        g.seg_bytes = round_up(seg_of(g.S), 128);
        g.op_bytes = g.nseg * g.seg_bytes;
        if (g.op_bytes < 20480) g.op_bytes = 20480;      // the last reduction borrows the region: (512 + 128) x 4 doubles
        s.smem = fixed + g.op_bytes;
        if (s.smem <= 227 * 1024 && g.plane16 < (1 << 14)) return true;
        if (g.BN < 32) return false;
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// in: [P, cin] float / fixed point (in_mode 0) or bf16 (in_mode 1); out, partner and the BN input of a
// data gradient must be plain (unsplit) tensors of cout channels
bool run_fused(Exec &ex, const char *what, int in_mode, const void *in, float in_q, BnRef bn, Geom geo, int cin, int cout, int k,
               const float *Wsrc, const bf16 *prepacked, bool transposed, Pair out, Pair partner, int sign, EpiReq req, bf16 *a_out) {
    FusedShape s;
    if (out.c1 != 0 || (sign && partner.c1 != 0) || (req.bnbwd && req.bnbwd->t.c1 != 0)) return false;
    if (!fused_shape(geo, cin, cout, k, ex.ctx->sm_count, s)) return false;
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
    float *part = defer ? req.stats->part : (reduce ? ex.ws.get<float>((size_t)ctas * 2 * cout) : nullptr);
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
        FusedLayer &p = A.ly;
        p.in_mode = in_mode == 0 && in_q != 0.f ? 2 : in_mode; p.in = in; p.in_q = in_q; p.bn = bn; p.a_out = a_out;
        p.aux = req.bnbwd ? req.bnbwd->t.p0 : (sign ? partner.p0 : out.p0);
        p.wide_in = ((uintptr_t)in & 31) == 0;
        p.wide_out = ((uintptr_t)out.p0 & 31) == 0 && ((uintptr_t)p.aux & 31) == 0 && cout % 8 == 0;
        p.w_early = prepacked ? 1 : 0;
        A.status = ex.ctx->dev_status; A.stamp = ex.stamp_slot();
        FusedEpi &e = p.epi;
        e.mode = req.bnbwd ? EPI_BNBWD : (sign ? EPI_COUPLE : EPI_PLAIN);
        e.out = out.p0; e.q = req.bnbwd ? req.bnbwd->t.q : out.q; e.sign = sign; e.n_cols = cout;
        e.part = part; e.counter = (reduce && !defer) ? ex.ctx->counter() : nullptr;
        e.inv_count = 1.0 / (double)geo.P(); e.eps = ex.eps;
        if (req.stats) { e.mean = req.stats->mean; e.rstd = req.stats->rstd; }
        if (req.bnbwd) { e.bn = req.bnbwd->bn; e.dgamma = req.bnbwd->dgamma; e.dbeta = req.bnbwd->dbeta; e.coef = req.bnbwd->coef; }
        static OncePerDevice once;
        if (once.first(ex.ctx->device)) {
            cudaFuncSetAttribute(conv_fused_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
            cudaFuncSetAttribute(conv_fused_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        }
        dim3 grid((unsigned)ctas, (unsigned)s.n_tiles);
        const int EW = s.g.BN == 16 ? 8 : 16;
        launch(ex, EW == 16 ? conv_fused_kernel<16> : conv_fused_kernel<8>, grid, fused_threads(EW), s.smem, A);
        const double bytes = (double)geo.P() * cin * (in_mode == 0 ? 4 : 2) + (double)geo.P() * cout * (sign || req.bnbwd ? 8 : 4) +
                             (double)cout * taps * cin * 2 + (a_out ? (double)geo.P() * cin * 2 : 0.0);
        ex.check(what, bytes, 2.0 * geo.P() * cout * cin * taps);
    }
    ex.ws.release(m);
    return true;
}

}  // namespace

// whether conv_fprop_fused takes layer L on images gi (and so adds pending statistics of its input itself)
bool conv_fused_takes(Exec &ex, Geom gi, const Layer &L) {
    FusedShape s;
    return L.stride == 1 && fused_shape(gi, L.cin, L.cout, L.k, ex.ctx->sm_count, s);
}

// out = partner + sign * conv(ReLU(BN(t)));  a_out (optional): the activated tensor, for the weight gradient
bool conv_fprop_fused(Exec &ex, Pair t, BnRef bn, Geom gi, const Layer &L, Pair out, Pair partner, int sign, Moments *stats, bf16 *a_out) {
    if (L.stride != 1 || t.c1 != 0) return false;
    EpiReq req; req.stats = stats;
    return run_fused(ex, "conv_fprop_fused", 0, t.p0, t.q, bn, gi, L.cin, L.cout, L.k, L.W, L.Wp_fprop, false, out, partner, sign, req, a_out);
}

// da = conv^T(g) for a stride-1 layer, g bf16 [P, cout]
bool conv_dgrad_fused(Exec &ex, const void *g, Geom gi, const Layer &L, float *da, const BnBwdReq *bb) {
    if (L.stride != 1) return false;
    EpiReq req; req.bnbwd = bb;
    return run_fused(ex, "conv_dgrad_fused", 1, g, 0.f, BnRef{}, gi, L.cout, L.cin, L.k, L.W, L.Wp_dgrad, true, single(da, L.cin), Pair{}, 0, req, nullptr);
}
