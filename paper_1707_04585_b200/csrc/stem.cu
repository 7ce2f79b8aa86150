// The stem: a bare convolution of the 3-channel image (3x3 stride 1, or 7x7 stride 2), fp32 in both
// precision modes, forward and weight gradient.  With so few input channels the contraction per
// output pixel is short (K = k*k*3 = 27 or 147) and a tensor-core tile would be mostly padding, so
// these are register-tiled CUDA-core kernels.  The stems that the networks have (three channels; 3x3
// stride 1, 7x7 stride 2) take the row kernels: image rows in shared memory, a lane per one or two output
// channels, a window of image values that slides along the row in registers.  Other shapes take the patch
// kernels: the image patches of a tile of output pixels (128 forward, 64 for the weight gradient) are
// gathered into shared memory once and every thread keeps a small block of the result in registers.
//
//   fprop: out[p, co]      = sum_{kh,kw,ci} img[p*s + (kh,kw) - pad, ci] * W[co, kh, kw, ci]
//   wgrad: dW[co, kh,kw,ci] = sum_p g[p, co] * img[p*s + (kh,kw) - pad, ci]
// (the stem has no data gradient: nothing lies below the image).
#include "common.cuh"

namespace {

constexpr int kPx = 64;            // output pixels per chunk of the weight gradient
constexpr int kFPx = 128;          // output pixels per tile of the forward kernel

struct StemGeom { int N, H, W, Ci, Ho, Wo, Co, k, s, pad, K; };

// patch element kk = (kh, kw, ci) of the output pixel whose window starts at (y0, x0) of image n; zero outside
// the image.  Without branches (the load of an outside element reads the image's first pixel and is dropped),
// so that the loads of an unrolled gather loop are in flight together.
__device__ __forceinline__ float patch_at(const float *__restrict__ img, const StemGeom &g, size_t nbase, int y0, int x0, int koff, bool live) {
    const int kh = koff >> 16, kw = (koff >> 8) & 0xff, ci = koff & 0xff;
    const int y = y0 + kh, x = x0 + kw;
    const bool in = live && (unsigned)y < (unsigned)g.H && (unsigned)x < (unsigned)g.W;
    const size_t idx = in ? nbase + ((size_t)y * g.W + x) * g.Ci + ci : 0;
    const float v = __ldg(img + idx);
    return in ? v : 0.f;
}

__device__ __forceinline__ void fill_koff(const StemGeom &g, int *koff, int tid, int nthreads) {
    for (int kk = tid; kk < g.K; kk += nthreads) {
        const int ci = kk % g.Ci, tap = kk / g.Ci, kw = tap % g.k, kh = tap / g.k;
        koff[kk] = (kh << 16) | (kw << 8) | ci;
    }
}

// 256 threads, tiles of 128 output pixels: thread (tx = tid & 7, ty = tid >> 3) owns pixels ty*4 .. ty*4+3 of the tile and, per pass,
// output channels co0 + tx*CO_T .. + CO_T-1.  Shared memory: the weights transposed to [K][cop]
// (cop = Co rounded up to 8*CO_T), the tile's patches [K][128], the tap table.
template <int CO_T>
__global__ void __launch_bounds__(256) stem_fprop_kernel(const float *__restrict__ img, const float *__restrict__ W, Pair out,
                                                         StemGeom g, int cop, int n_tiles) {
    extern __shared__ float sm[];
    float *Ws = sm;                               // [K][cop]
    float *As = Ws + (size_t)g.K * cop;           // [K][kFPx]
    int *koff = reinterpret_cast<int *>(As + (size_t)g.K * kFPx);
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    fill_koff(g, koff, tid, 256);
    for (int e = tid; e < g.K * cop; e += 256) {
        const int co = e % cop, kk = e / cop;
        Ws[e] = co < g.Co ? W[(size_t)co * g.K + kk] : 0.f;
    }
    pdl_enter();
    const int P = g.N * g.Ho * g.Wo;
    const int px = tid & (kFPx - 1), kk0 = tid >> 7;      // this thread gathers pixel px, patch elements kk0, kk0 + 2, ...
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        __syncthreads();                                   // tables ready / the previous tile's patches consumed
        {
            const int p = t * kFPx + px;
            const bool live = p < P;
            const int wo = p % g.Wo, r = p / g.Wo, ho = r % g.Ho, n = r / g.Ho;
            const size_t nbase = (size_t)n * g.H * g.W * g.Ci;
            const int y0 = ho * g.s - g.pad, x0 = wo * g.s - g.pad;
#pragma unroll 8
            for (int kk = kk0; kk < g.K; kk += 2) As[kk * kFPx + px] = patch_at(img, g, nbase, y0, x0, koff[kk], live);
        }
        __syncthreads();
        for (int co0 = 0; co0 < cop; co0 += 8 * CO_T) {
            float acc[4][CO_T];
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < CO_T; j++) acc[i][j] = 0.f;
            const float *wrow = Ws + co0 + tx * CO_T;
#pragma unroll 3
            for (int kk = 0; kk < g.K; kk++) {
                const float4 a = *reinterpret_cast<const float4 *>(As + kk * kFPx + ty * 4);
                float w[CO_T];
#pragma unroll
                for (int j = 0; j < CO_T; j += 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(wrow + (size_t)kk * cop + j);
                    w[j] = v.x; w[j + 1] = v.y; w[j + 2] = v.z; w[j + 3] = v.w;
                }
#pragma unroll
                for (int j = 0; j < CO_T; j++) {
                    acc[0][j] = fmaf(a.x, w[j], acc[0][j]); acc[1][j] = fmaf(a.y, w[j], acc[1][j]);
                    acc[2][j] = fmaf(a.z, w[j], acc[2][j]); acc[3][j] = fmaf(a.w, w[j], acc[3][j]);
                }
            }
            const int co = co0 + tx * CO_T;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const int p = t * kFPx + ty * 4 + i;
                if (p >= P) continue;
#pragma unroll
                for (int j = 0; j < CO_T; j += 4)
                    if (co + j < g.Co) out.store4((size_t)p, co + j, make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]));
            }
        }
    }
}

// 256 threads = G groups x S pixel lanes.  Group (cg, kg) owns the CO_T x KK_T block of dW at output channels
// cg*CO_T.., patch elements kg*KK_T..; lane `sub` of the group adds the pixels sub, sub + S, ... of every
// 64-pixel chunk the CTA walks.  At the end the lanes are added in order through shared memory and the CTA
// writes one partial [Co][K]; splitk_reduce adds the partials in order.
template <int CO_T, int KK_T>
__global__ void __launch_bounds__(256) stem_wgrad_kernel(const float *__restrict__ img, const float *__restrict__ gout, float *__restrict__ part,
                                                         StemGeom g, int cop, int kp, int n_cg, int G, int S, int n_chunks) {
    extern __shared__ float sm[];
    float *Gs = sm;                               // [kPx][cop]
    float *As = Gs + (size_t)kPx * cop;           // [kPx][kp]
    int *koff = reinterpret_cast<int *>(As + (size_t)kPx * kp);
    const int tid = threadIdx.x;
    fill_koff(g, koff, tid, 256);
    pdl_enter();
    const int grp = tid % G, sub = tid / G;
    const bool worker = sub < S;
    const int cg = grp % n_cg, kg = grp / n_cg;
    float acc[CO_T][KK_T];
#pragma unroll
    for (int i = 0; i < CO_T; i++)
#pragma unroll
        for (int j = 0; j < KK_T; j++) acc[i][j] = 0.f;
    const int P = g.N * g.Ho * g.Wo;
    const int px = tid & (kPx - 1), kk0 = tid >> 6;      // gathers pixel px, patch elements kk0, kk0 + 4, ...
    for (int c = blockIdx.x; c < n_chunks; c += gridDim.x) {
        __syncthreads();
        {
            const int p = c * kPx + px;
            const bool live = p < P;
            const int wo = p % g.Wo, r = p / g.Wo, ho = r % g.Ho, n = r / g.Ho;
            const size_t nbase = (size_t)n * g.H * g.W * g.Ci;
            const int y0 = ho * g.s - g.pad, x0 = wo * g.s - g.pad;
#pragma unroll 8
            for (int kk = kk0; kk < kp; kk += 4) As[px * kp + kk] = patch_at(img, g, nbase, y0, x0, koff[kk < g.K ? kk : 0], live && kk < g.K);
        }
        for (int e = tid; e < kPx * cop; e += 256) {
            const int co = e % cop, q = e / cop;
            const int p = c * kPx + q;
            Gs[e] = (p < P && co < g.Co) ? gout[(size_t)p * g.Co + co] : 0.f;
        }
        __syncthreads();
        if (worker) {
            for (int q = sub; q < kPx; q += S) {
                float gv[CO_T], av[KK_T];
#pragma unroll
                for (int i = 0; i < CO_T; i += 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(Gs + q * cop + cg * CO_T + i);
                    gv[i] = v.x; gv[i + 1] = v.y; gv[i + 2] = v.z; gv[i + 3] = v.w;
                }
#pragma unroll
                for (int j = 0; j < KK_T; j += 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(As + q * kp + kg * KK_T + j);
                    av[j] = v.x; av[j + 1] = v.y; av[j + 2] = v.z; av[j + 3] = v.w;
                }
#pragma unroll
                for (int i = 0; i < CO_T; i++)
#pragma unroll
                    for (int j = 0; j < KK_T; j++) acc[i][j] = fmaf(gv[i], av[j], acc[i][j]);
            }
        }
    }
    // lanes of a group are added in order, one block element at a time through shared memory
    __syncthreads();
    float *red = sm;                              // [S][G] floats (S*G <= 256)
    float *mine = part + (size_t)blockIdx.x * g.Co * g.K;
#pragma unroll
    for (int i = 0; i < CO_T; i++)
#pragma unroll
        for (int j = 0; j < KK_T; j++) {
            if (worker) red[sub * G + grp] = acc[i][j];
            __syncthreads();
            if (worker && sub == 0) {
                float s = red[grp];
                for (int y = 1; y < S; y++) s += red[y * G + grp];
                const int co = cg * CO_T + i, kk = kg * KK_T + j;
                if (co < g.Co && kk < g.K) mine[(size_t)co * g.K + kk] = s;
            }
            __syncthreads();
        }
}

// ------------------------------------------------------------------ three channels, 3x3 stride 1 or 7x7 stride 2
// Image rows y0 .. y0 + rows - 1 of image n into shared memory, element (row, column, channel) at
// row * rp + (column + pad) * xp + channel * cp; rows outside the image become zeros, the columns beside it stay as they are
// (zero since the start of the kernel).  Asynchronous: the caller waits.
__device__ __forceinline__ void stage_rows(const float *__restrict__ img, const StemGeom &g, FastDiv rowdiv, int n, int y0, int rows, float *dst, int rp, int xp, int cp) {
    const int row_e = g.W * 3;
    for (int e = threadIdx.x; e < rows * row_e; e += blockDim.x) {
        uint32_t r, q;
        rowdiv.divmod((uint32_t)e, r, q);
        const uint32_t x = q / 3, c = q - 3 * x;
        const int y = y0 + (int)r;
        const bool ok = (unsigned)y < (unsigned)g.H && n < g.N;
        const float *src = img + (ok ? ((size_t)n * g.H + y) * row_e + q : 0);
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + (int)r * rp + ((int)x + g.pad) * xp + (int)c * cp);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(ok ? 4 : 0) : "memory");
    }
}
template <int K> struct StemRow {
    static constexpr int S = K == 3 ? 1 : 2;
    // weight gradient: KH rows of the filter per warp, RS output rows per CTA, U pixels per turn (a multiple of K: the window has
    // turned), CBW channel groups of 32 at most per CTA
    static constexpr int KH = K == 3 ? 3 : 1, HG = K / KH, RS = K == 3 ? 8 : 1, U = K == 3 ? 12 : 7, CBW = K == 3 ? 1 : 4;
    // forward (7x7): output rows per CTA, warps
    static constexpr int FR = 2, FW = 14;
};

// Weight gradient.  A warp has KH filter rows and 32 output channels, a lane each, and goes along output rows: per pixel S new image
// columns and one gradient value come in, KH * K * 3 FMAs follow from registers.  Every 128 pixels or more the
// sums are added to totals in shared memory, which are added over the warps of a filter row and written as one partial per CTA.
// Bound by the FMA pipes.  Measured: 131072 pixels x 32 channels, 3x3: 59 -> 20 us; 802816 x 128, 7x7: 1405 -> 1045 us (29 TFLOP/s;
// single FMAs reach 56).
template <int K>
__global__ void __launch_bounds__(K == 3 ? 256 : 896) stem_wgrad_row_kernel(const float *__restrict__ img, const float *__restrict__ gout, float *__restrict__ part,
                                                                           StemGeom g, FastDiv rowdiv, int cols, int tiles_per_img, int n_tiles, int cbw) {
    using T = StemRow<K>;
    constexpr int S = T::S, KH = T::KH, A = KH * K * 3, U = T::U, ROWS = (T::RS - 1) * S + K;
    extern __shared__ float sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
    const int hg = warp % T::HG, cb = (warp / T::HG) % cbw, rs = warp / (T::HG * cbw);
    const int co = ((int)blockIdx.y * cbw + cb) * 32 + lane;
    const int rp = cols * 4, buf_floats = ROWS * rp;
    float *tot = sm + 2 * buf_floats;                                  // [warp][A][32]
    for (int i = tid; i < 2 * buf_floats + nw * A * 32; i += blockDim.x) sm[i] = 0.f;
    __syncthreads();
    pdl_enter();
    float acc[A];
#pragma unroll
    for (int a = 0; a < A; a++) acc[a] = 0.f;
    auto stage = [&](int t, int b) {
        const int n = t / tiles_per_img, y0 = (t - n * tiles_per_img) * T::RS;
        stage_rows(img, g, rowdiv, n, y0 * S - g.pad, ROWS, sm + b * buf_floats, rp, 4, 1);
    };
    float *mytot = tot + (size_t)warp * A * 32 + lane;
    auto flush = [&]() {
#pragma unroll
        for (int a = 0; a < A; a++) { mytot[a * 32] += acc[a]; acc[a] = 0.f; }
    };
    int b = 0, held = 0;
    if ((int)blockIdx.x < n_tiles) stage(blockIdx.x, 0);
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, b ^= 1) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (t + (int)gridDim.x < n_tiles) stage(t + gridDim.x, b ^ 1);
        const int n = t / tiles_per_img, y = (t - n * tiles_per_img) * T::RS + rs;
        if (y < g.Ho && co < g.Co) {
            const float *gp = gout + (((size_t)n * g.Ho + y) * g.Wo) * g.Co + co;
            const float *rowp = sm + b * buf_floats + (rs * S + hg * KH) * rp;
            auto load_g = [&](int x, float (&v)[U]) {
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const bool in = x + u < g.Wo;
                    const float q = gp[(size_t)(in ? x + u : 0) * g.Co];
                    v[u] = in ? q : 0.f;
                }
            };
            float win[KH][K][3], gv[U], gn[U];
            auto column = [&](int c, int slot) {
#pragma unroll
                for (int r = 0; r < KH; r++) {
                    const float4 q = *reinterpret_cast<const float4 *>(rowp + r * rp + c * 4);
                    win[r][slot][0] = q.x; win[r][slot][1] = q.y; win[r][slot][2] = q.z;
                }
            };
#pragma unroll
            for (int c = 0; c < K - S; c++) column(c, c);
            load_g(0, gv);
#pragma unroll 1
            for (int x = 0; x < g.Wo; x += U) {
                load_g(x + U, gn);
#pragma unroll
                for (int u = 0; u < U; u++) {
#pragma unroll
                    for (int c = K - S; c < K; c++) column((x + u) * S + c, (u * S + c) % K);
#pragma unroll
                    for (int r = 0; r < KH; r++)
#pragma unroll
                        for (int kw = 0; kw < K; kw++)
#pragma unroll
                            for (int ci = 0; ci < 3; ci++)
                                acc[(r * K + kw) * 3 + ci] = fmaf(gv[u], win[r][(u * S + kw) % K][ci], acc[(r * K + kw) * 3 + ci]);
                }
#pragma unroll
                for (int u = 0; u < U; u++) gv[u] = gn[u];
            }
            held += g.Wo;
            if (held >= 128) { flush(); held = 0; }
        }
    }
    flush();
    __syncthreads();
    // one partial per CTA: dW[co][kh][kw][ci], the row warps added in order
    const int K27 = K * K * 3, n_co = cbw * 32, co0 = (int)blockIdx.y * n_co;
    float *mine = part + (size_t)blockIdx.x * g.Co * K27;
    const int n_rs = nw / (T::HG * cbw);
    for (int e = tid; e < n_co * K27; e += blockDim.x) {
        const int c = e / K27, kk = e - c * K27, h = kk / (KH * K * 3), a = kk - h * (KH * K * 3);
        if (co0 + c >= g.Co) continue;
        float v = 0.f;
        for (int r = 0; r < n_rs; r++) v += tot[((size_t)((r * cbw + c / 32) * T::HG + h) * A + a) * 32 + c % 32];
        mine[(size_t)(co0 + c) * K27 + kk] = v;
    }
}

// Forward, 7x7.  A warp takes eight pixels of an output row and 32 COL output channels: per filter row and channel the image values of
// its pixels (21 of them, planar rows in shared memory) and one weight row per column tap, 8 COL FMAs each.
// Bound by the FMA pipes.  Measured: 802816 pixels x 128 channels: 1610 -> 890 us.
template <int COL>
__global__ void __launch_bounds__(StemRow<7>::FW * 32) stem_fprop_row_kernel(const float *__restrict__ img, const float *__restrict__ W, Pair out,
                                                                           StemGeom g, FastDiv rowdiv, int cols, int tiles_per_img, int n_tiles, int cop) {
    constexpr int K = 7;
    using T = StemRow<K>;
    constexpr int S = T::S, ROWS = (T::FR - 1) * S + K, NX = (7 * S + K + 3) / 4;
    extern __shared__ float sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
    float *Ws = sm;                                                    // [kh][ci][kw][cop]
    float *rowsm = Ws + K * K * 3 * cop;                               // two buffers of [row][ci][cols]
    const int buf_floats = ROWS * 3 * cols;
    for (int i = tid; i < 2 * buf_floats; i += blockDim.x) rowsm[i] = 0.f;
    for (int e = tid; e < K * K * 3 * cop; e += blockDim.x) {
        const int co = e / (K * K * 3), kk = e - co * (K * K * 3), kh = kk / (K * 3), kw = kk / 3 % K, ci = kk % 3;
        Ws[((kh * 3 + ci) * K + kw) * cop + co] = co < g.Co ? W[(size_t)co * (K * K * 3) + kk] : 0.f;
    }
    __syncthreads();
    pdl_enter();
    auto stage = [&](int t, int b) {
        const int n = t / tiles_per_img, y0 = (t - n * tiles_per_img) * T::FR;
        stage_rows(img, g, rowdiv, n, y0 * S - g.pad, ROWS, rowsm + b * buf_floats, 3 * cols, 1, cols);
    };
    const int segs = (g.Wo + 7) / 8, cbs = cop / (32 * COL), tasks = T::FR * segs * cbs;
    int b = 0;
    if ((int)blockIdx.x < n_tiles) stage(blockIdx.x, 0);
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, b ^= 1) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (t + (int)gridDim.x < n_tiles) stage(t + gridDim.x, b ^ 1);
        const int n = t / tiles_per_img, y0 = (t - n * tiles_per_img) * T::FR;
        for (int task = warp; task < tasks; task += nw) {
            const int cb = task % cbs, q = task / cbs, seg = q % segs, r = q / segs;
            const int co = cb * 32 * COL + lane * COL;
            if (y0 + r >= g.Ho) break;
            const float *xp = rowsm + b * buf_floats + r * S * 3 * cols + seg * 8 * S;
            const float *wp = Ws + co;
            float acc[8][COL];
#pragma unroll
            for (int i = 0; i < 8; i++)
#pragma unroll
                for (int j = 0; j < COL; j++) acc[i][j] = 0.f;
#pragma unroll 3
            for (int kc = 0; kc < K * 3; kc++) {                       // filter row and channel
                float v[NX * 4];
#pragma unroll
                for (int i = 0; i < NX; i++) {
                    const float4 u = *reinterpret_cast<const float4 *>(xp + kc * cols + 4 * i);
                    v[4 * i] = u.x; v[4 * i + 1] = u.y; v[4 * i + 2] = u.z; v[4 * i + 3] = u.w;
                }
#pragma unroll
                for (int kw = 0; kw < K; kw++) {
                    float w[COL];
                    if constexpr (COL == 2) { const float2 u = *reinterpret_cast<const float2 *>(wp + (kc * K + kw) * cop); w[0] = u.x; w[1] = u.y; }
                    else w[0] = wp[(kc * K + kw) * cop];
#pragma unroll
                    for (int i = 0; i < 8; i++)
#pragma unroll
                        for (int j = 0; j < COL; j++) acc[i][j] = fmaf(v[i * S + kw], w[j], acc[i][j]);
                }
            }
            if (co < g.Co)
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    const int x = seg * 8 + i;
                    if (x >= g.Wo) continue;
                    const size_t p = ((size_t)n * g.Ho + y0 + r) * g.Wo + x;
                    if constexpr (COL == 2) out.couple2_with(p, co, make_float2(acc[i][0], acc[i][1]), make_float2(0.f, 0.f), 0);
                    else out.couple(p, co, acc[i][0], out, 0);
                }
        }
    }
}

// dW[i] = sum of the per-CTA partials, one warp per element: lane l adds the partials l, l + 32, ... and the
// lanes are combined by a shuffle tree, so the order of additions is fixed by `parts` alone
__global__ void stem_sum_kernel(const float *__restrict__ part, size_t n, int parts, float *__restrict__ out) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const size_t warp = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, n_warps = ((size_t)gridDim.x * blockDim.x) >> 5;
    for (size_t i = warp; i < n; i += n_warps) {
        float s = 0.f;
        for (int z = lane; z < parts; z += 32) s += part[(size_t)z * n + i];
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) out[i] = s;
    }
}

StemGeom stem_geom(Geom gi, const Layer &L) {
    StemGeom g;
    g.N = gi.N; g.H = gi.H; g.W = gi.W; g.Ci = L.cin; g.Co = L.cout; g.k = L.k; g.s = L.stride; g.pad = L.k / 2;
    g.Ho = conv_out(gi.H, L.k, L.stride); g.Wo = conv_out(gi.W, L.k, L.stride);
    g.K = L.k * L.k * L.cin;
    return g;
}
int round_up(int x, int m) { return (x + m - 1) / m * m; }

}  // namespace

// whether the row kernels take a stem, and their row pitch: columns -pad .. of the rows that the last turn of `turn` pixels reads
static bool row_stem(const StemGeom &g, int turn, int &cols) {
    if (g.Ci != 3 || !((g.k == 3 && g.s == 1) || (g.k == 7 && g.s == 2)) || (size_t)g.W * 3 * 32 > (1u << 30)) return false;
    cols = round_up((round_up(g.Wo, turn) - 1) * g.s + g.k, 4) + 4;
    if (cols < g.W + 2 * g.pad) cols = round_up(g.W + 2 * g.pad, 4);
    return true;
}
template <class F> static int row_grid(Exec &ex, F kernel, int threads, size_t smem, int n_tiles, int blocks_y) {
    int per_sm = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1) { cudaGetLastError(); per_sm = 1; }
    int ctas = ex.ctx->sm_count * per_sm / blocks_y; if (ctas < 1) ctas = 1;
    const int rounds = (n_tiles + ctas - 1) / ctas;
    return (n_tiles + rounds - 1) / rounds;
}
// (3x3: the patch kernel is the quicker one, 18 against 24 us for 131072 x 32)
template <int COL> static bool fprop_rows(Exec &ex, const float *img, const StemGeom &g, const float *W, Pair out) {
    constexpr int K = 7;
    using T = StemRow<K>;
    int cols;
    if (g.k != K || !row_stem(g, 8, cols)) return false;
    const int cop = round_up(g.Co, 32 * COL), tiles_per_img = (g.Ho + T::FR - 1) / T::FR, n_tiles = g.N * tiles_per_img;
    const size_t smem = ((size_t)g.K * cop + 2 * (size_t)((T::FR - 1) * T::S + K) * 3 * cols) * 4;
    if (smem > 200 * 1024) return false;
    if (ex.dry) return true;
    static OncePerDevice once;
    if (once.first(ex.ctx->device)) cudaFuncSetAttribute(stem_fprop_row_kernel<COL>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    const int grid = row_grid(ex, stem_fprop_row_kernel<COL>, T::FW * 32, smem, n_tiles, 1);
    launch(ex, stem_fprop_row_kernel<COL>, grid, T::FW * 32, smem, img, W, out, g, fast_div(g.W * 3), cols, tiles_per_img, n_tiles, cop);
    return true;
}
// Launch of the row weight gradient; false: shape not taken (decided here alone, for the sizing run and the real one)
struct RowWgrad { int cols, cbw, blocks_y, nw, tiles_per_img, n_tiles; size_t smem; };
template <int K> static bool wgrad_rows_shape(const StemGeom &g, RowWgrad &w) {
    using T = StemRow<K>;
    if (g.k != K || !row_stem(g, T::U, w.cols)) return false;
    const int cbs = (g.Co + 31) / 32;
    w.cbw = cbs < T::CBW ? cbs : T::CBW; w.blocks_y = (cbs + w.cbw - 1) / w.cbw;
    w.nw = T::HG * w.cbw * T::RS; w.tiles_per_img = (g.Ho + T::RS - 1) / T::RS; w.n_tiles = g.N * w.tiles_per_img;
    w.smem = (2 * (size_t)((T::RS - 1) * T::S + K) * w.cols * 4 + (size_t)w.nw * T::KH * K * 3 * 32) * 4;
    return w.smem <= 200 * 1024;
}
// part: room for `cap` partials; returns the number written
template <int K> static int wgrad_rows(Exec &ex, const float *img, const float *gout, const StemGeom &g, const RowWgrad &w, float *part, int cap) {
    static OncePerDevice once;
    if (once.first(ex.ctx->device)) cudaFuncSetAttribute(stem_wgrad_row_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    int parts = row_grid(ex, stem_wgrad_row_kernel<K>, w.nw * 32, w.smem, w.n_tiles, w.blocks_y);
    if (parts > cap) parts = cap;
    launch(ex, stem_wgrad_row_kernel<K>, dim3(parts, w.blocks_y), w.nw * 32, w.smem, img, gout, part, g, fast_div(g.W * 3), w.cols, w.tiles_per_img, w.n_tiles, w.cbw);
    return parts;
}

// image: fp32 [N,H,W,cin]; out: the stem's output (a plain tensor or the halves of stage 0's pair, float or fixed point)
bool stem_fprop(Exec &ex, const float *img, Geom gi, const Layer &L, Pair out) {
    const StemGeom g = stem_geom(gi, L);
    if (L.cin > 255 || L.k > 255 || L.cout % 4 || (out.c1 && out.c0 % 4)) return false;
    const bool wide = L.cout > 32;
    if (wide ? fprop_rows<2>(ex, img, g, L.W, out) : fprop_rows<1>(ex, img, g, L.W, out)) {
        const double P = (double)g.N * g.Ho * g.Wo;
        ex.flops += 2ull * g.N * g.Ho * g.Wo * g.Co * g.K;
        if (!ex.dry) ex.check("stem_fprop", (double)g.N * g.H * g.W * g.Ci * 4 + P * g.Co * 4 + (double)g.Co * g.K * 4, 2.0 * P * g.Co * g.K);
        return true;
    }
    const int CO_T = L.cout >= 64 ? 8 : 4;
    const int cop = round_up(L.cout, 8 * CO_T);
    const size_t smem = ((size_t)g.K * cop + (size_t)g.K * kFPx) * 4 + (size_t)g.K * 4;
    if (smem > 200 * 1024) return false;
    ex.flops += 2ull * g.N * g.Ho * g.Wo * g.Co * g.K;
    if (ex.dry) return true;
    const int P = g.N * g.Ho * g.Wo, n_tiles = (P + kFPx - 1) / kFPx;
    int per_sm = (int)((220 * 1024) / (smem + 1024)); if (per_sm > 8) per_sm = 8; if (per_sm < 1) per_sm = 1;
    int grid = ex.ctx->sm_count * per_sm; if (grid > n_tiles) grid = n_tiles;
    static OncePerDevice once;
    if (once.first(ex.ctx->device)) {
        cudaFuncSetAttribute(stem_fprop_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(stem_fprop_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    }
    if (CO_T == 8) launch(ex, stem_fprop_kernel<8>, grid, 256, smem, img, L.W, out, g, cop, n_tiles);
    else launch(ex, stem_fprop_kernel<4>, grid, 256, smem, img, L.W, out, g, cop, n_tiles);
    ex.check("stem_fprop", (double)g.N * g.H * g.W * g.Ci * 4 + (double)P * g.Co * 4 + (double)g.Co * g.K * 4, 2.0 * P * g.Co * g.K);
    return true;
}

// gout: fp32 [P, cout] gradient w.r.t. the stem output; dW: [cout][k][k][cin]
bool stem_wgrad(Exec &ex, const float *img, const float *gout, Geom gi, const Layer &L, float *dW) {
    const StemGeom g = stem_geom(gi, L);
    if (L.cin > 255 || L.k > 255) return false;
    const bool big = L.cout >= 64;
    const int CO_T = big ? 8 : 4, KK_T = big ? 12 : 4;
    const int cop = round_up(L.cout, CO_T), kp = round_up(g.K, KK_T);
    const int n_cg = cop / CO_T, n_kg = kp / KK_T, G = n_cg * n_kg;
    const int P = g.N * g.Ho * g.Wo, n_chunks = (P + kPx - 1) / kPx;
    const size_t smem = ((size_t)kPx * cop + (size_t)kPx * kp) * 4 + (size_t)g.K * 4;
    RowWgrad w;
    const bool rows = wgrad_rows_shape<3>(g, w) || wgrad_rows_shape<7>(g, w);
    if (!rows && (G > 256 || smem > 200 * 1024)) return false;
    int grid = ex.ctx->sm_count * (g.k == 3 ? 4 : 2); if (grid > n_chunks) grid = n_chunks;         // room for that many partials
    ex.flops += 2ull * P * g.Co * g.K;
    size_t m = ex.ws.mark();
    float *part = ex.ws.get<float>((size_t)grid * g.Co * g.K);
    if (!ex.dry) {
        if (rows) grid = g.k == 3 ? wgrad_rows<3>(ex, img, gout, g, w, part, grid) : wgrad_rows<7>(ex, img, gout, g, w, part, grid);
        else {
            if (grid > ex.ctx->sm_count * 2) grid = ex.ctx->sm_count * 2;
            const int S = 256 / G;
            static OncePerDevice once;
            if (once.first(ex.ctx->device)) {
                cudaFuncSetAttribute(stem_wgrad_kernel<8, 12>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
                cudaFuncSetAttribute(stem_wgrad_kernel<4, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
            }
            if (big) launch(ex, stem_wgrad_kernel<8, 12>, grid, 256, smem, img, gout, part, g, cop, kp, n_cg, G, S, n_chunks);
            else launch(ex, stem_wgrad_kernel<4, 4>, grid, 256, smem, img, gout, part, g, cop, kp, n_cg, G, S, n_chunks);
        }
        ex.check("stem_wgrad", (double)g.N * g.H * g.W * g.Ci * 4 + (double)P * g.Co * 4, 2.0 * P * g.Co * g.K);
        const size_t n = (size_t)g.Co * g.K;
        int sg = (int)((n + 7) / 8); if (sg > ex.ctx->sm_count * 8) sg = ex.ctx->sm_count * 8;      // eight warps per block
        launch(ex, stem_sum_kernel, sg, 256, 0, (const float *)part, n, grid, dW);
        ex.check("stem_sum", (double)n * 4 * (grid + 1));
    }
    ex.ws.release(m);
    return true;
}
