// Convolution forward / data-gradient / weight-gradient as fp32 implicit GEMMs on the CUDA cores.
// This is the strict-precision path, and the fallback for shapes the tensor-core
// kernels do not take.  Products and sums are fp32 FMA; operands may be float or bf16.
//
//   fprop: out[p,co]   = sum_{kh,kw,ci} a[p (+) (kh,kw), ci] * W[co,kh,kw,ci]        (Eq. 2, Conv_kxk)
//   dgrad: da[q,ci]    = sum_{kh,kw,co} g[p,co] * W[co,kh,kw,ci],  p*s + (kh,kw) - pad = q
//   wgrad: dW[co,kh,kw,ci] = sum_p g[p,co] * a[p (+) (kh,kw), ci]
//
// Four kernels.  conv3x3_direct_kernel takes fp32 3x3 stride-1 layers (forward and data gradient), wgrad3x3_strip_kernel the weight
// gradients of most of those of at most 48 channels (see wg_strip_shape), conv_gemm_kernel every other layer whose channel counts are multiples of four (all BN-ReLU-conv layers): quads of channels are loaded as vectors, a thread's pixel is decoded once, and the product is register-tiled.
// gemm_simt_kernel loads element by element and is left for the stem convolution's odd channel counts (an image has
// three), where the kernels of stem.cu do not take its size.
#include "common.cuh"
#include "conv_direct.cuh"
#include "conv_strips.cuh"
#include <algorithm>

template <class T> __device__ __forceinline__ float ldf(const T *p);
template <> __device__ __forceinline__ float ldf<float>(const float *p) { return *p; }
template <> __device__ __forceinline__ float ldf<bf16>(const bf16 *p) { return __bfloat162float(*p); }

struct ConvGeom {
    int N, H, W, Ci, Ho, Wo, Co, k, s, pad;
};

// ------------------------------------------------------------------ channel counts that are multiples of four
// C[M,N] = A[M,K] * B[K,N] in tiles of (64 WM) x (16 WN), 256 threads = 8 warps of which WK share the K range of a tile: a
// warp holds 64 x 16 accumulators, 8 x 4 per thread, so that one K step costs three 16-byte shared-memory reads (one wavefront
// each) per 32 FMAs.  K runs in chunks of 16 through two shared-memory buffers; the next chunk's quads are on their way
// from global memory while this one is multiplied.
// A sum of K products is taken in runs of 256 that are then added: the rounding error of one serial sum grows with the size
// of the running value (K = 7488, a 3x3 layer of 832 channels: 2e-7 to 5e-7 of the result's deviation, enough to turn the sign
// of a BN output close to zero), the runs keep it several times smaller, for 1.8 % of the time of a fp32 train
// step of the 38-layer network.
// Bound by the FMA pipes (and by issue: 35 instructions per 32 FMAs).  Measured on the 3x3 layers of the CIFAR-sized
// networks at batch 128: 16 channels at 32x32: 157 -> 33 us forward, 176 -> 27 us
// data gradient, 371 -> 49 us weight gradient (the element-wise kernel spent its time on index divisions and scalar loads).
// The forward pass and the data gradient of most 3x3 stride-1 layers now take the direct kernel further down.
template <class T> __device__ __forceinline__ float4 ldq(const T *p);
template <> __device__ __forceinline__ float4 ldq<float>(const float *p) { return *reinterpret_cast<const float4 *>(p); }
template <> __device__ __forceinline__ float4 ldq<bf16>(const bf16 *p) {
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ float round_w(float w, bool to_bf16) { return to_bf16 ? __bfloat162float(__float2bfloat16_rn(w)) : w; }
__device__ __forceinline__ float4 round_w4(float4 w, bool b) { return make_float4(round_w(w.x, b), round_w(w.y, b), round_w(w.z, b), round_w(w.w, b)); }

// Operands.  kAlongK: a quad is four consecutive K indices of one row (else four consecutive rows at one K index).
// row(m): what a thread keeps of its row (quad of rows); quad(state, k): the four values, zeros outside.
struct RowAt { int y, x; size_t base; bool ok; };
template <class TA> struct FpropA {           // m = output pixel, k = (kh, kw, ci)
    static constexpr bool kAlongK = true;
    const TA *a; ConvGeom g; FastDiv wo, ho, ci, kk; int M, K;
    __device__ __forceinline__ RowAt row(int m) const {
        uint32_t t, x, n, y;
        wo.divmod((uint32_t)m, t, x); ho.divmod(t, n, y);
        return RowAt{(int)y * g.s - g.pad, (int)x * g.s - g.pad, (size_t)n * g.H * g.W * g.Ci, m < M};
    }
    __device__ __forceinline__ float4 quad(const RowAt &r, int k) const {
        uint32_t tap, c, kh, kw;
        ci.divmod((uint32_t)k, tap, c); kk.divmod(tap, kh, kw);
        const int y = r.y + (int)kh, x = r.x + (int)kw;
        if (!r.ok || k >= K || (unsigned)y >= (unsigned)g.H || (unsigned)x >= (unsigned)g.W) return make_float4(0.f, 0.f, 0.f, 0.f);
        return ldq(a + r.base + ((size_t)y * g.W + x) * g.Ci + c);
    }
    __device__ __forceinline__ size_t out_row(int m) const { return (size_t)m; }
    __device__ __forceinline__ bool skip(int, int, int) const { return false; }
};
// m = input pixel, k = (kh, kw, co).  With stride 2 the pixels are numbered parity class by parity class ((y & 1, x & 1), then
// image, y / 2, x / 2), so that a tile lies in one class and the chunks of the taps that do not reach it are skipped.
template <class TG> struct DgradA {
    static constexpr bool kAlongK = true;
    const TG *gq; ConvGeom g; FastDiv w, h, co, kk, cls; bool classes; int M, K;       // w, h: columns and rows of a class (stride 1: of the image)
    __device__ __forceinline__ void place(int m, int &n, int &y, int &x) const {
        uint32_t c = 0, r = (uint32_t)m, t, xx, nn, yy;
        if (classes) cls.divmod(r, c, r);
        w.divmod(r, t, xx); h.divmod(t, nn, yy);
        n = (int)nn;
        y = classes ? (int)(2 * yy + (c >> 1)) : (int)yy; x = classes ? (int)(2 * xx + (c & 1)) : (int)xx;
    }
    __device__ __forceinline__ RowAt row(int m) const {
        int n, y, x;
        place(m, n, y, x);
        return RowAt{y + g.pad, x + g.pad, (size_t)n * g.Ho * g.Wo * g.Co, m < M};
    }
    __device__ __forceinline__ float4 quad(const RowAt &r, int k) const {
        uint32_t tap, c, kh, kw;
        co.divmod((uint32_t)k, tap, c); kk.divmod(tap, kh, kw);
        int y = r.y - (int)kh, x = r.x - (int)kw;
        bool ok = r.ok && k < K && y >= 0 && x >= 0;
        if (g.s == 2) { ok = ok && !((y | x) & 1); y >>= 1; x >>= 1; }
        if (!ok || y >= g.Ho || x >= g.Wo) return make_float4(0.f, 0.f, 0.f, 0.f);
        return ldq(gq + r.base + ((size_t)y * g.Wo + x) * g.Co + c);
    }
    __device__ __forceinline__ size_t out_row(int m) const {
        if (!classes) return (size_t)m;
        int n, y, x;
        place(m, n, y, x);
        return ((size_t)n * g.H + y) * g.W + x;
    }
    // whether the chunk k .. k + 15 adds nothing to the rows m0 .. m1
    __device__ __forceinline__ bool skip(int m0, int m1, int k) const {
        if (!classes) return false;
        const uint32_t c = cls.div((uint32_t)m0), tap = co.div((uint32_t)k);
        if (c != cls.div((uint32_t)(m1 < M ? m1 : M - 1)) || tap != co.div((uint32_t)(k + 15))) return false;
        uint32_t kh, kw;
        kk.divmod(tap, kh, kw);
        return (((c >> 1) + g.pad + kh) & 1) || (((c & 1) + g.pad + kw) & 1);
    }
};
template <class TA> struct WgradA {           // m = (kh, kw, ci), k = output pixel
    static constexpr bool kAlongK = false;
    const TA *a; ConvGeom g; FastDiv wo, ho, ci, kk; int M, K;
    __device__ __forceinline__ RowAt row(int m) const {
        uint32_t tap, c, kh, kw;
        ci.divmod((uint32_t)m, tap, c); kk.divmod(tap, kh, kw);
        return RowAt{(int)kh - g.pad, (int)kw - g.pad, c, m < M};
    }
    __device__ __forceinline__ float4 quad(const RowAt &r, int k) const {
        uint32_t t, xo, n, yo;
        wo.divmod((uint32_t)k, t, xo); ho.divmod(t, n, yo);
        const int y = (int)yo * g.s + r.y, x = (int)xo * g.s + r.x;
        if (!r.ok || k >= K || (unsigned)y >= (unsigned)g.H || (unsigned)x >= (unsigned)g.W) return make_float4(0.f, 0.f, 0.f, 0.f);
        return ldq(a + (((size_t)n * g.H + y) * g.W + x) * g.Ci + r.base);
    }
    __device__ __forceinline__ bool skip(int, int, int) const { return false; }
};
struct FpropB {                               // n = co, k = (kh, kw, ci): W[co][k];  wb: weights take part as bf16 values (mode 0)
    static constexpr bool kAlongK = true;
    const float *w; int N, K; bool wb;
    __device__ __forceinline__ float4 quad(int n, int k) const {
        return n < N && k < K ? round_w4(ldq(w + (size_t)n * K + k), wb) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
};
struct DgradB {                               // n = ci (four of them), k = (kh, kw, co): W[co][tap][ci]
    static constexpr bool kAlongK = false;
    const float *w; FastDiv co; int taps, N, K; bool wb;
    __device__ __forceinline__ float4 quad(int n, int k) const {
        uint32_t tap, c;
        co.divmod((uint32_t)k, tap, c);
        return n < N && k < K ? round_w4(ldq(w + ((size_t)c * taps + tap) * N + n), wb) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
};
template <class TG> struct WgradB {           // n = co (four of them), k = output pixel
    static constexpr bool kAlongK = false;
    const TG *gq; int N, K;
    __device__ __forceinline__ float4 quad(int n, int k) const { return n < N && k < K ? ldq(gq + (size_t)k * N + n) : make_float4(0.f, 0.f, 0.f, 0.f); }
};

// Epilogues: four consecutive N of row m
struct OutCouple {                            // out = partner + sign*acc (sign 0: plain store); out / partner may be split pairs
    static constexpr bool kTransposed = false;
    Pair out, partner; int sign;
    __device__ __forceinline__ void store(size_t row, int n, float4 v) const { out.couple4(row, n, v, partner, sign); }
    // the first `live` (one to eight) of eight rows `step` apart, columns n and n + 1; the partner's loads leave before the first
    // store (it may be in place), those of the other rows repeat row 0
    __device__ __forceinline__ void store8(size_t row, int step, int live, int n, const float (&v)[8][2]) const {
        float2 p[8];
        if (sign)
#pragma unroll
            for (int r = 0; r < 8; r++) p[r] = *reinterpret_cast<const float2 *>(partner.at(row + (size_t)(r < live ? r : 0) * step, n));
#pragma unroll
        for (int r = 0; r < 8; r++)
            if (r < live) out.couple2_with(row + (size_t)r * step, n, make_float2(v[r][0], v[r][1]), p[r], sign);
    }
};
struct OutPlain {
    static constexpr bool kTransposed = false;
    float *out; int N;
    __device__ __forceinline__ void store(size_t row, int n, float4 v) const { *reinterpret_cast<float4 *>(out + row * N + n) = v; }
    __device__ __forceinline__ void store8(size_t row, int step, int live, int n, const float (&v)[8][2]) const {
#pragma unroll
        for (int r = 0; r < 8; r++)
            if (r < live) *reinterpret_cast<float2 *>(out + (row + (size_t)r * step) * N + n) = make_float2(v[r][0], v[r][1]);
    }
};
struct OutSplit {                             // slice z of a split reduction: four consecutive M of column n, out[z][n][M]
    static constexpr bool kTransposed = true;
    float *out; int M; size_t slice;
    __device__ __forceinline__ void store(int n, int m, float4 v, int z) const { *reinterpret_cast<float4 *>(out + z * slice + (size_t)n * M + m) = v; }
};

template <int WM, int WN, int WK> struct GemmTile {
    static constexpr int BM = 64 * WM, BN = 16 * WN, BK = 16, PA = BM + 4, PB = BN + 4, kStage = BK * (PA + PB);
    static constexpr int kReduce = (WK - 1) * WM * WN * 1024;
    static constexpr int kSmem = (2 * kStage > kReduce ? 2 * kStage : kReduce) * 4;
    static_assert(WM * WN * WK == 8, "eight warps");
};

constexpr int kRun = 16;            // chunks of 16
// (127 registers, two CTAs per SM; the weight gradient of at most 16 output channels spills 52 bytes)
template <int WM, int WN, int WK, class AL, class BL, class EP>
__global__ void __launch_bounds__(256, 2) conv_gemm_kernel(AL al, BL bl, EP ep, int M, int N, int K, int k_per_split) {
    pdl_enter();
    using T = GemmTile<WM, WN, WK>;
    constexpr int BM = T::BM, BN = T::BN, BK = T::BK, PA = T::PA, PB = T::PB;
    constexpr int NA = BM / 64;               // A quads a thread loads per chunk
    extern __shared__ float sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lm = lane >> 2, ln = lane & 3;
    const int wk = warp % WK, wn = (warp / WK) % WN, wm = warp / (WK * WN);
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    const int kbeg = blockIdx.z * k_per_split, kend = kbeg + k_per_split < K ? kbeg + k_per_split : K;
    // this thread's A quads: along K, row tid % BM and K quads tid / BM + i * (256 / BM); along M, row quad tid % (BM / 4)
    const int am = AL::kAlongK ? tid % BM : (tid % (BM / 4)) * 4;
    const int ak = AL::kAlongK ? (tid / BM) * 4 : tid / (BM / 4);
    constexpr int AKS = AL::kAlongK ? (BM < 256 ? 1024 / BM : 4) : 1024 / BM;      // K step between the quads of a thread
    const bool b_on = tid < BN * 4;
    const int bn = BL::kAlongK ? tid % BN : (tid % (BN / 4)) * 4;
    const int bk = BL::kAlongK ? (tid / BN) * 4 : tid / (BN / 4);
    const RowAt ra = al.row(m0 + am);
    float4 va[NA], vb;
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < NA; i++) va[i] = k0 + ak + i * AKS < kend ? al.quad(ra, k0 + ak + i * AKS) : make_float4(0.f, 0.f, 0.f, 0.f);
        vb = b_on && k0 + bk < kend ? bl.quad(n0 + bn, k0 + bk) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto put = [&](float *As, float *Bs) {
#pragma unroll
        for (int i = 0; i < NA; i++) {
            const int k = ak + i * AKS;
            if (AL::kAlongK) { As[k * PA + am] = va[i].x; As[(k + 1) * PA + am] = va[i].y; As[(k + 2) * PA + am] = va[i].z; As[(k + 3) * PA + am] = va[i].w; }
            else *reinterpret_cast<float4 *>(As + k * PA + am) = va[i];
        }
        if (b_on) {
            if (BL::kAlongK) { Bs[bk * PB + bn] = vb.x; Bs[(bk + 1) * PB + bn] = vb.y; Bs[(bk + 2) * PB + bn] = vb.z; Bs[(bk + 3) * PB + bn] = vb.w; }
            else *reinterpret_cast<float4 *>(Bs + bk * PB + bn) = vb;
        }
    };
    float acc[8][4], sum[8][4];               // products of the current run of kRun chunks; sum of the runs before it
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = sum[i][j] = 0.f;
    auto next_chunk = [&](int k) { while (k < kend && al.skip(m0, m0 + BM - 1, k)) k += BK; return k; };
    int k0 = next_chunk(kbeg), buf = 0, run = 0;
    if (k0 < kend) { fetch(k0); put(sm, sm + BK * PA); }
    __syncthreads();
    while (k0 < kend) {
        const int kn = next_chunk(k0 + BK);
        if (kn < kend) fetch(kn);
        const float *As = sm + buf * T::kStage + wm * 64 + lm * 4, *Bs = sm + buf * T::kStage + BK * PA + wn * 16 + ln * 4;
#pragma unroll
        for (int kk = 0; kk < BK / WK; kk++) {
            const int k = wk * (BK / WK) + kk;
            const float4 a0 = *reinterpret_cast<const float4 *>(As + k * PA), a1 = *reinterpret_cast<const float4 *>(As + k * PA + 32);
            const float4 b = *reinterpret_cast<const float4 *>(Bs + k * PB);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
            for (int i = 0; i < 8; i++) {
                acc[i][0] = fmaf(a[i], b.x, acc[i][0]); acc[i][1] = fmaf(a[i], b.y, acc[i][1]);
                acc[i][2] = fmaf(a[i], b.z, acc[i][2]); acc[i][3] = fmaf(a[i], b.w, acc[i][3]);
            }
        }
        if (++run == kRun) {
            run = 0;
#pragma unroll
            for (int i = 0; i < 8; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) { sum[i][j] += acc[i][j]; acc[i][j] = 0.f; }
        }
        buf ^= 1;
        if (kn < kend) put(sm + buf * T::kStage, sm + buf * T::kStage + BK * PA);
        __syncthreads();
        k0 = kn;
    }
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] += sum[i][j];
    if (WK > 1) {
        // the warps that share a tile are added in order
        float *red = sm + (size_t)(wm * WN + wn) * 1024 + lane * 4;
        if (wk > 0)
#pragma unroll
            for (int i = 0; i < 8; i++)
                *reinterpret_cast<float4 *>(red + (size_t)(wk - 1) * WM * WN * 1024 + i * 128) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        __syncthreads();
        if (wk > 0) return;
        for (int w = 0; w < WK - 1; w++)
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const float4 v = *reinterpret_cast<const float4 *>(red + (size_t)w * WM * WN * 1024 + i * 128);
                acc[i][0] += v.x; acc[i][1] += v.y; acc[i][2] += v.z; acc[i][3] += v.w;
            }
    }
    const int n = n0 + wn * 16 + ln * 4;
    if constexpr (EP::kTransposed) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int m = m0 + wm * 64 + h * 32 + lm * 4;
            if (m < M)
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (n + j < N) ep.store(n + j, m, make_float4(acc[4 * h][j], acc[4 * h + 1][j], acc[4 * h + 2][j], acc[4 * h + 3][j]), blockIdx.z);
        }
    } else if (n < N) {
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int m = m0 + wm * 64 + (i >> 2) * 32 + lm * 4 + (i & 3);
            if (m < M) ep.store(al.out_row(m), n, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
        }
    }
}

template <int WM, int WN, int WK, class AL, class BL, class EP>
static void launch_tile(Exec &ex, AL al, BL bl, EP ep, int M, int N, int K, int splits, int k_per_split) {
    using T = GemmTile<WM, WN, WK>;
    static OncePerDevice once;
    if (T::kSmem > 48 * 1024 && once.first(ex.ctx->device))
        cudaFuncSetAttribute(conv_gemm_kernel<WM, WN, WK, AL, BL, EP>, cudaFuncAttributeMaxDynamicSharedMemorySize, T::kSmem);
    launch(ex, conv_gemm_kernel<WM, WN, WK, AL, BL, EP>, dim3((M + T::BM - 1) / T::BM, (N + T::BN - 1) / T::BN, splits), 256, T::kSmem, al, bl, ep, M, N, K, k_per_split);
}
// Tile of a forward / data-gradient GEMM (M = pixels): N tile as wide as the layer up to 64; the tallest M tile that still
// gives every SM two CTAs (the warps it does not need for rows share the K range instead)
template <class AL, class BL, class EP>
static void launch_pixels(Exec &ex, AL al, BL bl, EP ep, int M, int N, int K) {
    const long want = 2l * ex.ctx->sm_count;
    const int nt = (N + 63) / 64;
    if (N <= 16) {
        if ((M + 255) / 256 >= want) launch_tile<4, 1, 2>(ex, al, bl, ep, M, N, K, 1, K);
        else launch_tile<1, 1, 8>(ex, al, bl, ep, M, N, K, 1, K);
    } else if (N <= 32) {
        if ((M + 255) / 256 >= want) launch_tile<4, 2, 1>(ex, al, bl, ep, M, N, K, 1, K);
        else launch_tile<1, 2, 4>(ex, al, bl, ep, M, N, K, 1, K);
    } else if ((long)((M + 127) / 128) * nt >= want) launch_tile<2, 4, 1>(ex, al, bl, ep, M, N, K, 1, K);
    else if ((long)((M + 63) / 64) * nt >= ex.ctx->sm_count) launch_tile<1, 4, 2>(ex, al, bl, ep, M, N, K, 1, K);
    else launch_tile<1, 2, 4>(ex, al, bl, ep, M, N, K, 1, K);
}

// ------------------------------------------------------------------ 3x3 stride 1, forward and data gradient: direct
// out[p, n] = sum over taps and channels r of in[p + tap, r] * w[n][tap][r] with the input tile staged once, halo included,
// instead of once per tap (the implicit GEMM above spends half its instructions on that).
// A warp takes 8 rows x 4 columns of an image and 16 output channels: a lane one column, two output channels, eight rows.  Per
// channel quad and column tap a lane reads ten input quads (eight rows and the halo, shared by the three row taps) and six weight
// quads for 192 FMAs: 16 wavefronts of shared memory.  (Packed pairs, fma.rn.f32x2, reach 43.6 TFLOP/s here where single FMAs
// reach 56, and need a second partial sum per output.)
// A CTA is NW warps: CB groups of 16 output channels, NW / CB of those tiles (gx columns x gy rows x the rest images).  The input
// channels are staged in chunks of up to 32 (pixel pitch: an odd number of quads, so that the four columns of a warp and their
// 16-byte reads fall into different banks) by asynchronous copies into two buffers, the next chunk or tile while this one is
// worked on; the sums of a chunk, at most 288 products each, are added to the running sums.
// Bound by the FMA pipes, with about half of the time outside them: the start of a launch with one to four tiles per SM, the
// copies' address arithmetic, and (8x8 images) too few warps.  Measured at batch 128, whole launches: 16 channels at 32x32
// 33 -> 21 us, 32 at 16x16 41 -> 21 us, 56 at 8x8 41 -> 32 us against the implicit GEMM above.
// four channels r .. r + 3 of tap `tap` (of the sum above) for output n; forward: W[n][tap][r], data gradient: W[r][8 - tap][n]
struct DirectFprop {
    static constexpr bool kAlongK = true;
    const float *w; int Ci;
    __device__ __forceinline__ float4 along(int n, int tap, int r) const { return ldq(w + ((size_t)n * 9 + tap) * Ci + r); }
};
struct DirectDgrad {
    static constexpr bool kAlongK = false;
    const float *w; int Co;
    __device__ __forceinline__ float4 along(int n, int tap, int r) const { return ldq(w + ((size_t)r * 9 + 8 - tap) * Co + n); }     // n .. n + 3
};
// weights of a chunk in shared memory: [tap][quad of r][output n of the CTA, in each 16 the even ones first][4]
__device__ __forceinline__ int direct_slot(int n) { return (n & ~15) | ((n & 1) << 3) | ((n & 15) >> 1); }

template <class WL, class EP>
__global__ void __launch_bounds__(256, 2) conv3x3_direct_kernel(const float *__restrict__ in, WL wl, EP ep, const __grid_constant__ DirectGeom g) {
    extern __shared__ float sm[];
    const int tid = threadIdx.x, nth = blockDim.x, warp = tid >> 5, lane = tid & 31, lx = lane & 3, lg = lane >> 2;
    const int wpx = g.NW / g.CB, wt = warp % wpx, wc = warp / wpx;                  // tile and channel group of this warp
    const int wx = wt % g.gx, wy = (wt / g.gx) % g.gy, wi = wt / (g.gx * g.gy);
    const int cols = g.gx * 4 + 2, rows = g.gy * 8 + 2, nb = g.CB * 16, n0 = blockIdx.y * nb;
    const int quads = g.kc / 4, positions = rows * cols * g.gi, buf_floats = positions * g.pitch;
    float *acts = sm + 9 * g.kc * nb;
    const int at0 = ((wi * rows + wy * 8) * cols + wx * 4 + lx) * g.pitch;
    const float *myw = sm + wc * 64 + lg * 4;
    const int rowp = cols * g.pitch;
    pdl_enter();
    int x0, y0, i0;
    auto place = [&](int t) {
        uint32_t r0, bx, by, bi;
        g.dtx.divmod((uint32_t)t, r0, bx); g.dty.divmod(r0, bi, by);
        x0 = (int)bx * g.gx * 4; y0 = (int)by * g.gy * 8; i0 = (int)bi * g.gi;
    };
    // chunk c0 of tile t into buffer b; zeros outside the image and beyond the last channel
    auto stage = [&](int t, int c0, int b) {
        place(t);
        float *dst = acts + b * buf_floats;
        for (int e = tid; e < positions * quads; e += nth) {
            uint32_t pos, q, row, col, img, ry;
            g.dq.divmod((uint32_t)e, pos, q); g.dcol.divmod(pos, row, col); g.drow.divmod(row, img, ry);
            const int x = x0 + (int)col - 1, y = y0 + (int)ry - 1, i = i0 + (int)img;
            const bool ok = (unsigned)x < (unsigned)g.W && (unsigned)y < (unsigned)g.H && i < g.N && c0 + (int)q * 4 < g.Ci;
            const float *src = in + (ok ? (((size_t)i * g.H + y) * g.W + x) * g.Ci + c0 + q * 4 : 0);
            const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + (size_t)pos * g.pitch + q * 4);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
        }
    };
    int t = blockIdx.x, c0 = 0, b = 0;
    bool weights = true;
    float sum[8][2];
#pragma unroll
    for (int r = 0; r < 8; r++) sum[r][0] = sum[r][1] = 0.f;
    if (t < g.tiles) stage(t, 0, 0);
    while (t < g.tiles) {
        const int cq = (g.Ci - c0 < g.kc ? g.Ci - c0 : g.kc) / 4;                   // quads of this chunk
        __syncthreads();                                                            // the chunk before has been read
        if (weights) {
            if (WL::kAlongK) {
                for (int e = tid; e < 9 * nb * quads; e += nth) {
                    uint32_t k, q; g.dq.divmod((uint32_t)e, k, q);
                    const int tap = (int)k % 9, n = (int)k / 9;
                    const float4 v = n0 + n < g.Co && (int)q < cq ? wl.along(n0 + n, tap, c0 + (int)q * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
                    *reinterpret_cast<float4 *>(sm + ((size_t)(tap * quads + (int)q) * nb + direct_slot(n)) * 4) = v;
                }
            } else {
                const int nq = nb / 4;
                for (int e = tid; e < 9 * g.kc * nq; e += nth) {
                    const int n = e % nq * 4, k = e / nq, tap = k % 9, r = k / 9;
                    const float4 v = n0 + n < g.Co && c0 + r < g.Ci ? wl.along(n0 + n, tap, c0 + r) : make_float4(0.f, 0.f, 0.f, 0.f);
                    float *d = sm + (size_t)(tap * quads + r / 4) * nb * 4 + (r & 3);
                    d[direct_slot(n) * 4] = v.x; d[direct_slot(n + 1) * 4] = v.y; d[direct_slot(n + 2) * 4] = v.z; d[direct_slot(n + 3) * 4] = v.w;
                }
            }
            weights = g.kc < g.Ci;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        int tn = t, cn = c0 + g.kc;
        if (cn >= g.Ci) { tn += gridDim.x; cn = 0; }
        if (tn < g.tiles) stage(tn, cn, b ^ 1);
        const float *myact = acts + b * buf_floats + at0;
        float acc[8][2];
#pragma unroll
        for (int r = 0; r < 8; r++) acc[r][0] = acc[r][1] = 0.f;
#pragma unroll 1
        for (int q = 0; q < cq; q++) {
#pragma unroll
            for (int kw = 0; kw < 3; kw++) {
                float4 a[10];
#pragma unroll
                for (int r = 0; r < 10; r++) a[r] = *reinterpret_cast<const float4 *>(myact + r * rowp + kw * g.pitch + q * 4);
#pragma unroll
                for (int kh = 0; kh < 3; kh++) {
                    const float *w = myw + (size_t)((kh * 3 + kw) * quads + q) * nb * 4;
                    const float4 w0 = *reinterpret_cast<const float4 *>(w), w1 = *reinterpret_cast<const float4 *>(w + 32);
#pragma unroll
                    for (int r = 0; r < 8; r++) { acc[r][0] = fmaf(a[r + kh].x, w0.x, acc[r][0]); acc[r][1] = fmaf(a[r + kh].x, w1.x, acc[r][1]); }
#pragma unroll
                    for (int r = 0; r < 8; r++) { acc[r][0] = fmaf(a[r + kh].y, w0.y, acc[r][0]); acc[r][1] = fmaf(a[r + kh].y, w1.y, acc[r][1]); }
#pragma unroll
                    for (int r = 0; r < 8; r++) { acc[r][0] = fmaf(a[r + kh].z, w0.z, acc[r][0]); acc[r][1] = fmaf(a[r + kh].z, w1.z, acc[r][1]); }
#pragma unroll
                    for (int r = 0; r < 8; r++) { acc[r][0] = fmaf(a[r + kh].w, w0.w, acc[r][0]); acc[r][1] = fmaf(a[r + kh].w, w1.w, acc[r][1]); }
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 8; r++) { sum[r][0] += acc[r][0]; sum[r][1] += acc[r][1]; }
        if (tn != t) {
            place(t);
            const int n = n0 + wc * 16 + 2 * lg, x = x0 + wx * 4 + lx, y = y0 + wy * 8, i = i0 + wi;
            const int live = direct_live_rows(g, n, x, y, i);
            if (live > 0) ep.store8(((size_t)i * g.H + y) * g.W + x, g.W, live, n, sum);
#pragma unroll
            for (int r = 0; r < 8; r++) sum[r][0] = sum[r][1] = 0.f;
        }
        t = tn; c0 = cn; b ^= 1;
    }
}

template <class WL, class EP>
static void launch_direct(Exec &ex, const float *in, WL wl, EP ep, const DirectGeom &g) {
    const int smem = (9 * g.kc * g.CB * 16 + 2 * (g.gx * 4 + 2) * (g.gy * 8 + 2) * g.gi * g.pitch) * 4;      // at most 157 KB
    static OncePerDevice once;
    if (once.first(ex.ctx->device)) cudaFuncSetAttribute(conv3x3_direct_kernel<WL, EP>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    const int nbs = (g.Co + g.CB * 16 - 1) / (g.CB * 16);
    int per_sm = 16 / g.NW, fit = 227 * 1024 / (smem + 1024);
    if (per_sm > fit) per_sm = fit;
    int ctas = ex.ctx->sm_count * per_sm / nbs; if (ctas < 1) ctas = 1;
    const int rounds = (g.tiles + ctas - 1) / ctas;
    launch(ex, conv3x3_direct_kernel<WL, EP>, dim3((g.tiles + rounds - 1) / rounds, nbs), g.NW * 32, smem, in, wl, ep, g);
}

// ------------------------------------------------------------------ any channel count, element by element
// ---- operand loaders: element (m,k) of A and (k,n) of B of the implicit GEMM
template <class TA> struct AnyFpropA {           // m = output pixel, k = (kh,kw,ci)
    const TA *a; ConvGeom g;
    static constexpr bool k_fast = true;
    __device__ float operator()(int m, int kk) const {
        int wo = m % g.Wo, t = m / g.Wo, ho = t % g.Ho, n = t / g.Ho;
        int ci = kk % g.Ci, tap = kk / g.Ci, kw = tap % g.k, kh = tap / g.k;
        int y = ho * g.s + kh - g.pad, x = wo * g.s + kw - g.pad;
        if (y < 0 || y >= g.H || x < 0 || x >= g.W) return 0.f;
        return ldf(a + (((size_t)n * g.H + y) * g.W + x) * g.Ci + ci);
    }
};
struct AnyFpropB {                               // k = (kh,kw,ci), n = co ; W[co][kh][kw][ci]
    const float *w; int K; bool wb;           // wb: weights take part as bf16 values (mode 0)
    static constexpr bool k_fast = true;
    __device__ float operator()(int kk, int n) const { return round_w(w[(size_t)n * K + kk], wb); }
};
template <class TG> struct AnyWgradA {           // m = co, k = output pixel
    const TG *gq; ConvGeom g;
    static constexpr bool k_fast = false;
    __device__ float operator()(int m, int kk) const { return ldf(gq + (size_t)kk * g.Co + m); }
};
template <class TA> struct AnyWgradB {           // k = output pixel, n = (kh,kw,ci)
    const TA *a; ConvGeom g;
    static constexpr bool k_fast = false;
    __device__ float operator()(int kk, int n) const {
        int wo = kk % g.Wo, t = kk / g.Wo, ho = t % g.Ho, b = t / g.Ho;
        int ci = n % g.Ci, tap = n / g.Ci, kw = tap % g.k, kh = tap / g.k;
        int y = ho * g.s + kh - g.pad, x = wo * g.s + kw - g.pad;
        if (y < 0 || y >= g.H || x < 0 || x >= g.W) return 0.f;
        return ldf(a + (((size_t)b * g.H + y) * g.W + x) * g.Ci + ci);
    }
};

// ---- epilogues
struct EpiCouple {                            // out = partner + sign*acc (sign 0: plain store); out/partner may be split pairs
    Pair out, partner; int sign;
    __device__ void operator()(int m, int n, float v, int) const { out.couple(m, n, v, partner, sign); }
};
struct EpiPlain {                             // row-major [M][N] (+ split-K slice)
    float *out; int N; size_t slice;
    __device__ void operator()(int m, int n, float v, int z) const { out[z * slice + (size_t)m * N + n] = v; }
};

template <int BN, class AL, class BL, class EP>
__global__ __launch_bounds__(256) void gemm_simt_kernel(AL al, BL bl, EP ep, int M, int N, int K, int k_per_split) {
    pdl_enter();
    constexpr int BM = 64, BK = 16, TN = BN / 16;
    __shared__ float As[BK][BM + 1];
    __shared__ float Bs[BK][BN + 1];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    const int kbeg = blockIdx.z * k_per_split;
    int kend = kbeg + k_per_split; if (kend > K) kend = K;
    float acc[4][TN];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < TN; j++) acc[i][j] = 0.f;

    for (int k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
        for (int i = 0; i < (BM * BK) / 256; i++) {
            int e = tid + i * 256, mm, kk;
            if (AL::k_fast) { kk = e % BK; mm = e / BK; } else { mm = e % BM; kk = e / BM; }
            As[kk][mm] = (m0 + mm < M && k0 + kk < kend) ? al(m0 + mm, k0 + kk) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < (BN * BK + 255) / 256; i++) {
            int e = tid + i * 256, nn, kk;
            if (BL::k_fast) { kk = e % BK; nn = e / BK; } else { nn = e % BN; kk = e / BN; }
            if (e < BN * BK) Bs[kk][nn] = (n0 + nn < N && k0 + kk < kend) ? bl(k0 + kk, n0 + nn) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; kk++) {
            float a[4], b[TN];
#pragma unroll
            for (int i = 0; i < 4; i++) a[i] = As[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < TN; j++) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < TN; j++) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < TN; j++) {
            int m = m0 + ty * 4 + i, n = n0 + tx + 16 * j;
            if (m < M && n < N) ep(m, n, acc[i][j], blockIdx.z);
        }
}

template <class AL, class BL, class EP>
static void launch_gemm(Exec &ex, const char *what, AL al, BL bl, EP ep, int M, int N, int K, int splits, int k_per_split,
                        double bytes) {
    if (N <= 16) {
        dim3 grid((M + 63) / 64, (N + 15) / 16, splits);
        launch(ex, gemm_simt_kernel<16, AL, BL, EP>, grid, 256, 0, al, bl, ep, M, N, K, k_per_split);
    } else if (N <= 32) {
        dim3 grid((M + 63) / 64, (N + 31) / 32, splits);
        launch(ex, gemm_simt_kernel<32, AL, BL, EP>, grid, 256, 0, al, bl, ep, M, N, K, k_per_split);
    } else {
        dim3 grid((M + 63) / 64, (N + 63) / 64, splits);
        launch(ex, gemm_simt_kernel<64, AL, BL, EP>, grid, 256, 0, al, bl, ep, M, N, K, k_per_split);
    }
    ex.check(what, bytes, 2.0 * M * N * (double)K);
}

static ConvGeom geom_of(Geom gi, const Layer &L) {
    ConvGeom g;
    g.N = gi.N; g.H = gi.H; g.W = gi.W; g.Ci = L.cin; g.Co = L.cout; g.k = L.k; g.s = L.stride; g.pad = L.k / 2;
    g.Ho = conv_out(gi.H, L.k, L.stride); g.Wo = conv_out(gi.W, L.k, L.stride);
    return g;
}

void conv_fprop_simt(Exec &ex, const void *a, bool a_bf16, Geom gi, const Layer &L, Pair out, Pair partner, int sign) {
    ConvGeom g = geom_of(gi, L);
    const int M = g.N * g.Ho * g.Wo, N = g.Co, K = g.k * g.k * g.Ci;
    ex.flops += 2ull * M * N * K;
    if (ex.dry) return;
    const double bytes = (double)g.N * g.H * g.W * g.Ci * (a_bf16 ? 2 : 4) + (double)M * N * (sign ? 8 : 4) + (double)N * K * 4;
    if (g.Ci % 4) {
        EpiCouple ep{out, partner, sign};
        AnyFpropB bl{L.W, K, a_bf16};
        if (a_bf16) launch_gemm(ex, "conv_fprop_simt", AnyFpropA<bf16>{(const bf16 *)a, g}, bl, ep, M, N, K, 1, K, bytes);
        else launch_gemm(ex, "conv_fprop_simt", AnyFpropA<float>{(const float *)a, g}, bl, ep, M, N, K, 1, K, bytes);
        return;
    }
    const FastDiv wo = fast_div(g.Wo), ho = fast_div(g.Ho), ci = fast_div(g.Ci), kk = fast_div(g.k);
    const OutCouple ep{out, partner, sign};
    DirectGeom d;
    if (g.k == 3 && g.s == 1 && !a_bf16 && direct_shape(g.N, g.H, g.W, g.Ci, g.Co, ex.ctx->sm_count, d)) {
        launch_direct(ex, (const float *)a, DirectFprop{L.W, g.Ci}, ep, d);
        ex.check("conv_fprop_direct", bytes, 2.0 * M * N * (double)K);
        return;
    }
    const FpropB bl{L.W, N, K, a_bf16};
    if (a_bf16) launch_pixels(ex, FpropA<bf16>{(const bf16 *)a, g, wo, ho, ci, kk, M, K}, bl, ep, M, N, K);
    else launch_pixels(ex, FpropA<float>{(const float *)a, g, wo, ho, ci, kk, M, K}, bl, ep, M, N, K);
    ex.check("conv_fprop_gemm", bytes, 2.0 * M * N * (double)K);
}

void conv_dgrad_simt(Exec &ex, const void *gq, bool g_bf16, Geom gi, const Layer &L, float *da) {
    ConvGeom g = geom_of(gi, L);
    const int M = g.N * g.H * g.W, N = g.Ci, K = g.k * g.k * g.Co;
    ex.flops += 2ull * g.N * g.Ho * g.Wo * N * K;
    if (ex.dry) return;
    const double bytes = (double)g.N * g.Ho * g.Wo * g.Co * (g_bf16 ? 2 : 4) + (double)M * N * 4 + (double)N * K * 4;
    const OutPlain ep{da, N};
    DirectGeom d;
    if (g.k == 3 && g.s == 1 && !g_bf16 && g.Ci % 4 == 0 && direct_shape(g.N, g.H, g.W, g.Co, g.Ci, ex.ctx->sm_count, d)) {
        launch_direct(ex, (const float *)gq, DirectDgrad{L.W, g.Ci}, ep, d);
        ex.check("conv_dgrad_direct", bytes, 2.0 * g.N * g.Ho * g.Wo * N * (double)K);
        return;
    }
    // stride 2: parity classes of (H + 1) / 2 x (W + 1) / 2 pixels would be ragged on odd sizes; those keep the plain numbering
    const bool classes = g.s == 2 && g.H % 2 == 0 && g.W % 2 == 0;
    const FastDiv w = fast_div(classes ? g.W / 2 : g.W), h = fast_div(classes ? g.H / 2 : g.H), co = fast_div(g.Co), kk = fast_div(g.k);
    const FastDiv cls = fast_div(classes ? M / 4 : (uint32_t)M);
    const DgradB bl{L.W, co, g.k * g.k, N, K, g_bf16};
    if (g_bf16) launch_pixels(ex, DgradA<bf16>{(const bf16 *)gq, g, w, h, co, kk, cls, classes, M, K}, bl, ep, M, N, K);
    else launch_pixels(ex, DgradA<float>{(const float *)gq, g, w, h, co, kk, cls, classes, M, K}, bl, ep, M, N, K);
    ex.check("conv_dgrad_gemm", bytes, 2.0 * g.N * g.Ho * g.Wo * N * (double)K);
}

// fixed-order sum of split-K slices: a block takes 32 elements, eight threads each (every eighth slice), added in order
__global__ void splitk_reduce_kernel(const float *__restrict__ part, size_t n, int splits, float *__restrict__ out) {
    pdl_enter();
    __shared__ float sm[8][33];
    const int e = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const size_t i = (size_t)blockIdx.x * 32 + e;
    float s = 0.f;
    if (i < n)
#pragma unroll 4
        for (int z = grp; z < splits; z += 8) s += part[(size_t)z * n + i];
    sm[grp][e] = s;
    __syncthreads();
    if (grp == 0 && i < n) {
        for (int g = 1; g < 8; g++) s += sm[g][e];
        out[i] = s;
    }
}

// ------------------------------------------------------------------ weight gradient of fp32 3x3 stride-1 layers
// dW[co, (kh, kw), ci] = sum over pixels of g[y, x, co] a[y + kh - 1, x + kw - 1, ci], of at most 64 channels on either
// side and 144 pairs of channel quads (48 -> 48, 36 -> 64).
// A lane keeps four input channels x four output channels x the three column taps of one row tap: walking along a row of the image
// it reads one new quad of either tensor per pixel (the window of three input quads slides in registers) for 48 FMAs, where the
// implicit GEMM above reads three per 32 and works out the pixel of every quad that it stages.
// Warps: 3 row taps x nb blocks of 32 (input quad, output quad) pairs x R groups of rows; with at most 16 pairs a warp holds sl rows of
// them.  The rows of a strip (BH rows of an image, and the halo rows of the input) arrive by asynchronous copies in two
// buffers; the slices' sums are added through shared memory at the end, in order, and the CTAs' by splitk_reduce_kernel.
// Sums.  A lane adds at most kWgStripRun products in a row, then the sum of that run to a second set of registers (one CTA of 384 to 480
// threads per SM has them): rms error of dW against the runs of the implicit GEMM 0.98 (16 channels at 32x32, batch 128), 0.96
// (batch 256), 0.89 (32 channels at 16x16), 0.91 and 0.82 (40 and 48 channels at 32x32); serial sums of 64 to 480 products had 1.1 to 1.9.
// Bound by the FMA pipes, and by launch, first copies and the two reductions for a third of the time.  Block forward and backward, one layer per
// function, against the implicit GEMM: 16 channels at 32x32, batch 128, 328 -> 267 us, batch 256 602 -> 462; 8 channels 229 -> 173; 48 channels
// 1940 -> 1845; 32 channels at 16x16 267 -> 265; fp32 step of the 38-layer network 5.61 -> 5.18 ms.
__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void wg_fma(float (&acc)[16], const float4 &a, const float4 &g) {
    const float av[4] = {a.x, a.y, a.z, a.w}, gv[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[4 * j + i] = fmaf(av[i], gv[j], acc[4 * j + i]);
}
__global__ void __launch_bounds__(kWgStripThreads, 1) wgrad3x3_strip_kernel(const float *__restrict__ a, const float *__restrict__ g, float *__restrict__ part, const WgStrip p) {
    extern __shared__ float4 wg_smem[];
    float *buf = reinterpret_cast<float *>(wg_smem);
    pdl_enter();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
    const int s0 = blockIdx.x * p.per_cta, s1 = s0 + p.per_cta < p.strips ? s0 + p.per_cta : p.strips;
    const int stage = p.a_floats + p.g_floats, a_pitch = (p.W + 2) * p.Ci, g_pitch = p.W * p.Co;
    auto place = [&](int s, int &n, int &y0, int &rows) {
        uint32_t img, r;
        p.dimg.divmod((uint32_t)s, img, r);
        n = (int)img; y0 = (int)r * p.BH; rows = p.H - y0 < p.BH ? p.H - y0 : p.BH;
    };
    auto fetch = [&](int s, float *dst) {
        int n, y0, rows;
        place(s, n, y0, rows);
        const int na = (rows + 2) * (p.W + 2) * p.cq, ng = rows * p.W * p.oq;
        for (int i = tid; i < na; i += nt) {
            uint32_t t, q, r, x;
            p.dcq.divmod((uint32_t)i, t, q);
            p.dw2.divmod(t, r, x);
            const int yy = y0 + (int)r - 1, xx = (int)x - 1;
            const bool ok = (unsigned)yy < (unsigned)p.H && (unsigned)xx < (unsigned)p.W;
            cp_async16(dst + i * 4, ok ? a + (((size_t)n * p.H + yy) * p.W + xx) * p.Ci + q * 4 : a, ok);
        }
        const float *gs = g + ((size_t)n * p.H + y0) * p.W * p.Co;
        for (int i = tid; i < ng; i += nt) cp_async16(dst + p.a_floats + i * 4, gs + i * 4, true);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // this thread's work: row tap, pair of quads, slice of the rows
    const int kh = warp % 3;
    uint32_t rg, blk;
    p.dnb.divmod((uint32_t)(warp / 3), rg, blk);
    uint32_t sub = 0, pair = blk * 32 + lane;
    if (p.sl > 1) p.dpairs.divmod((uint32_t)lane, sub, pair);
    const bool active = (int)pair < p.pairs && (int)sub < p.sl;
    uint32_t oq, cq;
    p.dcq.divmod(pair, oq, cq);
    const int slice = (int)rg * p.sl + (int)sub, slices = p.R * p.sl;
    float acc[3][16], sum[3][16];            // products of the current run; sum of the runs before it
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
        for (int i = 0; i < 16; i++) acc[k][i] = sum[k][i] = 0.f;
    int run = 0;
    auto flush = [&]() {
        run = 0;
#pragma unroll
        for (int k = 0; k < 3; k++)
#pragma unroll
            for (int i = 0; i < 16; i++) { sum[k][i] += acc[k][i]; acc[k][i] = 0.f; }
    };
    fetch(s0, buf);
    for (int s = s0; s < s1; s++) {
        float *cur = buf + ((s - s0) & 1) * stage;
        if (s + 1 < s1) {
            fetch(s + 1, buf + ((s + 1 - s0) & 1) * stage);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        int n, y0, rows;
        place(s, n, y0, rows);
        if (active)
            for (int r = slice; r < rows; r += slices) {
                const float *pa = cur + (r + kh) * a_pitch + cq * 4, *pg = cur + p.a_floats + r * g_pitch + oq * 4;
                float4 a0 = *reinterpret_cast<const float4 *>(pa), a1 = *reinterpret_cast<const float4 *>(pa + p.Ci), a2;
                pa += 2 * p.Ci;
#pragma unroll 1
                for (int x = 0, end; x < p.W; x = end) {
                    end = x + kWgStripRun < p.W ? x + kWgStripRun : p.W;
                    if (run + end - x > kWgStripRun) flush();
                    run += end - x;
#pragma unroll 1
                    for (; x + 2 < end; x += 3) {
                        float4 gv = *reinterpret_cast<const float4 *>(pg);
                        a2 = *reinterpret_cast<const float4 *>(pa);
                        wg_fma(acc[0], a0, gv); wg_fma(acc[1], a1, gv); wg_fma(acc[2], a2, gv);
                        gv = *reinterpret_cast<const float4 *>(pg + p.Co);
                        a0 = *reinterpret_cast<const float4 *>(pa + p.Ci);
                        wg_fma(acc[0], a1, gv); wg_fma(acc[1], a2, gv); wg_fma(acc[2], a0, gv);
                        gv = *reinterpret_cast<const float4 *>(pg + 2 * p.Co);
                        a1 = *reinterpret_cast<const float4 *>(pa + 2 * p.Ci);
                        wg_fma(acc[0], a2, gv); wg_fma(acc[1], a0, gv); wg_fma(acc[2], a1, gv);
                        pa += 3 * p.Ci; pg += 3 * p.Co;
                    }
#pragma unroll 1
                    for (; x < end; x++) {
                        const float4 gv = *reinterpret_cast<const float4 *>(pg);
                        a2 = *reinterpret_cast<const float4 *>(pa);
                        wg_fma(acc[0], a0, gv); wg_fma(acc[1], a1, gv); wg_fma(acc[2], a2, gv);
                        a0 = a1; a1 = a2;
                        pa += p.Ci; pg += p.Co;
                    }
                }
            }
        __syncthreads();
    }
    flush();
    const int n_out = 9 * p.Ci * p.Co;
    float *out = part + (size_t)blockIdx.x * n_out, *dst = slices > 1 ? buf + (size_t)slice * n_out : out;
    if (active)
#pragma unroll
        for (int k = 0; k < 3; k++)
#pragma unroll
            for (int j = 0; j < 4; j++)
                *reinterpret_cast<float4 *>(dst + ((oq * 4 + j) * 9 + kh * 3 + k) * p.Ci + cq * 4) =
                    make_float4(sum[k][4 * j], sum[k][4 * j + 1], sum[k][4 * j + 2], sum[k][4 * j + 3]);
    if (slices > 1) {
        __syncthreads();
        for (int i = tid; i < n_out / 4; i += nt) {
            float4 v = reinterpret_cast<const float4 *>(buf)[i];
            for (int z = 1; z < slices; z++) {
                const float4 w = reinterpret_cast<const float4 *>(buf + (size_t)z * n_out)[i];
                v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
            }
            reinterpret_cast<float4 *>(out)[i] = v;
        }
    }
}
// dW as a GEMM of M = (tap, ci), N = co over the pixels; the pixels are split so that the grid fills the machine twice
template <class TG, class TA>
static void wgrad_launch(Exec &ex, const TG *gq, const TA *a, ConvGeom g, float *part, int splits, int kps) {
    const int M = g.k * g.k * g.Ci, N = g.Co, K = g.N * g.Ho * g.Wo;
    const WgradA<TA> al{a, g, fast_div(g.Wo), fast_div(g.Ho), fast_div(g.Ci), fast_div(g.k), M, K};
    const WgradB<TG> bl{gq, N, K};
    const OutSplit ep{part, M, (size_t)M * N};
    if (N <= 16) launch_tile<1, 1, 8>(ex, al, bl, ep, M, N, K, splits, kps);
    else if (N <= 32) launch_tile<1, 2, 4>(ex, al, bl, ep, M, N, K, splits, kps);
    else launch_tile<1, 4, 2>(ex, al, bl, ep, M, N, K, splits, kps);
}
void conv_wgrad_simt(Exec &ex, const void *gq, bool g_bf16, const void *a, bool a_bf16, Geom gi, const Layer &L, float *dW, size_t after) {
    ConvGeom g = geom_of(gi, L);
    const int Co = g.Co, KC = g.k * g.k * g.Ci, P = g.N * g.Ho * g.Wo;
    ex.flops += 2ull * Co * KC * (size_t)P;
    const bool quads = g.Ci % 4 == 0 && g.Co % 4 == 0;
    const int bn = Co <= 16 ? 16 : (Co <= 32 ? 32 : 64);
    const int tiles = quads ? ((KC + 63) / 64) * ((Co + bn - 1) / bn) : ((Co + 63) / 64) * ((KC + 63) / 64);
    int splits = (ex.ctx->sm_count * (quads ? 4 : 2) + tiles - 1) / tiles;
    int max_splits = (P + 255) / 256; if (splits > max_splits) splits = max_splits; if (splits < 1) splits = 1;
    int kps = (((P + splits - 1) / splits) + 15) / 16 * 16;
    splits = (P + kps - 1) / kps;
    // partials of strips: as many as the implicit GEMM would have, or as take no more workspace than what the caller allocates behind them
    const size_t room = after / ((size_t)Co * KC);
    const int most = (size_t)splits > room ? splits : (int)(room < (size_t)P ? room : (size_t)P);
    WgStrip st;
    int ctas, threads, smem;
    if (g.k == 3 && g.s == 1 && !g_bf16 && !a_bf16 && wg_strip_shape(g.N, g.H, g.W, g.Ci, g.Co, ex.ctx->sm_count, most, st, ctas, threads, smem)) {
        size_t m = ex.ws.mark();
        float *part = ctas > 1 ? ex.ws.get<float>((size_t)ctas * Co * KC) : dW;
        if (!ex.dry) {
            static OncePerDevice once;
            if (once.first(ex.ctx->device)) cudaFuncSetAttribute(wgrad3x3_strip_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
            launch(ex, wgrad3x3_strip_kernel, ctas, threads, smem, (const float *)a, (const float *)gq, part, st);
            ex.check("conv_wgrad_strip", (double)P * (g.Co + g.Ci) * 4 + (double)Co * KC * 4, 2.0 * Co * KC * (double)P);
            if (ctas > 1) {
                const size_t n = (size_t)Co * KC;
                launch(ex, splitk_reduce_kernel, (unsigned)((n + 31) / 32), 256, 0, part, n, ctas, dW);
                ex.check("splitk_reduce");
            }
        }
        ex.ws.release(m);
        return;
    }
    size_t m = ex.ws.mark();
    float *part = splits > 1 ? ex.ws.get<float>((size_t)splits * Co * KC) : dW;
    if (!ex.dry) {
        const double bytes = (double)P * g.Co * (g_bf16 ? 2 : 4) + (double)g.N * g.H * g.W * g.Ci * (a_bf16 ? 2 : 4) + (double)Co * KC * 4;
        if (quads && g_bf16 == a_bf16) {
            if (g_bf16) wgrad_launch(ex, (const bf16 *)gq, (const bf16 *)a, g, part, splits, kps);
            else wgrad_launch(ex, (const float *)gq, (const float *)a, g, part, splits, kps);
            ex.check("conv_wgrad_gemm", bytes, 2.0 * Co * KC * (double)P);
        } else {
            EpiPlain ep{part, KC, (size_t)Co * KC};
#define RV_WG(TG, TA) launch_gemm(ex, "conv_wgrad_simt", AnyWgradA<TG>{(const TG *)gq, g}, AnyWgradB<TA>{(const TA *)a, g}, ep, Co, KC, P, splits, kps, bytes)
            if (g_bf16 && a_bf16) RV_WG(bf16, bf16);
            else if (g_bf16) RV_WG(bf16, float);
            else if (a_bf16) RV_WG(float, bf16);
            else RV_WG(float, float);
#undef RV_WG
        }
        if (splits > 1) {
            const size_t n = (size_t)Co * KC;
            launch(ex, splitk_reduce_kernel, (unsigned)((n + 31) / 32), 256, 0, part, n, splits, dW);
            ex.check("splitk_reduce");
        }
    }
    ex.ws.release(m);
}
