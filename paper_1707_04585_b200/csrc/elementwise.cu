// HBM-bound kernels: BN batch statistics, BN+ReLU apply and backward, concat/cast, max-pool,
// classification head, SGD.  All reductions are two-stage with a fixed summation order, so a
// residual function recomputed in the backward pass reproduces the forward bit for bit.
#include "common.cuh"
#include "conv_epilogue.cuh"
#include <math.h>

cudaEvent_t revnet_ctx::next_event() {
    if (ev_used == ev_pool.size()) {
        cudaEvent_t e;
        cudaEventCreate(&e);
        ev_pool.push_back(e);
    }
    return ev_pool[ev_used++];
}

unsigned long long *Exec::stamp_slot() {
    if (dry || !ctx->stamping || !ctx->stamps || ctx->stamp_next >= kStampSlots) return nullptr;
    pending_slot = ctx->stamp_next++;
    return ctx->stamps + pending_slot;
}

void Exec::check(const char *what, double bytes, double flops) {
    launches++;
    if (pending_slot >= 0) { ctx->stamp_recs.push_back(StampRec{what, bytes, flops, pending_slot}); pending_slot = -1; }
    cudaError_t e = cudaPeekAtLastError();
    if (e != cudaSuccess && !failed) {
        failed = true;
        ctx->err = std::string(what) + ": " + cudaGetErrorString(e);
    }
    if (ctx->profiling) {
        cudaEvent_t ev = ctx->next_event();
        cudaEventRecord(ev, stream);
        ctx->prof.push_back(ProfRec{what, bytes, flops, ev});
    }
}
// Keeps the stream busy for `ns` nanoseconds (bounded) so that the host gets ahead of the device:
// the per-kernel events of a profiled step then measure kernels that were already queued, not the
// host's launch rate.
__global__ void profile_hold_kernel(unsigned long long ns) {
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (int i = 0; i < 100000; i++) {
        __nanosleep(1000);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 >= ns) break;
    }
}
void Exec::mark(const char *what) {
    if (ctx->profiling && !dry && hold_ns) {
        profile_hold_kernel<<<1, 1, 0, stream>>>(hold_ns);
        hold_ns = 0;
    }
    if (ctx->profiling && !dry) {
        cudaEvent_t ev = ctx->next_event();
        cudaEventRecord(ev, stream);
        ctx->prof.push_back(ProfRec{what, 0, 0, ev});
    }
}

static inline int cdiv(size_t a, size_t b) { return (int)((a + b - 1) / b); }

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ void st4(bf16 *p, float4 v) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    uint2 u;
    u.x = *reinterpret_cast<uint32_t *>(&lo);
    u.y = *reinterpret_cast<uint32_t *>(&hi);
    *reinterpret_cast<uint2 *>(p) = u;
}

// ------------------------------------------------------------------ column reductions
// Every per-channel reduction over a [P,C] tensor is one launch: a CTA of 256 threads owns a slab of SW <= 32 channel quads
// (512-byte row segments, or whole rows of narrow tensors) and a range of rows; threads of a slab column stride the rows
// with kRows loads in flight.  Each CTA writes a record of its slab's sums, and the CTA that finishes last in a slab adds
// the slab's records in a fixed order (double precision) and writes the results.  While it does, every other SM waits, and of
// the 592 records of a tensor of 64 to 128 channels a thread of it had 148: thirty dependent rounds of loads, 18 us.  Where that
// would take more than kTailRounds rounds, groups of consecutive CTAs of two rounds each add their own records (the last CTA
// of a group does) and the last group adds the groups' sums.
// Measured, 88 channels, 53580 pixels: 21 -> 12 us behind the kernel before (1x1 of 56 channels, 6200 pixels, 87 records: 9.0 in one level, 9.9 in two).
// Bound by HBM.  Measured (512 channels, 200704 pixels: 411 MB): 200 -> 99 us with the finalize launch gone (4.1 TB/s, 88 us
// with the whole L1;
// a row in flight per thread and a second kernel over uncoalesced partials before).
struct RedShape { int SW, RPP, slabs, chunks, rows_per_cta, group, groups; };     // group: CTAs of a group, 0: one level
constexpr int kTailRounds = 6;     // (two levels lose 1 us at four rounds and win as much at eight)
static RedShape red_shape(size_t P, int C, int sm, int rows_in_flight, int max_chunks = 0) {
    RedShape r;
    const int C4 = C / 4;
    r.slabs = cdiv(C4, 32);
    r.SW = cdiv(C4, r.slabs);
    r.RPP = 256 / r.SW;
    size_t want = (size_t)sm * 4 / r.slabs; if (want < 1) want = 1;
    if (max_chunks && want > (size_t)max_chunks) want = max_chunks;
    size_t rows = (P + want - 1) / want;
    const size_t pass = (size_t)r.RPP * rows_in_flight;       // rows of one pass over the loads in flight
    if (rows < pass) rows = pass;
    r.rows_per_cta = (int)rows;
    r.chunks = cdiv(P, rows);
    int rs = 4;
    while (rs < 2 * r.SW) rs <<= 1;
    const int round = 256 / rs * 5;                           // records of a slab that reduce_records<256> takes in a round of loads
    r.group = r.chunks > kTailRounds * round ? 2 * round : 0;
    r.groups = r.group ? cdiv(r.chunks, r.group) : 0;
    return r;
}
// floats of scratch: the records, then the groups' sums in double precision
static size_t red_floats(const RedShape &r, int C) { return (size_t)r.chunks * 2 * C + (size_t)r.groups * 4 * C; }
static dim3 red_grid(const RedShape &r) {
    const int z = cdiv(r.slabs, 65535);
    return dim3(r.chunks, cdiv(r.slabs, z), z);
}
// counter words: per slab one for the slab and one for each group; a slab of one CTA counts nothing
static int red_words(const RedShape &r) { return r.chunks > 1 ? r.slabs * (1 + r.groups) : 0; }
constexpr int kStatRows = 8, kBwdRows = 4;

// Where the result goes.  MODE 0: mean, rstd; MODE 1: dgamma, dbeta and coef[3][C] = gamma*rstd, gamma*rstd*dbeta/M, gamma*rstd*dgamma/M
struct RedOut { float *mean, *rstd, *dgamma, *dbeta, *coef; double inv_count; float eps; };
// Where the records go and who adds them
struct RedPlan {
    int SW, rows, chunks;         // quads of a slab, rows of a CTA, CTAs of a slab
    int group, groups;            // two levels: CTAs of a group, groups of a slab
    int pending;                  // the records stay: their consumer adds them
    float *part;                  // [chunk][C/4][2][4] (per channel quad: 4 sums, 4 second sums)
    double *gsum;                 // [group][C/4][2][4]
    unsigned int *counters;       // per slab 1 + groups zeroed words, left zero
};

// Grid: chunks along x, slabs along y and, beyond 65535 of them, z
// (64 registers for four CTAs per SM: 52 to 60 bytes of spills in mode 0, 92 to 96 in mode 1, around the reduction behind the loop.  Two
// kernels, because a small launch fetches every instruction of its tail anew: with both forms in one, each launch of the smallest block
// calls took 0.5 to 0.7 us longer)
template <int MODE, bool GROUPS>   // MODE 0: sum t, sum t^2 ; 1: sum db, sum db*xhat (BN+ReLU backward); GROUPS: records added in two levels
__global__ void __launch_bounds__(256, 4) col_reduce_kernel(Pair t, const float *__restrict__ da, size_t P, BnRef bn, const RedPlan pl, RedOut out) {
    pdl_enter();
    constexpr int NR = MODE == 0 ? kStatRows : kBwdRows;
    __shared__ double red[256 * 4], tot[128 * 4];
    __shared__ unsigned int last;
    const int C = t.C(), C4 = C / 4, SW = pl.SW, RPP = 256 / SW, tid = threadIdx.x;
    const int chunk = blockIdx.x, slab = blockIdx.y + blockIdx.z * gridDim.y;
    if (slab * SW >= C4) return;
    const int tx = tid % SW, ty = tid / SW, q = slab * SW + tx;
    const bool valid = q < C4 && ty < RPP;
    const size_t r0 = (size_t)chunk * pl.rows;
    size_t r1 = r0 + pl.rows; if (r1 > P) r1 = P;
    float4 s = make_float4(0, 0, 0, 0), ss = s;
    if (valid) {
        float4 sc, sh, mu, rs;
        if (MODE == 1) bn_coef4(bn, q * 4, sc, sh, mu, rs);
        for (size_t rb = r0 + ty; rb < r1; rb += (size_t)NR * RPP) {
            // all loads leave before anything waits on one: rows beyond the end read the last row again and are not added
            float4 v[NR], g[NR];
#pragma unroll
            for (int j = 0; j < NR; j++) {
                size_t row = rb + (size_t)j * RPP; if (row >= r1) row = r1 - 1;
                v[j] = t.ld4_raw(row, q * 4);
                if (MODE == 1) g[j] = ld4(da + row * C + q * 4);
            }
#pragma unroll
            for (int j = 0; j < NR; j++) {
                if (rb + (size_t)j * RPP >= r1) continue;
                v[j] = t.from_raw(v[j]);
                if (MODE == 0) {
                    s.x += v[j].x; s.y += v[j].y; s.z += v[j].z; s.w += v[j].w;
                    ss.x += v[j].x * v[j].x; ss.y += v[j].y * v[j].y; ss.z += v[j].z * v[j].z; ss.w += v[j].w * v[j].w;
                } else {
                    const float dx = fmaf(sc.x, v[j].x, sh.x) > 0.f ? g[j].x : 0.f, dy = fmaf(sc.y, v[j].y, sh.y) > 0.f ? g[j].y : 0.f;
                    const float dz = fmaf(sc.z, v[j].z, sh.z) > 0.f ? g[j].z : 0.f, dw = fmaf(sc.w, v[j].w, sh.w) > 0.f ? g[j].w : 0.f;
                    s.x += dx; s.y += dy; s.z += dz; s.w += dw;
                    ss.x += dx * ((v[j].x - mu.x) * rs.x); ss.y += dy * ((v[j].y - mu.y) * rs.y);
                    ss.z += dz * ((v[j].z - mu.z) * rs.z); ss.w += dw * ((v[j].w - mu.w) * rs.w);
                }
            }
        }
    }
    float4 *sm4 = reinterpret_cast<float4 *>(red);       // [256][2]
    sm4[tid * 2] = s; sm4[tid * 2 + 1] = ss;
    // the threads of a slab column, halved until one is left (narrow tensors: up to 128 of them)
    for (int n = RPP; n > 1;) {
        const int h = (n + 1) >> 1;
        __syncthreads();
        if (valid && ty + h < n) {
            const float4 a = sm4[((ty + h) * SW + tx) * 2], b = sm4[((ty + h) * SW + tx) * 2 + 1];
            s.x += a.x; s.y += a.y; s.z += a.z; s.w += a.w;
            ss.x += b.x; ss.y += b.y; ss.z += b.z; ss.w += b.w;
            sm4[tid * 2] = s; sm4[tid * 2 + 1] = ss;
        }
        n = h;
    }
    __syncthreads();
    if (ty == 0 && valid) {
        float *mine = pl.part + ((size_t)chunk * C4 + q) * 8;
        st4(mine, s); st4(mine + 4, ss);
    }
    if (pl.pending) return;
    const int q0 = slab * SW, nq = C4 - q0 < SW ? C4 - q0 : SW;
    unsigned int *cnt = pl.counters + (size_t)slab * (GROUPS ? 1 + pl.groups : 1);
    // whether this CTA is the last of n to come here (the word is left zero)
    auto last_of = [&](unsigned int *word, int n) {
        __syncthreads();
        if (tid == 0) {
            // (one thread's fences, on either side, order what all the CTA's threads wrote before the barrier and read after the next;
            // the word is cleared behind them: a fence waits for the stores in front of it)
            bool l = true;
            if (n > 1) {
                __threadfence();
                l = atomicAdd(word, 1u) == (unsigned int)n - 1;
                __threadfence();
                if (l) *word = 0u;
            }
            last = l ? 1u : 0u;
        }
        __syncthreads();
        return last != 0u;
    };
    if constexpr (GROUPS) {
        const int g = chunk / pl.group, first = g * pl.group, n = pl.chunks - first < pl.group ? pl.chunks - first : pl.group;
        if (!last_of(cnt + 1 + g, n)) return;
        tc::reduce_records<256>(pl.part + (size_t)first * 2 * C, n, C, 2 * q0, 2 * nq, red, tot, tid);
        for (int i = tid; i < nq * 8; i += 256) pl.gsum[(size_t)g * 2 * C + q0 * 8 + i] = tot[i];
        if (!last_of(cnt, pl.groups)) return;
        for (int i = tid; i < nq * 8; i += 256) {
            double v = 0;
#pragma unroll 8
            for (int j = 0; j < pl.groups; j++) v += __ldcg(pl.gsum + (size_t)j * 2 * C + q0 * 8 + i);
            tot[i] = v;
        }
        __syncthreads();
    } else {
        if (!last_of(cnt, pl.chunks)) return;
        tc::reduce_records<256>(pl.part, pl.chunks, C, 2 * q0, 2 * nq, red, tot, tid);
    }
    if (tid < nq * 4) {
        const int k = tid >> 2, j = tid & 3, ch = (q0 + k) * 4 + j;
        const double sum = tot[(2 * k) * 4 + j], sum2 = tot[(2 * k + 1) * 4 + j];
        if (MODE == 0) tc::moments_of(sum, sum2, out.inv_count, out.eps, out.mean[ch], out.rstd[ch]);
        else {
            out.dbeta[ch] = (float)sum; out.dgamma[ch] = (float)sum2;
            const double gr = (double)bn.gamma[ch] * (double)bn.rstd[ch];
            out.coef[ch] = (float)gr; out.coef[C + ch] = (float)(gr * sum * out.inv_count); out.coef[2 * C + ch] = (float)(gr * sum2 * out.inv_count);
        }
    }
}

static RedPlan red_plan(Exec &ex, const RedShape &r, int C, float *part, bool pending) {
    return RedPlan{r.SW, r.rows_per_cta, r.chunks, pending ? 0 : r.group, pending ? 0 : r.groups, pending ? 1 : 0, part,
                   reinterpret_cast<double *>(part + (size_t)r.chunks * 2 * C), pending ? nullptr : ex.ctx->counter(red_words(r))};
}

Moments mom_alloc(Exec &ex, int C, bool with_part) {
    Moments m;
    float *p = ex.ws.get<float>((size_t)2 * C);
    m.mean = p; m.rstd = p + C;
    if (with_part) {
        m.part_cap = mom_records(ex, C);
        m.part = ex.ws.get<float>(m.part_cap);
    }
    return m;
}
// records of 2C floats that a producer may leave: one per CTA of a convolution (conv_tc_kernel runs at most two CTAs per SM, the
// others one), kPendingRecords of a stand-alone reduction
size_t mom_records(const Exec &ex, int C) { return (size_t)2 * ex.ctx->sm_count * 2 * C; }

__global__ void __launch_bounds__(256) moments_finalize_kernel(const float *part, int parts, int C, double inv_count, float eps,
                                                             float *mean, float *rstd) {
    pdl_enter();
    __shared__ double red[256 * 4], tot[128 * 4];
    const int R = C >> 1, tid = threadIdx.x;
    for (int slot0 = 0; slot0 < R; slot0 += 128) {
        const int cw = R - slot0 < 128 ? R - slot0 : 128;
        tc::reduce_records<256>(part, parts, C, slot0, cw, red, tot, tid);
        for (int lc = tid; lc < cw * 2; lc += 256) {
            const int k = lc >> 2, j = lc & 3, ch = (slot0 >> 1) * 4 + lc;
            tc::moments_of(tot[(2 * k) * 4 + j], tot[(2 * k + 1) * 4 + j], inv_count, eps, mean[ch], rstd[ch]);
        }
        tc::named_barrier(1, 256);
    }
}

void mom_finalize(Exec &ex, Moments &m, int C) {
    if (!m.pending) return;
    if (!ex.dry) {
        launch(ex, moments_finalize_kernel, 1, 256, 0, (const float *)m.part, m.parts, C, m.inv_count, ex.eps, m.mean, m.rstd);
        ex.check("bn_stats_finalize");
    }
    m.pending = false;
}

// A consumer that adds pending records takes 160 of them in one round of loads (see reduce_records: 32 threads per slot, five
// each).  The last CTA's tail goes (basic block of 16 channels at 32x32: 260 -> 256 us for four such launches, of the odd-sized
// one 177 -> 171); a handful of records stays with the last CTA.
constexpr int kPendingRecords = 160, kFewRecords = 8;
void bn_stats(Exec &ex, Pair t, size_t P, Moments &mo) {
    const int C = t.C();
    RedShape r = red_shape(P, C, ex.ctx->sm_count, kStatRows);
    const bool defer = mo.defer && mo.part && (size_t)kPendingRecords * 2 * C <= mo.part_cap && r.chunks > kFewRecords;
    if (defer) r = red_shape(P, C, ex.ctx->sm_count, kStatRows, kPendingRecords);
    size_t m = ex.ws.mark();
    float *part = defer ? mo.part : ex.ws.get<float>(red_floats(r, C));
    mo.pending = defer; mo.parts = r.chunks; mo.inv_count = 1.0 / (double)P;
    if (!ex.dry) {
        launch_stream(ex, (double)P * C * 4, 30, r.group && !defer ? col_reduce_kernel<0, true> : col_reduce_kernel<0, false>, red_grid(r), 256, 0, t, nullptr, P, BnRef{}, red_plan(ex, r, C, part, defer),
               RedOut{mo.mean, mo.rstd, nullptr, nullptr, nullptr, 1.0 / (double)P, ex.eps});
        ex.check("bn_stats", (double)P * C * 4);
    }
    ex.ws.release(m);
}

// ------------------------------------------------------------------ streaming kernels over [P,C]
// A CTA of 256 threads takes a block of consecutive rows: a thread keeps V channels (their coefficients stay in registers) and
// walks the block in passes of 256 / SW rows, NR of them in flight; V is 8 (32-byte accesses) where size, channel counts and
// pointers allow, else 4.  The last rows go first: they are the ones that the kernel before has left in L2.
// Bound by HBM.  Many short CTAs instead of one resident wave of striding ones: the loads of a new CTA cover the stores
// and the start of the others.  Measured with BN-ReLU of 200704 x 512, 616 MB, alone: resident wave, four 16-byte loads in
// flight 6.1 TB/s; short CTAs 6.5 to 6.8 TB/s (two to four 32-byte loads, one to four passes; sixteen passes 6.2).
// In the train step of the large-image network: BN-ReLU 19.9 -> 17.5 ms, its backward with partner and bf16 copy
// 7.1 -> 5.3 ms, bf16 copies 1.4 -> 0.84 ms (summed over launches, some overlapped; see launch_stream for the larger part).
struct RowTile { int SW, rows; dim3 grid; };
static RowTile row_tile(size_t P, int CV, int NR, int sm, int per_sm) {     // per_sm: CTAs that an SM holds at least; 0: never several passes for the sake of one wave
    const int slabs = cdiv(CV, 256);
    RowTile r;
    r.SW = cdiv(CV, slabs);
    const size_t pass = (size_t)(256 / r.SW) * NR, n = (P + pass - 1) / pass;
    // up to four passes per CTA (the coefficients are read once per CTA) while sixteen CTAs per SM are left; what fits less
    // than four waves goes in one, with as many passes as that takes (no partly filled last wave)
    const size_t wave = (size_t)sm * per_sm;
    size_t passes = n * slabs / ((size_t)sm * 16);
    if (passes > 4) passes = 4;
    if (n * slabs < 4 * wave) passes = (n * slabs + wave - 1) / wave;
    if (passes < 1) passes = 1;
    r.rows = (int)(pass * passes);
    r.grid = dim3((unsigned)((n + passes - 1) / passes), slabs);
    return r;
}
// 32-byte accesses only where they leave every SM its four CTAs: below, twice the threads with half the bytes each are
// quicker (fp32 BN-ReLU of 131072 x 16: 3.1 against 2.4 us of a step's time per launch)
static bool wide_pays(size_t P, int C, int NR, int sm) { return (P * C) / ((size_t)256 * 8 * NR) >= (size_t)4 * sm; }
static bool wide_rows(const Pair &t) {
    return t.c0 % 8 == 0 && t.c1 % 8 == 0 && (uintptr_t)t.p0 % 32 == 0 && (t.c1 == 0 || (uintptr_t)t.p1 % 32 == 0);
}
template <int V> __device__ __forceinline__ void ldv(const float *p, float (&v)[V]) {
    if constexpr (V == 8) {
        uint32_t u[8];
        ld8(p, u, true);
#pragma unroll
        for (int i = 0; i < 8; i++) v[i] = __uint_as_float(u[i]);
    } else { const float4 a = ld4(p); v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; }
}
template <int V> __device__ __forceinline__ void stv(float *p, const float (&v)[V]) {
    if constexpr (V == 8) {
        uint32_t u[8];
#pragma unroll
        for (int i = 0; i < 8; i++) u[i] = __float_as_uint(v[i]);
        st8(p, u, true);
    } else st4(p, make_float4(v[0], v[1], v[2], v[3]));
}
template <int V> __device__ __forceinline__ void stv(bf16 *p, const float (&v)[V]) {
    if constexpr (V == 8) {
        uint4 u;
        uint32_t *w = reinterpret_cast<uint32_t *>(&u);
#pragma unroll
        for (int i = 0; i < 4; i++) { const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]); w[i] = *reinterpret_cast<const uint32_t *>(&h); }
        *reinterpret_cast<uint4 *>(p) = u;
    } else st4(p, make_float4(v[0], v[1], v[2], v[3]));
}
// raw words of a fixed-point tensor (q != 0) -> values
template <int V> __device__ __forceinline__ void values(float (&v)[V], float q) {
    if (q != 0.f)
#pragma unroll
        for (int i = 0; i < V; i++) v[i] = __int2float_rn(__float_as_int(v[i])) * q;
}
template <int V> struct BnCoef {
    float sc[V], sh[V], mu[V], rs[V];
    __device__ __forceinline__ BnCoef(const BnRef &bn, int c) {
#pragma unroll
        for (int i = 0; i < V; i += 4) {
            const float4 g = ld4(bn.gamma + c + i), b = ld4(bn.beta + c + i), m = ld4(bn.mean + c + i), r = ld4(bn.rstd + c + i);
            const float gg[4] = {g.x, g.y, g.z, g.w}, bb[4] = {b.x, b.y, b.z, b.w}, mm[4] = {m.x, m.y, m.z, m.w}, rr[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
            for (int j = 0; j < 4; j++) { mu[i + j] = mm[j]; rs[i + j] = rr[j]; bn_sc_sh(gg[j], bb[j], mm[j], rr[j], sc[i + j], sh[i + j]); }
        }
    }
};
constexpr int kApplyRows = 4;

// (64 registers for four CTAs per SM: with eight channels per thread the coefficients spill 20 to 24 bytes)
template <class TO, int V>
__global__ void __launch_bounds__(256, 4) bn_relu_apply_kernel(Pair t, size_t P, int SW, int rows, BnRef bn, TO *__restrict__ a, unsigned long long *stamp) {
    pdl_enter();
    stamp_begin(stamp);
    const int C = t.C(), rpp = 256 / SW, tx = threadIdx.x % SW, ty = threadIdx.x / SW, c = (blockIdx.y * SW + tx) * V;
    const size_t r0 = (size_t)(gridDim.x - 1 - blockIdx.x) * rows, r1 = r0 + rows < P ? r0 + rows : P;
    if (c < C && ty < rpp) {
        const BnCoef<V> k(bn, c);
#pragma unroll 1
        for (size_t rb = r0 + ty; rb < r1; rb += kApplyRows * rpp) {
            // all loads leave before anything waits on one: rows beyond the end read the last row again and are not stored
            float v[kApplyRows][V];
#pragma unroll
            for (int j = 0; j < kApplyRows; j++) {
                const size_t row = rb + j * rpp;
                ldv<V>(t.at(row < r1 ? row : r1 - 1, c), v[j]);
            }
#pragma unroll
            for (int j = 0; j < kApplyRows; j++) {
                const size_t row = rb + j * rpp;
                if (row >= r1) continue;
                values<V>(v[j], t.q);
#pragma unroll
                for (int i = 0; i < V; i++) v[j][i] = fmaxf(fmaf(k.sc[i], v[j][i], k.sh[i]), 0.f);
                stv<V>(a + row * C + c, v[j]);
            }
        }
    }
    stamp_end(stamp);
}

static int ew_grid(size_t n, int sm) {
    size_t g = (n + 255) / 256, cap = (size_t)sm * 8;
    return (int)(g < cap ? (g ? g : 1) : cap);
}
void bn_relu_apply(Exec &ex, Pair t, size_t P, BnRef bn, void *a, bool a_bf16) {
    if (ex.dry) return;
    const bool wide = wide_pays(P, t.C(), kApplyRows, ex.ctx->sm_count) && wide_rows(t) && (uintptr_t)a % 32 == 0;
    const RowTile r = row_tile(P, t.C() / (wide ? 8 : 4), kApplyRows, ex.ctx->sm_count, 4);
    const double bytes = (double)P * t.C() * (a_bf16 ? 6 : 8);
    unsigned long long *stamp = ex.stamp_slot();
#define RV_APPLY(TO, V) launch_stream(ex, bytes, 0, bn_relu_apply_kernel<TO, V>, r.grid, 256, 0, t, P, r.SW, r.rows, bn, (TO *)a, stamp)
    if (a_bf16) { if (wide) RV_APPLY(bf16, 8); else RV_APPLY(bf16, 4); }
    else { if (wide) RV_APPLY(float, 8); else RV_APPLY(float, 4); }
#undef RV_APPLY
    ex.check("bn_relu_apply", bytes);
}

// dt = coef0*db - coef1 - coef2*xhat ; db = da*[scale*t+shift > 0]
// OUT 0: out[P,C] = dt (float or bf16) ; 1: outp = dt (fp32 pair) ; 2: outp = add + dt
// CAST (OUT 1, 2): also write the result as one bf16 [P,C] tensor
template <int V> constexpr int kApplyBwdRows = V == 8 ? 2 : 4;
template <class TO, int OUT, bool CAST, int V>
__global__ void __launch_bounds__(256, 2) bn_relu_bwd_apply_kernel(const float *__restrict__ da, Pair t, size_t P, int SW, int rows, BnRef bn,
                                         const float *__restrict__ coef, TO *__restrict__ out, Pair add, Pair outp,
                                         bf16 *__restrict__ cast, unsigned long long *stamp) {
    pdl_enter();
    stamp_begin(stamp);
    constexpr int NR = kApplyBwdRows<V>;
    const int C = t.C(), rpp = 256 / SW, tx = threadIdx.x % SW, ty = threadIdx.x / SW, c = (blockIdx.y * SW + tx) * V;
    const size_t r0 = (size_t)(gridDim.x - 1 - blockIdx.x) * rows, r1 = r0 + rows < P ? r0 + rows : P;
    if (c < C && ty < rpp) {
        const BnCoef<V> k(bn, c);
        float k0[V], k1[V], k2[V];
        ldv<V>(coef + c, k0); ldv<V>(coef + C + c, k1); ldv<V>(coef + 2 * C + c, k2);
#pragma unroll 1
        for (size_t rb = r0 + ty; rb < r1; rb += NR * rpp) {
            // all loads leave before anything waits on one: rows beyond the end read the last row again and are not stored
            float v[NR][V], g[NR][V], pa[NR][V];
#pragma unroll
            for (int j = 0; j < NR; j++) {
                const size_t row = rb + j * rpp, rr = row < r1 ? row : r1 - 1;
                ldv<V>(t.at(rr, c), v[j]); ldv<V>(da + rr * C + c, g[j]);
                if (OUT == 2) ldv<V>(add.at(rr, c), pa[j]);
            }
#pragma unroll
            for (int j = 0; j < NR; j++) {
                const size_t row = rb + j * rpp;
                if (row >= r1) continue;
                values<V>(v[j], t.q);
                if (OUT == 2) values<V>(pa[j], add.q);
                float o[V];
#pragma unroll
                for (int i = 0; i < V; i++) {
                    const float x = v[j][i];
                    o[i] = k0[i] * (fmaf(k.sc[i], x, k.sh[i]) > 0.f ? g[j][i] : 0.f) - k1[i] - k2[i] * ((x - k.mu[i]) * k.rs[i]);
                    if (OUT == 2) o[i] += pa[j][i];
                }
                if (OUT == 0) stv<V>(out + row * C + c, o);
                else stv<V>(outp.at(row, c), o);
                if (CAST) stv<V>(cast + row * C + c, o);
            }
        }
    }
    stamp_end(stamp);
}

void bn_relu_bwd(Exec &ex, const float *da, Pair t, size_t P, BnRef bn, float *dgamma, float *dbeta, float *coef,
                 bool sums_done, void *out_single, bool out_bf16, Pair add, Pair out_pair, bf16 *out_cast) {
    const int C = t.C();
    RedShape r = red_shape(P, C, ex.ctx->sm_count, kBwdRows);
    size_t m = ex.ws.mark();
    float *part = sums_done ? nullptr : ex.ws.get<float>(red_floats(r, C));
    if (!ex.dry) {
        if (!sums_done) {
            launch_stream(ex, (double)P * C * 8, 30, r.group ? col_reduce_kernel<1, true> : col_reduce_kernel<1, false>, red_grid(r), 256, 0, t, da, P, bn, red_plan(ex, r, C, part, false),
                   RedOut{nullptr, nullptr, dgamma, dbeta, coef, 1.0 / (double)P, ex.eps});
            ex.check("bn_bwd_sums", (double)P * C * 8);
        }
        const bool pair = out_pair.p0 != nullptr, plus = pair && add.p0;
        const bool wide = wide_pays(P, C, kApplyBwdRows<8>, ex.ctx->sm_count) && wide_rows(t) && (uintptr_t)da % 32 == 0 && (uintptr_t)coef % 32 == 0 &&
                          (!pair || wide_rows(out_pair)) && (!plus || wide_rows(add)) && (uintptr_t)out_single % 32 == 0 && (uintptr_t)out_cast % 32 == 0;
        const RowTile rt = row_tile(P, C / (wide ? 8 : 4), wide ? kApplyBwdRows<8> : kApplyBwdRows<4>, ex.ctx->sm_count, 2);
        const double bytes = (double)P * C * ((pair ? (add.p0 ? 16 : 12) : (out_bf16 ? 10 : 12)) + (out_cast ? 2 : 0));
        unsigned long long *stamp = ex.stamp_slot();
#define RV_BWD(TO, OUT, CAST, dst) do { \
        if (wide) launch_stream(ex, bytes, 0, bn_relu_bwd_apply_kernel<TO, OUT, CAST, 8>, rt.grid, 256, 0, da, t, P, rt.SW, rt.rows, bn, coef, (TO *)(dst), add, out_pair, out_cast, stamp); \
        else launch_stream(ex, bytes, 0, bn_relu_bwd_apply_kernel<TO, OUT, CAST, 4>, rt.grid, 256, 0, da, t, P, rt.SW, rt.rows, bn, coef, (TO *)(dst), add, out_pair, out_cast, stamp); } while (0)
        if (plus) { if (out_cast) RV_BWD(float, 2, true, nullptr); else RV_BWD(float, 2, false, nullptr); }
        else if (pair) { if (out_cast) RV_BWD(float, 1, true, nullptr); else RV_BWD(float, 1, false, nullptr); }
        else if (out_bf16) RV_BWD(bf16, 0, false, out_single);
        else RV_BWD(float, 0, false, out_single);
#undef RV_BWD
        ex.check("bn_relu_bwd_apply", bytes);
    }
    ex.ws.release(m);
}

// bn_relu_bwd_apply_kernel on tensors of at most 64 channels from sums that are still the records of the data gradient's CTAs:
// ADD: the last step of a function's backward, out = add + dt, CAST: with a bf16 copy; else between its layers, the bf16 copy of dt alone.  Every CTA adds them, with its first rows already on the way: the records and the
// coefficients take it 2 us, where the reduction by the last CTA of the data gradient kept the GPU waiting for 4.  So a CTA takes all its rows
// in one or two rounds of loads, and the grid stays at two CTAs per SM.
constexpr int kSumsRows = 4;
template <bool ADD, bool CAST>
__global__ void __launch_bounds__(256, 2) bn_relu_bwd_sums_kernel(const float *__restrict__ da, Pair t, int P, int rows, BnRef bn, float *__restrict__ dgamma,
                                                                  float *__restrict__ dbeta, const float *add, float *out,
                                                                  bf16 *__restrict__ cast, unsigned long long *stamp) {
    __shared__ double red[256 * 4], tot[32 * 4];
    __shared__ __align__(16) float cf[7][64];
    pdl_enter();
    stamp_begin(stamp);
    const int C = t.c0, C4 = C >> 2, rpp = 256 / C4, tid = threadIdx.x, q = tid % C4, r = tid / C4;
    const int r0 = (int)blockIdx.x * rows, r1 = r0 + rows < P ? r0 + rows : P;
    float4 v[kSumsRows], g[kSumsRows], a[kSumsRows];
    auto load = [&](int rb) {
#pragma unroll
        for (int j = 0; j < kSumsRows; j++) {
            const int row = rb + j * rpp;
            if (row >= r1) continue;          // (out may be add: a row is read by the thread that stores it, and by no other)
            const size_t off = (size_t)row * C + q * 4;
            v[j] = ld4(t.p0 + off); g[j] = ld4(da + off);
            if (ADD) a[j] = ld4(add + off);
        }
    };
    if (r < rpp && r0 + r < r1) load(r0 + r);
    float gam = 0.f, bet = 0.f, mean = 0.f, rstd = 0.f;
    if (tid < C) { gam = bn.gamma[tid]; bet = bn.beta[tid]; mean = bn.mean[tid]; rstd = bn.rstd[tid]; }
    tc::reduce_records<256>(bn.part, bn.parts, C, 0, C >> 1, red, tot, tid);
    if (tid < C) {
        const double sum = tot[(2 * (tid >> 2)) * 4 + (tid & 3)], sum2 = tot[(2 * (tid >> 2) + 1) * 4 + (tid & 3)], gr = (double)gam * (double)rstd;
        float sc, sh;
        bn_sc_sh(gam, bet, mean, rstd, sc, sh);
        cf[0][tid] = sc; cf[1][tid] = sh; cf[2][tid] = mean; cf[3][tid] = rstd;
        cf[4][tid] = (float)gr; cf[5][tid] = (float)(gr * sum * bn.inv_count); cf[6][tid] = (float)(gr * sum2 * bn.inv_count);
        if (blockIdx.x == 0) { dbeta[tid] = (float)sum; dgamma[tid] = (float)sum2; }
    }
    __syncthreads();
    if (r < rpp) {
        float4 k[7];
#pragma unroll
        for (int i = 0; i < 7; i++) k[i] = ld4(&cf[i][q * 4]);
#pragma unroll 1
        for (int rb = r0 + r; rb < r1; rb += kSumsRows * rpp) {
            if (rb != r0 + r) load(rb);
#pragma unroll
            for (int j = 0; j < kSumsRows; j++) {
                const int row = rb + j * rpp;
                if (row >= r1) continue;
                float x[4] = {v[j].x, v[j].y, v[j].z, v[j].w}, o[4];
                values<4>(x, t.q);
                const float d[4] = {g[j].x, g[j].y, g[j].z, g[j].w}, p[4] = {ADD ? a[j].x : 0.f, ADD ? a[j].y : 0.f, ADD ? a[j].z : 0.f, ADD ? a[j].w : 0.f};
#define RV_K(n, i) (i == 0 ? k[n].x : i == 1 ? k[n].y : i == 2 ? k[n].z : k[n].w)
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    o[i] = RV_K(4, i) * (fmaf(RV_K(0, i), x[i], RV_K(1, i)) > 0.f ? d[i] : 0.f) - RV_K(5, i) - RV_K(6, i) * ((x[i] - RV_K(2, i)) * RV_K(3, i));
                    if (ADD) o[i] += p[i];
                }
#undef RV_K
                const float4 s = make_float4(o[0], o[1], o[2], o[3]);
                if (ADD) st4(out + (size_t)row * C + q * 4, s);
                if (CAST) st4(cast + (size_t)row * C + q * 4, s);
            }
        }
    }
    stamp_end(stamp);
}
// (larger tensors: the streaming kernel's wider accesses are worth more than the reduction in front of it)
bool bn_relu_bwd_sums_takes(size_t P, int C) { return C <= 64 && C % 4 == 0 && P * C <= (size_t)1 << 22; }
void bn_relu_bwd_sums(Exec &ex, const float *da, Pair t, size_t P, BnRef bn, float *dgamma, float *dbeta, const BwdSums &sums, Pair add, Pair out, bf16 *out_cast) {
    if (ex.dry) return;
    const int C = t.C(), rpp = 256 / (C / 4);
    int ctas = cdiv(P, (size_t)rpp * kSumsRows);
    if (ctas > 2 * ex.ctx->sm_count) ctas = 2 * ex.ctx->sm_count;
    const int rows = cdiv(P, ctas);
    bn.part = sums.part; bn.parts = sums.parts; bn.inv_count = sums.inv_count; bn.eps = ex.eps;
    unsigned long long *stamp = ex.stamp_slot();
    launch(ex, !add.p0 ? bn_relu_bwd_sums_kernel<false, true> : (out_cast ? bn_relu_bwd_sums_kernel<true, true> : bn_relu_bwd_sums_kernel<true, false>), dim3(cdiv(P, rows)), 256, 0, da, t, (int)P, rows, bn, dgamma, dbeta, (const float *)add.p0, out.p0, out_cast, stamp);
    ex.check("bn_relu_bwd_apply", (double)P * C * (add.p0 ? 16 + (out_cast ? 2 : 0) : 10));
}

template <class TO, int V>
__global__ void __launch_bounds__(256) concat_cast_kernel(Pair src, size_t P, int SW, int rows, TO *__restrict__ dst) {
    pdl_enter();
    const int C = src.C(), rpp = 256 / SW, tx = threadIdx.x % SW, ty = threadIdx.x / SW, c = (blockIdx.y * SW + tx) * V;
    const size_t r0 = (size_t)(gridDim.x - 1 - blockIdx.x) * rows, r1 = r0 + rows < P ? r0 + rows : P;
    if (c >= C || ty >= rpp) return;
#pragma unroll 1
    for (size_t rb = r0 + ty; rb < r1; rb += kApplyRows * rpp) {
        float v[kApplyRows][V];
#pragma unroll
        for (int j = 0; j < kApplyRows; j++) {
            const size_t row = rb + j * rpp;
            ldv<V>(src.at(row < r1 ? row : r1 - 1, c), v[j]);
        }
#pragma unroll
        for (int j = 0; j < kApplyRows; j++) {
            const size_t row = rb + j * rpp;
            if (row >= r1) continue;
            values<V>(v[j], src.q);
            stv<V>(dst + row * C + c, v[j]);
        }
    }
}

void concat_cast(Exec &ex, Pair src, size_t P, void *dst, bool dst_bf16) {
    if (ex.dry) return;
    const bool wide = wide_pays(P, src.C(), kApplyRows, ex.ctx->sm_count) && wide_rows(src) && (uintptr_t)dst % 32 == 0;
    // no coefficients to read once per CTA: one pass each (38 images of 47x30 x 88 channels 8.0 -> 5.9 us, 32 of 28x28 x 512 14.4 -> 13.5)
    const RowTile r = row_tile(P, src.C() / (wide ? 8 : 4), kApplyRows, ex.ctx->sm_count, 0);
    const double bytes = (double)P * src.C() * (dst_bf16 ? 6 : 8);
#define RV_CAST(TO, V) launch_stream(ex, bytes, 0, concat_cast_kernel<TO, V>, r.grid, 256, 0, src, P, r.SW, r.rows, (TO *)dst)
    if (dst_bf16) { if (wide) RV_CAST(bf16, 8); else RV_CAST(bf16, 4); }
    else { if (wide) RV_CAST(float, 8); else RV_CAST(float, 4); }
#undef RV_CAST
    ex.check("concat_cast", bytes);
}

// ------------------------------------------------------------------ max-pool 3x3 stride 2 pad 1 (NHWC)
__global__ void maxpool_fwd_kernel(const float *__restrict__ in, float *__restrict__ out, int N, int H, int W, int C4, int Ho, int Wo) {
    pdl_enter();
    size_t n = (size_t)N * Ho * Wo * C4;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        int q = (int)(i % C4); size_t p = i / C4;
        int j = (int)(p % Wo); p /= Wo; int io = (int)(p % Ho); int b = (int)(p / Ho);
        float4 m = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        for (int kh = 0; kh < 3; kh++) for (int kw = 0; kw < 3; kw++) {
            int y = io * 2 + kh - 1, x = j * 2 + kw - 1;
            if (y < 0 || y >= H || x < 0 || x >= W) continue;
            float4 v = ld4(in + (((size_t)b * H + y) * W + x) * C4 * 4 + q * 4);
            m.x = fmaxf(m.x, v.x); m.y = fmaxf(m.y, v.y); m.z = fmaxf(m.z, v.z); m.w = fmaxf(m.w, v.w);
        }
        st4(out + i * 4, m);
    }
}

// Gradient goes to the first maximum met in (kh,kw) row-major scan of each window.
// A CTA takes 8 x 8 input pixels x 8 channel quads of one image: it loads them with the halo their windows reach
// (11 x 11 pixels; outside the image: -inf) and the 5 x 5 gradients of those windows into shared memory, finds
// every window's first maximum once, and each input element then asks its (at most four) windows whether it is
// theirs -- one global read per element instead of one per window tap.
__global__ void __launch_bounds__(256) maxpool_bwd_kernel(const float *__restrict__ in, const float *__restrict__ dout, float *__restrict__ din,
                                                          int N, int H, int W, int C4, int Ho, int Wo, int tiles_y, int tiles_x, int tiles_q) {
    pdl_enter();
    __shared__ float4 tin[11 * 11 * 8];
    __shared__ float4 tg[5 * 5 * 8];
    __shared__ int4 tam[5 * 5 * 8];
    int t = blockIdx.x;
    const int tq = t % tiles_q; t /= tiles_q;
    const int tx = t % tiles_x; t /= tiles_x;
    const int ty = t % tiles_y; const int b = t / tiles_y;
    const int y0 = ty * 8, x0 = tx * 8, q0 = tq * 8;
    const int tid = threadIdx.x;
    const float ninf = -INFINITY;
    for (int idx = tid; idx < 11 * 11 * 8; idx += 256) {
        const int q = idx & 7, pos = idx >> 3, ry = pos / 11, rx = pos - ry * 11;
        const int yy = y0 - 1 + ry, xx = x0 - 1 + rx;
        float4 v = make_float4(ninf, ninf, ninf, ninf);
        if (yy >= 0 && yy < H && xx >= 0 && xx < W && q0 + q < C4) v = ld4(in + ((((size_t)b * H + yy) * W + xx) * C4 + q0 + q) * 4);
        tin[idx] = v;
    }
    if (tid < 5 * 5 * 8) {
        const int q = tid & 7, wpos = tid >> 3, wi = wpos / 5, wj = wpos - wi * 5;
        const int io = y0 / 2 + wi, j = x0 / 2 + wj;
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        if (io < Ho && j < Wo && q0 + q < C4) g = ld4(dout + ((((size_t)b * Ho + io) * Wo + j) * C4 + q0 + q) * 4);
        tg[tid] = g;
    }
    __syncthreads();
    if (tid < 5 * 5 * 8) {
        // window (wi, wj) covers tile rows 2wi .. 2wi+2, columns 2wj .. 2wj+2
        const int q = tid & 7, wpos = tid >> 3, wi = wpos / 5, wj = wpos - wi * 5;
        float4 best = make_float4(ninf, ninf, ninf, ninf);
        int4 at = make_int4(-1, -1, -1, -1);
        for (int kh = 0; kh < 3; kh++)
            for (int kw = 0; kw < 3; kw++) {
                const int pos = (2 * wi + kh) * 11 + 2 * wj + kw;
                const float4 v = tin[pos * 8 + q];
                if (v.x > best.x) { best.x = v.x; at.x = pos; }
                if (v.y > best.y) { best.y = v.y; at.y = pos; }
                if (v.z > best.z) { best.z = v.z; at.z = pos; }
                if (v.w > best.w) { best.w = v.w; at.w = pos; }
            }
        tam[tid] = at;
    }
    __syncthreads();
    for (int idx = tid; idx < 8 * 8 * 8; idx += 256) {
        const int q = idx & 7, lp = idx >> 3, ly = lp >> 3, lx = lp & 7;
        const int y = y0 + ly, x = x0 + lx;
        if (y >= H || x >= W || q0 + q >= C4) continue;
        const int mine = (ly + 1) * 11 + lx + 1;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int wi = ly / 2; wi <= (ly + 1) / 2; wi++)
            for (int wj = lx / 2; wj <= (lx + 1) / 2; wj++) {
                const int w = (wi * 5 + wj) * 8 + q;        // windows beyond the pooled image carry a zero gradient
                const int4 at = tam[w];
                const float4 g = tg[w];
                if (at.x == mine) acc.x += g.x;
                if (at.y == mine) acc.y += g.y;
                if (at.z == mine) acc.z += g.z;
                if (at.w == mine) acc.w += g.w;
            }
        st4(din + ((((size_t)b * H + y) * W + x) * C4 + q0 + q) * 4, acc);
    }
}

void maxpool_fwd(Exec &ex, const float *in, float *out, int N, int H, int W, int C) {
    if (ex.dry) return;
    int Ho = conv_out(H, 3, 2), Wo = conv_out(W, 3, 2);
    size_t n = (size_t)N * Ho * Wo * (C / 4);
    launch(ex, maxpool_fwd_kernel, ew_grid(n, ex.ctx->sm_count), 256, 0, in, out, N, H, W, C / 4, Ho, Wo);
    ex.check("maxpool_fwd");
}
void maxpool_bwd(Exec &ex, const float *in, const float *dout, float *din, int N, int H, int W, int C) {
    if (ex.dry) return;
    int Ho = conv_out(H, 3, 2), Wo = conv_out(W, 3, 2);
    const int C4 = C / 4, tiles_y = (H + 7) / 8, tiles_x = (W + 7) / 8, tiles_q = (C4 + 7) / 8;
    launch(ex, maxpool_bwd_kernel, (unsigned)((size_t)N * tiles_y * tiles_x * tiles_q), 256, 0, in, dout, din, N, H, W, C4, Ho, Wo, tiles_y, tiles_x, tiles_q);
    ex.check("maxpool_bwd");
}

// ------------------------------------------------------------------ head: avgpool -> FC -> softmax CE -> argmax
__global__ void avgpool_kernel(Pair y, int HW, float *__restrict__ feat) {
    pdl_enter();
    extern __shared__ float4 sm4[];
    const int C = y.C(), C4 = C / 4, SW = blockDim.x, RPP = blockDim.y;
    const int q = blockIdx.y * SW + threadIdx.x, n = blockIdx.x;
    const bool valid = q < C4;
    float4 s = make_float4(0, 0, 0, 0);
    if (valid)
        for (int r = threadIdx.y; r < HW; r += RPP) {
            float4 v = y.ld4((size_t)n * HW + r, q * 4);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
    sm4[threadIdx.y * SW + threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && valid) {
        for (int yy = 1; yy < RPP; yy++) { float4 a = sm4[yy * SW + threadIdx.x]; s.x += a.x; s.y += a.y; s.z += a.z; s.w += a.w; }
        float inv = 1.f / (float)HW;
        s.x *= inv; s.y *= inv; s.z *= inv; s.w *= inv;
        st4(feat + (size_t)n * C + q * 4, s);
    }
}

// one warp per (n,k)
__global__ void fc_fwd_kernel(const float *__restrict__ feat, const float *__restrict__ Wfc, const float *__restrict__ bfc,
                              int N, int C, int K, float *__restrict__ logits) {
    pdl_enter();
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= N * K) return;
    int n = warp / K, k = warp - n * K;
    float s = 0.f;
    for (int c = lane; c < C; c += 32) s = fmaf(feat[(size_t)n * C + c], Wfc[(size_t)k * C + c], s);
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) logits[warp] = s + bfc[k];
}

// one warp per sample: stable log-sum-exp, dlogits = (softmax - onehot)/N, arg-max (lowest index on ties)
// A label outside [0, K) is reported, not followed: nothing is read at it, the sample's loss becomes NaN and the
// context's status word is set to REVNET_E_INVALID_ARG (revnet_check_device returns it).
__global__ void softmax_ce_kernel(const float *__restrict__ logits, const int32_t *__restrict__ labels, int N, int K,
                                  float *__restrict__ dlogits, float *__restrict__ loss_n, int32_t *__restrict__ pred, int *status) {
    pdl_enter();
    int n = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (n >= N) return;
    const float *z = logits + (size_t)n * K;
    float m = -INFINITY; int mi = 0x7fffffff;
    for (int k = lane; k < K; k += 32) { float v = z[k]; if (v > m) { m = v; mi = k; } }
    for (int o = 16; o; o >>= 1) {
        float om = __shfl_xor_sync(0xffffffffu, m, o); int oi = __shfl_xor_sync(0xffffffffu, mi, o);
        if (om > m || (om == m && oi < mi)) { m = om; mi = oi; }
    }
    float s = 0.f;
    for (int k = lane; k < K; k += 32) s += expf(z[k] - m);
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const int lab = labels[n];
    const bool lab_ok = lab >= 0 && lab < K;
    const float inv = 1.f / s, invN = 1.f / (float)N;
    for (int k = lane; k < K; k += 32) dlogits[(size_t)n * K + k] = (expf(z[k] - m) * inv - (k == lab ? 1.f : 0.f)) * invN;
    if (lane == 0) {
        loss_n[n] = lab_ok ? m + logf(s) - z[lab] : __int_as_float(0x7fc00000);
        pred[n] = mi;
        if (!lab_ok && status) atomicCAS(status, 0, (int)REVNET_E_INVALID_ARG);
    }
}

__global__ void mean_kernel(const float *__restrict__ v, int N, float *out) {
    pdl_enter();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0; for (int i = 0; i < N; i++) s += v[i];
        *out = (float)(s / N);
    }
}

void head_fwd(Exec &ex, Pair y, int N, int HW, const float *Wfc, const float *bfc, const int32_t *labels,
              int K, float *feat, float *logits, float *dlogits, float *loss, int32_t *pred) {
    const int C = y.C();
    ex.flops += 2ull * N * C * K;
    size_t m = ex.ws.mark();
    float *loss_n = ex.ws.get<float>(N);
    if (!ex.dry) {
        int C4 = C / 4, SW = C4 < 128 ? C4 : 128, RPP = 256 / SW; if (RPP < 1) RPP = 1;
        dim3 grid(N, cdiv(C4, SW)), block(SW, RPP);
        launch(ex, avgpool_kernel, grid, block, (size_t)SW * RPP * 16, y, HW, feat);
        ex.check("avgpool");
        launch(ex, fc_fwd_kernel, cdiv((size_t)N * K * 32, 256), 256, 0, feat, Wfc, bfc, N, C, K, logits);
        ex.check("fc_fwd");
        launch(ex, softmax_ce_kernel, cdiv((size_t)N * 32, 256), 256, 0, logits, labels, N, K, dlogits, loss_n, pred, ex.ctx->dev_status);
        ex.check("softmax_ce");
        launch(ex, mean_kernel, 1, 32, 0, loss_n, N, loss);
        ex.check("loss_mean");
    }
    ex.ws.release(m);
}

__global__ void fc_wgrad_kernel(const float *__restrict__ dlogits, const float *__restrict__ feat, int N, int C, int K,
                                float *__restrict__ dW, float *__restrict__ db) {
    pdl_enter();
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < (size_t)K * C) {
        int k = (int)(i / C), c = (int)(i - (size_t)k * C);
        float s = 0.f;
        for (int n = 0; n < N; n++) s = fmaf(dlogits[(size_t)n * K + k], feat[(size_t)n * C + c], s);
        dW[i] = s;
    }
    if (i < (size_t)K) { float s = 0.f; for (int n = 0; n < N; n++) s += dlogits[(size_t)n * K + i]; db[i] = s; }
}
// the same for a small layer: one warp per element of dW (and of db), lanes over the samples, added by a shuffle tree
__global__ void fc_wgrad_warp_kernel(const float *__restrict__ dlogits, const float *__restrict__ feat, int N, int C, int K,
                                     float *__restrict__ dW, float *__restrict__ db) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const size_t w = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const size_t n_out = (size_t)K * C + K;
    if (w >= n_out) return;
    float s = 0.f;
    if (w < (size_t)K * C) {
        const int k = (int)(w / C), c = (int)(w - (size_t)k * C);
        for (int n = lane; n < N; n += 32) s = fmaf(dlogits[(size_t)n * K + k], feat[(size_t)n * C + c], s);
    } else {
        const int k = (int)(w - (size_t)K * C);
        for (int n = lane; n < N; n += 32) s += dlogits[(size_t)n * K + k];
    }
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) { if (w < (size_t)K * C) dW[w] = s; else db[w - (size_t)K * C] = s; }
}
__global__ void fc_dgrad_kernel(const float *__restrict__ dlogits, const float *__restrict__ Wfc, int N, int C, int K,
                                float scale, float *__restrict__ dfeat) {
    pdl_enter();
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)N * C) return;
    int n = (int)(i / C), c = (int)(i - (size_t)n * C);
    float s = 0.f;
    for (int k = 0; k < K; k++) s = fmaf(dlogits[(size_t)n * K + k], Wfc[(size_t)k * C + c], s);
    dfeat[i] = s * scale;
}
__global__ void avgpool_bwd_kernel(const float *__restrict__ dfeat, Pair dy, size_t nquads, int C4, int HW) {
    pdl_enter();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nquads; i += (size_t)gridDim.x * blockDim.x) {
        size_t row = i / C4; int q = (int)(i - row * C4); size_t n = row / HW;
        st4(dy.at(row, q * 4), ld4(dfeat + n * C4 * 4 + q * 4));
    }
}

void head_bwd(Exec &ex, Pair dy, int N, int HW, const float *Wfc, const float *feat, const float *dlogits,
              int K, float *dWfc, float *dbfc, float *dfeat) {
    const int C = dy.C();
    ex.flops += 4ull * N * C * K;
    if (ex.dry) return;
    if ((size_t)K * C <= 65536) launch(ex, fc_wgrad_warp_kernel, cdiv(((size_t)K * C + K) * 32, 256), 256, 0, dlogits, feat, N, C, K, dWfc, dbfc);
    else launch(ex, fc_wgrad_kernel, cdiv((size_t)K * C, 256), 256, 0, dlogits, feat, N, C, K, dWfc, dbfc);
    ex.check("fc_wgrad");
    launch(ex, fc_dgrad_kernel, cdiv((size_t)N * C, 256), 256, 0, dlogits, Wfc, N, C, K, 1.f / (float)HW, dfeat);
    ex.check("fc_dgrad");
    size_t nq = (size_t)N * HW * (C / 4);
    launch(ex, avgpool_bwd_kernel, ew_grid(nq, ex.ctx->sm_count), 256, 0, dfeat, dy, nq, C / 4, HW);
    ex.check("avgpool_bwd");
}

// ------------------------------------------------------------------ shortcut of a down-sampling unit
// S(x): 2x2 average pooling with stride 2, then zero channels up to cout; x and S(x) in the coupling-state format
// (on a fixed-point state the mean of the four grid values is rounded to the grid, ties to even).
__global__ void shortcut_fwd_kernel(const float *__restrict__ x, float *__restrict__ out, int N, int H, int W, int cin, int cout, float q) {
    pdl_enter();
    const int Ho = H >> 1, Wo = W >> 1, C4 = cout >> 2;
    const size_t n = (size_t)N * Ho * Wo * C4;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % C4) * 4; size_t p = i / C4;
        const int xo = (int)(p % Wo); p /= Wo;
        const int yo = (int)(p % Ho); const size_t b = p / Ho;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        if (c < cin) {
            const float *s0 = x + (((b * H + 2 * yo) * W + 2 * xo) * (size_t)cin + c);
            const float *s1 = s0 + (size_t)W * cin;
            if (q == 0.f) {
                const float4 a = ld4(s0), bq = ld4(s0 + cin), cq = ld4(s1), d = ld4(s1 + cin);
                o = make_float4((a.x + bq.x + cq.x + d.x) * 0.25f, (a.y + bq.y + cq.y + d.y) * 0.25f,
                                (a.z + bq.z + cq.z + d.z) * 0.25f, (a.w + bq.w + cq.w + d.w) * 0.25f);
            } else {
                const int4 a = *reinterpret_cast<const int4 *>(s0), bq = *reinterpret_cast<const int4 *>(s0 + cin);
                const int4 cq = *reinterpret_cast<const int4 *>(s1), d = *reinterpret_cast<const int4 *>(s1 + cin);
                auto avg = [](int u, int v, int w, int z) {
                    const int sum = u + v + w + z;
                    int k = sum >> 2; const int r = sum & 3;             // floor and remainder (in quarters)
                    if (r == 3 || (r == 2 && (k & 1))) k++;              // nearest, ties to even
                    return __int_as_float(k);
                };
                o = make_float4(avg(a.x, bq.x, cq.x, d.x), avg(a.y, bq.y, cq.y, d.y), avg(a.z, bq.z, cq.z, d.z), avg(a.w, bq.w, cq.w, d.w));
            }
        }
        st4(out + i * 4, o);
    }
}
// S^T d: the first cin channels of d [N, H/2, W/2, cout], each value spread over its 2x2 window with weight 1/4 -> [N, H, W, cin]
__global__ void shortcut_bwd_kernel(const float *__restrict__ d, float *__restrict__ gx, int N, int H, int W, int cin, int cout) {
    pdl_enter();
    const int Ho = H >> 1, Wo = W >> 1, C4 = cin >> 2;
    const size_t n = (size_t)N * H * W * C4;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % C4) * 4; size_t p = i / C4;
        const int xx = (int)(p % W); p /= W;
        const int yy = (int)(p % H); const size_t b = p / H;
        const float4 v = ld4(d + (((b * Ho + (yy >> 1)) * Wo + (xx >> 1)) * (size_t)cout + c));
        st4(gx + i * 4, make_float4(v.x * 0.25f, v.y * 0.25f, v.z * 0.25f, v.w * 0.25f));
    }
}
void shortcut_fwd(Exec &ex, const float *x, float *out, int N, int H, int W, int cin, int cout, float q) {
    if (ex.dry) return;
    const size_t n = (size_t)N * (H / 2) * (W / 2) * (cout / 4);
    launch(ex, shortcut_fwd_kernel, ew_grid(n, ex.ctx->sm_count), 256, 0, x, out, N, H, W, cin, cout, q);
    ex.check("shortcut_fwd", (double)N * H * W * cin * 4 + (double)n * 16);
}
void shortcut_bwd(Exec &ex, const float *d, float *gx, int N, int H, int W, int cin, int cout) {
    if (ex.dry) return;
    const size_t n = (size_t)N * H * W * (cin / 4);
    launch(ex, shortcut_bwd_kernel, ew_grid(n, ex.ctx->sm_count), 256, 0, d, gx, N, H, W, cin, cout);
    ex.check("shortcut_bwd", (double)n * 16 * 1.25);
}

// ------------------------------------------------------------------ SGD with momentum and weight decay
// v <- mu v + (g + wd w [decayed segments only]); w <- w - lr v   (Appendix 6.1).  Every segment but the last starts and ends
// on a multiple of four floats (channel counts are multiples of four), so a quad lies in one segment; the floats behind
// the last whole quad go one by one.
// A CTA takes 2048 consecutive floats, two quads per thread; each warp finds the segment of its first quad with a 32-way
// search (two dependent reads for a thousand segments) while its loads are on their way, and walks on from there.
// Bound by HBM.  Measured on the parameters of the large-image network: 2.39 ms (4.0 TB/s) with a binary search per quad in a
// striding grid, now 1.42 ms (6.8 TB/s).
__device__ __forceinline__ int sgd_segment(const uint32_t *__restrict__ seg_end, int n_seg, size_t i) {
    int lo = 0, hi = n_seg - 1;                  // first segment whose end is > i
    while (lo < hi) { int mid = (lo + hi) >> 1; if (seg_end[mid] > i) hi = mid; else lo = mid + 1; }
    return lo;
}
__device__ __forceinline__ int sgd_segment_warp(const uint32_t *__restrict__ seg_end, int n_seg, size_t i) {
    const int lane = threadIdx.x & 31;
    int lo = 0, len = n_seg;
    while (true) {
        const int step = (len + 31) >> 5, last = lo + (lane + 1) * step - 1;        // lane's run of `step` segments: its last one
        const int skip = __popc(__ballot_sync(0xffffffffu, (lane + 1) * step <= len && seg_end[last] <= i));
        lo += skip * step;
        if (step <= 1) break;
        len = len - skip * step < step ? len - skip * step : step;
    }
    return lo < n_seg ? lo : n_seg - 1;
}
constexpr int kSgdQuads = 2;
__global__ void __launch_bounds__(256) sgd_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ v, size_t n,
                                                  const uint32_t *__restrict__ seg_end, const uint8_t *__restrict__ seg_decay, int n_seg,
                                                  float lr, float mu, float wd) {
    pdl_enter();
    const size_t n4 = n >> 2;
    float4 *p4 = reinterpret_cast<float4 *>(p), *v4 = reinterpret_cast<float4 *>(v);
    const float4 *g4 = reinterpret_cast<const float4 *>(g);
    const size_t base = (size_t)blockIdx.x * (256 * kSgdQuads) + (threadIdx.x & ~31u) * kSgdQuads, i0 = base + (threadIdx.x & 31);
    if (base < n4) {
        float4 w[kSgdQuads], gg[kSgdQuads], vv[kSgdQuads];
#pragma unroll
        for (int j = 0; j < kSgdQuads; j++) {
            const size_t i = i0 + j * 32;
            if (i < n4) { w[j] = p4[i]; gg[j] = g4[i]; vv[j] = v4[i]; }
        }
        int seg = sgd_segment_warp(seg_end, n_seg, base * 4);
#pragma unroll
        for (int j = 0; j < kSgdQuads; j++) {
            const size_t i = i0 + j * 32;
            if (i >= n4) continue;
            while (seg < n_seg - 1 && seg_end[seg] <= i * 4) seg++;
            const float d = seg_decay[seg] ? wd : 0.f;
            float4 o;
            o.x = fmaf(mu, vv[j].x, gg[j].x + d * w[j].x); o.y = fmaf(mu, vv[j].y, gg[j].y + d * w[j].y);
            o.z = fmaf(mu, vv[j].z, gg[j].z + d * w[j].z); o.w = fmaf(mu, vv[j].w, gg[j].w + d * w[j].w);
            v4[i] = o;
            p4[i] = make_float4(w[j].x - lr * o.x, w[j].y - lr * o.y, w[j].z - lr * o.z, w[j].w - lr * o.w);
        }
    }
    if (blockIdx.x == 0)
        for (size_t i = n4 * 4 + threadIdx.x; i < n; i += blockDim.x) {
            const float w = p[i];
            const float gg = g[i] + (seg_decay[sgd_segment(seg_end, n_seg, i)] ? wd * w : 0.f);
            const float vv = fmaf(mu, v[i], gg);
            v[i] = vv;
            p[i] = w - lr * vv;
        }
}
// the same, one float at a time: for a parameter layout in which some segment does not start on a multiple of four
__global__ void sgd_scalar_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ v, size_t n,
                                  const uint32_t *__restrict__ seg_end, const uint8_t *__restrict__ seg_decay, int n_seg,
                                  float lr, float mu, float wd) {
    pdl_enter();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float w = p[i];
        const float gg = g[i] + (seg_decay[sgd_segment(seg_end, n_seg, i)] ? wd * w : 0.f);
        const float vv = fmaf(mu, v[i], gg);
        v[i] = vv;
        p[i] = w - lr * vv;
    }
}
void sgd_update(Exec &ex, float *params, const float *grads, float *mom, size_t n, const uint32_t *seg_end,
                const uint8_t *seg_decay, int n_seg, float lr, float momentum, float wd, bool quad_aligned) {
    if (ex.dry) return;
    if (quad_aligned) launch_stream(ex, (double)n * 20, 0, sgd_kernel, cdiv(n / 4 + 1, 256 * kSgdQuads), 256, 0, params, grads, mom, n, seg_end, seg_decay, n_seg, lr, momentum, wd);
    else launch(ex, sgd_scalar_kernel, ew_grid(n, ex.ctx->sm_count), 256, 0, params, grads, mom, n, seg_end, seg_decay, n_seg, lr, momentum, wd);
    ex.check("sgd", (double)n * 20);
}

__global__ void max_abs_diff_kernel(const float *__restrict__ a, const float *__restrict__ b, size_t n, float q, float *out) {
    pdl_enter();
    float m = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        if (q == 0.f) m = fmaxf(m, fabsf(a[i] - b[i]));
        else m = fmaxf(m, fabsf((float)(reinterpret_cast<const int *>(a)[i] - reinterpret_cast<const int *>(b)[i])) * q);
    }
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int *>(out), __float_as_int(m));   // m >= 0
}
void max_abs_diff(Exec &ex, const float *a, const float *b, size_t n, float q, float *out) {
    if (ex.dry) return;
    launch(ex, max_abs_diff_kernel, ew_grid(n, ex.ctx->sm_count), 256, 0, a, b, n, q, out);
    ex.check("max_abs_diff");
}
void fill_zero(Exec &ex, void *p, size_t bytes) {
    if (ex.dry) return;
    cudaMemsetAsync(p, 0, bytes, ex.stream);
}

__global__ void upsample_zero_kernel(const uint4 *__restrict__ in, uint4 *__restrict__ out, int N, int Ho, int Wo, int C8) {
    pdl_enter();
    const size_t n = (size_t)N * Ho * 2 * Wo * 2 * C8;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % C8); size_t p = i / C8;
        const int x = (int)(p % (2 * Wo)); p /= 2 * Wo;
        const int y = (int)(p % (2 * Ho)); const size_t b = p / (2 * Ho);
        uint4 v = make_uint4(0, 0, 0, 0);
        if (!(x & 1) && !(y & 1)) v = in[((b * Ho + (y >> 1)) * Wo + (x >> 1)) * C8 + c];
        out[i] = v;
    }
}
void upsample_zero_bf16(Exec &ex, const bf16 *in, bf16 *out, int N, int Ho, int Wo, int C) {
    if (ex.dry) return;
    const size_t n = (size_t)N * Ho * 2 * Wo * 2 * (C / 8);
    launch(ex, upsample_zero_kernel, ew_grid(n, ex.ctx->sm_count), 256, 0, (const uint4 *)in, (uint4 *)out, N, Ho, Wo, C / 8);
    ex.check("upsample_zero", (double)n * 16 * 1.25);
}
