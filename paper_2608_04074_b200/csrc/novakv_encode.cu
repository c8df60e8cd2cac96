// Write path of append-sized batches: forward transforms (binary64) + brute-force nearest-codeword search + paged store; the
// search of given coefficients; the staging kernels of the BF16 band.  (Prompt-sized batches: novakv_prefill.cu.)
// Side 0 = keys, 1 = values.  The search is ALU-bound (256 distance evaluations per group, per token, per side).
//
// The index the write path stores is the exact Euclidean nearest codeword of the binary64 coefficient
// (lowest index on a tie).  The 256 distances are evaluated in binary32; beside the minimum the search
// keeps the second smallest distance, and whenever the two are closer than a rigorous bound on what the
// binary32 evaluation (coefficient rounding included) can have moved them, the group is searched again in
// binary64 by the whole warp (certified search).  The binary32 result is kept only where it provably
// equals the binary64 one.
#include <math_constants.h>
#ifdef NOVAKV_TIMING
#include <cstdio>
#endif

#include <cooperative_groups.h>

#include "novakv_search.cuh"

namespace {

constexpr int ENC_THREADS = 512;
constexpr int ENC_TILE = 64;   // tokens per tile (search granularity)
// Shared-memory plan of the search-only kernel: codebook, one tile of coefficients, its indices.
template <int D>
struct EncSmem {
    static constexpr int L = D / NOVAKV_G;
    static constexpr int RSTRIDE = D + 4;                       // floats; keeps 128-bit row reads conflict-free
    static constexpr size_t cb_bytes = (size_t)L * NOVAKV_C * NOVAKV_G * sizeof(float);
    static constexpr size_t r_bytes = (size_t)ENC_TILE * RSTRIDE * sizeof(float);
    static constexpr size_t idx_bytes = (size_t)ENC_TILE * L;
    static constexpr size_t total = cb_bytes + r_bytes + idx_bytes;
};

#ifdef NOVAKV_SCALAR_SEARCH
// Scalar form of the binary32 distance: fma(e3,e3,fma(e2,e2,fma(e1,e1,e0*e0))).
__device__ __forceinline__ float dist4(const float4 r, const float4 c) {
    const float e0 = __fsub_rn(r.x, c.x), e1 = __fsub_rn(r.y, c.y);
    const float e2 = __fsub_rn(r.z, c.z), e3 = __fsub_rn(r.w, c.w);
    return __fmaf_rn(e3, e3, __fmaf_rn(e2, e2, __fmaf_rn(e1, e1, __fmul_rn(e0, e0))));
}
#endif

// Packed binary32 pairs: two IEEE operations per instruction (same roundings as the scalar forms).
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1,%2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// Distances of one coefficient vector (each component duplicated into a pair) to two codewords at once:
// cw[i] = (codeword c, component i ; codeword c+1, component i).  Same chain as dist4, per half.
__device__ __forceinline__ void dist4x2(const uint64_t (&r2)[4], const uint64_t (&cw)[4], float& d0, float& d1) {
#ifdef NOVAKV_SCALAR_SEARCH
    float r[4], lo[4], hi[4], dummy;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        asm("mov.b64 {%0,%1}, %2;" : "=f"(r[i]), "=f"(dummy) : "l"(r2[i]));
        asm("mov.b64 {%0,%1}, %2;" : "=f"(lo[i]), "=f"(hi[i]) : "l"(cw[i]));
    }
    d0 = dist4(make_float4(r[0], r[1], r[2], r[3]), make_float4(lo[0], lo[1], lo[2], lo[3]));
    d1 = dist4(make_float4(r[0], r[1], r[2], r[3]), make_float4(hi[0], hi[1], hi[2], hi[3]));
#else
    const uint64_t e0 = sub2(r2[0], cw[0]), e1 = sub2(r2[1], cw[1]), e2 = sub2(r2[2], cw[2]), e3 = sub2(r2[3], cw[3]);
    const uint64_t d = fma2(e3, e3, fma2(e2, e2, fma2(e1, e1, mul2(e0, e0))));
    asm("mov.b64 {%0,%1}, %2;" : "=f"(d0), "=f"(d1) : "l"(d));
#endif
}

// Shared-memory image of a (head, side) codebook for the search: [L][128 codeword pairs][4 components][2].
__device__ __forceinline__ void fill_codebook_pairs(float* cb_s, const float4* __restrict__ cb_g, int n_groups) {
    for (int i = threadIdx.x; i < n_groups * NOVAKV_C; i += ENC_THREADS) {
        const float4 v = cb_g[i];
        float* dst = cb_s + (size_t)(i >> 1) * 8 + (i & 1);
        dst[0] = v.x; dst[2] = v.y; dst[4] = v.z; dst[6] = v.w;
    }
}

__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Warp-cooperative exact search of one (token, group) in binary64: all 32 lanes call it with the same
// arguments and get the same result.  The binary32 coefficients in shared memory ARE the vector to encode.
// Lane i evaluates the codewords i, i+32, ... in ascending order with a strict '<'; the warp then keeps the
// smallest distance and, among equal distances, the lowest index.
__device__ __noinline__ int exact_search_group(const float* r_row_s, int l, const float* cb_pairs_s /* [L][128][4][2] */) {
    const int lane = threadIdx.x & 31;
    double r[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) r[c] = (double)r_row_s[l * 4 + c];
    double best = CUDART_INF;
    int bi = lane;
    const float* cb = cb_pairs_s + (size_t)l * NOVAKV_C * 4;
#pragma unroll
    for (int j = 0; j < NOVAKV_C / 32; ++j) {
        const int code = lane + 32 * j;
        const float* cw = cb + (size_t)(code >> 1) * 8 + (code & 1);
        double dd = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double e = r[c] - (double)cw[2 * c];
            dd = __dadd_rn(dd, __dmul_rn(e, e));
        }
        if (dd < best) { best = dd; bi = code; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob < best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    return bi;
}

// Search of the tile's coefficients (r_s, [ENC_TILE][RSTRIDE] float) against the paired codebook image.
// Warp w of n_warps owns groups w, w+n_warps, ...; lane t owns tokens t and t+32.
// The binary32 pass finds the first minimum in ascending codeword order (what a scan with a strict '<' keeps)
// in two steps that need far fewer compare/select instructions than a per-codeword running argmin:
//   1. blocks of 8 codewords: the block minimum (a tree of 3-input minima) updates the running minimum with a
//      strict '<', which keeps the first block that attains the overall minimum; the second smallest block
//      minimum is tracked beside it (two more min/max per block);
//   2. the 8 distances of that block are recomputed (same instructions, same bits); the first one equal to
//      the minimum gives the index and the others enter the second smallest distance.
// Then the certification: a group whose two smallest distances are too close to tell apart in binary32 is
// searched again in binary64 by the whole warp (exact_search_group).
template <int D>
__device__ __forceinline__ void search_tile(const float* r_s, const float4* cb_s, uint8_t* idx_s, int n_valid, int warp, int n_warps) {
    constexpr int L = D / NOVAKV_G;
    constexpr int RS = EncSmem<D>::RSTRIDE;
    const int lane = threadIdx.x & 31;
    for (int l = warp; l < L; l += n_warps) {
        const float4 ra = *reinterpret_cast<const float4*>(r_s + (size_t)lane * RS + l * 4);
        const float4 rb = *reinterpret_cast<const float4*>(r_s + (size_t)(lane + 32) * RS + l * 4);
        const uint64_t ra2[4] = {pk2(ra.x, ra.x), pk2(ra.y, ra.y), pk2(ra.z, ra.z), pk2(ra.w, ra.w)};
        const uint64_t rb2[4] = {pk2(rb.x, rb.x), pk2(rb.y, rb.y), pk2(rb.z, rb.z), pk2(rb.w, rb.w)};
        float best_a = CUDART_INF_F, best_b = CUDART_INF_F, sec_a = CUDART_INF_F, sec_b = CUDART_INF_F;
        int blk_a = 0, blk_b = 0;
        const ulonglong2* cb = reinterpret_cast<const ulonglong2*>(cb_s) + (size_t)l * NOVAKV_C;   // 2 x 16 B per pair
#pragma unroll 4
        for (int blk = 0; blk < NOVAKV_C / 8; ++blk) {
            float da[8], db[8];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const ulonglong2 q0 = cb[8 * blk + 2 * p], q1 = cb[8 * blk + 2 * p + 1];
                const uint64_t cw[4] = {q0.x, q0.y, q1.x, q1.y};
                dist4x2(ra2, cw, da[2 * p], da[2 * p + 1]);
                dist4x2(rb2, cw, db[2 * p], db[2 * p + 1]);
            }
            const float ma = fmin3(fmin3(da[0], da[1], da[2]), fmin3(da[3], da[4], da[5]), fminf(da[6], da[7]));
            const float mb = fmin3(fmin3(db[0], db[1], db[2]), fmin3(db[3], db[4], db[5]), fminf(db[6], db[7]));
            sec_a = fminf(sec_a, fmaxf(best_a, ma));
            sec_b = fminf(sec_b, fmaxf(best_b, mb));
            if (ma < best_a) { best_a = ma; blk_a = blk; }
            if (mb < best_b) { best_b = mb; blk_b = blk; }
        }
        // the winning blocks again: first codeword whose distance equals the minimum; the block's other
        // distances compete for the second place
        int ia = 8 * blk_a, ib = 8 * blk_b;
        {
            float da[8], db[8];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const ulonglong2 qa0 = cb[8 * blk_a + 2 * p], qa1 = cb[8 * blk_a + 2 * p + 1];
                const uint64_t cwa[4] = {qa0.x, qa0.y, qa1.x, qa1.y};
                dist4x2(ra2, cwa, da[2 * p], da[2 * p + 1]);
                const ulonglong2 qb0 = cb[8 * blk_b + 2 * p], qb1 = cb[8 * blk_b + 2 * p + 1];
                const uint64_t cwb[4] = {qb0.x, qb0.y, qb1.x, qb1.y};
                dist4x2(rb2, cwb, db[2 * p], db[2 * p + 1]);
            }
            int ka = 0, kb = 0;
#pragma unroll
            for (int k = 7; k >= 0; --k) {
                if (da[k] == best_a) ka = k;
                if (db[k] == best_b) kb = k;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k != ka) sec_a = fminf(sec_a, da[k]);
                if (k != kb) sec_b = fminf(sec_b, db[k]);
            }
            ia += ka; ib += kb;
        }
        // certification
        const bool ta = lane < n_valid && needs_exact_search(best_a, sec_a, 0.f);
        const bool tb = lane + 32 < n_valid && needs_exact_search(best_b, sec_b, 0.f);
        unsigned todo_a = __ballot_sync(0xffffffffu, ta), todo_b = __ballot_sync(0xffffffffu, tb);
        while (todo_a) {
            const int src = __ffs(todo_a) - 1;
            todo_a &= todo_a - 1;
            const int res = exact_search_group(r_s + (size_t)src * RS, l, reinterpret_cast<const float*>(cb_s));
            if (lane == src) ia = res;
        }
        while (todo_b) {
            const int src = __ffs(todo_b) - 1;
            todo_b &= todo_b - 1;
            const int res = exact_search_group(r_s + (size_t)(src + 32) * RS, l, reinterpret_cast<const float*>(cb_s));
            if (lane == src) ib = res;
        }
        if (lane < n_valid) idx_s[lane * L + l] = (uint8_t)ia;
        if (lane + 32 < n_valid) idx_s[(lane + 32) * L + l] = (uint8_t)ib;
    }
}

// Append-sized batches (a decode step appends one token per sequence): the prompt encoder would
// pad every (head, side) to a 256-token tile.  Here one warp owns one
// group of one (head, side) and stages only its 4 columns of the transform (4 KB of binary64) and its
// group's codebook (4 KB), so the work spreads over L/4 * Hkv * 2 CTAs per chunk of the token list.  A pass covers tp
// tokens (tp = 1, 2, 4, 8, the smallest power of two that holds the batch, at most 8): lane = grp * tp + token.
// Chunk c of n takes the passes c, c + n, ...: batches of more than 8 tokens get as many chunks as CTAs fit on the
// machine at once (128 tokens, d = 128: 30.5 us with one CTA per four groups and four passes of 32 tokens).
// The 32 / tp lane groups of a token share its transform (each takes one block of the input dimension, at most 8
// blocks; a butterfly adds the partial sums, so every lane holds the same coefficients) and search disjoint
// ranges of the codebook; their minima are merged with the lowest index winning ties.
// Everything that depends only on the calibration is staged before the grid-dependency wait, so it
// overlaps the tail of the preceding kernel in the stream.
// The coefficients are accumulated in binary64 (index order inside a block, then the blocks pairwise).  The
// search is certified like search_tile: binary32 ranking, and a binary64 search by the whole warp
// wherever the two nearest codewords are closer than binary32 rounding can resolve (the binary64 pipe is the
// slowest unit of the SM: a binary64 search of every token was 60 % of this kernel's time after the launch).
// KSC (key format with a per-token scale): the L/4 CTAs of a (head, side) form a thread-block cluster;
// each publishes the sums of squares of its 16 coefficients per token in its shared memory, a cluster
// barrier makes them visible, and every CTA adds the L/4 x 4 partial sums in the same fixed order through
// distributed shared memory, so that all of them normalise by the same rho.
// Binary64 search of one coefficient vector (the same in every lane) against a group's 256 codewords by the
// whole warp: lane i takes codewords i, i + 32, ... in ascending order with a strict '<'; the lanes' minima are
// merged with the lowest index winning ties.  The distance is the plain sum of the four squares, every
// operation rounded to binary64.
__device__ __forceinline__ int exact_search_warp(const double (&rd)[4], const float4* cb /* shared, [256] */, int lane) {
    double best = CUDART_INF;
    int bi = lane;
#pragma unroll
    for (int j = 0; j < NOVAKV_C / 32; ++j) {
        const float4 c = cb[lane + 32 * j];
        const double e0 = rd[0] - (double)c.x, e1 = rd[1] - (double)c.y, e2 = rd[2] - (double)c.z, e3 = rd[3] - (double)c.w;
        const double dd = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(e0, e0), __dmul_rn(e1, e1)), __dmul_rn(e2, e2)), __dmul_rn(e3, e3));
        if (dd < best) { best = dd; bi = lane + 32 * j; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob < best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    return bi;
}

constexpr int SMALL_CTAS_PER_SM = 5;             // (shared memory allows six at d = 128; five leave a thread 96 registers)
constexpr int SMALL_TP_LOG2 = 3;
// Chunks of the token list that run side by side: all of their CTAs are resident together.
int small_append_chunks(const novakv_ctx* ctx) {
    return max(1, SMALL_CTAS_PER_SM * ctx->n_sm / (ctx->n_groups / 4 * ctx->cfg.n_kv_heads * 2));
}
// Batches up to this size take the append kernel, larger ones the prompt encoder.  The append kernel's time grows with every
// pass of 8 tokens of its longest chunk, and fewer KV heads leave room for more chunks; the encoder's is one unit per SM.  So the
// line lies behind two passes (never above 256 tokens).  us in a stream of calls, append kernel / encoder:
//                 heads   two passes at most                      three or more
//   d = 128 plain     1   256: 10.2 / 20.0
//                     2   128: 10.3 / 17.8   256: 17.7 / 21.7
//                     4    64: 10.2 / 17.7   160: 18.4 / 22.2     192: 25.2 / 22.3   256: 26.0 / 24.4
//                     8    32: 10.2 / 19.0    64: 17.7 / 19.5      96: 25.2 / 20.1   256: 55.8 / 25.6
//           scaled    1, 2, 4, 8 heads: 256: 11.9 / 30.7   256: 21.2 / 28.5   160: 21.8 / 26.5   64: 21.2 / 21.8, 96: 30.4 / 22.1
//           deployed                    256: 14.0 / 30.8   256: 25.5 / 27.2   160: 26.2 / 26.5   64: 25.4 / 21.8, 96: 36.4 / 21.9
//   d = 64  plain                       256:  5.0 / 16.6   256:  8.2 / 17.2   256: 14.4 / 18.3  160: 14.7 / 17.9, 192: 20.3 / 18.3
//           scaled                      256:  6.5 / 17.7   256:  9.5 / 19.6   256: 17.0 / 21.2  160: 17.0 / 19.3, 192: 24.2 / 19.4
// With eight heads and more it lies a little or a lot too high (16 / 32 heads, d = 128, 64 tokens: 32.5 / 20.0, 62 / 30): up to 64
// (d = 128) or 192 tokens (d = 64) the append kernel keeps its calls, whose bounds are derived where the encoder's are measured.
constexpr int SMALL_PASSES = 2;
constexpr int small_always(int d) { return d == 128 ? 64 : 192; }
int small_append_tokens(const novakv_ctx* ctx) {
    return max(small_always(ctx->cfg.head_dim), min(256, (small_append_chunks(ctx) * SMALL_PASSES) << SMALL_TP_LOG2));
}
template <int D, int FMT>
__global__ void __launch_bounds__(128, SMALL_CTAS_PER_SM)
novakv_encode_small_kernel(const __nv_bfloat16* __restrict__ k_new, const __nv_bfloat16* __restrict__ v_new,
                           const int32_t* __restrict__ tok_seq, const int32_t* __restrict__ tok_pos, int n_tokens,
                           int tp_log2,
                           const double* __restrict__ rk_d, const double* __restrict__ rv_d,
                           const double* __restrict__ k_mean_d, const double* __restrict__ v_mean_d,
                           const float* __restrict__ cb_k, const float* __restrict__ cb_v,
                           uint8_t* __restrict__ k_pages, uint8_t* __restrict__ v_pages,
                           __nv_bfloat16* __restrict__ k_scales, __nv_bfloat16* __restrict__ v_meta, int n_pages,
                           const int32_t* __restrict__ page_table, int max_pages_per_seq, int n_seq,
                           int32_t* __restrict__ seq_lens, int n_kv_heads, uint32_t* __restrict__ dev_status) {
    constexpr int L = D / NOVAKV_G;
    constexpr bool KSC = FMT >= 1, VSQ = FMT == 2;
    // Rows of the transform and the mean are indexed by i + i / (D / 4): one row of padding after every quarter of
    // the input dimension, so that lane groups working on different blocks of it read different banks.
    constexpr int DP = D + 4;
    auto padded = [](int i) { return i + i / (D / 4); };
    __shared__ __align__(16) double R_s[4][DP][4];
    __shared__ float4 cb_s[4][NOVAKV_C];
    __shared__ double mean_s[DP];
    __shared__ double ss_s[4][32];                  // KSC: sum of squares of a warp's 4 coefficients, per token of the pass
    __shared__ float mx_s[4][32];                   // VSQ: maximum of a warp's 4 value coefficients (the minimum rides in ss_s)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int l = blockIdx.x * 4 + warp, kvh = blockIdx.y, side = blockIdx.z & 1;
    const int chunk = blockIdx.z >> 1, n_chunks = gridDim.z >> 1;
    const __nv_bfloat16* x_new = side == 0 ? k_new : v_new;
    const double* R = (side == 0 ? rk_d : rv_d) + (size_t)kvh * D * D;
    const double* mean = (side == 0 ? k_mean_d : v_mean_d) + (size_t)kvh * D;
    const float4* cb_g = reinterpret_cast<const float4*>((side == 0 ? cb_k : cb_v) + ((size_t)kvh * L + l) * NOVAKV_C * NOVAKV_G);
#ifdef NOVAKV_TIMING
    long long tm[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    long long t_prev = clock64();
    unsigned long long g_a0, g_a1;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_a0));
#define NOVAKV_ETICK(i) { const long long t_now = clock64(); tm[i] += t_now - t_prev; t_prev = t_now; }
#else
#define NOVAKV_ETICK(i)
#endif
    {
        // calibration constants -> shared memory; every load is issued before the first store
        double2 ra[D / 32], rb[D / 32];
        float4 cw[NOVAKV_C / 32];
#pragma unroll
        for (int k = 0; k < D / 32; ++k) {
            ra[k] = *reinterpret_cast<const double2*>(R + ((size_t)l * D + lane + 32 * k) * 4);
            rb[k] = *reinterpret_cast<const double2*>(R + ((size_t)l * D + lane + 32 * k) * 4 + 2);
        }
#pragma unroll
        for (int k = 0; k < NOVAKV_C / 32; ++k) cw[k] = cb_g[lane + 32 * k];
        const double mv = threadIdx.x < D ? mean[threadIdx.x] : 0.0;
#pragma unroll
        for (int k = 0; k < D / 32; ++k) {
            *reinterpret_cast<double2*>(&R_s[warp][padded(lane + 32 * k)][0]) = ra[k];
            *reinterpret_cast<double2*>(&R_s[warp][padded(lane + 32 * k)][2]) = rb[k];
        }
#pragma unroll
        for (int k = 0; k < NOVAKV_C / 32; ++k) cb_s[warp][lane + 32 * k] = cw[k];
        if (threadIdx.x < D) mean_s[padded(threadIdx.x)] = mv;
    }
    __syncthreads();
    NOVAKV_ETICK(0)
    novakv_grid_dependency_wait();           // inputs and the cache may be written by preceding kernels
    NOVAKV_ETICK(1)

    const int tp = 1 << tp_log2;
    const int tok_in_pass = lane & (tp - 1), grp = lane >> tp_log2;
    const int codes_per_grp = NOVAKV_C >> (5 - tp_log2);
    const int c0 = grp * codes_per_grp;
    const bool reporter = blockIdx.x == 0 && warp == 0 && kvh == 0 && side == 0 && grp == 0;
    // the lane groups of a token also share its transform: each takes one block of the input dimension
    // (at most 8 blocks), and a butterfly over the lane groups adds the partial sums
    const int ts_log2 = min(5 - tp_log2, 3);
    const int part = grp & ((1 << ts_log2) - 1);
    constexpr int PER_MAX = (D / 8) >> (5 - SMALL_TP_LOG2);
    const int per = (D / 8) >> ts_log2;             // 16-byte chunks of the token row per lane (1 .. PER_MAX)

    for (int t0 = chunk * tp; t0 < n_tokens; t0 += n_chunks * tp) {
        const int tkn = t0 + tok_in_pass;
        const bool in_range = tkn < n_tokens;
        int s = -1, pos = 0;
        if (in_range) { s = tok_seq[tkn]; pos = tok_pos[tkn]; }
        // this lane's block of its token's row (the loads are in flight together with the token list's)
        uint4 xr[PER_MAX];
        const uint4* xrow = reinterpret_cast<const uint4*>(x_new + ((size_t)(in_range ? tkn : 0) * n_kv_heads + kvh) * D) + part * per;
#pragma unroll
        for (int c = 0; c < PER_MAX; ++c)
            if (c < per) xr[c] = xrow[c];
        // a pass whose entries are all unused does nothing (the same decision in every warp and CTA: it depends
        // on the token list alone)
        if (!__any_sync(0xffffffffu, s != -1)) continue;
        // destination: the page-table entry is requested here and looked at after the transform
        const bool ok = s >= 0 && s < n_seq && pos >= 0 && pos / NOVAKV_PAGE_TOKENS < max_pages_per_seq;
        if (s != -1 && !ok && reporter) atomicOr(dev_status, NOVAKV_DEV_BAD_TOKEN);
        int page_raw = -1;
        if (ok) page_raw = page_table[(size_t)s * max_pages_per_seq + pos / NOVAKV_PAGE_TOKENS];
        const int slot = pos % NOVAKV_PAGE_TOKENS;
        NOVAKV_ETICK(2)
        // coefficients of group l in binary64: every block of the input dimension in index order, then the blocks
        // pairwise (neighbours first); all lanes of a token end with the same bits
        double acc0 = 0.0, acc1 = 0.0, acc2 = 0.0, acc3 = 0.0;
#pragma unroll
        for (int c = 0; c < PER_MAX; ++c) {
            if (c < per) {
                const __nv_bfloat16* xb = reinterpret_cast<const __nv_bfloat16*>(&xr[c]);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = padded((part * per + c) * 8 + j);
                    const double xc = (double)__bfloat162float(xb[j]) - mean_s[i];
                    const double2 r01 = *reinterpret_cast<const double2*>(&R_s[warp][i][0]);
                    const double2 r23 = *reinterpret_cast<const double2*>(&R_s[warp][i][2]);
                    acc0 = fma(xc, r01.x, acc0);
                    acc1 = fma(xc, r01.y, acc1);
                    acc2 = fma(xc, r23.x, acc2);
                    acc3 = fma(xc, r23.y, acc3);
                }
            }
        }
        for (int b = 0; b < ts_log2; ++b) {
            const int off = tp << b;
            acc0 += __shfl_xor_sync(0xffffffffu, acc0, off);
            acc1 += __shfl_xor_sync(0xffffffffu, acc1, off);
            acc2 += __shfl_xor_sync(0xffffffffu, acc2, off);
            acc3 += __shfl_xor_sync(0xffffffffu, acc3, off);
        }
        int page = -1;
        if (ok) {
            if (page_raw < 0 || page_raw >= n_pages) {
                if (reporter) atomicOr(dev_status, NOVAKV_DEV_BAD_PAGE);
            } else {
                page = page_raw;
                if (reporter) atomicMax(&seq_lens[s], pos + 1);
            }
        }
        float4 r = make_float4((float)acc0, (float)acc1, (float)acc2, (float)acc3);
        NOVAKV_ETICK(3)
        int vsq_byte = 0;
        if (KSC) {
            namespace cg = cooperative_groups;
            cg::cluster_group cluster = cg::this_cluster();
            if (side == 0 && grp == 0) {
                double ss = (double)r.x * (double)r.x;
                ss = fma((double)r.y, (double)r.y, ss);
                ss = fma((double)r.z, (double)r.z, ss);
                ss = fma((double)r.w, (double)r.w, ss);
                ss_s[warp][tok_in_pass] = ss;
            }
            cluster.sync();                             // every CTA of the (head, side) has published its partial sums
            if (side == 0) {
                double tot = 0.0;
                for (unsigned cr = 0; cr < cluster.num_blocks(); ++cr) {
                    const double* remote = cluster.map_shared_rank(&ss_s[0][0], cr);
#pragma unroll
                    for (int w = 0; w < 4; ++w) tot += remote[w * 32 + tok_in_pass];
                }
                float rho = __bfloat162float(__float2bfloat16_rn((float)sqrt(tot / (double)D)));
                if (!(rho > 0.f) || !isfinite(rho)) rho = 1.f;
                r = make_float4(__fdiv_rn(r.x, rho), __fdiv_rn(r.y, rho), __fdiv_rn(r.z, rho), __fdiv_rn(r.w, rho));
                if (blockIdx.x == 0 && warp == 0 && grp == 0 && page >= 0)
                    k_scales[((size_t)page * n_kv_heads + kvh) * NOVAKV_PAGE_TOKENS + slot] = __float2bfloat16_rn(rho);
            }
            if (VSQ && side == 1 && grp == 0) {
                // value side: the warp's minimum and maximum travel in the same slots (as doubles)
                ss_s[warp][tok_in_pass] = (double)fminf(fminf(r.x, r.y), fminf(r.z, r.w));
                mx_s[warp][tok_in_pass] = fmaxf(fmaxf(r.x, r.y), fmaxf(r.z, r.w));
            }
            if (VSQ) cluster.sync();
            if (VSQ && side == 1) {
                float mn = CUDART_INF_F, mx = -CUDART_INF_F;
                for (unsigned cr = 0; cr < cluster.num_blocks(); ++cr) {
                    const double* rmn = cluster.map_shared_rank(&ss_s[0][0], cr);
                    const float* rmx = cluster.map_shared_rank(&mx_s[0][0], cr);
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        mn = fminf(mn, (float)rmn[w * 32 + tok_in_pass]);
                        mx = fmaxf(mx, rmx[w * 32 + tok_in_pass]);
                    }
                }
                const float zero = __bfloat162float(__float2bfloat16_rn(mn));
                float scale = __bfloat162float(__float2bfloat16_rn(__fdiv_rn(__fsub_rn(mx, zero), 3.0f)));
                if (!(scale > 0.f) || !isfinite(scale)) scale = 1.f;
                auto level = [&](float x) {
                    float u = rintf(__fdiv_rn(__fsub_rn(x, zero), scale));
                    if (!(u > 0.f)) u = 0.f;
                    return (int)fminf(u, 3.f);
                };
                vsq_byte = level(r.x) | (level(r.y) << 2) | (level(r.z) << 4) | (level(r.w) << 6);
                if (blockIdx.x == 0 && warp == 0 && grp == 0 && page >= 0)
                    reinterpret_cast<__nv_bfloat162*>(v_meta)[((size_t)page * n_kv_heads + kvh) * NOVAKV_PAGE_TOKENS + slot] =
                        __floats2bfloat162_rn(scale, zero);
            }
            cluster.sync();                             // partial sums may be overwritten by the next pass / CTAs may exit
        }
        // The vector to encode is the binary64 coefficient; for normalised keys it is the binary32 quotient.
        double rd[4] = {acc0, acc1, acc2, acc3};
        if (KSC && side == 0) { rd[0] = (double)r.x; rd[1] = (double)r.y; rd[2] = (double)r.z; rd[3] = (double)r.w; }
        // Certified search, as in search_tile: this lane group's range of the codebook is ranked in binary32
        // from the coefficient rounded to binary32 (first minimum in ascending order), with the second-smallest
        // distance tracked beside the smallest (equal distances count as two: their gap is zero).
        // The range is a whole number of blocks of 8 codewords.  Per block the 8 distances are independent; the block
        // minimum updates the running minimum with a strict '<' (keeps the first block that attains it), and the
        // larger of the two feeds the second-smallest value.  The winning block is then evaluated again (same
        // instructions, same bits): its first distance equal to the minimum gives the index, the others are the
        // remaining candidates for the second-smallest value.
        const float4* cbw = &cb_s[warp][c0];
        auto dist8 = [&](int blk, float (&d)[8]) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float4 cw = cbw[blk * 8 + k];
                const float e0 = r.x - cw.x, e1 = r.y - cw.y, e2 = r.z - cw.z, e3 = r.w - cw.w;
                d[k] = fmaf(e3, e3, fmaf(e2, e2, fmaf(e1, e1, e0 * e0)));
            }
        };
        float best = CUDART_INF_F, sec = CUDART_INF_F;
        int bblk = 0;
#pragma unroll 2
        for (int blk = 0; blk < codes_per_grp / 8; ++blk) {
            float d[8];
            dist8(blk, d);
            const float m = fminf(fminf(fminf(d[0], d[1]), fminf(d[2], d[3])), fminf(fminf(d[4], d[5]), fminf(d[6], d[7])));
            sec = fminf(sec, fmaxf(best, m));
            if (m < best) { best = m; bblk = blk; }
        }
        int bi;
        {
            float d[8];
            dist8(bblk, d);
            int kb = 7;
#pragma unroll
            for (int k = 6; k >= 0; --k)
                if (d[k] == best) kb = k;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k != kb) sec = fminf(sec, d[k]);
            bi = c0 + bblk * 8 + kb;
        }
        NOVAKV_ETICK(6)
        // merge the groups of a token: smaller distance wins, equal distances keep the lower index
        for (int off = tp; off < 32; off <<= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best, off);
            const float os = __shfl_xor_sync(0xffffffffu, sec, off);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
            sec = fminf(fminf(sec, os), fmaxf(best, ob));
            if (ob < best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        NOVAKV_ETICK(7)
        // Where binary32 rounding (of the coefficient: at most 2^-24 per component, none for the quotient, which is
        // a binary32 number; and of the distance) can have changed the order of the two nearest codewords, the whole
        // warp searches that token's group again in binary64.
        {
            float delta = 0.f;
            if (!(KSC && side == 0))
                delta = 5.97e-8f * sqrtf(fmaf(r.x, r.x, fmaf(r.y, r.y, fmaf(r.z, r.z, r.w * r.w)))) * 1.0001f;
            const bool need = grp == 0 && s != -1 && !(VSQ && side == 1) && needs_exact_search(best, sec, delta);
            unsigned todo = __ballot_sync(0xffffffffu, need);
#ifdef NOVAKV_TIMING
            tm[8] += __popc(todo);
#endif
            while (todo) {
                const int src = __ffs(todo) - 1;             // (a lane of lane group 0: its index is the token's)
                todo &= todo - 1;
                const double rs[4] = {__shfl_sync(0xffffffffu, rd[0], src), __shfl_sync(0xffffffffu, rd[1], src),
                                      __shfl_sync(0xffffffffu, rd[2], src), __shfl_sync(0xffffffffu, rd[3], src)};
                const int res = exact_search_warp(rs, cb_s[warp], lane);
                if (tok_in_pass == src) bi = res;
            }
        }
        NOVAKV_ETICK(4)
        if (VSQ && side == 1) bi = vsq_byte;             // scalar codec: the byte holds four levels, no search result
        if (grp == 0 && page >= 0) {
            const size_t base = ((size_t)page * n_kv_heads + kvh) * (NOVAKV_PAGE_TOKENS * L);
            if (side == 0) k_pages[base + novakv_k_offset<L>(slot, l)] = (uint8_t)bi;
            else v_pages[base + novakv_v_offset<L>(slot, l)] = (uint8_t)bi;
        }
    }
#ifdef NOVAKV_TIMING
    NOVAKV_ETICK(5)
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_a1));
    if (threadIdx.x == 0 && blockIdx.y == 0 && blockIdx.z < 2 && (blockIdx.x == 0 || blockIdx.x == gridDim.x - 1))
        printf("append cta (%d,%d,%d) clocks: constants %lld dependency wait %lld rows+lookup %lld transform %lld ranking %lld merge %lld certificate+re-search %lld (%lld re-searches) store %lld | ns start %llu end %llu\n",
               blockIdx.x, blockIdx.y, blockIdx.z, tm[0], tm[1], tm[2], tm[3], tm[6], tm[7], tm[4], tm[8], tm[5], g_a0, g_a1);
#endif
}

// Search only, from given binary32 coefficients [n][Hkv][D]; logical indices out [n][Hkv][L].
template <int D>
__global__ void __launch_bounds__(ENC_THREADS, 1)
novakv_search_kernel(const float* __restrict__ coef, int n, const float* __restrict__ cb_all, int n_kv_heads,
                     uint8_t* __restrict__ idx_out) {
    constexpr int L = D / NOVAKV_G;
    constexpr int RS = EncSmem<D>::RSTRIDE;
    extern __shared__ __align__(16) unsigned char smem[];
    float4* cb_s = reinterpret_cast<float4*>(smem);
    float* r_s = reinterpret_cast<float*>(smem + EncSmem<D>::cb_bytes);
    uint8_t* idx_s = smem + EncSmem<D>::cb_bytes + EncSmem<D>::r_bytes;
    const int kvh = blockIdx.y;
    const float4* cb_g = reinterpret_cast<const float4*>(cb_all + (size_t)kvh * L * NOVAKV_C * NOVAKV_G);
    fill_codebook_pairs(reinterpret_cast<float*>(cb_s), cb_g, L);
    const int n_tiles = (n + ENC_TILE - 1) / ENC_TILE;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int t0 = tile * ENC_TILE;
        const int n_valid = min(ENC_TILE, n - t0);
        __syncthreads();
        for (int i = threadIdx.x; i < ENC_TILE * D; i += ENC_THREADS) {
            const int t = i / D, c = i - t * D;
            r_s[(size_t)t * RS + c] = t < n_valid ? coef[((size_t)(t0 + t) * n_kv_heads + kvh) * D + c] : 0.f;
        }
        __syncthreads();
        search_tile<D>(r_s, cb_s, idx_s, n_valid, threadIdx.x >> 5, ENC_THREADS / 32);
        __syncthreads();
        for (int i = threadIdx.x; i < n_valid * L; i += ENC_THREADS) {
            const int t = i / L, l = i - t * L;
            idx_out[((size_t)(t0 + t) * n_kv_heads + kvh) * L + l] = idx_s[i];
        }
    }
}

template <int D>
novakv_status launch_encode_t(novakv_ctx* ctx, const novakv_layer& ly, const __nv_bfloat16* k_new,
                              const __nv_bfloat16* v_new, const int32_t* tok_seq, const int32_t* tok_pos,
                              int n_tokens, uint8_t* k_pages, uint8_t* v_pages, int n_pages,
                              const int32_t* page_table, int max_pages_per_seq, int n_seq, int32_t* seq_lens,
                              cudaStream_t stream, __nv_bfloat16* k_scales, __nv_bfloat16* v_meta) {
    // (the append kernel reads the new rows in 16-byte pieces; rows on a 4-byte boundary take the prompt encoder, which can
    // copy them in words, whatever their number)
    const bool rows16 = (((uintptr_t)k_new | (uintptr_t)v_new) & 15) == 0;
    if (n_tokens <= small_append_tokens(ctx) && rows16) {
        int tp_log2 = 0;
        while ((1 << tp_log2) < n_tokens && tp_log2 < SMALL_TP_LOG2) ++tp_log2;
        // chunks of the token list: as many as there are passes, while all CTAs are resident together, and no more than the
        // longest chunk needs (every chunk stages the constants): 64 tokens, d = 128, plain: 5 chunks 23.4 us cold and 18.0
        // warm, 4 chunks 20.5 and 17.4
        const int passes = (n_tokens + (1 << tp_log2) - 1) >> tp_log2, resident = min(passes, small_append_chunks(ctx));
        const int longest = (passes + resident - 1) / resident, chunks = (passes + longest - 1) / longest;
        dim3 grid(D / NOVAKV_G / 4, ctx->cfg.n_kv_heads, 2 * chunks);
        novakv_prof_scope ps(ctx, 1, stream);
        auto small = v_meta ? novakv_encode_small_kernel<D, 2>
                            : (k_scales ? novakv_encode_small_kernel<D, 1> : novakv_encode_small_kernel<D, 0>);
        if (k_scales == nullptr) {
            novakv_launch_pdl(novakv_encode_small_kernel<D, 0>, grid, dim3(128), 0, stream, k_new, v_new, tok_seq, tok_pos,
                              n_tokens, tp_log2, ly.rk_d, ly.rv_d, ly.k_mean_d, ly.v_mean_d, ly.cb_k, ly.cb_v, k_pages, v_pages,
                              (__nv_bfloat16*)nullptr, (__nv_bfloat16*)nullptr, n_pages, page_table, max_pages_per_seq, n_seq, seq_lens,
                              ctx->cfg.n_kv_heads, ctx->dev_status);
        } else {
            // scaled key format: the L/4 CTAs of a (head, side) are one cluster (8 at d = 128, 4 at d = 64)
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = grid;
            cfg.blockDim = dim3(128);
            cfg.stream = stream;
            cudaLaunchAttribute attr[2];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            attr[1].id = cudaLaunchAttributeClusterDimension;
            attr[1].val.clusterDim.x = grid.x;
            attr[1].val.clusterDim.y = 1;
            attr[1].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 2;
            const int hkv = ctx->cfg.n_kv_heads;
            if (cudaLaunchKernelEx(&cfg, small, k_new, v_new, tok_seq, tok_pos, n_tokens, tp_log2,
                                   (const double*)ly.rk_d, (const double*)ly.rv_d, (const double*)ly.k_mean_d,
                                   (const double*)ly.v_mean_d, (const float*)ly.cb_k, (const float*)ly.cb_v, k_pages, v_pages,
                                   k_scales, v_meta, n_pages, page_table, max_pages_per_seq, n_seq, seq_lens, hkv,
                                   ctx->dev_status) != cudaSuccess)
                return NOVAKV_ECUDA;
        }
        ps.end();
        ctx->launches++;
        return cudaGetLastError() == cudaSuccess ? NOVAKV_OK : NOVAKV_ECUDA;
    }
    return novakv_launch_prefill(ctx, ly, k_new, v_new, tok_seq, tok_pos, n_tokens, k_pages, v_pages, n_pages, page_table,
                                 max_pages_per_seq, n_seq, seq_lens, stream, k_scales, v_meta);
}

template <int D>
novakv_status launch_search_t(novakv_ctx* ctx, const novakv_layer& ly, int which, const float* coef, int n,
                              uint8_t* idx_out, cudaStream_t stream) {
    auto kern = novakv_search_kernel<D>;
    const size_t smem = EncSmem<D>::total;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return NOVAKV_ECUDA;
    const int n_tiles = (n + ENC_TILE - 1) / ENC_TILE;
    // CTAs per head: about two whole waves of the machine
    dim3 grid(max(1, min(n_tiles, (2 * ctx->n_sm) / ctx->cfg.n_kv_heads)), ctx->cfg.n_kv_heads);
    kern<<<grid, ENC_THREADS, smem, stream>>>(coef, n, which == 0 ? ly.cb_k : ly.cb_v, ctx->cfg.n_kv_heads, idx_out);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? NOVAKV_OK : NOVAKV_ECUDA;
}

}  // namespace

int novakv_append_kernel_tokens(const novakv_ctx* ctx) { return small_append_tokens(ctx); }

novakv_status novakv_launch_encode(novakv_ctx* ctx, const novakv_layer& ly, const __nv_bfloat16* k_new,
    const __nv_bfloat16* v_new, const int32_t* tok_seq, const int32_t* tok_pos, int n_tokens,
    uint8_t* k_pages, uint8_t* v_pages, int n_pages, const int32_t* page_table,
    int max_pages_per_seq, int n_seq, int32_t* seq_lens, cudaStream_t stream, __nv_bfloat16* k_scales,
    __nv_bfloat16* v_meta) {
    if (v_meta != nullptr && k_scales == nullptr) return NOVAKV_EUNSUPPORTED;   // INT2 values come with scaled keys
    if (ctx->cfg.head_dim == 128)
        return launch_encode_t<128>(ctx, ly, k_new, v_new, tok_seq, tok_pos, n_tokens, k_pages, v_pages, n_pages,
                                    page_table, max_pages_per_seq, n_seq, seq_lens, stream, k_scales, v_meta);
    return launch_encode_t<64>(ctx, ly, k_new, v_new, tok_seq, tok_pos, n_tokens, k_pages, v_pages, n_pages,
                               page_table, max_pages_per_seq, n_seq, seq_lens, stream, k_scales, v_meta);
}

// Gather of up to 5 page-locked host buffers into device staging: every word crosses the bus once, consecutive threads take
// consecutive words, 16 bytes each where a buffer allows it (a quarter of the read requests).  The buffers are one list of
// words over all threads of the grid, so that every read is in flight at once: a thread that went through the buffers one
// after the other waited for a round trip over the bus (about 2 us) in each.  4 sequences of the d = 64 shape with eight heads
// (44 KB), host-buffer step with the wait: 47.5 -> 42.7 us; one sequence of the d = 128 shape 41.5 -> 38.2.
__device__ __forceinline__ bool stage_in_16(const novakv_stage_args& a, int sgm) {
    return ((reinterpret_cast<uintptr_t>(a.src[sgm]) | reinterpret_cast<uintptr_t>(a.dst[sgm])) & 15) == 0 && (a.words[sgm] & 3) == 0;
}
__global__ void __launch_bounds__(256) novakv_stage_kernel(const __grid_constant__ novakv_stage_args a) {
    // an append behind this kernel may start its prologue (calibration constants) now; it waits for this grid's completion
    // before it touches the staged inputs.  (The query blocks of a decode call do not wait: see novakv_prepare_kernel.)
    if (a.release) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x;; i += gridDim.x * blockDim.x) {
        unsigned j = i;                                     // place in its buffer
        int sgm = 0;
        bool by16 = false;
#pragma unroll 1
        for (; sgm < a.n; ++sgm) {
            by16 = stage_in_16(a, sgm);
            const unsigned units = by16 ? a.words[sgm] / 4 : a.words[sgm];
            if (j < units) break;
            j -= units;
        }
        if (sgm == a.n) break;
        if (by16) reinterpret_cast<uint4*>(a.dst[sgm])[j] = reinterpret_cast<const uint4*>(a.src[sgm])[j];
        else a.dst[sgm][j] = a.src[sgm][j];
    }
}

novakv_status novakv_launch_stage(novakv_ctx* ctx, const novakv_stage_args& a, cudaStream_t stream) {
    unsigned total = 0;
    for (int i = 0; i < a.n; ++i) {
        const bool by16 = ((reinterpret_cast<uintptr_t>(a.src[i]) | reinterpret_cast<uintptr_t>(a.dst[i])) & 15) == 0 && (a.words[i] & 3) == 0;
        total += by16 ? a.words[i] / 4 : a.words[i];
    }
    if (total == 0) return NOVAKV_OK;
    unsigned blocks = (total + 255) / 256;              // a word for every thread
    if (blocks > (unsigned)(8 * ctx->n_sm)) blocks = 8 * ctx->n_sm;
    novakv_stage_kernel<<<blocks, 256, 0, stream>>>(a);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? NOVAKV_OK : NOVAKV_ECUDA;
}

// ------------------------------------------------------------------------------------------------
// BF16 band, write side: one new token per sequence (App. B "Sink-plus-recent band")
// ------------------------------------------------------------------------------------------------
// One block per sequence.  Thread 0 advances the sequence's (sink_cnt, ring_start, ring_len, quantised
// length); the block copies the new token into its band slot and, when the ring has reached n_rec + block
// tokens, copies the block oldest ring tokens to the staging rows b * block + i with their (sequence,
// position) entries.  Rows of sequences that flush nothing get the "unused" marker (sequence -1).
__global__ void __launch_bounds__(256)
novakv_band_insert_kernel(const uint4* __restrict__ k_new, const uint4* __restrict__ v_new, uint4* __restrict__ band_k,
                          uint4* __restrict__ band_v, int band_cap, int n_sink, int n_rec, int block,
                          int32_t* __restrict__ band_meta, int32_t* __restrict__ quant_lens, int row_u4 /* Hkv * d / 8 */,
                          uint4* __restrict__ stage_k, uint4* __restrict__ stage_v, int32_t* __restrict__ tok_seq,
                          int32_t* __restrict__ tok_pos) {
    const int b = blockIdx.x;
    const int ring_cap = band_cap - n_sink;
    __shared__ int s_slot, s_flush, s_rs, s_q;
    if (threadIdx.x == 0) {
        int sc = band_meta[b * 3], rs = band_meta[b * 3 + 1], rl = band_meta[b * 3 + 2], q = quant_lens[b];
        // (state written by this kernel stays in range; a caller's out-of-range state is pulled back into it)
        sc = min(max(sc, 0), n_sink);
        rs = min(max(rs, 0), ring_cap - 1);
        rl = min(max(rl, 0), n_rec + block - 1);
        q = max(q, 0);
        int slot;
        if (sc < n_sink) { slot = sc; ++sc; }
        else { slot = n_sink + (rs + rl) % ring_cap; ++rl; }
        const int flush = rl >= n_rec + block;
        s_slot = slot; s_flush = flush; s_rs = rs; s_q = q;
        if (flush) { rs = (rs + block) % ring_cap; rl -= block; q += block; }
        band_meta[b * 3] = sc; band_meta[b * 3 + 1] = rs; band_meta[b * 3 + 2] = rl;
        quant_lens[b] = q;
    }
    __syncthreads();
    {
        const size_t dst = ((size_t)b * band_cap + s_slot) * row_u4, src = (size_t)b * row_u4;
        for (int i = threadIdx.x; i < row_u4; i += blockDim.x) { band_k[dst + i] = k_new[src + i]; band_v[dst + i] = v_new[src + i]; }
    }
    if (s_flush) {
        // the new token's slot is not among the block oldest ones (the ring holds at least n_rec > 0 more)
        for (int i = threadIdx.x; i < block * row_u4; i += blockDim.x) {
            const int t = i / row_u4, w = i - t * row_u4;
            const size_t src = ((size_t)b * band_cap + n_sink + (s_rs + t) % ring_cap) * row_u4 + w;
            const size_t dst = ((size_t)b * block + t) * row_u4 + w;
            stage_k[dst] = band_k[src];
            stage_v[dst] = band_v[src];
        }
    }
    for (int t = threadIdx.x; t < block; t += blockDim.x) {
        tok_seq[b * block + t] = s_flush ? b : -1;
        tok_pos[b * block + t] = n_sink + s_q + t;
    }
}

novakv_status novakv_launch_band_insert(novakv_ctx* ctx, const void* k_new, const void* v_new, int batch, void* band_k,
    void* band_v, int band_cap, int n_sink, int n_rec, int block, int32_t* band_meta, int32_t* quant_lens,
    void* stage_k, void* stage_v, int32_t* tok_seq, int32_t* tok_pos, cudaStream_t stream) {
    const int row_u4 = ctx->cfg.n_kv_heads * ctx->cfg.head_dim / 8;
    novakv_band_insert_kernel<<<batch, 256, 0, stream>>>((const uint4*)k_new, (const uint4*)v_new, (uint4*)band_k, (uint4*)band_v,
                                                        band_cap, n_sink, n_rec, block, band_meta, quant_lens, row_u4,
                                                        (uint4*)stage_k, (uint4*)stage_v, tok_seq, tok_pos);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? NOVAKV_OK : NOVAKV_ECUDA;
}

novakv_status novakv_launch_search(novakv_ctx* ctx, const novakv_layer& ly, int which, const float* coef,
    int n, uint8_t* idx_out, cudaStream_t stream) {
    if (ctx->cfg.head_dim == 128) return launch_search_t<128>(ctx, ly, which, coef, n, idx_out, stream);
    return launch_search_t<64>(ctx, ly, which, coef, n, idx_out, stream);
}
