// Read path: decode-step attention straight from the packed index cache.
//
//   prepare  : q' = sm_scale*log2(e) * q rk_inv_t  per head.  (For large batches also a prefix sum of page counts, the
//              work list of the scan kernel: one unit = one 64-token page of one (sequence, KV head); the scan forms it
//              itself otherwise.)
//   stage 1  : persistent scan kernel, one CTA per SM.  Each CTA takes a contiguous range of the
//              global page sequence, so that consecutive pages mostly belong to the same
//              (sequence, KV head) and reuse its score table.  Per (sequence, KV head) segment:
//                - score table LUT[code][l][h] = <q'_h[4l..4l+3], cb_k[l][code] - centre_l> in shared memory,
//                  all heads of the KV head side by side in one entry.  The first K32 groups, which carry
//                  the high-variance coordinates and hence the large entries, are kept in binary32; the
//                  others (head dimension 128 only) in binary16,
//                - every warp streams its own 32-token tiles with coalesced 128-bit loads straight into
//                  registers, the next tile's loads in flight while the current tile is consumed (the
//                  cache layout is such that each lane's bytes are exactly the ones it consumes),
//                - key side: lane <-> token, L table lookups summed in registers (no cross-lane
//                  reduction): binary32 adds for the binary32 entries, short binary16 chains, each
//                  flushed into the binary32 sum, for the others,
//                - online softmax per 32-token tile with a lazily updated running maximum,
//                - value side: sum_j p_j * value-codeword_j in the value-transform domain, a dense
//                  [heads x tokens] x [tokens x d] contraction, run on tensor cores (mma.sync, binary16
//                  operands, binary32 accumulators) or, as the selectable alternative, on CUDA cores in
//                  binary32; value codewords are 7-bit grid indices (4 bytes per codeword) that expand to
//                  binary16 with one byte permutation per pair,
//                - the warps' partial (m, l, acc) are merged and written once per segment.
//   merge    : exact log-sum-exp merge of the partials of every (sequence, KV head), then the inverse
//              value transform o = o' rv^T + v_mean, once per head.
//
// Shared-memory gathers are laid out against bank conflicts: byte j of a token's key bytes holds group
// j ^ (token % 8) (j ^ (token % 16) for j >= 16), so that at every step the lanes of a quarter warp read 8
// different 16-byte columns of a binary32 table row and the lanes of a half warp 16 different 8-byte
// columns of a binary16 row (steps 8..15 meet only 8 groups: those groups are stored a second time in the
// unused first columns of the row and the upper half of a half warp reads the copy); on the value
// side the 32 lanes of a warp read 32 different 4-byte slots, because the lane columns fc = 0,1 and fc = 2,3
// use two copies of the value codebook whose slots are rotated by 16, and odd columns take the group
// blocks in swapped order (the cache stores their bytes in that order, and the byte permutation that widens a
// codeword for the tensor core picks it from the swapped register).
// The kernel contains no spin wait.
#include <math_constants.h>
#ifdef NOVAKV_TIMING
#include <cstdio>
#endif

#include "novakv_internal.cuh"

namespace {

#ifndef NOVAKV_NCW
#define NOVAKV_NCW 16
#endif
#ifndef NOVAKV_CHAIN
#define NOVAKV_CHAIN 4        // table lookups summed in binary16 before a flush into the binary32 logit
#endif
#ifndef NOVAKV_KSC_CHAIN
#define NOVAKV_KSC_CHAIN 2
#endif
#ifndef NOVAKV_WINDOW
#define NOVAKV_WINDOW 8       // tiles whose tensor-core sums are accumulated before the centre of the value grid is removed
#endif
constexpr int NCW = NOVAKV_NCW;               // warps of the scan kernel
constexpr int S1_THREADS = NCW * 32;
constexpr int T16_BYTES = 65536;              // binary16 table: 256 codes x 256-byte rows
constexpr int T16_ROW = 256;
constexpr int VCB_COPY_BYTES = 32768;         // 256 codes x 32 slots x 4 bytes
constexpr int VCB_ROW = 128;
constexpr int S1_SMEM_BYTES = 229376;         // dynamic shared memory requested (224 KB; the CTA also has a few static words)
constexpr float M_INIT = -1.0e30f;
#ifndef NOVAKV_M_SLACK
#define NOVAKV_M_SLACK 4
#endif
constexpr float M_SLACK = (float)NOVAKV_M_SLACK;   // headroom (bits) a running maximum gets when it moves
constexpr int MAX_SCAN_CTAS = 255;            // scan CTAs (one per SM) the boundary table has room for
constexpr int MMA_MIN_PAGES = 5;              // pages per SM from which on the d = 64 kernel with tensor-core logits is taken
constexpr int PFX_CAP = 511;                  // batches up to this size keep their page / cost prefixes in shared memory

// VM selects the value side: true = tensor cores (mma.sync m16n8k16, fp16 weights and codewords,
// fp32 accumulators), false = CUDA cores (fp32 FMA).
template <int D, int HG, bool VM>
struct S1 {
    static constexpr int L = D / NOVAKV_G;
    static constexpr int NGB = L / 8;                         // group blocks of 8 groups (value side)
    static constexpr int KPL = L / 16;                        // 16-byte planes of a key tile: 2 or 1
    static constexpr int HSETS = HG <= 4 ? 1 : 2;             // sets of 4 heads
    static constexpr int HPAD = HSETS * 4;
    // Score table.  Groups 0 .. K32-1 (the equal-volume dealing puts the coordinates of largest variance there)
    // have binary32 entries, 16 bytes per head set: T32[hs][code][K32][4 heads].  The other groups have
    // binary16 entries, 8 bytes: T16[code][32 columns][4 heads], rows of 256 bytes (only for d = 128, where
    // Hq/Hkv <= 4).  For d = 64 every group is binary32.
    static constexpr int K32 = D == 128 ? 8 : L;
    static constexpr bool HAS16 = K32 < L;
    static_assert(!HAS16 || HSETS == 1, "binary16 entries hold one head set");
    static constexpr int ROW32 = 256;
    static constexpr int PLANE32 = 256 * ROW32;
    static constexpr int T32_BYTES = HSETS * PLANE32;
    static constexpr int TILE_BYTES = 32 * L;                 // index bytes of a 32-token tile, K or V
    // per-warp staging of the softmax weights of one 32-token tile
    //   VM: fp16 [HPAD][4 k-slot pairs][8 tokens]        otherwise: fp32 [32 tokens][HPAD]
    static constexpr int P_WARP_BYTES = VM ? HPAD * 64 : 32 * HPAD * 4;
    static constexpr int P_BYTES = NCW * P_WARP_BYTES;
    // Shared-window addresses, fixed so that they are immediates of the gathers.  Rows of 256 bytes: one byte permutation
    // puts a code above a column byte.  (The window's first KB and the static words lie below; checked at run time.)
    static constexpr int T16 = 4096;
    static constexpr int T32 = T16 + (HAS16 ? T16_BYTES : 0);
    static constexpr int VCB = T32 + T32_BYTES;                         // two copies of the value codebook
    static constexpr int P = VCB + 2 * VCB_COPY_BYTES;
    static constexpr int Q_BYTES = HPAD * D * 4;
    static constexpr int Q = P + P_BYTES;                               // fp32 [HPAD][D], of the present and of the next pair
    static constexpr int BND = Q + 2 * Q_BYTES;                        // long [MAX_SCAN_CTAS + 1]: first unit of every CTA
    static constexpr int PFX = BND + (MAX_SCAN_CTAS + 1) * 8;           // int [2][PFX_CAP + 1]: page and cost prefix of small batches
    static constexpr int SMEM = PFX + 2 * (PFX_CAP + 1) * 4;
    // merge buffer (aliases the larger table once a segment's scan is done)
    static constexpr int MROW = D + 4;                                  // floats per (warp, head) row of the merge buffer: 16 bytes of padding
                                                                        // keep the four head rows a warp writes at once on different banks
    static constexpr int MERGE_ACC_BYTES = NCW * HPAD * MROW * 4;
    static_assert(MERGE_ACC_BYTES + NCW * HPAD * 16 <= (HAS16 ? T16_BYTES : T32_BYTES), "merge buffer must fit in a table");
    static_assert(SMEM <= S1_SMEM_BYTES, "shared memory budget");
    static_assert(S1_THREADS % L == 0, "table build mapping");
};

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ int clamp_len(int len, int max_pages) {
    const int cap = max_pages * NOVAKV_PAGE_TOKENS;
    return len < 0 ? 0 : (len > cap ? cap : len);
}

// ------------------------------------------------------------------------------------------------
// prepare: query transform + page prefix
// ------------------------------------------------------------------------------------------------
// One block per KV head and run of `seqs_per_block` sequences: its share of rk_inv_t is read once into registers, and the
// Hg queries of a (sequence, head) share it.  512 threads = D columns x (512/D) row parts; each thread's loads are
// independent and all in flight.  Small batches take one sequence per block, in an instantiation without the loop (RUNS =
// false: the loop's registers cost 0.7 us of 4.1, cold, at 8 sequences x 8 heads); once there are more pairs than the
// machine holds blocks, runs save the 64 KB per pair that re-reading the transform costs: 128 sequences x 8 heads,
// d = 128: 13.5 -> 8.2 us.
constexpr int PREPARE_RUN = 8;                 // sequences per block at most
template <int D, int HG, bool RUNS>
__global__ void __launch_bounds__(512)
novakv_prepare_kernel(const __nv_bfloat16* __restrict__ q, const float* __restrict__ rk_inv_t,
                      const int32_t* __restrict__ seq_lens, int batch, int n_q_heads, int n_kv_heads,
                      int max_pages_per_seq, float scale_log2, float* __restrict__ qp,
                      int32_t* __restrict__ page_prefix, uint32_t* __restrict__ dev_status,
                      const float* __restrict__ k_mean /* [Hkv][D] */, float* __restrict__ qk_off /* [batch][Hq] or null */,
                      int32_t* __restrict__ cost_prefix /* [batch + 1] */, int seg_weight,
                      const float* __restrict__ k_center /* [Hkv][D], transform domain */, float* __restrict__ qc /* [batch][Hq] or null */,
                      int32_t* __restrict__ pair_count /* [Hkv * batch] arrival counters of the fused merge, or null */,
                      void* __restrict__ out_fused /* outputs, when the scan kernel itself merges */, int out_is_fp32,
                      int seqs_per_block, int form_prefix /* 0: the scan kernel forms the prefixes */) {
    const int blk = blockIdx.x;
#ifdef NOVAKV_TIMING
    unsigned long long g_p0, g_p1;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_p0));
#endif
    constexpr int PARTS = 512 / D, ROWS = D / PARTS;
    const int run = blk / n_kv_heads, kvh = blk - run * n_kv_heads;
    const int c = threadIdx.x % D, part = threadIdx.x / D;
    // The query transform depends on nothing the preceding kernel of the stream (normally the append of this
    // step's tokens) writes: queries are produced before that kernel started, the transform is a constant.  So
    // the blocks that transform queries run beside the preceding kernel.  They write nothing before it has completed: it
    // may still read what shares memory with this call's workspace (the partials of another call on that scratch, new
    // rows whose tensor has been freed).  The blocks keep their place until then, so the scan's come later: append + decode of
    // 1 x 777 18.1 -> 18.3 us, 32 x 8191 scaled 80.8 -> 82.2, the 128-sequence mix 281 -> 286 against writing at once.  (Fewer blocks, as
    // many as SMs: the mix 285, but 64 x 200 36.2 -> 38.9.)
    const int n_query_blocks = (int)gridDim.x - form_prefix;
    float rv[ROWS];
    if (blk < n_query_blocks) {
        const float* R = rk_inv_t + (size_t)kvh * D * D + (size_t)part * ROWS * D + c;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) rv[r] = R[(size_t)r * D];
    }
    if (blk == n_query_blocks) {
        novakv_grid_dependency_wait();
        // exclusive prefix over sequences of their page counts; small, done by one warp.  Beside it the same
        // prefix in "cost" units, in which every non-empty sequence weighs seg_weight pages more: the scan
        // kernel splits the walk evenly in cost, so that a CTA that has to set up several (sequence, KV head)
        // segments gets fewer pages.
        if (threadIdx.x < 32) {
            int carry = 0, carry_ne = 0;
            for (int b0 = 0; b0 < batch; b0 += 32) {
                const int b = b0 + threadIdx.x;
                int v = 0;
                if (b < batch) {
                    const int raw = seq_lens[b];
                    const int len = clamp_len(raw, max_pages_per_seq);
                    if (raw != len) atomicOr(dev_status, NOVAKV_DEV_BAD_LENGTH);
                    v = (len + NOVAKV_PAGE_TOKENS - 1) / NOVAKV_PAGE_TOKENS;
                }
                const int ne = v > 0 ? 1 : 0;
                int incl = v, incl_ne = ne;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, o);
                    const int tn = __shfl_up_sync(0xffffffffu, incl_ne, o);
                    if ((int)threadIdx.x >= o) { incl += t; incl_ne += tn; }
                }
                if (b < batch) {
                    page_prefix[b] = carry + incl - v;
                    cost_prefix[b] = carry + incl - v + seg_weight * (carry_ne + incl_ne - ne);
                }
                // no scan CTA ever visits an empty sequence: with the merge fused into the scan its zeros are written here
                if (out_fused != nullptr) {
                    const unsigned empties = __ballot_sync(0xffffffffu, b < batch && v == 0);
                    for (unsigned m = empties; m; m &= m - 1) {
                        const size_t row = (size_t)(b0 + __ffs(m) - 1) * n_q_heads * D;
                        for (int i = threadIdx.x; i < n_q_heads * D; i += 32) {
                            if (out_is_fp32) reinterpret_cast<float*>(out_fused)[row + i] = 0.f;
                            else reinterpret_cast<__nv_bfloat16*>(out_fused)[row + i] = __float2bfloat16_rn(0.f);
                        }
                    }
                }
                carry += __shfl_sync(0xffffffffu, incl, 31);
                carry_ne += __shfl_sync(0xffffffffu, incl_ne, 31);
            }
            if (threadIdx.x == 0) { page_prefix[batch] = carry; cost_prefix[batch] = carry + seg_weight * carry_ne; }
        }
#ifdef NOVAKV_TIMING
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_p1));
        if (threadIdx.x == 0) printf("prepare prefix block | ns start %llu end %llu\n", g_p0, g_p1);
#endif
        return;
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    static_assert(HG * D <= 512, "a thread for every coordinate of a KV head's queries");
    constexpr int RUN = RUNS ? PREPARE_RUN : 1;
    __shared__ float q_s[HG][D];
    __shared__ float red_s[PARTS][HG][D];
    __shared__ float qp_s[RUN][HG * D], qk_s[RUN][HG], qc_s[RUN][HG];            // results, until they may be written
    const int b0 = RUNS ? run * seqs_per_block : run, b_end = RUNS ? min(batch, b0 + seqs_per_block) : run + 1;
    for (int b = b0; b < b_end; ++b) {
        if (RUNS && b != b0) __syncthreads();                  // the shared arrays are free
        for (int i = threadIdx.x; i < HG * D; i += 512)
            q_s[i / D][i % D] = __bfloat162float(q[((size_t)b * n_q_heads + kvh * HG) * D + i]);
        __syncthreads();
        float acc[HG];
#pragma unroll
        for (int h = 0; h < HG; ++h) acc[h] = 0.f;
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
#pragma unroll
            for (int h = 0; h < HG; ++h) acc[h] = fmaf(q_s[h][part * ROWS + r], rv[r], acc[h]);
#pragma unroll
        for (int h = 0; h < HG; ++h) red_s[part][h][c] = acc[h];
        __syncthreads();
        if (threadIdx.x < HG * D) {
            const int h = threadIdx.x / D, cc = threadIdx.x % D;
            float v = 0.f;
#pragma unroll
            for (int p = 0; p < PARTS; ++p) v += red_s[p][h][cc];
            v *= scale_log2;
            qp_s[b - b0][threadIdx.x] = v;
            if (qc != nullptr) red_s[0][h][cc] = v * k_center[(size_t)kvh * D + cc];       // (each thread rewrites only what it read)
        }
        // the constant the read path drops from every logit of a query, q . k_mean * sm_scale (base-2 units):
        // only a learned sink logit and the BF16 band need it (they must be shifted by the same amount)
        if (qk_off != nullptr && (threadIdx.x >> 5) < HG) {
            const int h = threadIdx.x >> 5, lane = threadIdx.x & 31;
            float acc = 0.f;
            for (int i = lane; i < D; i += 32) acc = fmaf(q_s[h][i], k_mean[(size_t)kvh * D + i], acc);
            acc = warp_sum_f(acc);
            if (lane == 0) qk_s[b - b0][h] = acc * scale_log2;
        }
        // scaled key format: the table is built from centred codewords, and the centre's share <q', centre> of
        // every logit is added back before the per-token scale multiplies it
        if (qc != nullptr) {
            __syncthreads();
            if ((threadIdx.x >> 5) < HG) {
                const int h = threadIdx.x >> 5, lane = threadIdx.x & 31;
                float acc = 0.f;
                for (int i = lane; i < D; i += 32) acc += red_s[0][h][i];
                acc = warp_sum_f(acc);
                if (lane == 0) qc_s[b - b0][h] = acc;
            }
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (qk_off != nullptr || qc != nullptr) __syncthreads();    // (qp_s: every thread writes out what it put there)
    for (int b = b0; b < b_end; ++b) {
        const size_t row = (size_t)b * n_q_heads + kvh * HG;
        if (threadIdx.x < HG * D) qp[row * D + threadIdx.x] = qp_s[b - b0][threadIdx.x];
        if (threadIdx.x < HG) {
            if (qk_off != nullptr) qk_off[row + threadIdx.x] = qk_s[b - b0][threadIdx.x];
            if (qc != nullptr) qc[row + threadIdx.x] = qc_s[b - b0][threadIdx.x];
        }
        if (pair_count != nullptr && threadIdx.x == 0) pair_count[kvh * batch + b] = 0;
    }
#ifdef NOVAKV_TIMING
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_p1));
    if (threadIdx.x == 0 && (blk == 0 || blk == n_query_blocks - 1))
        printf("prepare block %d | ns start %llu end %llu\n", blk, g_p0, g_p1);
#endif
}

// ------------------------------------------------------------------------------------------------
// stage 1 helpers
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint4 lds_u128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
// Byte permutation with the full selector of the instruction: bit 3 of a selector nibble replaces the chosen
// byte by eight copies of its top bit (the intrinsic __byte_perm documents only the low three bits).
__device__ __forceinline__ uint32_t prmt_rep(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
// reads at an address plus a constant of the instruction
template <int OFF>
__device__ __forceinline__ uint4 lds_u128_at(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4+%5];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ uint2 lds_u64_at(uint32_t addr) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(addr), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ uint32_t lds_u32_at(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFF));
    return v;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1,%2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0,%1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// packed binary32 pairs (two IEEE operations per instruction)
__device__ __forceinline__ void fadd2(uint64_t& d, uint64_t a) {
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(a));
}
__device__ __forceinline__ void ffma2(uint64_t& d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ void fmul2(uint64_t& d, uint64_t a) {
    asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(a));
}
// packed binary16 pairs
__device__ __forceinline__ uint32_t hadd2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
// lo += low half of h, hi += high half of h (binary16 widened exactly, binary32 addition)
__device__ __forceinline__ void flush_h2(uint32_t h, float& lo, float& hi) {
    asm("{\n\t.reg .b16 l, u;\n\tmov.b32 {l, u}, %2;\n\tadd.rn.f32.f16 %0, l, %0;\n\tadd.rn.f32.f16 %1, u, %1;\n\t}"
        : "+f"(lo), "+f"(hi) : "r"(h));
}
__device__ __forceinline__ uint32_t pack_h2(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
// to +-60000, both halves; a NaN becomes -60000
__device__ __forceinline__ uint32_t clamp_h2(uint32_t h) {
    asm("max.f16x2 %0, %0, %1;\n\tmin.f16x2 %0, %0, %2;" : "+r"(h) : "r"(0xfb53fb53u), "r"(0x7b537b53u));
    return h;
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float warp_max(float v) {
    int i = __float_as_int(v);
    i ^= (i >> 31) & 0x7fffffff;               // order-preserving map to signed integers
    i = __reduce_max_sync(0xffffffffu, i);
    i ^= (i >> 31) & 0x7fffffff;
    return __int_as_float(i);
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// two grid indices u 2^-24 -> (u - 64) 2^-10, exact
__device__ __forceinline__ uint32_t grid_steps(uint32_t u) {
    uint32_t d;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(u), "r"(0x74007400u), "r"(0xac00ac00u));
    return d;
}
// the same with a zero accumulator
__device__ __forceinline__ void mma_f16_zero(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

struct Segment {
    int b, kvh, pg0, npg, len;
};

// Page and cost prefixes of a batch of at most PFX_CAP sequences in shared memory (pfx: [2][PFX_CAP + 1]), by all threads of a
// scan CTA; CTA 0 also writes the prefixes for the merge kernel and reports lengths out of range.  Every CTA does it by
// itself: a block of the kernel in front would have to wait for the append, load the lengths and write, and the scan for that
// block (append + decode, that block / here: 1 x 777 19.0 / 18.4 us, 8 x 16384 42.4 / 42.0, 128 x 1000 102.9 / 102.3; 5 x 100 of the
// d = 64 shape 17.0 / 16.5).
static_assert(PFX_CAP < S1_THREADS, "a thread for every sequence");
__device__ __forceinline__ void form_prefixes(int32_t* pfx, int (*s_part)[NCW], const int32_t* __restrict__ seq_lens, int batch, int max_pages,
                                              int seg_weight, int32_t* __restrict__ page_prefix, int32_t* __restrict__ cost_prefix,
                                              uint32_t* dev_status) {
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    int pages = 0;
    if (t < batch) {
        const int raw = seq_lens[t], len = clamp_len(raw, max_pages);
        if (raw != len && blockIdx.x == 0) atomicOr(dev_status, NOVAKV_DEV_BAD_LENGTH);
        pages = (len + NOVAKV_PAGE_TOKENS - 1) / NOVAKV_PAGE_TOKENS;
    }
    int incl = pages, incl_ne = pages > 0;
    if (warp * 32 < batch) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, incl, o), b = __shfl_up_sync(0xffffffffu, incl_ne, o);
            if (lane >= o) { incl += a; incl_ne += b; }
        }
    }
    if (batch > 32) {
        if (lane == 31) { s_part[0][warp] = incl; s_part[1][warp] = incl_ne; }
        __syncthreads();
        if (warp * 32 < batch)                                 // (the others would only keep everybody waiting)
            for (int w = 0; w < warp; ++w) { incl += s_part[0][w]; incl_ne += s_part[1][w]; }
    }
    if (t < batch) {
        const int p0 = incl - pages, c0 = p0 + seg_weight * (incl_ne - (pages > 0));
        pfx[t] = p0;
        pfx[PFX_CAP + 1 + t] = c0;
        if (blockIdx.x == 0) { page_prefix[t] = p0; cost_prefix[t] = c0; }
        if (t == batch - 1) {
            const int c1 = incl + seg_weight * incl_ne;
            pfx[batch] = incl;
            pfx[PFX_CAP + 1 + batch] = c1;
            if (blockIdx.x == 0) { page_prefix[batch] = incl; cost_prefix[batch] = c1; }
        }
    }
    __syncthreads();
}

// A scan CTA that cannot run leaves an empty range; the merge kernel reads the prefixes all the same and needs them whole.
__device__ __noinline__ void leave_unscanned(long* cta_range, int form_prefix, const int32_t* seq_lens, int batch, int max_pages, int seg_weight,
                                             int32_t* page_prefix, int32_t* cost_prefix, uint32_t* dev_status) {
    novakv_grid_dependency_wait();
    if (threadIdx.x != 0) return;
    atomicOr(dev_status, NOVAKV_DEV_SMEM_LAYOUT);
    cta_range[blockIdx.x * 2] = 0;
    cta_range[blockIdx.x * 2 + 1] = 0;
    if (!form_prefix || blockIdx.x != 0) return;
    int pages = 0, cost = 0;
    for (int b = 0; b <= batch; ++b) {
        page_prefix[b] = pages;
        cost_prefix[b] = cost;
        const int n = b < batch ? (clamp_len(seq_lens[b], max_pages) + NOVAKV_PAGE_TOKENS - 1) / NOVAKV_PAGE_TOKENS : 0;
        pages += n;
        cost += n > 0 ? n + seg_weight : 0;
    }
}

// Locate the (KV head, sequence, page) of global page unit u.  Units are ordered KV-head-major:
// u = kvh * P + page_prefix[b] + page, with P = page_prefix[batch] the pages of all sequences, so that
// consecutive segments of a CTA share the KV head (and its value codebook).  page_prefix is exclusive,
// length batch + 1.  Cooperative: every thread tests one sequence (all loads independent, one memory
// latency), the owner publishes sequence, length, first page and KV head through shared memory (found); a barrier, then
// segment_at().  A CTA looks its next segment up before the scan of the present one.
__device__ __forceinline__ void find_segment(const int32_t* __restrict__ page_prefix, const int32_t* __restrict__ seq_lens,
                                             int batch, int max_pages, long u, int kvh, int* found) {
    const long r = u - (long)kvh * page_prefix[batch];
    for (int t = threadIdx.x; t < batch; t += S1_THREADS) {
        const int lo = page_prefix[t], hi = page_prefix[t + 1];
        if ((long)lo <= r && r < (long)hi) { found[0] = t; found[1] = clamp_len(seq_lens[t], max_pages); found[2] = lo; found[3] = kvh; }
    }
}
__device__ __forceinline__ Segment segment_at(const int32_t* __restrict__ page_prefix, int batch, long u, long u_end, const int* found) {
    Segment s;
    s.b = found[0];
    s.len = found[1];
    s.kvh = found[3];
    const long r = u - (long)s.kvh * page_prefix[batch];
    const int pages_b = (s.len + NOVAKV_PAGE_TOKENS - 1) / NOVAKV_PAGE_TOKENS;
    s.pg0 = (int)(r - found[2]);
    const long left = u_end - u;
    s.npg = (int)(left < (long)(pages_b - s.pg0) ? left : (long)(pages_b - s.pg0));
    return s;
}

// ------------------------------------------------------------------------------------------------
// stage 1: persistent index scan
// ------------------------------------------------------------------------------------------------
// Streaming 128-/64-bit loads of index bytes: read once, keep them out of L1.
__device__ __forceinline__ uint4 ldg_stream_128(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ldg_stream_32(const void* p) {
    uint32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ldg_stream_16(const void* p) {
    uint32_t v;
    asm volatile("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ldg_stream_64(const void* p) {
    uint2 v;
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}

// Value codebook of a KV head (32 KB image, uint8 [256 codes][32 slots][4], slot = group) -> two copies in
// shared memory, copy c holding group g in slot (g + 16 c) % 32, without registers: asynchronous 16-byte
// copies that land while the caller does other work (segment lookup, page ids, table build);
// async_copies_wait() before the barrier that publishes the copies.  A 16-byte chunk holds 4 slots, so the
// rotation by 16 slots moves whole chunks.
__device__ __forceinline__ void stage_value_codebook_async(uint32_t d0, const uint8_t* __restrict__ src_g) {
    for (int i = threadIdx.x; i < VCB_COPY_BYTES / 16; i += S1_THREADS) {
        const int row = i >> 3, ch = i & 7;
        const uint8_t* src = src_g + (size_t)i * 16;
#pragma unroll
        for (int c = 0; c < 2; ++c)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d0 + c * VCB_COPY_BYTES + row * VCB_ROW + ((ch + 4 * c) & 7) * 16), "l"(src) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void async_copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The table build is kept out of line so that its load batches do not disturb the register allocation of
// the scan loop.  Entry (code, l, h) = <q'_h segment of group l, centred key codeword (l, code)>, heads beyond
// HG zero: binary32 in T32 for l < K32, binary16 in T16 otherwise.
template <int D, int HG, bool VM>
__device__ __noinline__ void build_score_table(unsigned char* t32, unsigned char* t16,
                                               const float* __restrict__ cb_k_lut /* [256][L][4] of the KV head */,
                                               const float* q_s /* shared: q' of the pair, [HPAD][D] */) {
    using C = S1<D, HG, VM>;
    constexpr int L = C::L, HPAD = C::HPAD, HSETS = C::HSETS, K32 = C::K32;
    if constexpr (C::HAS16) {
        // Hybrid table: whole warps take one kind of entry, so that no warp runs both store paths.  Threads
        // 0 .. 16 K32 - 1 build the binary32 part (group = t % K32, 16 codes per pass), the others the binary16
        // part (group = K32 + t' % (L - K32), 16 codes per pass); 16 passes either way.
        static_assert(K32 == 8 && L == 32 && S1_THREADS == 512 && HPAD == 4, "work split of the hybrid table build");
        constexpr int T32_THREADS = 16 * K32;                   // 128 = 4 warps
        constexpr int BATCH = 4;                                // (8 or 16 in flight: spills around the call, 10 % of the scan)
        const bool is32 = threadIdx.x < T32_THREADS;
        const int tl = is32 ? threadIdx.x : threadIdx.x - T32_THREADS;
        const int g = is32 ? tl % K32 : K32 + tl % (L - K32);
        const int code0 = is32 ? tl / K32 : tl / (L - K32);
        // q' of two heads side by side: one packed multiply-add serves both
        uint64_t q01[4], q23[4];
        {
            const float4 h0 = *reinterpret_cast<const float4*>(q_s + g * 4), h1 = *reinterpret_cast<const float4*>(q_s + D + g * 4);
            const float4 h2 = *reinterpret_cast<const float4*>(q_s + 2 * D + g * 4), h3 = *reinterpret_cast<const float4*>(q_s + 3 * D + g * 4);
            q01[0] = pack2(h0.x, h1.x); q01[1] = pack2(h0.y, h1.y); q01[2] = pack2(h0.z, h1.z); q01[3] = pack2(h0.w, h1.w);
            q23[0] = pack2(h2.x, h3.x); q23[1] = pack2(h2.y, h3.y); q23[2] = pack2(h2.z, h3.z); q23[3] = pack2(h2.w, h3.w);
        }
        const float4* cbk = reinterpret_cast<const float4*>(cb_k_lut) + g;
        const uint32_t a32 = smem_u32(t32) + g * 16, a16 = smem_u32(t16) + g * 8;
        float4 cw[BATCH];
        auto load = [&](int it0) {
#pragma unroll
            for (int u = 0; u < BATCH; ++u) cw[u] = cbk[(size_t)(code0 + (it0 + u) * 16) * L];
        };
        load(0);
#pragma unroll 1
        for (int it0 = 0; it0 < 16; it0 += BATCH) {
            float4 now[BATCH];                                  // the next codewords fly while these are multiplied
#pragma unroll
            for (int u = 0; u < BATCH; ++u) now[u] = cw[u];
            if (it0 + BATCH < 16) load(it0 + BATCH);
#pragma unroll
            for (int u = 0; u < BATCH; ++u) {
                const int code = code0 + (it0 + u) * 16;
                const uint64_t x = pack2(now[u].x, now[u].x), y = pack2(now[u].y, now[u].y), z = pack2(now[u].z, now[u].z), w = pack2(now[u].w, now[u].w);
                uint64_t o01 = q01[0], o23 = q23[0];
                fmul2(o01, x); fmul2(o23, x);
                ffma2(o01, q01[1], y); ffma2(o23, q23[1], y);
                ffma2(o01, q01[2], z); ffma2(o23, q23[2], z);
                ffma2(o01, q01[3], w); ffma2(o23, q23[3], w);
                float o[HPAD];
                unpack2(o01, o[0], o[1]);
                unpack2(o23, o[2], o[3]);
                if (is32) {
                    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(a32 + code * C::ROW32),
                                 "f"(o[0]), "f"(o[1]), "f"(o[2]), "f"(o[3]) : "memory");
                } else {
                    // (a table entry beyond the binary16 range would be a logit share of 2^16 bits; clamped to 60000, never inf)
                    const uint32_t e0 = clamp_h2(pack_h2(o[0], o[1])), e1 = clamp_h2(pack_h2(o[2], o[3]));
                    asm volatile("st.shared.v2.b32 [%0], {%1,%2};" ::"r"(a16 + code * T16_ROW), "r"(e0), "r"(e1) : "memory");
                    // groups 8..15 a second time in columns 0..7: the 16 lanes of a half warp then read 16 different columns
                    if (g < 16) asm volatile("st.shared.v2.b32 [%0], {%1,%2};" ::"r"(a16 + code * T16_ROW - 64), "r"(e0), "r"(e1) : "memory");
                }
            }
        }
        return;
    }
    constexpr int CSTEP = S1_THREADS / L;                       // codes per pass of the CTA
    constexpr int NIT = (256 + CSTEP - 1) / CSTEP;
    constexpr int BATCH = 8;                                    // loads in flight per thread
    const int g = threadIdx.x % L, code0 = threadIdx.x / L;
    float4 qs[HPAD];
#pragma unroll
    for (int h = 0; h < HPAD; ++h) qs[h] = *reinterpret_cast<const float4*>(q_s + h * D + g * 4);
    const float4* cbk = reinterpret_cast<const float4*>(cb_k_lut);
#pragma unroll 1
    for (int it0 = 0; it0 < NIT; it0 += BATCH) {
        float4 cw[BATCH];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int code = code0 + (it0 + u) * CSTEP;
            if (it0 + u < NIT && code < 256) cw[u] = cbk[(size_t)code * L + g];
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int code = code0 + (it0 + u) * CSTEP;
            if (it0 + u < NIT && code < 256) {
                float o[HPAD];
#pragma unroll
                for (int h = 0; h < HPAD; ++h)
                    o[h] = fmaf(qs[h].w, cw[u].w, fmaf(qs[h].z, cw[u].z, fmaf(qs[h].y, cw[u].y, qs[h].x * cw[u].x)));
#pragma unroll
                for (int hs = 0; hs < HSETS; ++hs)
                    *reinterpret_cast<float4*>(t32 + hs * C::PLANE32 + code * C::ROW32 + g * 16) =
                        make_float4(o[hs * 4], o[hs * 4 + 1], o[hs * 4 + 2], o[hs * 4 + 3]);
            }
        }
    }
}

// Index bytes of one 32-token tile as one lane holds them.
//   kw: this lane's token (lane = token within the tile), L bytes: byte j holds the code of group
//       j ^ (lane % 8) for j < 16 and j ^ (lane % 16) for j >= 16.
//   vw: per 16-token block, the codes of this lane's MMA coordinates (fr = lane/4, fc = lane%4):
//       word gb holds, for the four tokens 4u + fc of the block (byte u), the code of group 8 gb + fr.
template <int L>
struct TileRegs {
    uint32_t kw[L / 4];
    uint32_t vw[2][L / 8];
    uint32_t ks;          // this lane's token: bfloat16 key scale in the low half, if used
    uint32_t vm;          // this lane's token: bfloat16 value scale (low half) and zero-point (high half), if used
};

// First unit of scan CTA c of G (c = G gives the end of the walk).  The walk is cut evenly in cost units,
// cost = pages + seg_weight per (sequence, KV head) pair: cost point t lies in the pair whose cost interval
// contains it and maps to unit  start + clamp(t - cost_start - seg_weight, 0, pages)  (the first seg_weight cost
// units of a pair stand for setting up its score table).  seg_weight = 0 is the even split in pages.
__device__ __forceinline__ long scan_boundary(int c, int G, const int32_t* __restrict__ page_prefix,
                                              const int32_t* __restrict__ cost_prefix, int batch, int n_kv_heads, int seg_weight) {
    const long P = page_prefix[batch], U = P * n_kv_heads;
    if (seg_weight == 0) return ((long)c * U) / G;
    const long cper = cost_prefix[batch], T = cper * n_kv_heads;
    const long t = ((long)c * T) / G;
    if (cper <= 0 || t >= T) return U;
    const long kv = t / cper, rem = t - kv * cper;
    int lo = 0, hi = batch - 1;                   // the last sequence whose cost interval starts at or before rem
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((long)cost_prefix[mid] <= rem) lo = mid; else hi = mid - 1;
    }
    const long p0 = page_prefix[lo], pg = page_prefix[lo + 1] - p0;
    return kv * P + p0 + min(max(rem - cost_prefix[lo] - seg_weight, 0l), pg);
}

// Merge of one (sequence, KV head) pair inside the scan kernel, run by the CTA that wrote the pair's last
// partial: exact log-sum-exp combination of the partials of the CTAs first .. last (those with an empty
// range skipped), normalisation, inverse value transform o = o' rv^T + v_mean.  scratch: shared memory,
// (1 + S1_THREADS / D) * HG * D floats.  Partials of other CTAs are read past the L1 (they were written by
// other SMs; the arrival counter orders the accesses).
template <int D, int HG>
__device__ __noinline__ void fused_merge(float* scratch, const float* part_ml, const float* part_acc, int pair, int first,
                                         int last, const long* s_bnd, const float* __restrict__ rv_t,
                                         const float* __restrict__ v_mean, int kvh, void* __restrict__ out, int out_is_fp32,
                                         size_t out_row /* (b * Hq + kvh * HG) * D */) {
    constexpr int PARTS = S1_THREADS / D, COLS = D / PARTS;
    float* o_s = scratch;                         // [HG][D]
    float* red_s = scratch + HG * D;              // [PARTS][HG][D]
    for (int i = threadIdx.x; i < HG * D; i += S1_THREADS) {
        const int h = i / D, c = i - h * D;
        float M = M_INIT;
        for (int cta = first; cta <= last; ++cta)
            if (s_bnd[cta] < s_bnd[cta + 1]) M = fmaxf(M, __ldcg(part_ml + (((size_t)pair + cta) * HG + h) * 2));
        float a = 0.f, lsum = 0.f;
        for (int cta = first; cta <= last; ++cta) {
            if (s_bnd[cta] >= s_bnd[cta + 1]) continue;
            const size_t pidx = (size_t)pair + cta;
            const float sc = ex2(__ldcg(part_ml + (pidx * HG + h) * 2) - M);
            a = fmaf(sc, __ldcg(part_acc + (pidx * HG + h) * D + c), a);
            lsum = fmaf(sc, __ldcg(part_ml + (pidx * HG + h) * 2 + 1), lsum);
        }
        o_s[i] = lsum > 0.f ? a / lsum : 0.f;
    }
    __syncthreads();
    {
        const int r = threadIdx.x % D, part = threadIdx.x / D;
        const float* R = rv_t + (size_t)kvh * D * D + (size_t)part * COLS * D + r;      // rv_t[c][r] = R_V[r][c]
        float acc[HG];
#pragma unroll
        for (int h = 0; h < HG; ++h) acc[h] = 0.f;
#pragma unroll 8
        for (int c = 0; c < COLS; ++c) {
            const float rv = R[(size_t)c * D];
#pragma unroll
            for (int h = 0; h < HG; ++h) acc[h] = fmaf(o_s[h * D + part * COLS + c], rv, acc[h]);
        }
#pragma unroll
        for (int h = 0; h < HG; ++h) red_s[(part * HG + h) * D + r] = acc[h];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < HG * D; i += S1_THREADS) {
        const int h = i / D, r = i - h * D;
        float o = v_mean[(size_t)kvh * D + r];
#pragma unroll
        for (int p = 0; p < PARTS; ++p) o += red_s[(p * HG + h) * D + r];
        if (out_is_fp32) reinterpret_cast<float*>(out)[out_row + i] = o;
        else reinterpret_cast<__nv_bfloat16*>(out)[out_row + i] = __float2bfloat16_rn(o);
    }
}

// KSC: the key format carries a per-token bfloat16 scale (k_scales [n_pages][Hkv][64]); the logits of a
// token are multiplied by it once, after the table lookups are summed (and the centre's share added back).
// VSQ: scalar INT2 values with a per-token bfloat16 scale and zero-point (v_meta [n_pages][Hkv][64][2]).
// A byte holds four 2-bit codes (levels 0 .. 3) of a group.  Both halves of a word get the byte, and a mask leaves two levels
// where they stand, as the binary16 subnormals l 4^i 2^-24: no gather, and the accumulators of level i are divided by 4^i in
// the epilogue.  64 sequences of 32768 tokens with band: 441 -> 418 us a call against a gather from the 256 products
// {0,1,2,3}^4 in shared memory; error against binary64 at 700 / 6000 tokens 3.2e-4 / 4.4e-4 -> 2.4e-4 / 3.1e-4, because the
// tensor core aligns subnormals without normalising them, so larger ones lose less.  (Both levels of a word from two
// tokens, 16 tokens a product, saves 32 instructions per 32 tokens but doubles the accumulators: 421 us, and 4.0e-4.)
// The weight of a token's codes is p * scale and the zero-points enter through one extra running sum per head,
// sum_j p_j zero_j, added to every coefficient in the epilogue.
//
// Numerics of the tensor-core value side.  A softmax weight enters the product as the binary16 number
// w = fp16(2^15 p) (p <= 1 relative to the running maximum, so w <= 2^15; weights down to 2^-39 stay
// non-zero), and the same rounded w is what the normaliser sums: the result is an exact softmax of slightly
// perturbed logits.  A value codeword is four 7-bit grid indices u (bytes with the top bit clear); the byte
// permutation that widens them pairs every byte with its replicated top bit, i.e. with a zero byte: the
// binary16 numbers u 2^-24 (subnormal, exact; the tensor core multiplies them exactly).  The same permutation
// picks the bytes from one of two registers by lane, which undoes the block swap of the odd lane columns.
// Every NOVAKV_WINDOW tiles, and before any rescaling, the grid centre is removed with the weight sum of
// the same tokens (every lane adds up the rounded weights of its own tokens; a shuffle reduction per window
// gives each lane column the sum of its head): acc -= 64 2^-24 sum_j w_j leaves 2^-24 sum_j w_j (u_j - 64),
// so that the long-running sums stay centred.  (An all-ones operand on the tensor core gave the same sums at
// four more matrix instructions per tile, which cost more issue time than the shuffles.)
template <int D, int HG, bool VM, bool KSC, bool VSQ>
__global__ void __launch_bounds__(S1_THREADS, 1)
novakv_decode_stage1_kernel(const float* __restrict__ qp, const float* __restrict__ cb_k_lut,
                            const uint8_t* __restrict__ cb_v_img, const float* __restrict__ v_scale,
                            const float* __restrict__ v_off, const uint8_t* __restrict__ k_pages,
                            const uint8_t* __restrict__ v_pages, const __nv_bfloat16* __restrict__ k_scales,
                            const __nv_bfloat16* __restrict__ v_meta, int n_pages,
                            const int32_t* __restrict__ page_table, int max_pages_per_seq,
                            const int32_t* __restrict__ seq_lens, int32_t* __restrict__ page_prefix_g,
                            int batch, int n_q_heads, int n_kv_heads, float* __restrict__ part_ml,
                            float* __restrict__ part_acc, uint32_t* __restrict__ dev_status, int pt_stride,
                            int32_t* __restrict__ cost_prefix_g, int seg_weight, long* __restrict__ cta_range,
                            const float* __restrict__ qc,
                            int32_t* __restrict__ pair_count, const float* __restrict__ rv_t,
                            const float* __restrict__ v_mean, void* __restrict__ out_fused, int out_is_fp32, int form_prefix) {
    // out_fused != null: the CTA that writes the last partial of a (sequence, KV head) pair also merges the pair's
    // partials and applies the inverse value transform (no merge kernel follows); pair_count holds one arrival
    // counter per pair, zero on entry and reset to zero by the merging CTA.  Nothing waits on another CTA.
    // page_table points at the first column that is scanned; rows are pt_stride entries apart and
    // max_pages_per_seq bounds the pages of a row that may be read from there
    using C = S1<D, HG, VM>;
    constexpr int L = C::L, HPAD = C::HPAD, HSETS = C::HSETS, NGB = C::NGB, KPL = C::KPL, K32 = C::K32;
    constexpr bool HAS16 = C::HAS16;
    constexpr int TILE_BYTES = C::TILE_BYTES, PAGE_BYTES = 2 * TILE_BYTES;
    constexpr float SH = VM ? 15.f : 0.f;                     // weights are scaled by 2^SH before the binary16 rounding
    constexpr float U_UNIT = 5.9604644775390625e-08f;         // 2^-24: a grid index u enters a product as the binary16 subnormal u 2^-24
    constexpr float CEN = VSQ ? 0.f : 64.f * U_UNIT;          // what one unit of weight adds to a tensor-core sum beyond u - centre
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ int s_found[2][4], s_part[2][NCW];
    __shared__ int s_arrived, s_first, s_last;
    const uint32_t s_base = smem_u32(smem);
    if (s_base > C::T16 || C::SMEM - s_base > (uint32_t)S1_SMEM_BYTES) {
        // cannot happen with the shared address window of this architecture; reported, never trapped
        leave_unscanned(cta_range, form_prefix, seq_lens, batch, max_pages_per_seq, seg_weight, page_prefix_g, cost_prefix_g, dev_status);
        return;
    }
    unsigned char* const s_abs = smem - s_base;               // s_abs + a: the byte at shared-window address a
    unsigned char* const t32_p = s_abs + C::T32;
    unsigned char* const t16_p = s_abs + C::T16;

    // With the KV-head-major walk the first KV head of CTA c is floor(c * Hkv / G) whatever the lengths are:
    // its (constant) value codebook starts flowing into shared memory before the grid-dependency wait and
    // lands behind the segment lookup and the first table build.
    int vcb_head = (int)(((long)blockIdx.x * n_kv_heads) / gridDim.x);   // KV head whose value codebook is resident
    if (!VSQ) stage_value_codebook_async(C::VCB, cb_v_img + (size_t)vcb_head * VCB_COPY_BYTES);
    // With the merge fused in this grid writes the outputs: its dependents are not let in before it is done.
    if (out_fused != nullptr) asm volatile("griddepcontrol.wait;" ::: "memory");
    else novakv_grid_dependency_wait();

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // The two prefixes are read many times (boundaries, segment look-ups): small batches form them in shared memory.
    const int32_t *page_prefix = page_prefix_g, *cost_prefix = cost_prefix_g;
    if (form_prefix) {                                        // (batches of at most PFX_CAP sequences)
        int32_t* pfx = reinterpret_cast<int32_t*>(s_abs + C::PFX);
        form_prefixes(pfx, s_part, seq_lens, batch, max_pages_per_seq, seg_weight, page_prefix_g, cost_prefix_g, dev_status);
        page_prefix = pfx;
        cost_prefix = pfx + PFX_CAP + 1;
    } else if (batch <= PFX_CAP) {
        int32_t* pfx = reinterpret_cast<int32_t*>(s_abs + C::PFX);
        for (int i = threadIdx.x; i <= batch; i += S1_THREADS) { pfx[i] = page_prefix_g[i]; pfx[PFX_CAP + 1 + i] = cost_prefix_g[i]; }
        __syncthreads();
        page_prefix = pfx;
        cost_prefix = pfx + PFX_CAP + 1;
    }
    // First unit of every CTA (see scan_boundary): one thread per boundary.  This CTA owns [s_bnd[c], s_bnd[c + 1]).
    long* const s_bnd = reinterpret_cast<long*>(s_abs + C::BND);
    for (int c = threadIdx.x; c <= (int)gridDim.x; c += S1_THREADS)
        s_bnd[c] = scan_boundary(c, gridDim.x, page_prefix, cost_prefix, batch, n_kv_heads, seg_weight);
    __syncthreads();
    const long u_begin = s_bnd[blockIdx.x], u_end = s_bnd[blockIdx.x + 1];
    if (threadIdx.x == 0) { cta_range[blockIdx.x * 2] = u_begin; cta_range[blockIdx.x * 2 + 1] = u_end; }
    if (u_begin >= u_end) { async_copies_wait(); return; }

    // ---- lane roles and constants
    const int fr = lane >> 2, fc = lane & 3;          // value side: MMA fragment coordinates
    // key side: token = lane; its byte j holds group j ^ (lane & 7) (j < 16) or j ^ (lane & 15) (j >= 16).  The column of
    // step j is one byte below 128 (columns from 128 on come as an immediate), four steps to a word; a byte permutation of
    // (index word, column word) makes a gather address: column, code, and twice the column's replicated top bit, a zero.
    uint32_t col32[2], col16[HAS16 ? 4 : 1];
#pragma unroll
    for (int w = 0; w < 2; ++w) col32[w] = (0x30201000u ^ ((uint32_t)(lane & 7) * 0x10101010u)) ^ (w * 0x40404040u);
#pragma unroll
    for (int w = 0; w < (HAS16 ? 4 : 1); ++w) col16[w] = (0x18100800u ^ ((uint32_t)(lane & 15) * 0x08080808u)) ^ (w * 0x20202020u);
#pragma unroll
    for (int w = 0; w < 2; ++w) asm volatile("" : "+r"(col32[w]));               // (kept in registers: formed again in every tile otherwise)
#pragma unroll
    for (int w = 0; w < (HAS16 ? 4 : 1); ++w) asm volatile("" : "+r"(col16[w]));
    // value side: lane column fc reads copy fc / 2 of the value codebook; odd columns take the group blocks in
    // swapped order (x ^ 1), so that the 32 lanes of a gather hit 32 different slots.  Address = pos + code * 128, a byte
    // dot product: the permutations above and those that widen a codeword fill the integer pipe (55 % busy), dot products run
    // on the one of the multiply-adds.  With the columns above 55 -> 45 %; 64 sequences of 65536 tokens 655 -> 639 us a call.
    uint32_t pos[NGB];
#pragma unroll
    for (int x = 0; x < NGB; ++x) pos[x] = (fc >> 1) * VCB_COPY_BYTES + ((8 * (x ^ (fc & 1)) + fr + 16 * (fc >> 1)) & 31) * 4;
    // codeword whose code is byte b of word w, for load x
    auto vgather = [&](uint32_t w, int b, int x) -> uint32_t { return lds_u32_at<C::VCB>(__dp4a(w, (uint32_t)VCB_ROW << (8 * b), pos[x])); };
    const bool odd_col = fc & 1;
    // widening selectors: byte pairs (u, replicated top bit of u = 0) of the low / high half of a codeword, taken
    // from the first operand in even columns and from the second in odd columns
    const uint32_t sel_lv = odd_col ? 0x4444u : 0u;
    const uint32_t sel_lo = odd_col ? 0xD5C4u : 0x9180u, sel_hi = odd_col ? 0xF7E6u : 0xB3A2u;
    // B fragments carry a weight in the low or high half depending on the column parity (fr & 1)
    const uint32_t sel_b0 = (fr & 1) ? 0x1044u : 0x4410u, sel_b1 = (fr & 1) ? 0x3244u : 0x4432u;
    const uint32_t s_pw = C::P + warp * C::P_WARP_BYTES;

    // ---- per-warp running state
    float m_run[HPAD];                           // running maximum of the logits (base 2), the same in every lane
    float macc[HSETS][NGB][4];                   //  VM: lane (fr, fc): head 4 hs + fc, group 8 gb + fr, 4 coefficients
    float wsum[HPAD];                            //  VM: this lane's tokens: sums of the (rounded) weights per head since the last offset removal
    float l_run[HPAD];                           //  VM: [hs] weight sum of head 4 hs + fc (every lane); else this lane's tokens, per head
    float lz_run[VSQ ? HPAD : 1];                //  VSQ: running sum_j p_j zero_j per head (this lane's tokens)
    uint64_t acc[VM ? 1 : NGB][VM ? 1 : HPAD][2];  // !VM: lane (fr, fc): group 8 gb + fr, head, 4 coefficients, its own tokens
    float esh_pow = 0.f;                         //  VSQ: 2^E with E >= log2 of every value scale seen so far (weights carry 2^-E)
#pragma unroll
    for (int h = 0; h < HPAD; ++h) { m_run[h] = M_INIT; l_run[h] = 0.f; }
#pragma unroll
    for (int h = 0; h < (VSQ ? HPAD : 1); ++h) lz_run[h] = 0.f;
#pragma unroll
    for (int hs = 0; hs < HSETS; ++hs) {
#pragma unroll
        for (int gb = 0; gb < NGB; ++gb)
#pragma unroll
            for (int i = 0; i < 4; ++i) macc[hs][gb][i] = 0.f;
    }
#pragma unroll
    for (int h = 0; h < HPAD; ++h) wsum[h] = 0.f;
#pragma unroll
    for (int x = 0; x < (VM ? 1 : NGB); ++x)
#pragma unroll
        for (int h = 0; h < (VM ? 1 : HPAD); ++h) { acc[x][h][0] = 0ull; acc[x][h][1] = 0ull; }

    // remove the centre of the value grid from the sums of the tiles since the last call (tensor-core value side)
    auto flush_window = [&]() {
        if (VSQ) return;          // INT2 levels carry no grid centre, and that format sums its normaliser per lane
#pragma unroll
        for (int hs = 0; hs < HSETS; ++hs) {
            // weight sum of head 4 hs + fc over the whole warp's tokens: transposing reduction inside the quad (each
            // step halves the heads a lane keeps), then a butterfly over the eight quads
            const float k0 = fc & 1 ? wsum[hs * 4 + 1] : wsum[hs * 4 + 0], s0 = fc & 1 ? wsum[hs * 4 + 0] : wsum[hs * 4 + 1];
            const float k1 = fc & 1 ? wsum[hs * 4 + 3] : wsum[hs * 4 + 2], s1 = fc & 1 ? wsum[hs * 4 + 2] : wsum[hs * 4 + 3];
            const float lo = k0 + __shfl_xor_sync(0xffffffffu, s0, 1), hi = k1 + __shfl_xor_sync(0xffffffffu, s1, 1);
            float w = (fc & 2 ? hi : lo) + __shfl_xor_sync(0xffffffffu, fc & 2 ? lo : hi, 2);
#pragma unroll
            for (int o = 4; o <= 16; o <<= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
#pragma unroll
            for (int gb = 0; gb < NGB; ++gb)
#pragma unroll
                for (int i = 0; i < 4; ++i) macc[hs][gb][i] = fmaf(-CEN, w, macc[hs][gb][i]);
            l_run[hs] += w;
#pragma unroll
            for (int i = 0; i < 4; ++i) wsum[hs * 4 + i] = 0.f;
        }
    };

#ifdef NOVAKV_TIMING
    long long tm[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    unsigned long long g_start;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_start));
    long long t_prev = clock64();
    const long long t_start = t_prev;
    int n_seg = 0;
#define NOVAKV_TICK(i) { const long long t_now = clock64(); tm[i] += t_now - t_prev; t_prev = t_now; }
#else
#define NOVAKV_TICK(i)
#endif
    // q' of a pair's heads -> shared memory (rows beyond HG stay zero), without registers and without a wait
    auto stage_query = [&](int b, int kvh, int buf) {
        const float4* src = reinterpret_cast<const float4*>(qp + ((size_t)b * n_q_heads + kvh * HG) * D);
        for (int i = threadIdx.x; i < HG * D / 4; i += S1_THREADS)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(C::Q + buf * C::Q_BYTES + i * 16), "l"(src + i) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (HG < HPAD)
        for (int i = threadIdx.x; i < 2 * (HPAD - HG) * D; i += S1_THREADS)
            reinterpret_cast<float*>(s_abs + C::Q + i / ((HPAD - HG) * D) * C::Q_BYTES)[HG * D + i % ((HPAD - HG) * D)] = 0.f;
    // What a segment needs before its table can be built is on its way early: its place in the batch is looked up and its
    // query copied during the scan of the segment before, its first page ids fly during that segment's merge.  With the packed
    // table build, scaled 32 x 8191 84.0 -> 80.0 us a call, 128-sequence mix 303 -> 298.
    int rem = (int)(u_end - u_begin);            // units of this CTA that are left; the present one is s_bnd[its end] - rem
    int cur_seg = 0;                             // which half of s_found and of the q' buffers holds the present segment
    find_segment(page_prefix, seq_lens, batch, max_pages_per_seq, u_begin, (int)(u_begin / page_prefix[batch]), s_found[0]);
    __syncthreads();
    Segment sg = segment_at(page_prefix, batch, u_begin, u_end, s_found[0]);
    for (int i = threadIdx.x; i < HG * D / 4; i += S1_THREADS)                // (the first one with plain loads: a wait for copies
        reinterpret_cast<float4*>(s_abs + C::Q)[i] =                          // would be one for the value codebook as well)
            reinterpret_cast<const float4*>(qp + ((size_t)sg.b * n_q_heads + sg.kvh * HG) * D)[i];
    int n_it = 0, ids_cur = 0, ids_next = 0;
    const int32_t* pt = nullptr;
    // page ids of 32 consecutive tiles of this warp, one per lane (coalesced gather, loaded a batch ahead)
    auto load_ids = [&](int batch_i) {
        const int it = batch_i * 32 + lane;
        int page = 0;
        if (it < n_it) {
            page = pt[(warp + NCW * it) >> 1];
            if (page < 0 || page >= n_pages) { atomicOr(dev_status, NOVAKV_DEV_BAD_PAGE); page = 0; }
        }
        return page;
    };
    auto fetch_ids = [&]() {
        // this warp's tiles of the segment: half pages hp = warp, warp + NCW, ...
        const int n_half = min(2 * sg.npg, (sg.len - sg.pg0 * NOVAKV_PAGE_TOKENS + 31) / 32);
        n_it = n_half > warp ? (n_half - warp + NCW - 1) / NCW : 0;
        pt = page_table + (size_t)sg.b * pt_stride + sg.pg0;
        ids_cur = load_ids(0);
        ids_next = load_ids(1);
    };
    fetch_ids();
    __syncthreads();
    while (rem > 0) {
        NOVAKV_TICK(0)
        const int pair = sg.kvh * batch + sg.b;            // grows along the walk
        rem -= sg.npg;

        // ---- segment prologue -----------------------------------------------------------------
        if (!VSQ && vcb_head != sg.kvh) {
            stage_value_codebook_async(C::VCB, cb_v_img + (size_t)sg.kvh * VCB_COPY_BYTES);
            vcb_head = sg.kvh;
        }
        if (rem > 0) {
            const long u_next = s_bnd[blockIdx.x + 1] - rem;
            find_segment(page_prefix, seq_lens, batch, max_pages_per_seq, u_next,
                         sg.kvh + (u_next >= (long)(sg.kvh + 1) * page_prefix[batch]), s_found[cur_seg ^ 1]);
        }
        float qcen[KSC ? HPAD : 1];
        if (KSC) {
#pragma unroll
            for (int h = 0; h < HPAD; ++h) qcen[h] = h < HG ? qc[(size_t)sg.b * n_q_heads + sg.kvh * HG + h] : 0.f;
        }

        // a warp's tiles are all first or all second halves of their pages (an even number of warps)
        static_assert(NCW % 2 == 0, "half of a page is a constant of the warp");
        const uint32_t k_step = (uint32_t)n_kv_heads * PAGE_BYTES;                       // bytes of a page
        const uint8_t* const kb = k_pages + (size_t)sg.kvh * PAGE_BYTES + (warp & 1) * TILE_BYTES + lane * 16;
        const uint8_t* const vb = v_pages + (size_t)sg.kvh * PAGE_BYTES + (warp & 1) * TILE_BYTES + lane * (NGB * 4);
        const size_t m0 = (size_t)sg.kvh * NOVAKV_PAGE_TOKENS + (warp & 1) * 32 + lane;  // this lane's token in the pools of scales
        // tiles are loaded in ascending order, one ahead of the tile being consumed
        auto load_tile = [&](int it, TileRegs<L>& t) {
            if ((it & 31) == 0 && it > 0) { ids_cur = ids_next; ids_next = load_ids((it >> 5) + 1); }
            const int page = __shfl_sync(0xffffffffu, ids_cur, it & 31);
            const uint8_t* const kp = kb + (size_t)(uint32_t)page * k_step;
            const uint8_t* const vp = vb + (size_t)(uint32_t)page * k_step;
            const size_t mi = m0 + (size_t)(uint32_t)page * (uint32_t)(n_kv_heads * NOVAKV_PAGE_TOKENS);
            // (kept as loaded: a shift here waits for the load, a tile ahead of its use; 64 scaled sequences of 32768 tokens
            // 431 -> 368 us a call without it)
            if (KSC) t.ks = ldg_stream_16(reinterpret_cast<const unsigned short*>(k_scales) + mi);
            if (VSQ) t.vm = ldg_stream_32(reinterpret_cast<const uint32_t*>(v_meta) + mi);
#pragma unroll
            for (int p = 0; p < KPL; ++p) {
                const uint4 w = ldg_stream_128(kp + p * 512);
                t.kw[4 * p + 0] = w.x; t.kw[4 * p + 1] = w.y; t.kw[4 * p + 2] = w.z; t.kw[4 * p + 3] = w.w;
            }
#pragma unroll
            for (int blk = 0; blk < 2; ++blk) {
                if (NGB == 4) {
                    const uint4 w = ldg_stream_128(vp + blk * (L * 16));
                    t.vw[blk][0] = w.x; t.vw[blk][1] = w.y; t.vw[blk][NGB - 2] = w.z; t.vw[blk][NGB - 1] = w.w;
                } else {
                    const uint2 w = ldg_stream_64(vp + blk * (L * 16));
                    t.vw[blk][0] = w.x; t.vw[blk][1] = w.y;
                }
            }
        };

        // ---- one 32-token tile -------------------------------------------------------------------
        const int left = sg.len - sg.pg0 * NOVAKV_PAGE_TOKENS - warp * 32;     // tokens from this warp's first tile on
        auto process = [&](const TileRegs<L>& cur, int it) {
            const int nvalid = left - it * (NCW * 32);

            // ---- key side: lane <-> token; step j gathers the entry of (code_j, group j ^ lane bits) ------
            float zf[HPAD];
            {
                uint64_t z2[HPAD / 2];
#pragma unroll
                for (int k = 0; k < HPAD / 2; ++k) z2[k] = 0ull;
#pragma unroll
                for (int j = 0; j < K32; ++j) {
                    const uint32_t a = prmt_rep(cur.kw[j >> 2], col32[(j >> 2) & 1], 0xcc04u + (j & 3) * 0x1111u);
#pragma unroll
                    for (int hs = 0; hs < HSETS; ++hs) {
                        const uint4 v = j < 8 ? (hs ? lds_u128_at<C::T32 + C::PLANE32>(a) : lds_u128_at<C::T32>(a))
                                              : (hs ? lds_u128_at<C::T32 + C::PLANE32 + 128>(a) : lds_u128_at<C::T32 + 128>(a));
                        fadd2(z2[2 * hs], (uint64_t)v.x | ((uint64_t)v.y << 32));
                        fadd2(z2[2 * hs + 1], (uint64_t)v.z | ((uint64_t)v.w << 32));
                    }
                }
#pragma unroll
                for (int k = 0; k < HPAD / 2; ++k) unpack2(z2[k], zf[2 * k], zf[2 * k + 1]);
            }
            if (HAS16) {
                // (with a per-token key scale the sum is multiplied by rho afterwards, which carries the rounding of the
                // binary16 chains into tokens of large norm: shorter chains there)
                constexpr int CHAIN = KSC ? NOVAKV_KSC_CHAIN : NOVAKV_CHAIN;
                uint32_t ch[2];
#pragma unroll
                for (int j = K32; j < L; ++j) {
                    const uint32_t a = prmt_rep(cur.kw[j >> 2], col16[HAS16 ? (j >> 2) & 3 : 0], 0xcc04u + (j & 3) * 0x1111u);
                    const uint2 v = j < 16 ? lds_u64_at<C::T16>(a) : lds_u64_at<C::T16 + 128>(a);
                    if ((j - K32) % CHAIN == 0) { ch[0] = v.x; ch[1] = v.y; }
                    else { ch[0] = hadd2(ch[0], v.x); ch[1] = hadd2(ch[1], v.y); }
                    if ((j - K32) % CHAIN == CHAIN - 1 || j == L - 1) {
                        flush_h2(ch[0], zf[0], zf[1]);
                        flush_h2(ch[1], zf[2], zf[3]);
                    }
                }
            }
            float vscale = 1.f, vzero = 0.f, vsmax = 0.f;     // vsmax: this lane's scale as it enters the running bound (0 beyond the length)
            if (KSC) {
                const float rho = __uint_as_float(cur.ks << 16);
#pragma unroll
                for (int h = 0; h < HPAD; ++h) zf[h] = (zf[h] + qcen[h]) * rho;
            }
            if (VSQ && lane < nvalid) {
                // (slots beyond the length hold no metadata; a scale that is not positive and finite counts as 1)
                vscale = __uint_as_float(cur.vm << 16);
                vzero = __uint_as_float(cur.vm & 0xffff0000u);
                if (!(vscale > 0.f && vscale < CUDART_INF_F)) vscale = 1.f;
                vsmax = vscale;
            }
            if (nvalid < 32 && lane >= nvalid) {
#pragma unroll
                for (int h = 0; h < HPAD; ++h) zf[h] = -CUDART_INF_F;
            }
            // ---- online softmax (base 2): the running maximum moves only when a logit exceeds it ---------
            {
                bool up = false;
#pragma unroll
                for (int h = 0; h < HPAD; ++h) up |= zf[h] > m_run[h];
                if (VSQ) up |= vsmax >= esh_pow;
                if (__any_sync(0xffffffffu, up)) {
                    float alpha[HPAD];
#pragma unroll
                    for (int h = 0; h < HPAD; ++h) {
                        // a head whose maximum moved gets M_SLACK bits of headroom above the new maximum: the next
                        // few record logits then need no update (the reference point of a softmax is free; weights
                        // stay <= 2^SH, and those below 2^(SH - 24 + M_SLACK) of the maximum vanish)
                        const float wm = warp_max(zf[h]);
                        const float m_new = wm > m_run[h] ? wm + M_SLACK : m_run[h];
                        alpha[h] = ex2(m_run[h] - m_new);
                        m_run[h] = m_new;
                    }
                    float vsc = 1.f;                     // VSQ: 2^(E_old - E_new)
                    if (VSQ) {
                        // E = exponent of the largest scale so far + 1 (scale < 2^E), an exact power of two
                        const float smax = warp_max(vsmax);
                        const float e_new = __uint_as_float((__float_as_uint(smax) & 0x7f800000u) + 0x00800000u);
                        if (e_new > esh_pow) { vsc = esh_pow / e_new; esh_pow = e_new; }
                    }
                    if (VM) {
#pragma unroll
                        for (int hs = 0; hs < HSETS; ++hs) {
                            const float a01 = fc & 1 ? alpha[hs * 4 + 1] : alpha[hs * 4 + 0];
                            const float a23 = fc & 1 ? alpha[hs * 4 + 3] : alpha[hs * 4 + 2];
                            const float al = fc & 2 ? a23 : a01;
#pragma unroll
                            for (int gb = 0; gb < NGB; ++gb)
#pragma unroll
                                for (int i = 0; i < 4; ++i) macc[hs][gb][i] *= al * vsc;
                            if (!VSQ) {
                                l_run[hs] *= al;
                                // the weight sums still waiting for their window flush move with the accumulators
#pragma unroll
                                for (int i = 0; i < 4; ++i) wsum[hs * 4 + i] *= alpha[hs * 4 + i];
                            }
                        }
                        if (VSQ) {
#pragma unroll
                            for (int h = 0; h < HPAD; ++h) { l_run[h] *= alpha[h]; lz_run[h] *= alpha[h]; }
                        }
                    } else {
#pragma unroll
                        for (int h = 0; h < HPAD; ++h) {
                            const uint64_t a2 = pack2(alpha[h], alpha[h]);
#pragma unroll
                            for (int x = 0; x < NGB; ++x) { fmul2(acc[VM ? 0 : x][VM ? 0 : h][0], a2); fmul2(acc[VM ? 0 : x][VM ? 0 : h][1], a2); }
                            l_run[h] *= alpha[h];
                        }
                    }
                }
            }
            // weights
            uint32_t ph[HPAD / 2];
            if (VSQ) {
                // INT2 values: the tensor-core product needs the weight of the token's integer codes,
                // w = p * scale (times 2^15 / 2^E), in binary16.  The rounding must not separate numerator and
                // normaliser: the weight that counts is p' = fp16(w) / (scale 2^-E), used for the normaliser and
                // for the zero-point sum as well (an exact softmax of perturbed logits).
                const float wmul = __fdividef(vscale, esh_pow), winv = __fdividef(esh_pow, vscale);
#pragma unroll
                for (int h = 0; h < HPAD; h += 2) {
                    const float w0 = ex2(zf[h] - m_run[h] + SH) * wmul, w1 = ex2(zf[h + 1] - m_run[h + 1] + SH) * wmul;
                    ph[h / 2] = pack_h2(w0, w1);
                    const float2 wf = __half22float2(*reinterpret_cast<const __half2*>(&ph[h / 2]));
                    const float p0 = wf.x * winv, p1 = wf.y * winv;
                    l_run[h] += p0; l_run[h + 1] += p1;
                    lz_run[h] = fmaf(p0, vzero, lz_run[h]); lz_run[h + 1] = fmaf(p1, vzero, lz_run[h + 1]);
                }
            } else if (VM) {
#pragma unroll
                for (int h = 0; h < HPAD; h += 2)
                {
                    ph[h / 2] = pack_h2(ex2(zf[h] - m_run[h] + SH), ex2(zf[h + 1] - m_run[h + 1] + SH));
                    flush_h2(ph[h / 2], wsum[h], wsum[h + 1]);       // the rounded weights are what the normaliser sums
                }
            } else {
#pragma unroll
                for (int h = 0; h < HPAD; ++h) { zf[h] = ex2(zf[h] - m_run[h]); l_run[h] += zf[h]; }
            }

            if (VM) {
                // ---- value side on tensor cores ---------------------------------------------------------
                // D[m][n] += sum_k A[m][k] B[k][n], m16 n8 k16, per 8-token sub-tile and group block gb:
                //   k = (token j of the sub-tile, sub-coefficient i in {0,1}),
                //   A[m][(j,i)] = 2^-24 x grid index of codeword(token j, group 8gb + (m & 7))[2 (m >> 3) + i]     fp16 (subnormal)
                //   B[(j,i)][(h,i')] = w_h(token j) * [i == i']                                                fp16
                //   D[m][(h,i')] = partial of head h, group 8gb + (m & 7), coefficient 2 (m >> 3) + i'
                // weights -> shared memory as fp16, [head][k-slot pair = token & 3][token >> 3, (token >> 2) & 1]
                __syncwarp();      // previous tile's readers of the P area are done
                {
                    const uint32_t wa = s_pw + (lane & 3) * 16 + ((lane >> 3) * 2 + ((lane >> 2) & 1)) * 2;
#pragma unroll
                    for (int h = 0; h < HPAD; ++h)
                        asm volatile("st.shared.u16 [%0], %1;" ::"r"(wa + h * 64),
                                     "h"((unsigned short)((h & 1) ? (ph[h / 2] >> 16) : (ph[h / 2] & 0xffffu))) : "memory");
                }
                __syncwarp();
                // B-fragment sources: 8 weights of head (4 hs + fr/2) for the tokens with (token & 3) == fc
                uint4 pw[HSETS];
#pragma unroll
                for (int hs = 0; hs < HSETS; ++hs) pw[hs] = lds_u128(s_pw + (hs * 4 + (fr >> 1)) * 64 + fc * 16);
#pragma unroll
                for (int blk = 0; blk < 2; ++blk) {
#pragma unroll
                    for (int ts = 0; ts < 2; ++ts) {                       // 8-token sub-tiles of the block
                        const int t = blk * 2 + ts;                         // sub-tile index within the 32-token tile
                        uint32_t b0[HSETS], b1[HSETS];
#pragma unroll
                        for (int hs = 0; hs < HSETS; ++hs) {
                            const uint32_t w = t == 0 ? pw[hs].x : (t == 1 ? pw[hs].y : (t == 2 ? pw[hs].z : pw[hs].w));
                            b0[hs] = __byte_perm(w, 0u, sel_b0);
                            b1[hs] = __byte_perm(w, 0u, sel_b1);
                        }
                        // gather: X[x][u] = codeword of token 8ts + 4u + fc of the block, group block x ^ (fc & 1), row fr
                        uint32_t X[NGB][2];
#pragma unroll
                        for (int x = 0; x < (VSQ ? 0 : NGB); ++x) {
                            const uint32_t vwd = cur.vw[blk][x];      // codes of the group block this load fetches (x ^ 1 in odd columns)
                            X[x][0] = vgather(vwd, 2 * ts, x);
                            X[x][1] = vgather(vwd, 2 * ts + 1, x);
                        }
#pragma unroll
                        for (int gb = 0; gb < NGB; ++gb) {
                            uint32_t a0, a1, a2, a3;
                            if (VSQ) {
                                // the token's byte of four levels into both halves of a word, from the even or odd columns' word,
                                // and two levels kept in place: the accumulators of level i carry 4^i
                                const uint32_t d0 = __byte_perm(cur.vw[blk][gb], cur.vw[blk][gb ^ 1], sel_lv + 0x1111u * (2 * ts));
                                const uint32_t d1 = __byte_perm(cur.vw[blk][gb], cur.vw[blk][gb ^ 1], sel_lv + 0x1111u * (2 * ts + 1));
                                a0 = d0 & 0x000c0003u; a1 = d0 & 0x00c00030u;
                                a2 = d1 & 0x000c0003u; a3 = d1 & 0x00c00030u;
                            } else {
                                // bytes (u, 0) pairs from X[gb] (even columns) or X[gb ^ 1] (odd columns)
                                a0 = prmt_rep(X[gb][0], X[gb ^ 1][0], sel_lo); a1 = prmt_rep(X[gb][0], X[gb ^ 1][0], sel_hi);
                                a2 = prmt_rep(X[gb][1], X[gb ^ 1][1], sel_lo); a3 = prmt_rep(X[gb][1], X[gb ^ 1][1], sel_hi);
                            }
#pragma unroll
                            for (int hs = 0; hs < HSETS; ++hs) mma_f16(macc[hs][gb], a0, a1, a2, a3, b0[hs], b1[hs]);
                        }
                    }
                }
                if ((it & (NOVAKV_WINDOW - 1)) == NOVAKV_WINDOW - 1) flush_window();
            } else {
                // ---- value side on CUDA cores (fp32): same lane coordinates and gathers, FMA instead of MMA ----
                __syncwarp();      // previous tile's readers of the P area are done
#pragma unroll
                for (int h = 0; h < HPAD; h += 4)
                    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(s_pw + lane * (HPAD * 4) + h * 4),
                                 "f"(zf[h]), "f"(zf[h + 1]), "f"(zf[h + 2]), "f"(zf[h + 3]) : "memory");
                __syncwarp();
#pragma unroll
                for (int blk = 0; blk < 2; ++blk)
#pragma unroll
                    for (int tq = 0; tq < 4; ++tq) {                       // this lane's 4 tokens of the block: 4 tq + fc
                        const int tok = blk * 16 + tq * 4 + fc;
                        float pf[HPAD];
#pragma unroll
                        for (int h = 0; h < HPAD; h += 4)
                            asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(pf[h]), "=f"(pf[h + 1]), "=f"(pf[h + 2]), "=f"(pf[h + 3])
                                         : "r"(s_pw + tok * (HPAD * 4) + h * 4));
#pragma unroll
                        for (int x = 0; x < NGB; ++x) {
                            // (odd lane columns fetch group block x ^ 1 with load x; their accumulator x holds that block)
                            const uint32_t cwd = vgather(cur.vw[blk][x], tq, x);
                            // grid indices -> binary32, centred: bytes (u, 0) are the binary16 subnormals u 2^-24
                            const __half2 c64 = __halves2half2(__ushort_as_half((unsigned short)64), __ushort_as_half((unsigned short)64));
                            const uint32_t h01 = __byte_perm(cwd, 0u, 0x4140u), h23 = __byte_perm(cwd, 0u, 0x4342u);
                            const float2 f01 = __half22float2(__hsub2(*reinterpret_cast<const __half2*>(&h01), c64));
                            const float2 f23 = __half22float2(__hsub2(*reinterpret_cast<const __half2*>(&h23), c64));
                            const uint64_t v01 = pack2(f01.x, f01.y), v23 = pack2(f23.x, f23.y);
#pragma unroll
                            for (int h = 0; h < HPAD; ++h) {
                                const uint64_t p2 = pack2(pf[h], pf[h]);
                                ffma2(acc[VM ? 0 : x][VM ? 0 : h][0], v01, p2);
                                ffma2(acc[VM ? 0 : x][VM ? 0 : h][1], v23, p2);
                            }
                        }
                    }
            }
        };

        // ---- score table (the first tile's loads are issued before, so that they fly during the build)
        TileRegs<L> ta;
        if (n_it > 0) load_tile(0, ta);
        NOVAKV_TICK(1)
        build_score_table<D, HG, VM>(t32_p, t16_p, cb_k_lut + (size_t)sg.kvh * 256 * L * 4,
                                     reinterpret_cast<const float*>(s_abs + C::Q + cur_seg * C::Q_BYTES));
        NOVAKV_TICK(2)
        async_copies_wait();
        __syncthreads();     // table and value codebook complete, next segment found
        if (rem > 0) stage_query(s_found[cur_seg ^ 1][0], s_found[cur_seg ^ 1][3], cur_seg ^ 1);
        NOVAKV_TICK(3)

        // ---- scan: 32-token tiles, the next tile's loads in flight while one is consumed
        for (int it = 0; it < n_it; ++it) {
            const TileRegs<L> cur = ta;
            if (it + 1 < n_it) load_tile(it + 1, ta);
            process(cur, it);
        }

        // ---- segment epilogue: merge the warps' partials, write one partial ---------------------
        NOVAKV_TICK(4)
        if (VM) flush_window();
        const Segment done = sg;
        if (rem > 0) {
            const long u_stop = s_bnd[blockIdx.x + 1];
            cur_seg ^= 1;
            sg = segment_at(page_prefix, batch, u_stop - rem, u_stop, s_found[cur_seg]);
            fetch_ids();
        }
        __syncthreads();                                   // scan done everywhere: the tables are dead
        NOVAKV_TICK(5)
        unsigned char* const merge_p = HAS16 ? t16_p : t32_p;
        float* m_acc = reinterpret_cast<float*>(merge_p);                              // [NCW][HPAD][MROW]
        float* m_ml = reinterpret_cast<float*>(merge_p + C::MERGE_ACC_BYTES);          // [NCW][HPAD][2]
        float* m_lz = m_ml + NCW * HPAD * 2;                                           // [NCW][HPAD]  (VSQ)
        if (VM && !VSQ) {
            // lane (fr = 0, fc) holds the weight sum of heads 4 hs + fc
            if (fr == 0) {
#pragma unroll
                for (int hs = 0; hs < HSETS; ++hs) {
                    const float ma01 = fc & 1 ? m_run[hs * 4 + 1] : m_run[hs * 4 + 0];
                    const float ma23 = fc & 1 ? m_run[hs * 4 + 3] : m_run[hs * 4 + 2];
                    m_ml[(warp * HPAD + hs * 4 + fc) * 2] = fc & 2 ? ma23 : ma01;
                    m_ml[(warp * HPAD + hs * 4 + fc) * 2 + 1] = l_run[hs];
                }
            }
        } else {
#pragma unroll
            for (int h = 0; h < HPAD; ++h) {
                const float lsum = warp_sum(l_run[h]);
                if (lane == 0) { m_ml[(warp * HPAD + h) * 2] = m_run[h]; m_ml[(warp * HPAD + h) * 2 + 1] = lsum; }
                if (VSQ) {
                    const float lz = warp_sum(lz_run[h]);
                    if (lane == 0) m_lz[warp * HPAD + h] = lz;
                    lz_run[h] = 0.f;
                }
            }
        }
#pragma unroll
        for (int h = 0; h < HPAD; ++h) { m_run[h] = M_INIT; l_run[h] = 0.f; }
        if (VM) {
            // VSQ: the sums carry 2^-E of the scales; E is per warp, so it is folded back here
            const float unsh = VSQ ? esh_pow : 1.f;
#pragma unroll
            for (int hs = 0; hs < HSETS; ++hs)
#pragma unroll
                for (int gb = 0; gb < NGB; ++gb) {
                    *reinterpret_cast<float4*>(m_acc + ((size_t)warp * HPAD + hs * 4 + fc) * C::MROW + (8 * gb + fr) * 4) =
                        VSQ ? make_float4(macc[hs][gb][0] * unsh, macc[hs][gb][1] * (unsh * 0.25f), macc[hs][gb][2] * (unsh * 0.0625f), macc[hs][gb][3] * (unsh * 0.015625f))
                            : make_float4(macc[hs][gb][0], macc[hs][gb][1], macc[hs][gb][2], macc[hs][gb][3]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) macc[hs][gb][i] = 0.f;
                }
            esh_pow = 0.f;
        } else {
            // every lane column holds a partial over its own tokens (accumulator x of an odd column belongs to group
            // block x ^ 1): add the four columns, column fc writes head 4 k + fc
#pragma unroll
            for (int x = 0; x < NGB; ++x) {
#pragma unroll
                for (int h = 0; h < HPAD; ++h) {
                    float a0, a1, a2, a3, b0, b1, b2, b3;
                    unpack2(acc[VM ? 0 : x][VM ? 0 : h][0], a0, a1);
                    unpack2(acc[VM ? 0 : x][VM ? 0 : h][1], a2, a3);
                    unpack2(acc[VM ? 0 : (x ^ 1)][VM ? 0 : h][0], b0, b1);
                    unpack2(acc[VM ? 0 : (x ^ 1)][VM ? 0 : h][1], b2, b3);
                    if (odd_col) { a0 = b0; a1 = b1; a2 = b2; a3 = b3; }           // now: this lane's partial of group block x
#pragma unroll
                    for (int o = 1; o <= 2; o <<= 1) {
                        a0 += __shfl_xor_sync(0xffffffffu, a0, o); a1 += __shfl_xor_sync(0xffffffffu, a1, o);
                        a2 += __shfl_xor_sync(0xffffffffu, a2, o); a3 += __shfl_xor_sync(0xffffffffu, a3, o);
                    }
                    if ((h & 3) == fc)
                        *reinterpret_cast<float4*>(m_acc + ((size_t)warp * HPAD + h) * C::MROW + (8 * x + fr) * 4) = make_float4(a0, a1, a2, a3);
                }
            }
#pragma unroll
            for (int x = 0; x < NGB; ++x)
#pragma unroll
                for (int h = 0; h < HPAD; ++h) { acc[VM ? 0 : x][VM ? 0 : h][0] = 0ull; acc[VM ? 0 : x][VM ? 0 : h][1] = 0ull; }
        }
        __syncthreads();
        {
            const size_t pidx = (size_t)pair + blockIdx.x;      // unique: pair and CTA index both grow along the walk
            const float unscale = VM ? 3.0517578125e-05f : 1.f;  // 2^-15: the weights carried 2^15
            for (int i = threadIdx.x; i < HG * D; i += S1_THREADS) {
                const int h = i / D, c = i - h * D;
                float M = M_INIT;
#pragma unroll
                for (int w = 0; w < NCW; ++w) M = fmaxf(M, m_ml[(w * HPAD + h) * 2]);
                float a = 0.f, lsum = 0.f, zsum = 0.f;
#pragma unroll
                for (int w = 0; w < NCW; ++w) {
                    const float sc = ex2(m_ml[(w * HPAD + h) * 2] - M);
                    a = fmaf(sc, m_acc[((size_t)w * HPAD + h) * C::MROW + c], a);
                    if (VSQ) zsum = fmaf(sc, m_lz[w * HPAD + h], zsum);              // zero-points: the same amount on every coefficient
                    lsum = fmaf(sc, m_ml[(w * HPAD + h) * 2 + 1], lsum);
                }
                // grid index sums -> value-transform coefficients: s (u - 64) + (lo + 64 s) per unit of weight
                a *= 16777216.f;                           // indices entered the sums as u 2^-24
                float val;
                if (VSQ) val = (a + zsum) * unscale;       // levels are the codes themselves (s = 1, no offset)
                else val = (v_scale[(size_t)done.kvh * D + c] * a + v_off[(size_t)done.kvh * D + c] * lsum) * unscale;
                part_acc[(pidx * HG + h) * D + c] = val;
                if (c == 0) { part_ml[(pidx * HG + h) * 2] = M; part_ml[(pidx * HG + h) * 2 + 1] = lsum * unscale; }
            }
        }
        if (out_fused != nullptr) {
            // arrival: this CTA's partial is visible before its count is; the CTA that completes the count merges
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) {
                s_arrived = atomicAdd(&pair_count[pair], 1) + 1;
                s_first = gridDim.x;
                s_last = -1;
            }
            __syncthreads();
            const long P = page_prefix[batch];
            const long pu0 = (long)done.kvh * P + page_prefix[done.b], pu1 = pu0 + (done.len + NOVAKV_PAGE_TOKENS - 1) / NOVAKV_PAGE_TOKENS;
            bool touches = false;                           // CTA threadIdx.x has a non-empty share of this pair
            if (threadIdx.x < gridDim.x) {
                const int c = threadIdx.x;
                touches = s_bnd[c] < s_bnd[c + 1] && s_bnd[c] < pu1 && s_bnd[c + 1] > pu0;
                if (touches) { atomicMin(&s_first, c); atomicMax(&s_last, c); }
            }
            const int expected = __syncthreads_count(touches);
            if (s_arrived == expected) {
                __threadfence();
                fused_merge<D, HG>(reinterpret_cast<float*>(t32_p), part_ml, part_acc, pair, s_first, s_last, s_bnd, rv_t, v_mean,
                                   done.kvh, out_fused, out_is_fp32, ((size_t)done.b * n_q_heads + done.kvh * HG) * D);
                if (threadIdx.x == 0) pair_count[pair] = 0;
            }
        }
        async_copies_wait();
        __syncthreads();                                   // merge buffer free, next query complete: the next table can be built
        NOVAKV_TICK(6)
#ifdef NOVAKV_TIMING
        ++n_seg;
#endif
    }
#ifdef NOVAKV_TIMING
    unsigned long long g_end;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_end));
    if (threadIdx.x == 0)
        printf("cta %3d segs %d pages %ld | clocks: pre-loop %lld locate+q %lld build %lld vcbwait %lld scan(w0) %lld barrier %lld epilogue %lld total %lld | ns start %llu end %llu\n",
               blockIdx.x, n_seg, (long)(u_end - u_begin), tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], tm[6], clock64() - t_start, g_start, g_end);
#endif
}

// ------------------------------------------------------------------------------------------------
// stage 1 for d = 64 and eight query heads per KV head: logits on tensor cores too
// ------------------------------------------------------------------------------------------------
// A score table costs 32 bytes of shared-memory reads and eight additions per (token, group) here.  A key codeword costs 16
// bytes - four binary16 coordinates and their binary16 remainders, about 22 bits - and the additions are matrix products
// over all eight heads at once, binary32 accumulators.
// The codewords belong to the KV head, so a segment has no table to build: its set-up is 16 numbers of q' per lane.
//   mma m16n8k16: rows 0-7 = q_hi and rows 8-15 = q_lo of the eight heads, columns = 8 tokens, K = 4 groups; one product
//   takes the codewords' hi halves and one their remainders, and a logit is the sum of its two rows.  The tensor core
//   truncates: the remainders have accumulators of their own, so that four truncations at the size of the logit are left
//   instead of eight, and what those lose on average (half an ulp each at a size that grows: 1.0e-7, measured) is given back
//   by the addition that the remainders need anyway.  Lane
//   (fr, fc) = (lane / 4, lane % 4) supplies groups 4 fc .. 4 fc + 3 (one per k-step) of the token in column fr: the two
//   64-bit halves of a 128-bit gather are the two B operands as they stand.  (Codewords as A, tokens as rows, need three
//   products for 16 tokens instead of four, but the operand then mixes two gathers: 64 register moves per 32 tokens.)
//   Column c of a block of 8 tokens is token c / 2 + 4 (c % 2): the weights of a lane then are the B operand of the value
//   product in the order in which the cache keeps the value bytes of a lane (tokens fc, 4 + fc, 8 + fc, 12 + fc).
//   value product: rows = (group 8 gb + fr, coordinate 2 cp) and, at fr + 8, coordinate 2 cp + 1; K = 16 tokens.  One byte
//   permutation takes the same coordinate of two codewords and widens it (bytes with a clear top bit pair with their
//   replicated top bit), and one multiply-add centres the grid.  (Sixteen products of one sign, truncated at the size of
//   their sum before its centre is removed, cost 0.4 % of the output error at 32 tokens and 5 % at 512.)
// Error against binary64, 96 sequences: outputs (rel) 6.47e-5 / 5.09e-5 / 5.89e-5 at 60 / 700 / 4000 tokens, the table kernel
// 6.49e-5 / 5.17e-5 / 6.23e-5; log-sum-exp at 512 tokens 1.357e-5 against 1.356e-5 (binary16 weights are what both show).
// Rows of 256 bytes, so that one byte permutation puts a code into an address.  Bank conflicts: the eight lanes of a quarter
// warp read four groups of two tokens; two copies of the key codewords, their columns 64 bytes apart, serve even and odd fr.
// Four copies of the value codewords, 32 bytes apart, serve the four fc.
// Measured (16 sequences of 65536 tokens, 8 KV heads, sink, whole call): score table 193 us, this kernel 161 us (145 us with one
// chain of products and the centre removed afterwards, 4 us of it the accumulators of the remainders and 12 us the
// multiply-adds, two chains of hi products 165 us).  No single bound.
struct S1M {
    static constexpr int D = 64, HG = 8, L = 16;
    static constexpr int KEY_COPY = 65536, VAL_BYTES = 65536;
    static constexpr int TILE_BYTES = 32 * L, PAGE_BYTES = 2 * TILE_BYTES;
    static constexpr int MROW = D + 4, MHEADS = 4;                         // merge buffer: four heads at a time
    // Shared-window addresses, fixed so that they are immediates of the gathers: 32 additions per 32 tokens otherwise.
    // (The window's first KB and the static words lie below; checked at run time.)
    static constexpr int KEY = 4096;                                       // [2 copies][256 codes][16 columns][16 B]
    static constexpr int VAL = KEY + 2 * KEY_COPY;                         // [256 codes][2 group blocks][4 copies][8 groups][4 B]
    static constexpr int MACC = VAL + VAL_BYTES;
    static constexpr int ML = MACC + NCW * MHEADS * MROW * 4;
    static constexpr int BND = ML + NCW * HG * 8;
    static constexpr int PFX = BND + (MAX_SCAN_CTAS + 1) * 8;
    static constexpr int SMEM = PFX + 2 * (PFX_CAP + 1) * 4;
    static_assert(SMEM <= S1_SMEM_BYTES, "shared memory budget");
};
__global__ void __launch_bounds__(S1_THREADS, 1)
novakv_decode_mma_kernel(const float* __restrict__ qp, const uint4* __restrict__ cb_k_mma /* [Hkv][256][16] (hi, lo) */,
                         const float* __restrict__ k_mma_scale /* [Hkv][64] */, const uint8_t* __restrict__ cb_v_img,
                         const float* __restrict__ v_scale, const float* __restrict__ v_off, const uint8_t* __restrict__ k_pages,
                         const uint8_t* __restrict__ v_pages, int n_pages, const int32_t* __restrict__ page_table,
                         int max_pages_per_seq, const int32_t* __restrict__ seq_lens, int32_t* __restrict__ page_prefix_g,
                         int batch, int n_q_heads, int n_kv_heads, float* __restrict__ part_ml, float* __restrict__ part_acc,
                         uint32_t* __restrict__ dev_status, int pt_stride, int32_t* __restrict__ cost_prefix_g,
                         int seg_weight, long* __restrict__ cta_range, int form_prefix) {
    using C = S1M;
    constexpr int D = C::D, HG = C::HG, L = C::L;
    constexpr float SH = 15.f;                                // weights are scaled by 2^SH before the binary16 rounding
    constexpr float LOST = 1.0e-7f;                           // share of a logit that four truncated accumulations lose on average
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ int s_found[2][4], s_part[2][NCW];
    const uint32_t s_base = smem_u32(smem);
    if (s_base > C::KEY || C::SMEM - s_base > (uint32_t)S1_SMEM_BYTES) {
        // cannot happen with the shared address window of this architecture; reported, never trapped
        leave_unscanned(cta_range, form_prefix, seq_lens, batch, max_pages_per_seq, seg_weight, page_prefix_g, cost_prefix_g, dev_status);
        return;
    }
    unsigned char* const s_abs = smem - s_base;               // s_abs + a: the byte at shared-window address a

    // codewords of a KV head -> shared memory
    auto stage_head = [&](int kvh) {
        const uint4* src = cb_k_mma + (size_t)kvh * 256 * L;
        for (int i = threadIdx.x; i < 256 * L; i += S1_THREADS) {
            const uint32_t dst = C::KEY + (i >> 4) * 256, col = (i & 3) * 4 + ((i >> 2) & 3);     // k-step, fc
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst + col * 16), "l"(src + i) : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst + C::KEY_COPY + (col ^ 4) * 16), "l"(src + i) : "memory");
        }
        const uint8_t* vsrc = cb_v_img + (size_t)kvh * VCB_COPY_BYTES;
        for (int i = threadIdx.x; i < 256 * (L / 4); i += S1_THREADS) {
            const int code = i >> 2, ch = i & 3;              // four groups of a codeword row
#pragma unroll
            for (int c = 0; c < 4; ++c)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(C::VAL + code * 256 + (ch >> 1) * 128 + c * 32 + (ch & 1) * 16),
                             "l"(vsrc + code * VCB_ROW + ch * 16) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int head = (int)(((long)blockIdx.x * n_kv_heads) / gridDim.x);   // KV head whose codewords are resident (see the other kernel)
    stage_head(head);
    novakv_grid_dependency_wait();

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int32_t *page_prefix = page_prefix_g, *cost_prefix = cost_prefix_g;
    if (form_prefix) {                                        // (batches of at most PFX_CAP sequences)
        int32_t* pfx = reinterpret_cast<int32_t*>(s_abs + C::PFX);
        form_prefixes(pfx, s_part, seq_lens, batch, max_pages_per_seq, seg_weight, page_prefix_g, cost_prefix_g, dev_status);
        page_prefix = pfx;
        cost_prefix = pfx + PFX_CAP + 1;
    } else if (batch <= PFX_CAP) {
        int32_t* pfx = reinterpret_cast<int32_t*>(s_abs + C::PFX);
        for (int i = threadIdx.x; i <= batch; i += S1_THREADS) { pfx[i] = page_prefix_g[i]; pfx[PFX_CAP + 1 + i] = cost_prefix_g[i]; }
        __syncthreads();
        page_prefix = pfx;
        cost_prefix = pfx + PFX_CAP + 1;
    }
    long* const s_bnd = reinterpret_cast<long*>(s_abs + C::BND);
    for (int c = threadIdx.x; c <= (int)gridDim.x; c += S1_THREADS)
        s_bnd[c] = scan_boundary(c, gridDim.x, page_prefix, cost_prefix, batch, n_kv_heads, seg_weight);
    __syncthreads();
    const long u_begin = s_bnd[blockIdx.x], u_end = s_bnd[blockIdx.x + 1];
    if (threadIdx.x == 0) { cta_range[blockIdx.x * 2] = u_begin; cta_range[blockIdx.x * 2 + 1] = u_end; }
    if (u_begin >= u_end) { async_copies_wait(); return; }

    // ---- lane roles and constants
    const int fr = lane >> 2, fc = lane & 3;
    const int tau = (fr >> 1) + 4 * (fr & 1);                 // this lane's token in a block of 8 (rows fr, fr + 8 of an operand)
    // byte j of a token holds group j ^ tau: the codes of groups 4 fc + ks lie in word fc ^ (tau / 4), byte ks ^ (tau % 4)
    const uint32_t key_word = (uint32_t)(fc ^ (tau >> 2)) * 4;
    uint32_t ksel[4], kcol[2];                                // gather offset = byte permutation of (codes, kcol[ks % 2]) by ksel[ks]
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        ksel[ks] = 0x7604u | ((uint32_t)(ks ^ (tau & 3)) << 4);
        asm volatile("" : "+r"(ksel[ks]));                    // (kept in registers: formed again in every tile otherwise)
    }
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
        kcol[ks] = (fr & 1) * C::KEY_COPY + ((4 * ks + fc) ^ (4 * (fr & 1))) * 16;
        asm volatile("" : "+r"(kcol[ks]));
    }
    const uint32_t vcol = fc * 32 + fr * 4;

    float m_run = M_INIT, l_run = 0.f, wsum[2] = {0.f, 0.f};  // head fr (wsum: even and odd columns)
    float macc[2][2][4];                                      // [gb][cp]: coordinate 2 cp of heads 2 fc, + 1, then 2 cp + 1
#pragma unroll
    for (int i = 0; i < 16; ++i) macc[i >> 3][(i >> 2) & 1][i & 3] = 0.f;
    auto flush_window = [&]() {
        l_run += wsum[0] + wsum[1];
        wsum[0] = wsum[1] = 0.f;
    };

    // What a segment needs from global memory before its first tile - query, page ids - is asked for while the partials of
    // the segment before are merged, and its place in the batch is looked up during the scan before that: 16 sequences of
    // 65536 tokens 151 -> 149 us, 5 of 5001 52.9 -> 52.4.  (The table kernel does not gain: its table build needs the SM
    // for twice the time of these loads, and the registers slow its scan by 0-2 %.)
    long u = u_begin;
    Segment sg;
    int n_it = 0, ids_cur = 0, ids_next = 0;
    const int32_t* pt = nullptr;
    float4 qv[4];                                             // q' of head fr, groups 4 fc + ks
    auto load_ids = [&](int batch_i) {
        const int it = batch_i * 32 + lane;
        int page = 0;
        if (it < n_it) {
            page = pt[(warp + NCW * it) >> 1];
            if (page < 0 || page >= n_pages) { atomicOr(dev_status, NOVAKV_DEV_BAD_PAGE); page = 0; }
        }
        return page;
    };
    auto fetch_segment = [&]() {
        // this warp's tiles of the segment: half pages hp = warp, warp + NCW, ...
        const int n_half = min(2 * sg.npg, (sg.len - sg.pg0 * NOVAKV_PAGE_TOKENS + 31) / 32);
        n_it = n_half > warp ? (n_half - warp + NCW - 1) / NCW : 0;
        pt = page_table + (size_t)sg.b * pt_stride + sg.pg0;
        const float4* q4 = reinterpret_cast<const float4*>(qp + ((size_t)sg.b * n_q_heads + sg.kvh * HG + fr) * D) + 4 * fc;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) qv[ks] = q4[ks];
        ids_cur = load_ids(0);
        ids_next = load_ids(1);
    };
    uint32_t kn[4];                                       // key codes of tokens tau, + 8, + 16, + 24
    uint2 vn[2];                                          // value codes of a 16-token block: group blocks fc % 2, 1 - fc % 2
    auto load_tile = [&](int it) {
        if ((it & 31) == 0 && it > 0) { ids_cur = ids_next; ids_next = load_ids((it >> 5) + 1); }
        const int page = __shfl_sync(0xffffffffu, ids_cur, it & 31);
        const int half = (warp + NCW * it) & 1;
        const size_t off = ((size_t)page * n_kv_heads + sg.kvh) * C::PAGE_BYTES + half * C::TILE_BYTES;
        const uint8_t* kp = k_pages + off + tau * 16 + key_word;
        const uint8_t* vp = v_pages + off + lane * 8;
#pragma unroll
        for (int i = 0; i < 4; ++i) kn[i] = ldg_stream_32(kp + 128 * i);
#pragma unroll
        for (int blk = 0; blk < 2; ++blk) vn[blk] = ldg_stream_64(vp + blk * (L * 16));
    };

    int found = 0;                                            // the half of s_found that holds the current segment
    find_segment(page_prefix, seq_lens, batch, max_pages_per_seq, u, (int)(u / page_prefix[batch]), s_found[0]);
    __syncthreads();
    sg = segment_at(page_prefix, batch, u, u_end, s_found[0]);
    fetch_segment();
    while (u < u_end) {
        const int pair = sg.kvh * batch + sg.b;
        if (n_it > 0) load_tile(0);
        if (head != sg.kvh) { stage_head(sg.kvh); head = sg.kvh; }       // (every warp is past the last segment's scan)
        const long u_next = u + sg.npg;
        if (u_next < u_end)
            find_segment(page_prefix, seq_lens, batch, max_pages_per_seq, u_next,
                         sg.kvh + (u_next >= (long)(sg.kvh + 1) * page_prefix[batch]), s_found[found ^ 1]);

        // q' of head fr, groups 4 fc + ks, in the key codewords' scale; per head a power of two brings the largest to
        // [2^9, 2^10), so that binary16 halves neither overflow nor lose small coordinates
        uint32_t qa[4][4];                                    // A operand of a k-step: hi, lo of coordinates 0, 1, then of 2, 3
        float us;
        {
            const float4* s4 = reinterpret_cast<const float4*>(k_mma_scale + (size_t)sg.kvh * D) + 4 * fc;
            float mx = 0.f;
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                const float4 a = qv[ks], s = s4[ks];
                qv[ks] = make_float4(a.x * s.x, a.y * s.y, a.z * s.z, a.w * s.w);
                mx = fmaxf(fmaxf(mx, fmaxf(fabsf(qv[ks].x), fabsf(qv[ks].y))), fmaxf(fabsf(qv[ks].z), fabsf(qv[ks].w)));
            }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            int e = (int)(__float_as_uint(mx) >> 23) - 127 - 9;
            e = max(-100, min(e, 110));
            const float down = __uint_as_float((uint32_t)(127 - e) << 23);
            us = __uint_as_float((uint32_t)(127 + e) << 23);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                const float v[4] = {qv[ks].x * down, qv[ks].y * down, qv[ks].z * down, qv[ks].w * down};
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const uint32_t hi = pack_h2(v[2 * i], v[2 * i + 1]);
                    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&hi));
                    qa[ks][2 * i] = hi;
                    qa[ks][2 * i + 1] = pack_h2(v[2 * i] - f.x, v[2 * i + 1] - f.y);
                }
            }
        }

        async_copies_wait();
        __syncthreads();                                      // codewords complete (and the last segment's merge is read out)

#pragma unroll 1
        for (int it = 0; it < n_it; ++it) {
            uint32_t kc[4];
            uint2 vc[2];
#pragma unroll
            for (int i = 0; i < 4; ++i) kc[i] = kn[i];
            vc[0] = vn[0]; vc[1] = vn[1];
            if (it + 1 < n_it) load_tile(it + 1);
            const int hp = warp + NCW * it;
            const int nvalid = min(32, sg.len - ((sg.pg0 + (hp >> 1)) * NOVAKV_PAGE_TOKENS + (hp & 1) * 32));

            // ---- logits of head fr, tokens 8 i + fc and 8 i + 4 + fc, over us
            float z[4][2];
            {
                float acc[4][4], rem[4][4];                       // products of the codewords' hi halves; of their remainders
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    uint4 c[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        c[i] = ks < 2 ? lds_u128_at<C::KEY>(prmt_rep(kc[i], kcol[ks & 1], ksel[ks]))
                                      : lds_u128_at<C::KEY + 128>(prmt_rep(kc[i], kcol[ks & 1], ksel[ks]));
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (ks == 0) mma_f16_zero(acc[i], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], c[i].x, c[i].y);
                        else mma_f16(acc[i], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], c[i].x, c[i].y);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (ks == 0) mma_f16_zero(rem[i], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], c[i].z, c[i].w);
                        else mma_f16(rem[i], qa[ks][0], qa[ks][1], qa[ks][2], qa[ks][3], c[i].z, c[i].w);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j) z[i][j] = acc[i][j] + fmaf(acc[i][j], LOST, (rem[i][j] + rem[i][2 + j]) + acc[i][2 + j]);
            }
            if (nvalid < 32) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (8 * (i >> 1) + 4 * (i & 1) + fc >= nvalid) z[i >> 1][i & 1] = -CUDART_INF_F;
            }
            // ---- online softmax (base 2), as in the other kernel; the four lanes of a quad share a head
            {
                float t = fmaxf(fmaxf(fmaxf(z[0][0], z[0][1]), fmaxf(z[1][0], z[1][1])), fmaxf(fmaxf(z[2][0], z[2][1]), fmaxf(z[3][0], z[3][1]))) * us;
                if (__any_sync(0xffffffffu, t > m_run)) {
                    t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, 1));
                    t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, 2));
                    const float m_new = t > m_run ? t + M_SLACK : m_run;
                    const float al = ex2(m_run - m_new);
                    m_run = m_new;
                    l_run *= al;
                    wsum[0] *= al;
                    wsum[1] *= al;
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const float a = __shfl_sync(0xffffffffu, al, 8 * fc + 4 * j);
#pragma unroll
                        for (int gb = 0; gb < 2; ++gb)
#pragma unroll
                            for (int cp = 0; cp < 2; ++cp) { macc[gb][cp][j] *= a; macc[gb][cp][2 + j] *= a; }
                    }
                }
            }
            // ---- weights: as they stand the B operand of the value product
            uint32_t bw[4];
            {
                const float o = SH - m_run;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    bw[i] = pack_h2(ex2(fmaf(z[i][0], us, o)), ex2(fmaf(z[i][1], us, o)));
                    flush_h2(bw[i], wsum[0], wsum[1]);        // the rounded weights are what the normaliser sums
                }
            }
            // ---- values
#pragma unroll
            for (int blk = 0; blk < 2; ++blk) {
                const uint32_t codes[2] = {fc & 1 ? vc[blk].y : vc[blk].x, fc & 1 ? vc[blk].x : vc[blk].y};
#pragma unroll
                for (int gb = 0; gb < 2; ++gb) {
                    uint32_t X[4];                            // codewords of tokens fc, 4 + fc, 8 + fc, 12 + fc
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        X[t] = gb ? lds_u32_at<C::VAL + 128>(__byte_perm(codes[gb], vcol, 0x7604u | (t << 4))) : lds_u32_at<C::VAL>(__byte_perm(codes[gb], vcol, 0x7604u | (t << 4)));
#pragma unroll
                    for (int cp = 0; cp < 2; ++cp) {
                        constexpr uint32_t SEL0 = 0xC480u;     // bytes (u0, 0, u4, 0): the same coordinate of two codewords
                        const uint32_t sa = SEL0 + 0x1111u * (2 * cp), sb = SEL0 + 0x1111u * (2 * cp + 1);
                        mma_f16(macc[gb][cp], grid_steps(prmt_rep(X[0], X[1], sa)), grid_steps(prmt_rep(X[0], X[1], sb)),
                                grid_steps(prmt_rep(X[2], X[3], sa)), grid_steps(prmt_rep(X[2], X[3], sb)), bw[2 * blk], bw[2 * blk + 1]);
                    }
                }
            }
            if ((it & (NOVAKV_WINDOW - 1)) == NOVAKV_WINDOW - 1) flush_window();
        }

        // ---- segment epilogue: merge the warps' partials, four heads at a time, and write one partial
        const float vs = v_scale[(size_t)sg.kvh * D + threadIdx.x % D], vo = v_off[(size_t)sg.kvh * D + threadIdx.x % D];
        flush_window();
        l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
        l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
        float* const m_acc = reinterpret_cast<float*>(s_abs + C::MACC);             // [NCW][MHEADS][MROW]
        float2* const m_ml = reinterpret_cast<float2*>(s_abs + C::ML);              // [NCW][HG]
        if (fc == 0) m_ml[warp * HG + fr] = make_float2(m_run, l_run);
        const size_t pidx = (size_t)pair + blockIdx.x;          // unique: pair and CTA index both grow along the walk
        if (u_next < u_end) {
            found ^= 1;
            sg = segment_at(page_prefix, batch, u_next, u_end, s_found[found]);
            fetch_segment();                                  // flies during the merge
        }
#pragma unroll 1
        for (int hp = 0; hp < HG / C::MHEADS; ++hp) {
            if ((fc >> 1) == hp) {
#pragma unroll
                for (int gb = 0; gb < 2; ++gb)
#pragma unroll
                    for (int cp = 0; cp < 2; ++cp)
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            *reinterpret_cast<float2*>(m_acc + (warp * C::MHEADS + 2 * (fc & 1) + j) * C::MROW + (8 * gb + fr) * 4 + 2 * cp) =
                                make_float2(macc[gb][cp][j], macc[gb][cp][2 + j]);
            }
            __syncthreads();
            for (int i = threadIdx.x; i < C::MHEADS * D; i += S1_THREADS) {
                const int hl = i / D, c = i - hl * D, h = hp * C::MHEADS + hl;
                float M = M_INIT;
#pragma unroll
                for (int w = 0; w < NCW; ++w) M = fmaxf(M, m_ml[w * HG + h].x);
                float a = 0.f, lsum = 0.f;
#pragma unroll
                for (int w = 0; w < NCW; ++w) {
                    const float2 ml = m_ml[w * HG + h];
                    const float sc = ex2(ml.x - M);
                    a = fmaf(sc, m_acc[(w * C::MHEADS + hl) * C::MROW + c], a);
                    lsum = fmaf(sc, ml.y, lsum);
                }
                // grid index sums -> value-transform coefficients: s (u - 64) + (lo + 64 s) per unit of weight
                const float val = (vs * (a * 1024.f) + vo * lsum) * 3.0517578125e-05f;
                part_acc[(pidx * HG + h) * D + c] = val;
                if (c == 0) { part_ml[(pidx * HG + h) * 2] = M; part_ml[(pidx * HG + h) * 2 + 1] = lsum * 3.0517578125e-05f; }
            }
            __syncthreads();
        }
        m_run = M_INIT;
        l_run = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) macc[i >> 3][(i >> 2) & 1][i & 3] = 0.f;
        u = u_next;
    }
}

// ------------------------------------------------------------------------------------------------
// merge + inverse value transform
// ------------------------------------------------------------------------------------------------
// One block per KV head and run of sequences, NP sequences at a time; it keeps its slice of the inverse transform in
// registers.  A warp finds the pieces of one sequence (the CTAs whose recorded ranges meet it), their common maximum and
// their scales; then every thread sums its coordinate over the pieces, all loads independent.  Bound by that chain of
// memory latencies (lengths and prefixes, ranges, (max, sum) pairs, accumulators: about 3 us), which the sequences of a
// block share: 256 pairs 11.5 -> 9.0 us, 1024 pairs 22.4 -> 19.3 us (cold caches).
// RUNS = false: one sequence per block (batches that give every SM at most one block).  Nothing is shared then, and the
// warp's 10 shuffles per head would only lengthen the chain: all threads fetch the candidates and their (max, sum) pairs, and
// every thread combines them itself.  16 sequences of the d = 64 shape with eight heads: 7.7 us with the shuffles, 6.5
// without (cold); d = 128, 8 sequences: 7.9 us where one warp searches, 7.1 so.
// EXT = the call carries a learned sink logit and/or a BF16 band partial; without it that code is compiled out.
// With eight heads per KV head runs do not pay: a block then has 512 threads and 126 registers, one an SM, and two sequences
// at a time.  One sequence per block in 64 registers (MINB = 2 blocks an SM) beyond one block per SM: whole calls of 100
// tokens, 37 / 64 / 192 sequences 23.0 / 35.4 / 77.0 us in runs, 19.8 / 33.6 / 72.5 so (with up to four heads and d = 128,
// 64 / 192: 38.1 / 96.5 and 40.6 / 103).
template <int D, int HG, bool EXT, bool RUNS, int MINB>
__global__ void __launch_bounds__(HG * D > 512 ? 512 : HG * D, MINB)
novakv_decode_merge_kernel(const float* __restrict__ part_ml, const float* __restrict__ part_acc,
                           const int32_t* __restrict__ page_prefix, const int32_t* __restrict__ seq_lens,
                           int batch, int n_q_heads, int n_kv_heads, int max_pages_per_seq, int grid_s1,
                           const float* __restrict__ rv_t, const float* __restrict__ v_mean,
                           void* __restrict__ out, int out_is_fp32,
                           const float* __restrict__ sink_logits /* [Hq] natural-log units, or null */,
                           const float* __restrict__ qk_off /* [batch][Hq], base-2 units */,
                           const float* __restrict__ band_ml /* [batch][Hq][2] (max, sum) of the BF16 band, or null */,
                           const float* __restrict__ band_acc /* [batch][Hq][D] sum p v of the band, original value domain */,
                           const int32_t* __restrict__ cost_prefix, int seg_weight, const long* __restrict__ cta_range,
                           int seqs_per_block) {
    constexpr int NP = RUNS ? 4 : 1, NT = HG * D > 512 ? 512 : HG * D, NW = NT / 32;
    constexpr int PARTS = NT / D, COLS = D / PARTS, PER = (HG * D + NT - 1) / NT;
    __shared__ float o_s[NP][HG * D];
    __shared__ float red_s[PARTS][HG][D];
    __shared__ short piece_s[RUNS ? NP : 1][RUNS ? MAX_SCAN_CTAS + 1 : 1];          // scan CTAs that hold a piece of the sequence
    __shared__ float scale_s[RUNS ? NP : 1][RUNS ? MAX_SCAN_CTAS + 1 : 1][HG];      // 2^(max of the piece - common max)
    __shared__ float2 ml_s[RUNS ? 1 : MAX_SCAN_CTAS + 1][HG];                       // (max, sum) of a candidate's piece
    __shared__ int cand_s[RUNS ? 1 : MAX_SCAN_CTAS + 1];                            // 1 = this candidate holds a piece
    __shared__ float m_s[NP][HG], l_s[NP][HG];                // common maximum and sum
    __shared__ float frac_s[NP][HG];                          // share of the softmax mass on quantised tokens (1 without sink and band)
    __shared__ float bsc_s[NP][HG];                           // multiplier of the band accumulator (0 without a band)
    __shared__ int n_s[NP];                                   // pieces; -1 = empty sequence
    const int run = blockIdx.x / n_kv_heads, kvh = blockIdx.x - run * n_kv_heads;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // constants of the inverse transform are fetched before the grid-dependency wait (they overlap the
    // tail of the scan kernel): this thread's slice of rv_t and the mean of its output coordinates
    float rv[COLS];
    {
        const float* R = rv_t + (size_t)kvh * D * D + (size_t)(threadIdx.x / D) * COLS * D + threadIdx.x % D;   // rv_t[c][r] = R_V[r][c]
#pragma unroll
        for (int c = 0; c < COLS; ++c) rv[c] = R[(size_t)c * D];
    }
    float vm[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) vm[k] = v_mean[(size_t)kvh * D + (threadIdx.x + k * NT) % D];
#ifdef NOVAKV_TIMING
    unsigned long long g_m0, g_m1, g_m2;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_m0));
#endif
    novakv_grid_dependency_wait();
#ifdef NOVAKV_TIMING
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_m1));
#endif
    const int b_end = RUNS ? min(batch, (run + 1) * seqs_per_block) : run + 1;
    for (int b0 = RUNS ? run * seqs_per_block : run; b0 < b_end; b0 += NP) {
        const int np = RUNS ? min(NP, b_end - b0) : 1;
        int c_first = 0, n_cand = 0;
        if (!RUNS) {
            // the same search, candidates and their (max, sum) pairs each fetched by as many threads
            const int pages_b = (clamp_len(seq_lens[b0], max_pages_per_seq) + NOVAKV_PAGE_TOKENS - 1) / NOVAKV_PAGE_TOKENS;
            if (pages_b > 0) {
                const long P = page_prefix[batch], cost_all = cost_prefix[batch];
                const long u0 = (long)kvh * P + page_prefix[b0], u1 = u0 + pages_b, T = cost_all * n_kv_heads;
                const long x0 = (long)kvh * cost_all + cost_prefix[b0] + seg_weight, x1 = x0 + pages_b - 1;
                c_first = max((int)(((x0 + 1) * grid_s1 - 1) / T) - 1, 0);
                n_cand = min((int)(((x1 + 1) * grid_s1 - 1) / T) + 1, grid_s1 - 1) - c_first + 1;
                for (int t = threadIdx.x; t < n_cand; t += NT) {
                    const long r0 = cta_range[(c_first + t) * 2], r1 = cta_range[(c_first + t) * 2 + 1];
                    cand_s[t] = r0 < r1 && r1 > u0 && r0 < u1;
                }
            }
            if (threadIdx.x == 0) n_s[0] = pages_b > 0 ? 0 : -1;
            __syncthreads();
            for (int i = threadIdx.x; i < n_cand * HG; i += NT)
                if (cand_s[i / HG])
                    ml_s[i / HG][i % HG] = *reinterpret_cast<const float2*>(part_ml + (((size_t)kvh * batch + b0 + c_first + i / HG) * HG + i % HG) * 2);
        }
        for (int p = RUNS ? warp : np; p < np; p += NW) {
            const int b = b0 + p;
            const int len = clamp_len(seq_lens[b], max_pages_per_seq);
            const int pages_b = (len + NOVAKV_PAGE_TOKENS - 1) / NOVAKV_PAGE_TOKENS;
            const size_t slot0 = (size_t)kvh * batch + b;          // the scan kernel's pair index (walk order)
            int n = pages_b > 0 ? 0 : -1;
            if (pages_b > 0) {
                // CTAs that may hold a piece: those whose cost range meets the pair's (the largest c with
                // floor(c*T/G) <= x for its first and last cost unit), widened by one on each side; the ranges the scan
                // CTAs recorded decide
                const long P = page_prefix[batch], cost_all = cost_prefix[batch];
                const long u0 = (long)kvh * P + page_prefix[b], u1 = u0 + pages_b;
                const long T = cost_all * n_kv_heads;
                const long x0 = (long)kvh * cost_all + cost_prefix[b] + seg_weight, x1 = x0 + pages_b - 1;
                const int c_first = max((int)(((x0 + 1) * grid_s1 - 1) / T) - 1, 0);
                const int c_last = min((int)(((x1 + 1) * grid_s1 - 1) / T) + 1, grid_s1 - 1);
                for (int c0 = c_first; c0 <= c_last; c0 += 32) {
                    bool has = false;
                    if (c0 + lane <= c_last) {
                        const long r0 = cta_range[(c0 + lane) * 2], r1 = cta_range[(c0 + lane) * 2 + 1];
                        has = r0 < r1 && r1 > u0 && r0 < u1;
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, has);
                    if (has) piece_s[p][n + __popc(m & ((1u << lane) - 1))] = (short)(c0 + lane);
                    n += __popc(m);
                }
                __syncwarp();
                // exact log-sum-exp combination: lane = (piece, head)
                float M[HG], l[HG];
#pragma unroll
                for (int h = 0; h < HG; ++h) { M[h] = M_INIT; l[h] = 0.f; }
                for (int k0 = 0; k0 < n; k0 += 32) {
#pragma unroll
                    for (int h = 0; h < HG; ++h) {
                        float2 ml = make_float2(M_INIT, 0.f);
                        if (k0 + lane < n) ml = *reinterpret_cast<const float2*>(part_ml + ((slot0 + piece_s[p][k0 + lane]) * HG + h) * 2);
                        float mx = ml.x;
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                        const float m_new = fmaxf(M[h], mx);
                        float sum = ex2(ml.x - m_new) * ml.y;
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                        l[h] = fmaf(l[h], ex2(M[h] - m_new), sum);
                        M[h] = m_new;
                        if (k0 + lane < n) scale_s[p][k0 + lane][h] = ml.x;
                    }
                }
                __syncwarp();
                for (int k = lane; k < n; k += 32)
#pragma unroll
                    for (int h = 0; h < HG; ++h) scale_s[p][k][h] = ex2(scale_s[p][k][h] - M[h]);
                if (lane == 0) {
#pragma unroll
                    for (int h = 0; h < HG; ++h) { m_s[p][h] = M[h]; l_s[p][h] = l[h]; }
                }
            } else if (lane < HG) {
                m_s[p][lane] = M_INIT; l_s[p][lane] = 0.f;
            }
            if (lane == 0) n_s[p] = n;
        }
        __syncthreads();
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (p >= np) break;
            const int b = b0 + p, n = n_s[p];
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int i = threadIdx.x + k * NT;
                if (i >= HG * D) break;
                const int h = i / D, c = i - h * D;
                float a = 0.f, M, lsum;
                if (RUNS) {
#pragma unroll 4
                    for (int j = 0; j < n; ++j)
                        a = fmaf(scale_s[p][j][h], part_acc[(((size_t)kvh * batch + b + piece_s[p][j]) * HG + h) * D + c], a);
                    M = m_s[p][h];
                    lsum = l_s[p][h];
                } else {
                    M = M_INIT;
                    lsum = 0.f;
                    for (int j = 0; j < n_cand; ++j)
                        if (cand_s[j]) M = fmaxf(M, ml_s[j][h].x);
                    for (int j = 0; j < n_cand; ++j) {
                        if (!cand_s[j]) continue;
                        const float sc = ex2(ml_s[j][h].x - M);
                        a = fmaf(sc, part_acc[(((size_t)kvh * batch + b + c_first + j) * HG + h) * D + c], a);
                        lsum = fmaf(sc, ml_s[j][h].y, lsum);
                    }
                }
                float lq = lsum;          // mass of the quantised tokens at the running scale
                float wb = 0.f;           // weight of the band accumulator at the running scale
                const int hq = kvh * HG + h;
                if (EXT && band_ml != nullptr) {
                    // BF16 sink-plus-recent band: one more partial, accumulated in the original value domain
                    const float mb = band_ml[((size_t)b * n_q_heads + hq) * 2], lb = band_ml[((size_t)b * n_q_heads + hq) * 2 + 1];
                    const float M2 = fmaxf(M, mb);
                    const float wq = ex2(M - M2);
                    wb = ex2(mb - M2);
                    a *= wq;
                    lq *= wq;
                    lsum = fmaf(lb, wb, lq);
                    M = M2;
                }
                if (EXT && sink_logits != nullptr) {
                    // learned sink: an extra logit in the normaliser, added exactly once, after the cross-split
                    // combine; it is shifted by the per-query constant the token logits dropped (q . k_mean)
                    const float s2 = sink_logits[hq] * 1.4426950408889634f - qk_off[(size_t)b * n_q_heads + hq];
                    const float M2 = fmaxf(M, s2);
                    const float w = ex2(M - M2);
                    a *= w;
                    lq *= w;
                    wb *= w;
                    lsum = fmaf(lsum, w, ex2(s2 - M2));
                }
                float val = 0.f, frac = 0.f, bsc = 0.f;
                if (lsum > 0.f) {
                    val = a / lsum;
                    if (EXT) { frac = lq / lsum; bsc = wb / lsum; }
                }
                if (EXT && c == 0) { frac_s[p][h] = frac; bsc_s[p][h] = bsc; }
                o_s[p][i] = val;
            }
        }
        __syncthreads();
        // o_h = o'_h rv^T + v_mean: threads = D outputs x PARTS column parts, all HG heads share each load
        for (int p = 0; p < np; ++p) {
            const int b = b0 + p;
            {
                const int r = threadIdx.x % D, part = threadIdx.x / D;
                float acc[HG];
#pragma unroll
                for (int h = 0; h < HG; ++h) acc[h] = 0.f;
                if (n_s[p] >= 0) {
#pragma unroll
                    for (int c = 0; c < COLS; ++c)
#pragma unroll
                        for (int h = 0; h < HG; ++h) acc[h] = fmaf(o_s[p][h * D + part * COLS + c], rv[c], acc[h]);
                }
#pragma unroll
                for (int h = 0; h < HG; ++h) red_s[part][h][r] = acc[h];
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int i = threadIdx.x + k * NT;
                if (i >= HG * D) break;
                const int h = i / D, r = i - h * D;
                float o = 0.f;
#pragma unroll
                for (int q = 0; q < PARTS; ++q) o += red_s[q][h][r];
                // sum_j p_j (s^_j R_V^T + v_mean): the mean carries the quantised-token mass (all of it without sink and band)
                if (EXT) o = fmaf(vm[k], frac_s[p][h], o);
                else if (n_s[p] >= 0) o += vm[k];
                const size_t oi = ((size_t)b * n_q_heads + kvh * HG + h) * D + r;
                if (EXT && band_acc != nullptr) o = fmaf(band_acc[oi], bsc_s[p][h], o);
                if (out_is_fp32) reinterpret_cast<float*>(out)[oi] = o;
                else reinterpret_cast<__nv_bfloat16*>(out)[oi] = __float2bfloat16_rn(o);
            }
            __syncthreads();
        }
    }
#ifdef NOVAKV_TIMING
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(g_m2));
    if (threadIdx.x == 0 && (blockIdx.x == 0 || blockIdx.x == gridDim.x - 1))
        printf("merge block %d | ns start %llu after-wait %llu end %llu\n", blockIdx.x, g_m0, g_m1, g_m2);
#endif
}

// ------------------------------------------------------------------------------------------------
// BF16 sink-plus-recent band: exact attention partial over the tokens that are not quantised
// ------------------------------------------------------------------------------------------------
// One CTA per (sequence, KV head), 8 warps.  A warp takes groups of 32 / Hg (at least 8) band tokens, one row per warp
// instruction, lanes hold D/32 dimensions, the next group's rows in flight; the group's Hg logits per token are reduced
// across the lanes by one transposing butterfly (31 shuffles for 32 logits; five per logit before), online softmax per
// warp, then a merge of the warps.  Output: (max, sum) and sum_j p_j v_j per query head, base-2 domain, unnormalised.
// Bound by memory latency: 64 sequences x 8 heads x 320 tokens, d = 128 (84 MB): 63 -> 30 us; two blocks an SM
// (128 registers) against one: 39 us.
// Band buffers: bf16 [batch][band_cap][Hkv][D]; of sequence b, slots 0 .. sink_cnt-1 hold the sink tokens
// and slots n_sink + (ring_start + i) % (band_cap - n_sink), i < ring_len, the recent tokens.
// The kernel reads nothing the scan writes: its blocks start as scan CTAs leave, and the dependency wait comes before the
// outputs (it is what orders the merge kernel behind the scan).
constexpr int BAND_WARPS = 8;
template <int N>
__device__ __forceinline__ void butterfly_halves(float (&v)[N], int s, int lane) {
    // lanes with bit s set keep the upper half, the others the lower half; the kept half receives the partner's share
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const bool up = (lane & s) != 0;
        const float send = up ? v[i] : v[i + N / 2];
        const float keep = up ? v[i + N / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
}
template <int D, int HG>
__global__ void __launch_bounds__(BAND_WARPS * 32, HG >= 4 ? 2 : 1)
novakv_band_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ band_k,
                   const __nv_bfloat16* __restrict__ band_v, int band_cap, int n_sink,
                   const int32_t* __restrict__ band_meta, int n_q_heads, int n_kv_heads, float scale_log2,
                   const float* __restrict__ k_mean, float* __restrict__ band_ml, float* __restrict__ band_acc) {
    constexpr int DPL = D / 32, WPL = DPL / 2;              // dimensions / 32-bit words of a row per lane
    constexpr int TG = HG >= 4 ? 8 : 32 / HG;               // tokens per group
    constexpr int NV = TG * HG, VPL = NV / 32;              // logits per group, of which a lane finishes VPL
    __shared__ float m_s[BAND_WARPS][HG], l_s[BAND_WARPS][HG];
    __shared__ float acc_s[BAND_WARPS][HG][D];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int b = blockIdx.x / n_kv_heads, kvh = blockIdx.x - b * n_kv_heads;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ring_cap = band_cap - n_sink;
    const int sink_cnt = min(max(band_meta[b * 3 + 0], 0), n_sink);
    const int ring_start = ring_cap > 0 ? max(band_meta[b * 3 + 1], 0) % ring_cap : 0;
    const int ring_len = ring_cap > 0 ? min(max(band_meta[b * 3 + 2], 0), ring_cap) : 0;
    const int n = sink_cnt + ring_len;
    float qr[HG][DPL];
#pragma unroll
    for (int h = 0; h < HG; ++h)
#pragma unroll
        for (int i = 0; i < DPL; ++i)
            qr[h][i] = __bfloat162float(q[((size_t)b * n_q_heads + kvh * HG + h) * D + lane * DPL + i]) * scale_log2;
    // the quantised tokens' logits omit the constant q . k_mean (Lemma S1): the band's logits must sit on the same scale,
    // so the same constant is subtracted; the lane finishes the logits with flat index lane * VPL + j = token * HG + head
    float zoff[VPL];
    {
        float z[HG];
#pragma unroll
        for (int h = 0; h < HG; ++h) {
            float t = 0.f;
#pragma unroll
            for (int i = 0; i < DPL; ++i) t = fmaf(qr[h][i], k_mean[(size_t)kvh * D + lane * DPL + i], t);
            z[h] = warp_sum_f(t);
        }
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            float v = z[0];
#pragma unroll
            for (int h = 1; h < HG; ++h) v = (lane * VPL + j) % HG == h ? z[h] : v;
            zoff[j] = v;
        }
    }
    const uint32_t* const kb = reinterpret_cast<const uint32_t*>(band_k) + (((size_t)b * band_cap * n_kv_heads + kvh) * D + lane * DPL) / 2;
    const uint32_t* const vb = reinterpret_cast<const uint32_t*>(band_v) + (((size_t)b * band_cap * n_kv_heads + kvh) * D + lane * DPL) / 2;
    const bool by8 = ((reinterpret_cast<uintptr_t>(band_k) | reinterpret_cast<uintptr_t>(band_v)) & 7) == 0;    // (4 is guaranteed)
    auto load_row = [&](const uint32_t* p, uint32_t (&w)[WPL]) {
        if (WPL == 2 && by8) {
            const uint2 x = *reinterpret_cast<const uint2*>(p);
            w[0] = x.x; w[WPL - 1] = x.y;
        } else {
            w[0] = p[0];
            if (WPL == 2) w[WPL - 1] = p[1];
        }
    };
    uint32_t kn[TG][WPL], vn[TG][WPL];
    auto load_group = [&](int i0) {
#pragma unroll
        for (int t = 0; t < TG; ++t) {
            const int i = min(i0 + t, n - 1);                // (a valid row; its weight is zeroed below)
            int r = ring_start + (i - sink_cnt);
            r = r >= ring_cap ? r - ring_cap : r;
            const size_t off = (size_t)(i < sink_cnt ? i : n_sink + r) * n_kv_heads * (D / 2);
            load_row(kb + off, kn[t]);
            load_row(vb + off, vn[t]);
        }
    };
    float m_run[VPL], l_run[VPL], acc[HG][DPL];
#pragma unroll
    for (int j = 0; j < VPL; ++j) { m_run[j] = M_INIT; l_run[j] = 0.f; }
#pragma unroll
    for (int h = 0; h < HG; ++h)
#pragma unroll
        for (int i = 0; i < DPL; ++i) acc[h][i] = 0.f;
    if (warp * TG < n) load_group(warp * TG);
    for (int i0 = warp * TG; i0 < n; i0 += BAND_WARPS * TG) {
        uint32_t kc[TG][WPL], vc[TG][WPL];
#pragma unroll
        for (int t = 0; t < TG; ++t)
#pragma unroll
            for (int w = 0; w < WPL; ++w) { kc[t][w] = kn[t][w]; vc[t][w] = vn[t][w]; }
        if (i0 + BAND_WARPS * TG < n) load_group(i0 + BAND_WARPS * TG);
        float z[NV];
#pragma unroll
        for (int t = 0; t < TG; ++t)
#pragma unroll
            for (int h = 0; h < HG; ++h) {
                float s = 0.f;
#pragma unroll
                for (int w = 0; w < WPL; ++w) {
                    s = fmaf(qr[h][2 * w], __uint_as_float(kc[t][w] << 16), s);
                    s = fmaf(qr[h][2 * w + 1], __uint_as_float(kc[t][w] & 0xffff0000u), s);
                }
                z[t * HG + h] = s;
            }
        butterfly_halves<NV>(z, 16, lane);
        butterfly_halves<NV / 2>(reinterpret_cast<float (&)[NV / 2]>(z), 8, lane);
        butterfly_halves<NV / 4>(reinterpret_cast<float (&)[NV / 4]>(z), 4, lane);
        butterfly_halves<NV / 8>(reinterpret_cast<float (&)[NV / 8]>(z), 2, lane);
        butterfly_halves<NV / 16>(reinterpret_cast<float (&)[NV / 16]>(z), 1, lane);
        // online softmax; the lanes that share a head differ in the lane bits above log2(HG / VPL)
        float p[VPL], alpha[VPL];
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            const float zz = i0 + (lane * VPL + j) / HG < n ? z[j] - zoff[j] : -CUDART_INF_F;
            float mx = zz;
#pragma unroll
            for (int s = HG / VPL; s < 32; s <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
            const float m_new = fmaxf(m_run[j], mx);
            alpha[j] = ex2(m_run[j] - m_new);
            m_run[j] = m_new;
            p[j] = ex2(zz - m_new);
            l_run[j] = fmaf(l_run[j], alpha[j], p[j]);
        }
#pragma unroll
        for (int h = 0; h < HG; ++h) {
            const float al = __shfl_sync(0xffffffffu, alpha[h % VPL], h / VPL);     // head h lives at flat index h (token 0)
#pragma unroll
            for (int i = 0; i < DPL; ++i) acc[h][i] *= al;
        }
#pragma unroll
        for (int t = 0; t < TG; ++t)
#pragma unroll
            for (int h = 0; h < HG; ++h) {
                const int flat = t * HG + h;
                const float ph = __shfl_sync(0xffffffffu, p[flat % VPL], flat / VPL);
#pragma unroll
                for (int w = 0; w < WPL; ++w) {
                    acc[h][2 * w] = fmaf(ph, __uint_as_float(vc[t][w] << 16), acc[h][2 * w]);
                    acc[h][2 * w + 1] = fmaf(ph, __uint_as_float(vc[t][w] & 0xffff0000u), acc[h][2 * w + 1]);
                }
            }
    }
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        float l = l_run[j];
#pragma unroll
        for (int s = HG / VPL; s < 32; s <<= 1) l += __shfl_xor_sync(0xffffffffu, l, s);
        const int flat = lane * VPL + j;
        if (flat < HG) { m_s[warp][flat] = m_run[j]; l_s[warp][flat] = l; }
    }
#pragma unroll
    for (int h = 0; h < HG; ++h)
#pragma unroll
        for (int i = 0; i < DPL; ++i) acc_s[warp][h][lane * DPL + i] = acc[h][i];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    for (int idx = threadIdx.x; idx < HG * D; idx += BAND_WARPS * 32) {
        const int h = idx / D, c = idx - h * D;
        float M = M_INIT;
#pragma unroll
        for (int w = 0; w < BAND_WARPS; ++w) M = fmaxf(M, m_s[w][h]);
        float a = 0.f, L = 0.f;
#pragma unroll
        for (int w = 0; w < BAND_WARPS; ++w) {
            const float sc = ex2(m_s[w][h] - M);
            a = fmaf(sc, acc_s[w][h][c], a);
            L = fmaf(sc, l_s[w][h], L);
        }
        const size_t o = (size_t)b * n_q_heads + kvh * HG + h;
        band_acc[o * D + c] = a;
        if (c == 0) { band_ml[o * 2] = M; band_ml[o * 2 + 1] = L; }
    }
}

// workspace layout
struct WsLayout {
    size_t qp, prefix, cost, range, qk, qc, cnt, bml, bacc, ml, acc, total;
};
WsLayout ws_layout(const novakv_ctx* ctx, int batch) {
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t d = ctx->cfg.head_dim, hq = ctx->cfg.n_q_heads;
    const size_t n_part = (size_t)batch * ctx->cfg.n_kv_heads + ctx->n_sm;
    WsLayout w;
    w.qp = 0;
    w.prefix = al(w.qp + (size_t)batch * hq * d * 4);
    w.cost = al(w.prefix + ((size_t)batch + 1) * 4);
    w.range = al(w.cost + ((size_t)batch + 1) * 4);
    w.qk = al(w.range + (size_t)ctx->n_sm * 2 * sizeof(long));
    w.qc = al(w.qk + (size_t)batch * hq * 4);
    w.cnt = al(w.qc + (size_t)batch * hq * 4);
    w.bml = al(w.cnt + (size_t)batch * ctx->cfg.n_kv_heads * 4);
    w.bacc = al(w.bml + (size_t)batch * hq * 2 * 4);
    w.ml = al(w.bacc + (size_t)batch * hq * d * 4);
    w.acc = al(w.ml + n_part * ctx->hg * 2 * 4);
    w.total = al(w.acc + n_part * ctx->hg * d * 4);
    return w;
}

template <int D, int HG, bool VM, bool KSC, bool VSQ>
novakv_status launch_decode_t(novakv_ctx* ctx, const novakv_layer& ly, const __nv_bfloat16* q,
                              const uint8_t* k_pages, const uint8_t* v_pages, const __nv_bfloat16* k_scales,
                              const __nv_bfloat16* v_meta, int n_pages,
                              const int32_t* page_table, int max_pages_per_seq, const int32_t* seq_lens,
                              int batch, float sm_scale, void* out, int out_is_fp32, void* workspace,
                              cudaStream_t stream, const float* sink_logits, const novakv_band_args* band) {
    using C = S1<D, HG, VM>;
    // with a BF16 band the index cache holds positions n_sink .. n_sink + seq_lens[b] - 1: the scan starts at
    // page column n_sink / 64 of every row
    const int pt_stride = max_pages_per_seq;
    if (band != nullptr) {
        const int shift = band->n_sink / NOVAKV_PAGE_TOKENS;
        page_table += shift;
        max_pages_per_seq -= shift;
    }
    const WsLayout w = ws_layout(ctx, batch);
    char* ws = (char*)workspace;
    float* qp = (float*)(ws + w.qp);
    int32_t* prefix = (int32_t*)(ws + w.prefix);
    int32_t* cost_prefix = (int32_t*)(ws + w.cost);
    long* cta_range = (long*)(ws + w.range);
    float* qk_off = sink_logits ? (float*)(ws + w.qk) : nullptr;
    float* qc = KSC ? (float*)(ws + w.qc) : nullptr;
    // what the token logits drop: q . k_mean, and for the unscaled key format also the share of the codebook
    // centres (k_mean_eff = k_mean + centre R_K^{-1}); with a per-token scale the centres are added back instead
    const float* k_off_vec = KSC ? ly.k_mean : ly.k_mean_eff;
    float* band_ml = band ? (float*)(ws + w.bml) : nullptr;
    float* band_acc = band ? (float*)(ws + w.bacc) : nullptr;
    float* part_ml = (float*)(ws + w.ml);
    float* part_acc = (float*)(ws + w.acc);
    int32_t* pair_count = (int32_t*)(ws + w.cnt);
    const int hq = ctx->cfg.n_q_heads, hkv = ctx->cfg.n_kv_heads;
    const int grid = ctx->scan_ctas > 0 ? (ctx->scan_ctas < ctx->n_sm ? ctx->scan_ctas : ctx->n_sm) : ctx->n_sm;
    if (grid > MAX_SCAN_CTAS) return NOVAKV_EUNSUPPORTED;
    // Optionally (novakv_debug_set_fused_merge), without a sink logit or a BF16 band, the scan kernel merges each
    // (sequence, KV head) pair itself (the CTA that writes the pair's last partial does it); otherwise the merge
    // kernel follows.
    const bool fuse = sink_logits == nullptr && band == nullptr && ctx->fused_merge;

    // (with the merge fused in, the outputs of empty sequences are written where the prefixes are formed)
    // Eight heads per KV head: only batches of one warp.  The append (d = 64, about 6 us) then ends before the queries are
    // transformed, and a block of the prepare kernel has formed the prefixes by the time the scan could (append + decode, a block
    // of the prepare kernel / the scan: 33 x 1000 32.7 / 33.2 us, 70 x 400 43.1 / 43.6, 128 x 1000 81.0 / 81.8; 5 x 100 17.0 / 16.5).
    const int scan_prefix = batch <= (HG == 8 ? 32 : PFX_CAP) && !fuse;
    // sequences per prepare block: one while all pairs fit on the machine twice over, then enough to make that so
    const int seqs_per_block = max(1, min(PREPARE_RUN, (batch * hkv + 2 * ctx->n_sm - 1) / (2 * ctx->n_sm)));
    auto prepare = seqs_per_block > 1 ? novakv_prepare_kernel<D, HG, true> : novakv_prepare_kernel<D, HG, false>;
    novakv_launch_pdl(prepare, dim3((batch + seqs_per_block - 1) / seqs_per_block * hkv + (scan_prefix ? 0 : 1)), dim3(512), 0, stream, q, ly.rk_inv_t, seq_lens,
                      batch, hq, hkv, max_pages_per_seq, sm_scale * 1.4426950408889634f, qp, prefix, ctx->dev_status,
                      k_off_vec, qk_off, cost_prefix, ctx->seg_weight, (const float*)ly.k_center, qc,
                      fuse ? pair_count : (int32_t*)nullptr, fuse ? out : (void*)nullptr, out_is_fp32, seqs_per_block, scan_prefix ? 0 : 1);
    ctx->launches++;

    // d = 64 with eight query heads per KV head, plain format: the kernel that takes the logits from tensor cores.  (At
    // d = 128 its two copies of the key codewords do not fit; with four heads a look-up in the table reads no more bytes than
    // a gather of a codeword; the scaled format has not been built with it.)  Not for short calls: its CTAs stage 192 KB of
    // codewords, which only pages pay back - 18 sequences of 100 tokens (2 pages an SM) 12.9 us with the table, 13.9 with
    // products; 1 of 5000 and 48 of 100 (4 and 5) within 3 % of each other; 8 of 2000 (14) 18.4 and 17.6.  The capacity stands
    // in for the lengths, which only the device knows.
    constexpr bool MMA = D == 64 && HG == 8 && VM && !KSC && !VSQ;
    if (MMA && !fuse && (long)batch * hkv * max_pages_per_seq >= (long)MMA_MIN_PAGES * ctx->n_sm) {
        constexpr unsigned mma_bit = 1u << 8;
        if (!(ctx->smem_opt_in & mma_bit)) {
            if (cudaFuncSetAttribute(novakv_decode_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, S1_SMEM_BYTES) != cudaSuccess) return NOVAKV_ECUDA;
            ctx->smem_opt_in |= mma_bit;
        }
        novakv_prof_scope ps(ctx, 0, stream);
        novakv_launch_pdl(novakv_decode_mma_kernel, dim3(grid), dim3(S1_THREADS), S1_SMEM_BYTES, stream, qp, (const uint4*)ly.cb_k_mma,
                          (const float*)ly.k_mma_scale, (const uint8_t*)ly.cb_v_u8, (const float*)ly.v_scale, (const float*)ly.v_off,
                          k_pages, v_pages, n_pages, page_table, max_pages_per_seq, seq_lens, prefix, batch, hq, hkv, part_ml, part_acc,
                          ctx->dev_status, pt_stride, cost_prefix, ctx->seg_weight, cta_range, scan_prefix);
        ps.end();
        ctx->launches++;
    } else {
        auto kern = novakv_decode_stage1_kernel<D, HG, VM, KSC, VSQ>;
        // the opt-in is per device and per kernel instantiation: remembered in the context (one device each)
        constexpr unsigned inst_bit = 1u << ((VM ? 1 : 0) + (KSC ? 2 : 0) + (VSQ ? 4 : 0));
        if (!(ctx->smem_opt_in & inst_bit)) {
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S1_SMEM_BYTES) != cudaSuccess) return NOVAKV_ECUDA;
            ctx->smem_opt_in |= inst_bit;
        }
        {
            novakv_prof_scope ps(ctx, 0, stream);
            novakv_launch_pdl(kern, dim3(grid), dim3(S1_THREADS), S1_SMEM_BYTES, stream, qp, ly.cb_k_lut,
                              (const uint8_t*)ly.cb_v_u8, (const float*)ly.v_scale,
                              (const float*)ly.v_off, k_pages, v_pages, k_scales, v_meta, n_pages, page_table, max_pages_per_seq,
                              seq_lens, prefix, batch, hq, hkv, part_ml, part_acc, ctx->dev_status, pt_stride,
                              cost_prefix, ctx->seg_weight, cta_range, (const float*)qc,
                              pair_count, (const float*)ly.rv_t, (const float*)ly.v_mean,
                              fuse ? out : (void*)nullptr, out_is_fp32, scan_prefix);
            ps.end();
            ctx->launches++;
        }
    }
    // (behind the scan, whose CTAs let it start when they have seen everything in front of this call complete)
    if (band != nullptr) {
        novakv_launch_pdl(novakv_band_kernel<D, HG>, dim3(batch * hkv), dim3(BAND_WARPS * 32), 0, stream, q, band->k, band->v,
                          band->cap, band->n_sink, band->meta, hq, hkv, sm_scale * 1.4426950408889634f, k_off_vec, band_ml,
                          band_acc);
        ctx->launches++;
    }
    if (fuse) return cudaGetLastError() == cudaSuccess ? NOVAKV_OK : NOVAKV_ECUDA;
    const bool ext = sink_logits != nullptr || band != nullptr;
    // (one block per SM, so that the slice of the transform stays in registers, and one wave of blocks where at most 8
    // sequences a block make that possible)
    constexpr bool NO_RUNS = HG == 8;
    const int one_wave = max(1, ctx->n_sm / hkv);
    int merge_run = NO_RUNS ? 1 : max(1, min(8, (batch + one_wave - 1) / one_wave));
    // Runs that would need a second pass of four sequences: two blocks an SM in 64 registers, half the run each (128
    // sequences, 8 heads, d = 128: whole call 284 -> 281 us; at 32 sequences, one pass either way, 80.4 against 80.7).
    const bool halves = merge_run > 4;
    if (halves) merge_run = max(4, min(8, (batch * hkv + 2 * ctx->n_sm - 1) / (2 * ctx->n_sm)));
    auto merge = ext ? novakv_decode_merge_kernel<D, HG, true, false, 1> : novakv_decode_merge_kernel<D, HG, false, false, 1>;
    if (halves)
        merge = ext ? novakv_decode_merge_kernel<D, HG, true, !NO_RUNS, 2> : novakv_decode_merge_kernel<D, HG, false, !NO_RUNS, 2>;
    else if (batch > one_wave)
        merge = ext ? novakv_decode_merge_kernel<D, HG, true, !NO_RUNS, NO_RUNS ? 2 : 1> : novakv_decode_merge_kernel<D, HG, false, !NO_RUNS, NO_RUNS ? 2 : 1>;
    novakv_launch_pdl(merge, dim3((batch + merge_run - 1) / merge_run * hkv), dim3(HG * D > 512 ? 512 : HG * D), 0, stream,
                      part_ml, part_acc, prefix, seq_lens, batch, hq, hkv, max_pages_per_seq, grid, ly.rv_t, ly.v_mean, out,
                      out_is_fp32, sink_logits, qk_off, (const float*)band_ml, (const float*)band_acc,
                      (const int32_t*)cost_prefix, ctx->seg_weight, (const long*)cta_range, merge_run);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? NOVAKV_OK : NOVAKV_ECUDA;
}

}  // namespace

size_t novakv_decode_ws_bytes(const novakv_ctx* ctx, int batch) { return ws_layout(ctx, batch).total; }

novakv_status novakv_launch_decode(novakv_ctx* ctx, const novakv_layer& ly, const __nv_bfloat16* q,
    const uint8_t* k_pages, const uint8_t* v_pages, int n_pages, const int32_t* page_table,
    int max_pages_per_seq, const int32_t* seq_lens, int batch, float sm_scale, void* out,
    int out_is_fp32, void* workspace, size_t workspace_bytes, cudaStream_t stream, const __nv_bfloat16* k_scales,
    const float* sink_logits, const novakv_band_args* band, const __nv_bfloat16* v_meta) {
    (void)workspace_bytes;
    const int d = ctx->cfg.head_dim, hg = ctx->hg;
    if (k_scales != nullptr && ctx->value_path == 0) return NOVAKV_EUNSUPPORTED;   // scaled keys: tensor-core value side only
    if (v_meta != nullptr && k_scales == nullptr) return NOVAKV_EUNSUPPORTED;      // INT2 values come with scaled keys (deployed format)
#define NOVAKV_DISPATCH(DD, HH)                                                                             \
    if (d == DD && hg == HH) {                                                                                   \
        if (v_meta != nullptr)                                                                                   \
            return launch_decode_t<DD, HH, true, true, true>(ctx, ly, q, k_pages, v_pages, k_scales, v_meta, n_pages, page_table, \
                                                  max_pages_per_seq, seq_lens, batch, sm_scale, out, out_is_fp32, \
                                                  workspace, stream, sink_logits, band);                         \
        if (k_scales != nullptr)                                                                                 \
            return launch_decode_t<DD, HH, true, true, false>(ctx, ly, q, k_pages, v_pages, k_scales, nullptr, n_pages, page_table, \
                                                  max_pages_per_seq, seq_lens, batch, sm_scale, out, out_is_fp32, \
                                                  workspace, stream, sink_logits, band);                               \
        if (ctx->value_path == 0)                                                                                \
            return launch_decode_t<DD, HH, false, false, false>(ctx, ly, q, k_pages, v_pages, nullptr, nullptr, n_pages, page_table, \
                                                  max_pages_per_seq, seq_lens, batch, sm_scale, out, out_is_fp32, \
                                                  workspace, stream, sink_logits, band);                               \
        return launch_decode_t<DD, HH, true, false, false>(ctx, ly, q, k_pages, v_pages, nullptr, nullptr, n_pages, page_table,  \
                                             max_pages_per_seq, seq_lens, batch, sm_scale, out, out_is_fp32,     \
                                             workspace, stream, sink_logits, band);                                    \
    }
    NOVAKV_DISPATCH(128, 1)
    NOVAKV_DISPATCH(128, 2)
    NOVAKV_DISPATCH(128, 4)
    NOVAKV_DISPATCH(64, 1)
    NOVAKV_DISPATCH(64, 2)
    NOVAKV_DISPATCH(64, 4)
    NOVAKV_DISPATCH(64, 8)
#undef NOVAKV_DISPATCH
    return NOVAKV_ESHAPE;
}
