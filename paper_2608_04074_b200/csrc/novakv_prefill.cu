// Write path for prompt-sized batches: transform and nearest-codeword search on the 5th-generation tensor cores.
//
// Work unit: 256 tokens of one (KV head, side) and 16 (or 8) groups; one persistent CTA per SM walks a contiguous run of
// units.  Per 128-token half tile (TMEM lane = token):
//   transform   D[128 x 64] = x R, three bfloat16 slices of the binary32 matrix R, binary32 accumulators in TMEM.  The
//               token's thread subtracts the mean's share m R and parks the coefficients in shared memory.
//   search      per group D[128 x 256] = |r - c|^2 / 2 for all codewords as ONE K = 16 product
//                   [rh rh rl 1 1 qh ql] . [-ch -cl -ch ph pl 1 1],   q = |r|^2 / 2, p = |c|^2 / 2,
//               (h, l: a binary16 number and its binary16 remainder), binary16 accumulators in TMEM; the thread takes the
//               minima of 32 rows of 8 codewords with packed three-input minima (a quarter instruction per codeword),
//               keeps every row that could hold the nearest codeword, and evaluates those rows - almost always one -
//               directly in binary32.
//   certificate the direct distances are trusted only where the two smallest are further apart than the error bounds of
//               coefficient and distance; every other (token, group) goes to one of two helper warps, which search it in
//               binary64 from the binary64 coefficient.  The stored index is the nearest codeword of the binary64
//               coefficient.
//
// Roles: four token warpgroups, two per half tile (thread = token, each takes half of the groups), whose first warp
// issues the search MMAs; one warp looks up destinations, copies token rows (TMA) and issues the transforms; one feeds the
// codebook rings; two search in binary64.  The round trip token warps -> MMA -> token warps takes some 400 cycles and more
// until the last warp is there, so the two warpgroups of a half tile take turns on its 256 columns: one reads all 256
// distances of a group in one go (the next 32 columns on their way while 32 are looked at) and then ranks, evaluates and
// stores while the other reads; each issues the other's MMA when it is done reading.  (One chunk of 128 columns for each
// warpgroup, two round trips a group: 522 us where this takes 505.)  Every wait is bounded (novakv_tcgen05.cuh): a wait that gives up sets NOVAKV_DEV_WAIT_TIMEOUT, and the CTA
// runs through the rest of its segment without waiting and leaves.  Three things hold on that way: the token warps take
// no destination that the flag has overtaken (tokens without one are neither stored nor looked at again), the named
// barriers among token warps and the waits for the search MMAs between them are never skipped (each of these MMAs is issued
// whatever has happened, so that they end; skipping one would let a warp overtake its warpgroup's barrier), and the
// tensor core and the copies are given time to finish before the CTA's memory goes away.
//
// What bounds it: instruction issue and latency of the selection, about 600 warp instructions per 32 tokens and group (of
// which 64 + 16 packed minima and comparisons on the half-rate pipe) with four token warps per scheduler; tensor pipe
// 16 %, issue slots 58 % busy.  The kernel lives at the limit of 96 registers: everything the rare paths need is
// formed there.  d = 128, 32768 tokens: 493 us a call in a stream of calls (binary32 search on the FMA pipe with a binary64 transform: 1971 us).
// Norms of the rows by the loading warp instead of the token warps: 528 us against 505 (the rows' way to the transform got longer).
// Measured on the way, with chunks: coefficients in TMEM and chunks of 64 codewords 945 us; releasing a chunk through an mbarrier
// instead of a hardware barrier +13 %; MMAs issued behind lane == 0 instead of elect.sync +40 cycles each; spills of 150
// bytes in the loop +15 %; one helper warp instead of two 665 us; direct distances one group late, to hide the round
// trip of the second chunk too: 635 us (longer register lifetimes cost more than the wait).
#include <cuda.h>
#include <math_constants.h>

#include <cmath>
#include <cstring>

#include "novakv_search.cuh"
#include "novakv_tcgen05.cuh"

namespace {

constexpr int PF_TOKEN_WARPS = 16;
constexpr int PF_HELPERS = 2;
constexpr int PF_THREADS = (PF_TOKEN_WARPS + 2 + PF_HELPERS) * 32;
constexpr int PF_TILE = 256;                 // tokens per unit: two half tiles
constexpr int PF_HALF = 128;
constexpr int PF_TOK_NS = 0, PF_AUX_NS = 200; // nanoseconds slept between tries of a wait: token warps, the others
constexpr int PF_OP_BYTES = 8192;            // a group's codebook as search operand
constexpr int PF_CW_BYTES = 4096;            // and in binary32
constexpr int PF_CW_STAGES = 6;              // (the binary32 codewords are needed one group longer than the operand)
static_assert(PF_OP_BYTES + PF_CW_BYTES == NOVAKV_PF_GROUP_BYTES, "codebook image");
constexpr int PF_QUEUE = 16;                 // entries of a helper's queue
constexpr int PF_QUEUE_LAST = 4;             // of which a segment's last tile fills so many (the CTA waits for what is queued at its end)
// Durations the work split reckons with, microseconds per unit: 18 to 19 for 16 groups of plain keys or values, about 26 for
// scaled keys, which transform and norm the whole row, 12 to 25 for INT2 values, whose unsure tokens take the binary64 row
// (32768 tokens, deployed / scaled: 464 / 634 us with 9 and 11 for the last two, 479 / 629 with 7 and 15, 462 / 617 so).
// Plain keys at d = 128 leave more to the helpers than values and take 7 % longer; the cut reckons with that where a CTA has
// enough units for it to matter (32768 tokens, 28 units a CTA: 505 -> 490 us).
constexpr double PF_KEYS = 1.07;
constexpr int PF_KEYS_UNITS = 8;
constexpr double PF_US_UNIT = 3.0, PF_US_GROUP = 1.0, PF_US_SCALED = 8.0, PF_US_INT2 = 13.0;
// |coefficient - binary64 coefficient| <= KAPPA (|x| + |mean|) |R column|.  The accumulation order of the tensor core is
// not specified; all-positive inputs (every truncation in the same direction) showed 2^-21.6, random signs 2^-23.3.
constexpr float KAPPA = 1.4e-6f;             // > 2^-19.5
// |D - |r - c|^2 / 2| <= EPS_S (|r| + |c|)^2: dropped rl.cl and remainders (3 2^-22 |r||c|) plus the accumulation
// (5.3e-7 of the largest term seen on random operands), with a factor of 4.
constexpr float EPS_S = 1.0e-6f;
constexpr float KEY_REL = 9.6e-7f;           // > 2^-20: the direct distances carry a codeword number in their low 3 bits

template <int D, int FMT>
struct PF {
    static constexpr int L = D / NOVAKV_G;
    static constexpr int KSTEPS = D / 16;
    static constexpr int GU = 16;                                 // groups of a unit, at most
    // a per-token scale needs the token's whole row: then all columns of R are resident, which leaves room for two slots
    static constexpr int R_COLS = FMT == 0 ? GU * NOVAKV_G : D;
    static constexpr int NX = D == 128 && FMT != 0 ? 2 : 3;
    static constexpr int NOP = D == 128 && FMT != 0 ? 3 : 4;      // stages of the operand ring
    static constexpr uint32_t R_SLICE = R_COLS * D * 2;
    static constexpr uint32_t R_IMG_SLICE = D * D * 2;
    static constexpr uint32_t X_BYTES = PF_HALF * D * 2;          // token rows of a half tile
    static constexpr uint32_t SLOT_BYTES = PF_HALF * GU * 16;     // the same memory later holds its coefficients [GU][128][4]
    static constexpr uint32_t A_BYTES = PF_HALF * 32;             // search operand of one group
    static constexpr int NCONST = NOVAKV_PF_CONSTS(D);            // mean share [D] | column norm [L] | scale [L] | 4 norms
    static constexpr uint32_t OFF_R = 0;
    static constexpr uint32_t OFF_X = OFF_R + 3 * R_SLICE;
    static constexpr uint32_t OFF_RING = OFF_X + NX * SLOT_BYTES;
    static constexpr uint32_t OFF_CW = OFF_RING + NOP * PF_OP_BYTES;
    static constexpr uint32_t OFF_A = OFF_CW + PF_CW_STAGES * PF_CW_BYTES;
    static constexpr uint32_t OFF_QUEUE = OFF_A + 4 * A_BYTES;
    static constexpr uint32_t OFF_PAGE = OFF_QUEUE + PF_HELPERS * PF_QUEUE * 16;  // int [NX][128], page of a token or -1
    static constexpr uint32_t OFF_TSLOT = OFF_PAGE + NX * PF_HALF * 4;            // uint8 [NX][128], its slot in the page
    static constexpr uint32_t OFF_CONST = OFF_TSLOT + NX * PF_HALF;
    static constexpr uint32_t OFF_BAR = OFF_CONST + ((NCONST * 4 + 15) & ~15);
    // ints: TMEM base, abort flag, finished token warps, -, queue counters [4], wait limit [2], -; unsure tokens [16]
    static constexpr uint32_t OFF_MISC = OFF_BAR + 288;
    static constexpr uint32_t BYTES = OFF_MISC + 128;
    static_assert(BYTES <= 232448, "shared memory budget");
    static_assert(X_BYTES <= SLOT_BYTES && R_SLICE % 1024 == 0 && SLOT_BYTES % 1024 == 0, "swizzled operands start on 1024 bytes");
};
// mbarriers
enum { B_R = 0, B_X = 1 /* +slot */, B_XFREE = 4 /* +slot */, B_T = 7 /* +half */, B_TFREE = 9 /* +half */, B_S = 11 /* +wg */,
       B_RING = 15 /* +stage */, B_RINGFREE = 19, B_CW = 23 /* +stage */, B_CWFREE = B_CW + PF_CW_STAGES,
       B_DRAIN = B_CW + 2 * PF_CW_STAGES, B_COUNT };
static_assert(B_COUNT * 8 <= 288, "barrier block");
// named barriers: 1 + wg among the four warps of a warpgroup, 5 + half among the eight of a half tile, 7 + wg: the other
// warpgroup of the half tile has read its distances, wg has written its operand
__device__ __forceinline__ void nbar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void nbar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

struct PrefillArgs {
    const __nv_bfloat16 *k_new, *v_new;
    const int32_t *tok_seq, *tok_pos;
    int n_tokens;
    const uint8_t* r_img;       // [2][Hkv][3 d d 2]
    const uint8_t* cb_img;      // [2][Hkv][L][stage]
    const float* consts;        // [2][Hkv][NCONST]
    const double *rk_d, *rv_d;  // [Hkv][L][d][4]
    const float *rk_rows, *rv_rows;   // [Hkv][d][d]
    const double *k_mean_d, *v_mean_d;
    const float *cb_k, *cb_v;   // [Hkv][L][256][4]
    uint8_t *k_pages, *v_pages;
    __nv_bfloat16 *k_scales, *v_meta;
    int n_pages;
    const int32_t* page_table;
    int max_pages_per_seq, n_seq;
    int32_t* seq_lens;
    int n_kv_heads;
    int gs;                     // parts a head's groups are cut into
    int cost_k, cost_v;         // relative cost of a key / value unit (the cut of the walk)
    int tma;                    // the token rows can be copied by the tensor maps (16-byte aligned)
    int words;                  // the pools can be written in words (4-byte aligned; single bytes otherwise)
    long wait_clocks;           // limit of a wait
    uint32_t* dev_status;
    CUtensorMap map_k, map_v;   // k_new / v_new as [n_tokens][Hkv d], boxes of 64 x 128
};

__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
__device__ __forceinline__ float2 unpack_half2(uint32_t h) { return __half22float2(*reinterpret_cast<const __half2*>(&h)); }
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float4 lds_f4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_f4(uint32_t addr, float4 v) {
    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ uint64_t dup2(float x) {
    uint64_t r;
    asm("mov.b64 %0, {%1,%1};" : "=l"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Binary32 codeword image of a group: rows of 8 codewords (128 bytes), a row as 4 codeword pairs of two 16-byte chunks:
// chunk 2 p + h of a row holds components 2 h, 2 h + 1 of its codewords 2 p, 2 p + 1, [c0.a c1.a c0.b c1.b].
__host__ __device__ __forceinline__ int codeword_offset(int code, int comp) {       // in floats
    return (code >> 3) * 32 + (((code & 7) >> 1) * 2 + (comp >> 1)) * 4 + (comp & 1) * 2 + (code & 1);
}

// Warp-cooperative exact search of one (token, group) among the rows of 8 codewords that its ranking has left (bit k:
// row 2 (k % 16) + k / 16): all lanes call it with the same arguments and get the same result.  rho > 0: the vector to
// encode is the binary32 quotient of the binary32 coefficient and rho (scaled key format).  Four rows at a time, lane =
// codeword; the smallest distance wins and, among equal distances, the lowest index.
// (It forms its pointers itself, so that the token warps keep none of them in registers.)
template <int D>
__device__ __noinline__ int exact_search_token(const PrefillArgs& a, int side, int kvh, int tkn, int l, float rho, uint32_t rows) {
    const int lane = threadIdx.x & 31;
    const __nv_bfloat16* x_row = (side == 0 ? a.k_new : a.v_new) + ((size_t)tkn * a.n_kv_heads + kvh) * D;
    const double* R = (side == 0 ? a.rk_d : a.rv_d) + (size_t)kvh * D * D + l * D * 4;
    const double* mean = (side == 0 ? a.k_mean_d : a.v_mean_d) + (size_t)kvh * D;
    const float4* cb = reinterpret_cast<const float4*>(side == 0 ? a.cb_k : a.cb_v) + ((size_t)kvh * (D / NOVAKV_G) + l) * NOVAKV_C;
    if (rows == 0u) rows = 0xffffffffu;                               // (the ranking was void)
    // this lane's codeword of the next four rows; -1 beyond the last
    auto next_code = [&]() {
        int code = -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = __ffs(rows) - 1;
            if (rows && (lane >> 3) == j) code = ((((k & 15) << 1) | (k >> 4)) << 3) | (lane & 7);
            rows &= rows - 1;
        }
        return code;
    };
    int code = next_code();
    float4 cw = cb[code < 0 ? 0 : code];                              // (requested before the coefficient is formed)
    double r[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) r[c] = 0.0;
#pragma unroll
    for (int j = 0; j < D / 32; ++j) {
        const int k = lane + 32 * j;
        const double xc = (double)__bfloat162float(x_row[k]) - mean[k];
        const double2 r01 = *reinterpret_cast<const double2*>(R + k * 4);
        const double2 r23 = *reinterpret_cast<const double2*>(R + k * 4 + 2);
        r[0] = fma(xc, r01.x, r[0]); r[1] = fma(xc, r01.y, r[1]);
        r[2] = fma(xc, r23.x, r[2]); r[3] = fma(xc, r23.y, r[3]);
    }
    {
        // sum over the lanes: lane bits 0 and 1 choose the component a lane goes on with, then every lane gets all four
        const double k0 = lane & 1 ? r[1] : r[0], s0 = lane & 1 ? r[0] : r[1], k1 = lane & 1 ? r[3] : r[2], s1 = lane & 1 ? r[2] : r[3];
        const double p0 = k0 + __shfl_xor_sync(0xffffffffu, s0, 1), p1 = k1 + __shfl_xor_sync(0xffffffffu, s1, 1);
        double p = (lane & 2 ? p1 : p0) + __shfl_xor_sync(0xffffffffu, lane & 2 ? p0 : p1, 2);
#pragma unroll
        for (int o = 4; o <= 16; o <<= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
#pragma unroll
        for (int c = 0; c < 4; ++c) r[c] = __shfl_sync(0xffffffffu, p, c);
    }
    if (rho > 0.f) {
#pragma unroll
        for (int c = 0; c < 4; ++c) r[c] = (double)__fdiv_rn((float)r[c], rho);
    }
    double best = CUDART_INF;
    int bi = 0x7fffffff;
    for (;;) {
        const double e0 = r[0] - (double)cw.x, e1 = r[1] - (double)cw.y, e2 = r[2] - (double)cw.z, e3 = r[3] - (double)cw.w;
        const double dd = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(e0, e0), __dmul_rn(e1, e1)), __dmul_rn(e2, e2)), __dmul_rn(e3, e3));
        if (code >= 0 && (dd < best || (dd == best && code < bi))) { best = dd; bi = code; }
        if (rows == 0u) break;
        code = next_code();
        cw = cb[code < 0 ? 0 : code];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob < best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    return bi == 0x7fffffff ? 0 : bi;                                 // (a coefficient that is not a number is nearest to none: index 0, as in
                                                                      // a scan with a strict '<')
}

// Whether any of the entries t0 .. t1 - 1 is used; a barrier of the whole CTA.
__device__ __forceinline__ bool any_used(const int32_t* tok_seq, int t0, int t1) {
    for (int t = t0; t < t1; t += PF_THREADS)
        if (__syncthreads_or(t + (int)threadIdx.x < t1 && tok_seq[t + threadIdx.x] != -1)) return true;
    return false;
}

// One token's coefficients in binary64, by the eight warps of a half tile: warp q sums an eighth of the input dimension
// into part_s[q][D]; after a barrier row_of() adds the parts.  Lane i holds columns D / 32 * i ...
template <int D>
__device__ __noinline__ void exact_row_part(const PrefillArgs& a, int side, int kvh, int tkn, int q, double* part_s) {
    constexpr int N = D / 32;
    const int lane = threadIdx.x & 31;
    const __nv_bfloat16* x_row = (side == 0 ? a.k_new : a.v_new) + ((size_t)tkn * a.n_kv_heads + kvh) * D + q * (D / 8);
    const float* R = (side == 0 ? a.rk_rows : a.rv_rows) + ((size_t)kvh * D + q * (D / 8)) * D + lane * N;
    const double* mean = (side == 0 ? a.k_mean_d : a.v_mean_d) + (size_t)kvh * D + q * (D / 8);
    double acc[N];
#pragma unroll
    for (int i = 0; i < N; ++i) acc[i] = 0.0;
    float rr[D / 8][N];
#pragma unroll
    for (int k = 0; k < D / 8; ++k) {
        if (N == 4) {
            const float4 v = *reinterpret_cast<const float4*>(R + k * D);
            rr[k][0] = v.x; rr[k][1] = v.y; rr[k][N - 2] = v.z; rr[k][N - 1] = v.w;
        } else {
            const float2 v = *reinterpret_cast<const float2*>(R + k * D);
            rr[k][0] = v.x; rr[k][1] = v.y;
        }
    }
#pragma unroll
    for (int k = 0; k < D / 8; ++k) {
        const double xc = (double)__bfloat162float(x_row[k]) - mean[k];
#pragma unroll
        for (int i = 0; i < N; ++i) acc[i] = fma(xc, (double)rr[k][i], acc[i]);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) part_s[q * D + lane * N + i] = acc[i];
}
template <int D>
__device__ __forceinline__ void row_of(const double* part_s, int lane, float (&r)[D / 32]) {
#pragma unroll
    for (int i = 0; i < D / 32; ++i) {
        double p[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) p[q] = part_s[q * D + lane * (D / 32) + i];
        r[i] = (float)(((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7])));
    }
}

// Stores the codes of groups l .. l + 3 of this lane's token (group l in the low byte); l a multiple of 4.
template <int L>
__device__ __forceinline__ void store_key_word(uint8_t* chunk, int slot, int l, uint32_t w) {
    const int x = slot & (l < 16 ? 7 : 15);
    const int jw = (l >> 2) ^ (x >> 2);
    *reinterpret_cast<uint32_t*>(chunk + ((((slot >> 5) * (L / 16) + (jw >> 2)) * 32 + (slot & 31)) * 16 + (jw & 3) * 4)) =
        __byte_perm(w, 0u, 0x3210u ^ ((x & 3) * 0x1111u));
}
// Values keep the codes of four tokens (4 apart) of one group in a word.  aligned: the warp's lanes are whole 16-token
// blocks in order, so that a 4 x 4 byte transpose among the lanes (4 apart) makes those words; otherwise single bytes.
template <int L>
__device__ __forceinline__ void store_value_word(uint8_t* chunk, int slot, int l, uint32_t w, bool aligned, bool valid, int lane) {
    if (aligned) {
        uint32_t t = __shfl_xor_sync(0xffffffffu, w, 8);
        w = __byte_perm(w, t, lane & 8 ? 0x3276u : 0x5410u);
        t = __shfl_xor_sync(0xffffffffu, w, 4);
        w = __byte_perm(w, t, lane & 4 ? 0x3715u : 0x6240u);
        const int gl = l + ((lane >> 2) & 3), fc = lane & 3;
        *reinterpret_cast<uint32_t*>(chunk + ((slot >> 4) * (L * 16) + ((gl & 7) * 4 + fc) * (L / 2) + ((gl >> 3) ^ (fc & 1)) * 4)) = w;
    } else if (valid) {
#pragma unroll
        for (int i = 0; i < 4; ++i) chunk[novakv_v_offset<L>(slot, l + i)] = (uint8_t)(w >> (8 * i));
    }
}

// FMT: 0 = 2-bit keys and values (vector quantised), 1 = keys with a per-token scale, 2 = those and scalar INT2 values.
// Per-token scale (keys): rho = bf16(sqrt(sum r^2 / d)) of the binary32 coefficients; it is taken from the tensor-core
// coefficients where no error within their bound can move the bfloat16 rounding, else from the binary64 row.
// INT2 values: zero, scale and the levels likewise; a token with any decision inside the bound takes the binary64 row.
template <int D, int FMT>
__global__ void __launch_bounds__(PF_THREADS, 1) novakv_prefill_kernel(const __grid_constant__ PrefillArgs a) {
    using P = PF<D, FMT>;
    constexpr int L = P::L;
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t sb = smem_u32(smem);
    if ((sb & 1023u) != 0u) {          // cannot happen without static shared memory; reported, never trapped
        if (threadIdx.x == 0) atomicOr(a.dev_status, NOVAKV_DEV_SMEM_LAYOUT);
        return;
    }
    novakv_grid_dependency_wait();      // (the launch overlaps the preceding kernel's tail, and the next kernel's launch this one's)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int* const misc = reinterpret_cast<volatile int*>(smem + P::OFF_MISC);
    volatile int* const abort_flag = misc + 1;
    int* const s_done = reinterpret_cast<int*>(smem + P::OFF_MISC) + 2;               // token warps that have finished the segment
    int* const s_count = reinterpret_cast<int*>(smem + P::OFF_MISC) + 4;              // [helper] entries in the queue
    int* const s_head = reinterpret_cast<int*>(smem + P::OFF_MISC) + 4 + PF_HELPERS;  // [helper] entries ever queued
    static_assert(4 + 2 * PF_HELPERS == 1 + MBAR_LIMIT, "the wait limit follows the queue counters");
    float* const cst = reinterpret_cast<float*>(smem + P::OFF_CONST);
    auto bar = [&](int i) -> uint32_t { return sb + P::OFF_BAR + i * 8; };

    // the walk: key units, then value units, cut evenly in cost
    const int n_tiles = (a.n_tokens + PF_TILE - 1) / PF_TILE;
    const int units_k = a.n_kv_heads * a.gs * n_tiles, gs_v = FMT == 2 ? 1 : a.gs, units_v = a.n_kv_heads * gs_v * n_tiles;
    auto first_unit = [&](int c) -> int {
        const long tk = (long)units_k * a.cost_k, t = (tk + (long)units_v * a.cost_v) * c / gridDim.x;
        return t < tk ? (int)(t / a.cost_k) : units_k + (int)((t - tk) / a.cost_v);
    };
    const int u_end = first_unit(blockIdx.x + 1);
    int u_next = first_unit(blockIdx.x);
    if (u_next >= u_end) return;
    // A CTA whose token entries are all unused (sequence -1) has nothing to do: rings of the BF16 band that flush nothing
    // send such lists (64 sequences x 8 entries, none used: 33 us without this).  The first entries decide for a prompt.
    {
        const int n = u_end - u_next, tile = (u_next < units_k ? u_next : u_next - units_k) % n_tiles;
        const bool whole = tile + n > n_tiles;                         // the walk goes on to another row of units
        if (!any_used(a.tok_seq, whole ? 0 : tile * PF_TILE, whole ? a.n_tokens : min(a.n_tokens, (tile + n) * PF_TILE))) return;
    }

    if (warp == 0) tmem_alloc<512>(sb + P::OFF_MISC);
    if (threadIdx.x == 0) {
        misc[1] = 0;
        *reinterpret_cast<volatile long long*>(abort_flag + MBAR_LIMIT) = a.wait_clocks;
#pragma unroll
        for (int h = 0; h < PF_HELPERS; ++h) { s_count[h] = 0; s_head[h] = 0; }
        mbar_init(bar(B_R), 1);
#pragma unroll
        for (int x = 0; x < P::NX; ++x) { mbar_init(bar(B_X + x), 2); mbar_init(bar(B_XFREE + x), 8); }
#pragma unroll
        for (int w = 0; w < 2; ++w) { mbar_init(bar(B_T + w), 1); mbar_init(bar(B_TFREE + w), 4); }
#pragma unroll
        for (int g = 0; g < 4; ++g) mbar_init(bar(B_S + g), 1);
#pragma unroll
        for (int s = 0; s < P::NOP; ++s) { mbar_init(bar(B_RING + s), 1); mbar_init(bar(B_RINGFREE + s), 2); }
#pragma unroll
        for (int s = 0; s < PF_CW_STAGES; ++s) { mbar_init(bar(B_CW + s), 1); mbar_init(bar(B_CWFREE + s), 8); }
        mbar_init(bar(B_DRAIN), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    for (int i = threadIdx.x; i < PF_HELPERS * PF_QUEUE; i += PF_THREADS) reinterpret_cast<uint4*>(smem + P::OFF_QUEUE)[i] = make_uint4(0, 0, 0, 0);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = (uint32_t)misc[0];

    // running phase counts of the barriers, over all segments
    int n_it = 0, n_use = 0, n_seg = 0;               // tiles; ring uses; segments
    uint32_t n_s = 0;                                 // token warps: groups seen
    int q_tail = 0;                                   // helpers: entries taken

    // ---- segments: units of one (KV head, side, part of the groups)
    while (u_next < u_end) {
        const bool is_v = u_next >= units_k;
        const int ul = is_v ? u_next - units_k : u_next, row_u = ul / n_tiles, tile0 = ul - row_u * n_tiles;
        const int gs = is_v ? gs_v : a.gs, kvh = row_u / gs, part = row_u - kvh * gs, side = is_v ? 1 : 0;
        const int n_local = min(n_tiles - tile0, (is_v ? u_end : min(u_end, units_k)) - u_next);
        const bool ksc = FMT >= 1 && side == 0, vsq = FMT == 2 && side == 1;
        const int ngh = vsq ? 0 : L / gs / 2;                              // groups a token warpgroup searches
        const int g0 = part * (L / gs);
        // columns of the transform: all of them where a token's whole row is needed
        const int c0 = ksc || vsq ? 0 : g0 * 4, nc = ksc || vsq ? D : L / gs * 4;
        u_next += n_local;
        const size_t sh = (size_t)side * a.n_kv_heads + kvh;
        auto chunk_of = [&](int page) -> uint8_t* {
            return (side == 0 ? a.k_pages : a.v_pages) + ((size_t)(page < 0 ? 0 : page) * a.n_kv_heads + kvh) * (NOVAKV_PAGE_TOKENS * L);
        };
        for (int i = threadIdx.x; i < P::NCONST; i += PF_THREADS) cst[i] = a.consts[sh * P::NCONST + i];
        if (threadIdx.x == 0) *s_done = 0;
        __syncthreads();

        if (warp == PF_TOKEN_WARPS) {
            // ---- token rows ([128][D] bfloat16 of a half tile, 128-byte rows per panel, 16-byte chunks swizzled by the
            //      row) and destinations, one half tile ahead of the transforms.  Half tile q of the CTA uses slot q % NX.
            const int q0 = 2 * n_it, q1 = q0 + 2 * n_local;
            int q_loaded = q0;
            bool ok = true;
            // destinations of half tile q's tokens (four per lane); its rows on their way into the L2
            int page[4], tslot[4];
            auto look_up = [&](int q) {
                const int t0 = tile0 * PF_TILE + (q - q0) * PF_HALF;
                if (a.tma && lane < D / 64 && t0 < a.n_tokens) tma_prefetch_2d(side == 0 ? &a.map_k : &a.map_v, kvh * D + lane * 64, t0);
                int sq[4], pos[4];
                bool named[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int tkn = t0 + lane + 32 * j;
                    sq[j] = -1; pos[j] = 0;
                    if (tkn < a.n_tokens) { sq[j] = a.tok_seq[tkn]; pos[j] = a.tok_pos[tkn]; }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    named[j] = sq[j] >= 0 && sq[j] < a.n_seq && pos[j] >= 0 && pos[j] / NOVAKV_PAGE_TOKENS < a.max_pages_per_seq;
                    page[j] = named[j] ? a.page_table[(size_t)sq[j] * a.max_pages_per_seq + pos[j] / NOVAKV_PAGE_TOKENS] : -1;
                    tslot[j] = pos[j] % NOVAKV_PAGE_TOKENS;
                    if (!named[j] && sq[j] != -1) atomicOr(a.dev_status, NOVAKV_DEV_BAD_TOKEN);   // (-1: unused entry, skipped)
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (named[j] && (page[j] < 0 || page[j] >= a.n_pages)) {
                        atomicOr(a.dev_status, NOVAKV_DEV_BAD_PAGE);
                        page[j] = -1;
                    } else if (named[j] && sh == 0 && g0 == 0) {
                        atomicMax(&a.seq_lens[sq[j]], pos[j] + 1);
                    }
                }
            };
            auto load_rows = [&](int q) {
                const int slot = q % P::NX;
                if (q >= P::NX) ok = mbar_wait<PF_AUX_NS>(bar(B_XFREE + slot), (q / P::NX - 1) & 1, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) { ok = false; return; }
                const int t0 = tile0 * PF_TILE + (q - q0) * PF_HALF;
                const uint32_t dst0 = sb + P::OFF_X + slot * P::SLOT_BYTES;
                if (a.tma) {
                    if (elect_one()) {
                        fence_proxy_async();                       // (the slot held coefficients written by threads)
                        mbar_expect_tx(bar(B_X + slot), P::X_BYTES);
#pragma unroll
                        for (int p = 0; p < D / 64; ++p)
                            tma_load_2d(dst0 + p * (PF_HALF * 128), side == 0 ? &a.map_k : &a.map_v, kvh * D + p * 64, t0, bar(B_X + slot));
                    }
                } else {
#pragma unroll 4
                    for (int e = lane; e < PF_HALF * (D / 2); e += 32) {        // 4-byte copies
                        const int t = e / (D / 2), c = e - t * (D / 2);
                        const uint32_t dst = dst0 + (c >> 5) * (PF_HALF * 128) + t * 128 + ((((c >> 2) & 7) ^ (t & 7)) * 16) + (c & 3) * 4;
                        const bool in = t0 + t < a.n_tokens;
                        const __nv_bfloat16* src = (side == 0 ? a.k_new : a.v_new) + ((size_t)(in ? t0 + t : 0) * a.n_kv_heads + kvh) * D + c * 2;
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
                    }
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    fence_proxy_async();
                    __syncwarp();
                    mbar_arrive_lane0(bar(B_X + slot), lane);
                }
                q_loaded = q + 1;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    reinterpret_cast<int*>(smem + P::OFF_PAGE)[slot * PF_HALF + lane + 32 * j] = page[j];
                    (smem + P::OFF_TSLOT)[slot * PF_HALF + lane + 32 * j] = (unsigned char)tslot[j];
                }
                __syncwarp();
                mbar_arrive_lane0(bar(B_X + slot), lane);
                __syncwarp();
            };
            look_up(q0);
            load_rows(q0);
            ok = __all_sync(0xffffffffu, ok && mbar_wait<PF_AUX_NS>(bar(B_R), n_seg & 1, abort_flag));
            const uint32_t id_t = umma_idesc(true, true, 128, 0) | ((uint32_t)(nc >> 3) << 17);
            for (int q = q0; q < q1 && ok; ++q) {
                const int w = q & 1, slot = q % P::NX;
                if (q + 1 < q1) look_up(q + 1);
                ok = mbar_wait<PF_AUX_NS>(bar(B_X + slot), (q / P::NX) & 1, abort_flag);
                if (q >= 2) ok = ok && mbar_wait<50>(bar(B_TFREE + w), ((q >> 1) - 1) & 1, abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    bool first = true;
                    // small slices first: their sums are added while the accumulator is small
#pragma unroll 1
                    for (int s = 2; s >= 0; --s)
#pragma unroll
                        for (int k = 0; k < P::KSTEPS; ++k) {
                            const uint32_t off = P::OFF_X + slot * P::SLOT_BYTES + (k >> 2) * (PF_HALF * 128) + (k & 3) * 32;
                            const uint32_t offr = P::OFF_R + s * P::R_SLICE + (k >> 2) * (P::R_COLS * 128) + (k & 3) * 32;
                            umma_f16(tmem + w * 256, umma_desc(sb + off, 16, 1024, 2), umma_desc(sb + offr, 16, 1024, 2), id_t, !first);
                            first = false;
                        }
                    umma_commit(bar(B_T + w));
                }
                __syncwarp();
                if (q + 1 < q1) load_rows(q + 1);
            }
            // (after a wait that gave up: the last copy must have landed before the CTA's memory goes away)
            if (q_loaded > q0) {
                int tries = 0;
                while (!mbar_try(bar(B_X + (q_loaded - 1) % P::NX), ((q_loaded - 1) / P::NX) & 1) && ++tries < 1000000) {}
            }
            n_it += n_local;
        } else if (warp == PF_TOKEN_WARPS + 1) {
            if (lane == 0) {
                // ---- the matrix slices (columns c0 .. c0 + nc - 1) once, then the codebook ring
                mbar_expect_tx(bar(B_R), 3 * (uint32_t)nc * D * 2);
#pragma unroll 1
                for (int s = 0; s < 3; ++s)
#pragma unroll 1
                    for (int p = 0; p < D / 64; ++p)
                        bulk_copy(sb + P::OFF_R + s * P::R_SLICE + p * (P::R_COLS * 128),
                                  a.r_img + sh * (3 * P::R_IMG_SLICE) + s * P::R_IMG_SLICE + p * (D * 128) + c0 * 128, (uint32_t)nc * 128, bar(B_R));
                const uint8_t* src = a.cb_img + (sh * L + g0) * NOVAKV_PF_GROUP_BYTES;
                const int n = n_local * 2 * ngh;
                bool ok = true;
                // use 2 g + h: group g of the half of the groups that warpgroups h take
                for (int j = 0, g = 0; j < n && ok; ++j, ++n_use) {
                    const int so = n_use % P::NOP, sc = n_use % PF_CW_STAGES;
                    const uint8_t* img = src + (size_t)((j & 1) * ngh + g) * NOVAKV_PF_GROUP_BYTES;
                    if (n_use >= P::NOP) ok = mbar_wait<PF_AUX_NS>(bar(B_RINGFREE + so), (n_use / P::NOP - 1) & 1, abort_flag);
                    if (!ok) break;
                    mbar_expect_tx(bar(B_RING + so), PF_OP_BYTES);
                    bulk_copy(sb + P::OFF_RING + so * PF_OP_BYTES, img, PF_OP_BYTES, bar(B_RING + so));
                    if (n_use >= PF_CW_STAGES) ok = mbar_wait<PF_AUX_NS>(bar(B_CWFREE + sc), (n_use / PF_CW_STAGES - 1) & 1, abort_flag);
                    if (!ok) { ++n_use; break; }
                    mbar_expect_tx(bar(B_CW + sc), PF_CW_BYTES);
                    bulk_copy(sb + P::OFF_CW + sc * PF_CW_BYTES, img + PF_OP_BYTES, PF_CW_BYTES, bar(B_CW + sc));
                    if (j & 1) g = g + 1 == ngh ? 0 : g + 1;
                }
                // no copy and no commit may be in flight when the segment (and the CTA's memory) goes away
                auto landed = [&](int b, int parity) {             // (after a wait that gave up, too)
                    int tries = 0;
                    while (!mbar_try(bar(b), parity) && ++tries < 1000000) {}
                };
                landed(B_R, n_seg & 1);
                for (int j = max(0, n_use - P::NOP); j < n_use; ++j) {
                    landed(B_RING + j % P::NOP, (j / P::NOP) & 1);
                    mbar_wait<PF_AUX_NS>(bar(B_RINGFREE + j % P::NOP), (j / P::NOP) & 1, abort_flag);
                }
                for (int j = max(0, n_use - PF_CW_STAGES); j < n_use - (ok ? 0 : 1); ++j) landed(B_CW + j % PF_CW_STAGES, (j / PF_CW_STAGES) & 1);
            }
            __syncwarp();
        } else if (warp > PF_TOKEN_WARPS + 1) {
            // ---- helpers: binary64 searches queued by the token warps
            const int h = warp - (PF_TOKEN_WARPS + 2);
            volatile uint32_t* const queue = reinterpret_cast<volatile uint32_t*>(smem + P::OFF_QUEUE) + h * PF_QUEUE * 4;
            for (;;) {
                const bool last = *reinterpret_cast<volatile int*>(s_done) == PF_TOKEN_WARPS;      // (read before the entry)
                volatile uint32_t* const e = queue + (q_tail % PF_QUEUE) * 4;
                const uint32_t tag = __shfl_sync(0xffffffffu, e[0], 0);
                if (tag == 0u) {
                    if (__all_sync(0xffffffffu, last || *abort_flag)) break;
                    __nanosleep(200);
                    continue;
                }
                // key scale (a bfloat16 number), a set bit, slot in the page, group | token | page | rows
                __threadfence_block();
                const int l = tag & 63, slot = (tag >> 6) & 63, tkn = (int)e[1], page = (int)e[2];
                const uint32_t rows = e[3];
                __syncwarp();
                if (lane == 0) {
                    e[0] = 0u;                                     // (the entry has been read: its place is free)
                    __threadfence_block();
                    atomicSub(&s_count[h], 1);
                }
                const int bi = exact_search_token<D>(a, side, kvh, tkn, l, __uint_as_float(tag & 0xffff0000u), rows);
                if (lane == 0) chunk_of(page)[side == 0 ? novakv_k_offset<L>(slot, l) : novakv_v_offset<L>(slot, l)] = (uint8_t)bi;
                __syncwarp();
                ++q_tail;
            }
        } else {
            // ---- token warps: thread = token; warpgroup wg = 2 * half tile + half of the groups
            const int wg = warp >> 2, w = wg >> 1, hf = wg & 1, row = threadIdx.x & (PF_HALF - 1);
            const uint32_t lane_base = (uint32_t)(warp & 3) << 21;
            const uint32_t d_t = tmem + w * 256 + lane_base, d_s = tmem + w * 256;
            const uint32_t a_s = sb + P::OFF_A + wg * P::A_BYTES;
            float* const x2_s = reinterpret_cast<float*>(smem + P::OFF_A);               // partial |x|^2, [wg][A_BYTES / 4]
            const float* const mr = cst;
            const int lx = lane & 7;
#pragma unroll 1
            for (int i = 0; i < n_local; ++i, ++n_it) {
                const int t0 = (tile0 + i) * PF_TILE + w * PF_HALF;            // first token of the half tile
                const int tw = t0 + (warp & 3) * 32;                           // first token of the warp
                const int tkn = t0 + row;
                const int q = 2 * n_it + w, xslot = q % P::NX;
                unsigned char* const x_s = smem + P::OFF_X + xslot * P::SLOT_BYTES;
                // |x| of the token; each warpgroup sums its half of the row
                mbar_wait<PF_TOK_NS>(bar(B_X + xslot), (q / P::NX) & 1, abort_flag);
                __syncwarp();
                // (the flag is read after the wait: while it is clear no wait of this thread was skipped, so this one counts)
                const int page = *abort_flag ? -1 : reinterpret_cast<const int*>(smem + P::OFF_PAGE)[xslot * PF_HALF + row];
                const int slot = (smem + P::OFF_TSLOT)[xslot * PF_HALF + row];
                const bool valid = page >= 0;
                {
                    float x2 = 0.f;
#pragma unroll
                    for (int cc = 0; cc < D / 16; ++cc) {
                        const int c = hf * (D / 16) + cc;
                        const uint4 v = *reinterpret_cast<const uint4*>(x_s + (c >> 3) * (PF_HALF * 128) + row * 128 + (((c & 7) ^ (row & 7)) * 16));
                        const uint32_t qv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float lo = __uint_as_float(qv[j] << 16), hi = __uint_as_float(qv[j] & 0xffff0000u);
                            x2 = fmaf(lo, lo, fmaf(hi, hi, x2));
                        }
                    }
                    x2_s[wg * (P::A_BYTES / 4) + row] = x2;
                }
                nbar_sync(5 + w, PF_TILE);                                     // the row has been read by everyone; partial sums visible
                float bound;                                                   // times a column norm: error of that coefficient
                {
                    const float x2 = x2_s[(2 * w) * (P::A_BYTES / 4) + row] + x2_s[(2 * w + 1) * (P::A_BYTES / 4) + row];
                    // (a sum of squares below 1e-30 may have lost terms to underflow: 1e-15 bounds |x| then)
                    bound = KAPPA * (sqrtf(fmaxf(x2, 1e-30f)) * 1.00001f + cst[D + 2 * L] /* |mean| */);
                }
                mbar_wait<PF_TOK_NS>(bar(B_T + w), n_it & 1, abort_flag);
                tc_fence_after();
                __syncwarp();

                // The tokens of the half tile whose decisions the tensor-core coefficients leave open get their coefficients
                // in binary64, one after the other by all eight warps (a warp alone took 18,000 cycles for one).  fn(lane of
                // the token, its row) runs in the two warps that own the token.
                auto exact_rows = [&](bool unsure, auto fn) {
                    volatile uint32_t* const masks = reinterpret_cast<volatile uint32_t*>(smem + P::OFF_MISC + 64) + w * 8;
                    double* const part_s = reinterpret_cast<double*>(smem + P::OFF_A + 2 * w * P::A_BYTES);
                    const unsigned mine = __ballot_sync(0xffffffffu, unsure);
                    if (lane == 0) masks[warp & 7] = mine;
                    nbar_sync(5 + w, PF_TILE);
#pragma unroll 1
                    for (int o = 0; o < 4; ++o) {
                        uint32_t todo = masks[o] | masks[o + 4];
                        while (todo) {
                            const int src = __ffs(todo) - 1;
                            todo &= todo - 1;
                            exact_row_part<D>(a, side, kvh, t0 + o * 32 + src, warp & 7, part_s);
                            nbar_sync(5 + w, PF_TILE);
                            if ((warp & 3) == o) {
                                float r[D / 32];
                                row_of<D>(part_s, lane, r);
                                fn(src, r);
                            }
                            nbar_sync(5 + w, PF_TILE);
                        }
                    }
                };
                float rho = 0.f, inv_rho = 1.f;
                if (ksc) {
                    float ss = 0.f;
#pragma unroll 1
                    for (int c = 0; c < D; c += 16) {
                        float f[16];
                        tmem_ld16(d_t + c, f);
                        tmem_wait_ld();
                        float s0 = 0.f, s1 = 0.f;
#pragma unroll
                        for (int j = 0; j < 16; j += 2) {
                            const float v0 = f[j] - mr[c + j], v1 = f[j + 1] - mr[c + j + 1];
                            s0 = fmaf(v0, v0, s0);
                            s1 = fmaf(v1, v1, s1);
                        }
                        ss += s0 + s1;
                    }
                    // relative error of the norm: that of the coefficients, their rounding, and the binary32 sum
                    const float nrm = sqrtf(ss), rel = bound * cst[D + 2 * L + 1] /* |R| */ / nrm + 4.0e-6f;
                    const float f = sqrtf(ss / (float)D);
                    rho = bf16_round(f);
                    const bool sure = bf16_round(f * (1.f - rel)) == rho && bf16_round(f * (1.f + rel)) == rho && rho > 0.f && rho < CUDART_INF_F;
                    exact_rows(valid && !sure, [&](int src, const float (&r)[D / 32]) {
                        double s2 = 0.0;
#pragma unroll
                        for (int j = 0; j < D / 32; ++j) s2 = fma((double)r[j], (double)r[j], s2);
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
                        float e = bf16_round((float)sqrt(s2 / (double)D));
                        if (!(e > 0.f) || !isfinite(e)) e = 1.f;
                        if (lane == src) rho = e;
                    });
                    if (!(rho > 0.f) || !isfinite(rho)) rho = 1.f;             // (lanes without a token)
                    inv_rho = __fdividef(1.f, rho);
                    bound *= inv_rho * 1.00001f;
                }
                // coefficients of this warpgroup's groups lb .. lb + ngh - 1 -> shared memory, [group][token][4]
                const int lb = g0 + hf * ngh;
                const uint32_t c_s = sb + P::OFF_X + xslot * P::SLOT_BYTES + (hf * (P::GU / 2) * PF_HALF + row) * 16;
#pragma unroll 1
                for (int g = 0; g < ngh; g += 4) {
                    float f[16];
                    tmem_ld16(d_t + 4 * (lb + g) - c0, f);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float4 m = *reinterpret_cast<const float4*>(mr + 4 * (lb + g + j));
                        float4 r = make_float4(f[4 * j] - m.x, f[4 * j + 1] - m.y, f[4 * j + 2] - m.z, f[4 * j + 3] - m.w);
                        if (ksc) { r.x *= inv_rho; r.y *= inv_rho; r.z *= inv_rho; r.w *= inv_rho; }
                        sts_f4(c_s + (g + j) * (PF_HALF * 16), r);
                    }
                }
                const int page0 = __shfl_sync(0xffffffffu, page, lane & 16), slot0 = __shfl_sync(0xffffffffu, slot, lane & 16);
                const bool aligned = a.words && __all_sync(0xffffffffu, valid && page == page0 && (slot & 15) == (lane & 15) && (slot ^ slot0) < 16);
                if (ksc && valid && g0 == 0 && hf == 0)
                    a.k_scales[((size_t)page * a.n_kv_heads + kvh) * NOVAKV_PAGE_TOKENS + slot] = __float2bfloat16_rn(rho);
                if (vsq) {
                    float mn = CUDART_INF_F, mx = -CUDART_INF_F;
#pragma unroll 1
                    for (int c = 0; c < D; c += 16) {
                        float f[16];
                        tmem_ld16(d_t + c, f);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const float v = f[j] - mr[c + j];
                            mn = fminf(mn, v);
                            mx = fmaxf(mx, v);
                        }
                    }
                    const float err = bound * cst[D + 2 * L + 2] /* longest column */ + 1.2e-7f * fmaxf(fabsf(mn), fabsf(mx));
                    float zero = bf16_round(mn);
                    float scale = bf16_round(__fdiv_rn(__fsub_rn(mx, zero), 3.0f));
                    bool sure = bf16_round(mn - err) == zero && bf16_round(mn + err) == zero &&
                                bf16_round(((mx - err) - zero) * 0.33333328f) == scale && bf16_round(((mx + err) - zero) * 0.33333339f) == scale &&
                                scale > 0.f && scale < CUDART_INF_F;
                    const float inv_scale = __fdividef(1.f, scale), uerr = err * inv_scale + 2.0e-6f;
                    uint32_t word[L / 8];                                      // this warpgroup's half of the levels
#pragma unroll
                    for (int qw = 0; qw < L / 8; ++qw) {
                        const int c = hf * (D / 2) + qw * 16;
                        float f[16];
                        tmem_ld16(d_t + c, f);
                        tmem_wait_ld();
                        uint32_t wd = 0;
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            // level = clamp(rint(t), 0, 3); t near a boundary 0.5, 1.5, 2.5 is inside the bound
                            const float t = (f[j] - mr[c + j] - zero) * inv_scale;
                            const float lv = fminf(fmaxf(rintf(t), 0.f), 3.f);
                            sure &= fminf(fminf(fabsf(t - 0.5f), fabsf(t - 1.5f)), fabsf(t - 2.5f)) > uerr;
                            wd |= (uint32_t)lv << (2 * j);
                        }
                        word[qw] = wd;
                    }
                    tc_fence_before();
                    exact_rows(valid && !sure, [&](int src, const float (&r)[D / 32]) {
                        float rmn = r[0], rmx = r[0];
#pragma unroll
                        for (int j = 1; j < D / 32; ++j) { rmn = fminf(rmn, r[j]); rmx = fmaxf(rmx, r[j]); }
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) {
                            rmn = fminf(rmn, __shfl_xor_sync(0xffffffffu, rmn, o));
                            rmx = fmaxf(rmx, __shfl_xor_sync(0xffffffffu, rmx, o));
                        }
                        const float ez = bf16_round(rmn);
                        float es = bf16_round(__fdiv_rn(__fsub_rn(rmx, ez), 3.0f));
                        if (!(es > 0.f) || !isfinite(es)) es = 1.f;
                        uint32_t mine = 0;                                     // this lane's D / 32 levels, 2 bits each
#pragma unroll
                        for (int j = 0; j < D / 32; ++j) {
                            float t = rintf(__fdiv_rn(__fsub_rn(r[j], ez), es));
                            if (!(t > 0.f)) t = 0.f;
                            mine |= (uint32_t)fminf(t, 3.f) << (2 * j);
                        }
#pragma unroll
                        for (int qw = 0; qw < L / 8; ++qw) {                   // 16 levels per word: 512 / D lanes each
                            uint32_t wd = 0;
#pragma unroll
                            for (int j = 0; j < 512 / D; ++j)
                                wd |= __shfl_sync(0xffffffffu, mine, hf * 16 + qw * (512 / D) + j) << (j * (D / 16));
                            if (lane == src) word[qw] = wd;
                        }
                        if (lane == src) { zero = ez; scale = es; }
                    });
                    // (a barrier has passed: the accumulators are read out, the row slot is free)
                    if (lane == 0) {
                        mbar_arrive(bar(B_XFREE + xslot));
                        if (hf == 0) mbar_arrive(bar(B_TFREE + w));
                    }
#pragma unroll
                    for (int qw = 0; qw < L / 8; ++qw) store_value_word<L>(chunk_of(page), slot, hf * (L / 2) + 4 * qw, word[qw], aligned, valid, lane);
                    if (valid && hf == 0)
                        reinterpret_cast<__nv_bfloat162*>(a.v_meta)[((size_t)page * a.n_kv_heads + kvh) * NOVAKV_PAGE_TOKENS + slot] =
                            __floats2bfloat162_rn(scale, zero);
                    continue;
                }
                tc_fence_before();
                nbar_sync(5 + w, PF_TILE);                                     // the transform's accumulators are read out

                // ---- search of groups lb .. lb + ngh - 1
                const int use0 = n_use + hf;
                // the search operand of group g into shared memory
                auto publish = [&](int g) {
                    const float4 r = lds_f4(c_s + g * (PF_HALF * 16));
                    const float sc = cst[D + L + lb + g];
                    const float s0 = r.x * sc, s1 = r.y * sc, s2 = r.z * sc, s3 = r.w * sc;
                    const float qq = fmaf(s0, s0, fmaf(s1, s1, fmaf(s2, s2, s3 * s3)));
                    const uint32_t h01 = pack_half2(s0, s1), h23 = pack_half2(s2, s3);
                    const float2 f01 = unpack_half2(h01), f23 = unpack_half2(h23);
                    const uint32_t l01 = pack_half2(s0 - f01.x, s1 - f01.y), l23 = pack_half2(s2 - f23.x, s3 - f23.y);
                    const float qh = 0.5f * qq, qhh = __half2float(__float2half_rn(qh));
                    const uint32_t qp = pack_half2(qhh, qh - qhh);
                    const uint32_t dst = a_s + row * 16;
                    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%1,%2};" ::"r"(dst), "r"(h01), "r"(h23) : "memory");
                    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst + PF_HALF * 16), "r"(l01), "r"(l23), "r"(0x3c003c00u), "r"(qp) : "memory");
                    fence_proxy_async();
                };
                // The two warpgroups of a half tile take turns on its 256 columns.  Group g of warpgroup x (distances to all
                // 256 codewords, one MMA) is issued by x's partner, when the partner's four warps have read their own
                // distances out of the columns and x's four warps have written the operand: x works on its previous group
                // meanwhile, so that neither waits for the round trip.
                auto issue = [&](int x, int g) {
                    const int use = n_use + (x & 1) + 2 * g, st = use % P::NOP;
                    tc_fence_after();
                    if (elect_one()) {
                        umma_f16(d_s, umma_desc(sb + P::OFF_A + x * P::A_BYTES, PF_HALF * 16, 128, 0),
                                 umma_desc(sb + P::OFF_RING + st * PF_OP_BYTES, 4096, 128, 0), umma_idesc(false, false, 128, 256), false);
                        umma_commit(bar(B_S + x));
                        umma_commit(bar(B_RINGFREE + st));
                    }
                    __syncwarp();
                };
                auto ring_wait = [&](int x, int g) {
                    const int use = n_use + (x & 1) + 2 * g;
                    mbar_wait<PF_TOK_NS>(bar(B_RING + use % P::NOP), (use / P::NOP) & 1, abort_flag);
                };
                // this warpgroup has read the columns: the partner's group g is next
                auto hand_over = [&](int g) {
                    tc_fence_before();
                    if ((warp & 3) != 0) {
                        nbar_arrive(7 + (wg ^ 1), PF_TILE);
                    } else {
                        ring_wait(wg ^ 1, g);
                        nbar_sync(7 + (wg ^ 1), PF_TILE);
                        issue(wg ^ 1, g);
                    }
                };
                // minima of 32 rows of 8 codewords, two rows per register.  (Distances are not negative, or tiny: their
                // binary16 patterns compare like integers.  A negative one sorts below every positive one, and every negative
                // row minimum passes the test below.)
                uint32_t rmin[16];
                auto minima = [&](int c, const uint32_t (&v)[16]) {
#pragma unroll
                    for (int qd = 0; qd < 2; ++qd)
                        rmin[2 * c + qd] = __vimin3_s16x2(__vimin3_s16x2(v[8 * qd], v[8 * qd + 1], v[8 * qd + 2]),
                                                          __vimin3_s16x2(v[8 * qd + 3], v[8 * qd + 4], v[8 * qd + 5]),
                                                          __vmins2(v[8 * qd + 6], v[8 * qd + 7]));
                };
                auto accumulators = [&](int c, uint32_t (&v)[16]) { tmem_ld32_h2(d_s + lane_base + c * 32, v); };
                publish(0);
                if (hf == 1) {
                    nbar_arrive(7 + wg, PF_TILE);
                } else if ((warp & 3) != 0) {
                    nbar_arrive(1 + wg, PF_HALF);
                } else {
                    ring_wait(wg, 0);
                    nbar_sync(1 + wg, PF_HALF);
                    issue(wg, 0);
                }
                uint32_t codes = 0, pend = 0;
#pragma unroll 1
                for (int g = 0; g < ngh; ++g) {
                    {
                        mbar_wait_mma(bar(B_S + wg), n_s & 1, abort_flag);
                        ++n_s;
                        tc_fence_after();
                        __syncwarp();
                        {
                            uint32_t v0[16], v1[16];                           // one half on its way while the other is looked at
                            accumulators(0, v0);
#pragma unroll
                            for (int c = 0; c < 8; c += 2) {
                                tmem_wait_ld16(v0);
                                accumulators(c + 1, v1);
                                minima(c, v0);
                                tmem_wait_ld16(v1);
                                if (c + 2 < 8) accumulators(c + 2, v0);
                                else if (g + hf < ngh) hand_over(g + hf);
                                else {                                         // (the second warpgroup is the last to read)
                                    tc_fence_before();
                                    __syncwarp();
                                    if (lane == 0) mbar_arrive(bar(B_TFREE + w));
                                }
                                minima(c + 1, v1);
                            }
                        }
                        if (g + 1 < ngh) {
                            publish(g + 1);
                            nbar_arrive(7 + wg, PF_TILE);
                        }
                        float mf;
                        {
                            uint32_t m = __vimin3_s16x2(__vimin3_s16x2(rmin[0], rmin[1], rmin[2]), __vimin3_s16x2(rmin[3], rmin[4], rmin[5]),
                                                        __vimin3_s16x2(rmin[6], rmin[7], rmin[8]));
                            m = __vimin3_s16x2(m, __vimin3_s16x2(rmin[9], rmin[10], rmin[11]), __vimin3_s16x2(rmin[12], rmin[13], rmin[14]));
                            const float2 f = unpack_half2(__vmins2(m, rmin[15]));
                            mf = fminf(f.x, f.y);
                            if (!(f.x == f.x) || !(f.y == f.y)) mf = CUDART_INF_F;
                        }
                        // A row can hold the nearest codeword only if its binary16 minimum is at most t: the rounding of two
                        // binary16 numbers (2^-11 each; below their normal range 2^-25, also of the operands), the error of the
                        // product (EPS_S) for both, and what the error of the coefficient moves the difference of two distances by.
                        const float4 r = lds_f4(c_s + g * (PF_HALF * 16));
                        if (g + 1 == ngh) {
                            __syncwarp();
                            mbar_arrive_lane0(bar(B_XFREE + xslot), lane);  // the coefficients are read out
                        }
                        const float rlen2 = fmaf(r.x, r.x, fmaf(r.y, r.y, fmaf(r.z, r.z, r.w * r.w)));
                        const float delta = fmaf(bound, cst[D + lb + g], (ksc ? 3.0e-7f : 6.0e-8f) * sqrt_approx(rlen2));
                        const float sc = cst[D + L + lb + g], dl = delta * sc, sq2 = sqrt_approx(2.f * fmaxf(mf, 0.f));
                        const float s2 = fmaf(1.1f, sq2, 2.f * sqrt_approx(fmaf(r.x * sc, r.x * sc, fmaf(r.y * sc, r.y * sc, fmaf(r.z * sc, r.z * sc, (r.w * sc) * (r.w * sc))))));
                        float t = fmaf(2.1f * EPS_S, s2 * s2, fmaf(fmaxf(mf, 0.f), 1.0025f, 2.5f * dl * (sq2 + dl) + 4.0e-7f));
                        t *= 1.0005f;
                        const uint32_t t1 = pack_half2(t, t);
                        uint32_t bits = 0;
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const uint32_t le = __hle2_mask(*reinterpret_cast<const __half2*>(&rmin[k]), *reinterpret_cast<const __half2*>(&t1));
                            bits |= le & (0x00010001u << k);
                        }
                        bool exact = !(mf < 60000.f) || bits == 0u;
                        // Direct binary32 distances of the rows that are left, two codewords per operation.  A lane reads
                        // the 8 chunks of its row in the order j ^ (lane % 8), so that the 8 lanes of a quarter warp read 8
                        // different 16-byte columns: odd lanes meet the chunk of components 2, 3 first.  The low 3 bits of a
                        // distance are replaced by the codeword's number in the row.
                        const int l = lb + g, use = use0 + 2 * g, st = use % PF_CW_STAGES;
                        const uint32_t rows = exact ? 0u : bits;               // (a void ranking leaves every row)
                        uint32_t best = 0x7f800000u, second = 0x7f800000u;
                        int brow = 0;
                        mbar_wait<PF_TOK_NS>(bar(B_CW + st), (use / PF_CW_STAGES) & 1, abort_flag);
                        __syncwarp();
                        const uint32_t cb = sb + P::OFF_CW + st * PF_CW_BYTES;
                        {
                            const bool odd = lane & 1;
                            const uint64_t ra0 = dup2(odd ? r.z : r.x), ra1 = dup2(odd ? r.w : r.y);
                            const uint64_t rb0 = dup2(odd ? r.x : r.z), rb1 = dup2(odd ? r.y : r.w);
                            do {
                                const int k = bits ? __ffs(bits) - 1 : 0;
                                const bool take = bits != 0u;
                                const int rowi = ((k & 15) << 1) | (k >> 4);
                                const uint32_t base = cb + rowi * 128;
                                uint32_t key[8];
#pragma unroll
                                for (int p = 0; p < 4; ++p) {
                                    uint64_t a0, a1, b0, b1;
                                    asm volatile("ld.shared.v2.u64 {%0,%1}, [%2];" : "=l"(a0), "=l"(a1) : "r"(base + (((2 * p) ^ lx) * 16)));
                                    asm volatile("ld.shared.v2.u64 {%0,%1}, [%2];" : "=l"(b0), "=l"(b1) : "r"(base + (((2 * p + 1) ^ lx) * 16)));
                                    a0 = f2_sub(ra0, a0); a1 = f2_sub(ra1, a1); b0 = f2_sub(rb0, b0); b1 = f2_sub(rb1, b1);
                                    const uint64_t d = f2_fma(b1, b1, f2_fma(b0, b0, f2_fma(a1, a1, f2_mul(a0, a0))));
                                    key[2 * p] = ((uint32_t)d & ~7u) | (2 * p);
                                    key[2 * p + 1] = ((uint32_t)(d >> 32) & ~7u) | (2 * p + 1);
                                }
                                // two smallest of the 8: pairs, then merges
                                uint32_t lo[4], hi[4];
#pragma unroll
                                for (int p = 0; p < 4; ++p) { lo[p] = min(key[2 * p], key[2 * p + 1]); hi[p] = max(key[2 * p], key[2 * p + 1]); }
#pragma unroll
                                for (int p = 0; p < 4; p += 2) {
                                    hi[p] = __vimin3_u32(max(lo[p], lo[p + 1]), hi[p], hi[p + 1]);
                                    lo[p] = min(lo[p], lo[p + 1]);
                                }
                                hi[0] = __vimin3_u32(max(lo[0], lo[2]), hi[0], hi[2]);
                                lo[0] = min(lo[0], lo[2]);
                                if (take) {
                                    second = __vimin3_u32(max(best, lo[0]), second, hi[0]);
                                    if (lo[0] < best) { best = lo[0]; brow = rowi; }
                                }
                                bits &= bits - 1;
                            } while (__any_sync(0xffffffffu, bits != 0u));
                        }
                        __syncwarp();
                        mbar_arrive_lane0(bar(B_CWFREE + st), lane);
                        const int bi = brow * 8 + (int)((best & 7u) ^ (lx & 6));
                        // where the two nearest codewords are closer than the errors can resolve, the search is repeated in binary64
                        exact |= needs_exact_search(__uint_as_float(best & ~7u), __uint_as_float(second | 7u), delta, KEY_REL);
                        unsigned todo = __ballot_sync(0xffffffffu, exact && valid);
                        if (todo) {
                            // to the helper's queue, or here when that is full
                            const int h = warp & (PF_HELPERS - 1), n = __popc(todo);
                            int base = -1;
                            if (lane == 0) {
                                if (atomicAdd(&s_count[h], n) + n <= (i + 1 < n_local ? PF_QUEUE : PF_QUEUE_LAST)) base = atomicAdd(&s_head[h], n);
                                else atomicSub(&s_count[h], n);
                            }
                            base = __shfl_sync(0xffffffffu, base, 0);
                            if (base >= 0) {
                                if ((todo >> lane) & 1u) {
                                    volatile uint32_t* e = reinterpret_cast<volatile uint32_t*>(smem + P::OFF_QUEUE) +
                                                           (h * PF_QUEUE + (base + __popc(todo & ((1u << lane) - 1))) % PF_QUEUE) * 4;
                                    e[1] = (uint32_t)tkn; e[2] = (uint32_t)page; e[3] = rows;
                                    __threadfence_block();
                                    e[0] = (__float_as_uint(rho) & 0xffff0000u) | 0x8000u | ((uint32_t)slot << 6) | (uint32_t)l;
                                }
                            } else {
                                while (todo) {
                                    const int src = __ffs(todo) - 1;
                                    todo &= todo - 1;
                                    const int res = exact_search_token<D>(a, side, kvh, tw + src, l, __shfl_sync(0xffffffffu, rho, src),
                                                                          __shfl_sync(0xffffffffu, rows, src));
                                    if (lane == src) chunk_of(page)[side == 0 ? novakv_k_offset<L>(slot, l) : novakv_v_offset<L>(slot, l)] = (uint8_t)res;
                                }
                            }
                        }
                        codes = (codes >> 8) | ((uint32_t)bi << 24);
                        pend = (pend >> 1) | (exact && valid ? 8u : 0u);
                        if ((l & 3) == 3) {
                            if (__any_sync(0xffffffffu, pend != 0u) || !a.words) {
                                // single bytes: those that are searched again are written by the search alone
                                if (valid) {
#pragma unroll
                                    for (int k = 0; k < 4; ++k)
                                        if (!((pend >> k) & 1u))
                                            chunk_of(page)[side == 0 ? novakv_k_offset<L>(slot, l - 3 + k) : novakv_v_offset<L>(slot, l - 3 + k)] =
                                                (uint8_t)(codes >> (8 * k));
                                }
                            } else if (side == 0) {
                                if (valid) store_key_word<L>(chunk_of(page), slot, l - 3, codes);
                            } else {
                                store_value_word<L>(chunk_of(page), slot, l - 3, codes, aligned, valid, lane);
                            }
                        }
                    }
                }
                n_use += 2 * ngh;
            }
            __syncwarp();
            if (lane == 0) { __threadfence_block(); atomicAdd(s_done, 1); }
        }
        ++n_seg;
        tc_fence_before();
        __syncthreads();                               // constants, matrix slices and TMEM are free for the next segment
        tc_fence_after();
        if (*abort_flag) break;                        // (the same in every warp: nobody waits before the next barrier)
    }
    if (*abort_flag) {
        // transforms may be under way: they have to end before TMEM is handed back
        if (warp == PF_TOKEN_WARPS) {
            if (elect_one()) umma_commit(bar(B_DRAIN));
            __syncwarp();
        }
        int tries = 0;
        while (!mbar_try(bar(B_DRAIN), 0) && ++tries < 1000000) {}
        __syncthreads();
    }
    if (warp == 0) tmem_dealloc<512>(tmem);
    if (threadIdx.x == 0 && misc[1] != 0) atomicOr(a.dev_status, NOVAKV_DEV_WAIT_TIMEOUT);
}

// Tensor map of [n_tokens][row] bfloat16 with boxes of 64 columns (128 bytes, swizzled) x 128 rows.
bool row_map(CUtensorMap* map, const void* base, int n_tokens, int row) {
    using encode_fn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                   const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const encode_fn encode = []() -> encode_fn {                 // (the driver's entry point, looked up once)
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &found) != cudaSuccess || found != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        return reinterpret_cast<encode_fn>(fn);
    }();
    if (encode == nullptr) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)row, (cuuint64_t)n_tokens}, strides[1] = {(cuuint64_t)row * 2};
    const cuuint32_t box[2] = {64, PF_HALF}, step[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D, int FMT>
novakv_status launch_prefill_t(novakv_ctx* ctx, const PrefillArgs& args, cudaStream_t stream) {
    using P = PF<D, FMT>;
    constexpr int L = P::L;
    PrefillArgs a = args;
    auto kern = novakv_prefill_kernel<D, FMT>;
    if (!(ctx->prefill_opt_in & (1u << FMT))) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P::BYTES) != cudaSuccess) return NOVAKV_ECUDA;
        ctx->prefill_opt_in |= 1u << FMT;
    }
    const int n_tiles = (a.n_tokens + PF_TILE - 1) / PF_TILE, hkv = ctx->cfg.n_kv_heads;
    // Units of 16 groups; of 8 (each repeats the transform's fixed costs) where that makes the longest run of units
    // cheaper: when there are too few units to give every SM one, or a few whole ones.
    double best = 1e30;
    int grid = 1;
    bool one_each = false;              // no more units than SMs
    for (int gs = L / P::GU; gs <= L / 8; gs *= 2) {
        const double cp = PF_US_UNIT + PF_US_GROUP * (L / gs), ck = cp + (FMT ? PF_US_SCALED : 0.0), cv = FMT == 2 ? PF_US_INT2 : cp;
        const int uk = hkv * gs * n_tiles, uv = FMT == 2 ? hkv * n_tiles : uk;
        const int g = uk + uv < ctx->n_sm ? uk + uv : ctx->n_sm;
        const double even = (uk * ck + uv * cv) / g, longest = ck * ceil(even / ck - 1e-6);       // units are whole
        if (longest < best) {
            best = longest;
            grid = g;
            a.gs = gs;
            // (then one unit per CTA: a cut in cost would hand some a key and a value unit)
            one_each = uk + uv <= ctx->n_sm;
            a.cost_k = one_each ? 1 : (int)(ck * (D == 128 && FMT == 0 && uk + uv >= PF_KEYS_UNITS * g ? PF_KEYS : 1.0) * 64.0);
            a.cost_v = one_each ? 1 : (int)(cv * 64.0);
        }
    }
    // tensor maps of the new rows (rebuilt on every call: the buffers are the caller's)
    a.tma = (((uintptr_t)a.k_new | (uintptr_t)a.v_new) & 15) == 0 &&
            row_map(&a.map_k, a.k_new, a.n_tokens, hkv * D) && row_map(&a.map_v, a.v_new, a.n_tokens, hkv * D);
    a.words = (((uintptr_t)a.k_pages | (uintptr_t)a.v_pages) & 3) == 0;
    novakv_prof_scope ps(ctx, 1, stream);
    // A short call's launch overlaps the kernel in front.  Not a long one's: its CTAs would land on SMs in the order in which
    // the kernel in front leaves them (32768 tokens, calls in a row: 490 us so, 501 overlapped).
    if (one_each) novakv_launch_pdl(kern, dim3(grid), dim3(PF_THREADS), P::BYTES, stream, a);
    else kern<<<grid, PF_THREADS, P::BYTES, stream>>>(a);
    ps.end();
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? NOVAKV_OK : NOVAKV_ECUDA;
}

}  // namespace

novakv_status novakv_launch_prefill(novakv_ctx* ctx, const novakv_layer& ly, const __nv_bfloat16* k_new, const __nv_bfloat16* v_new,
    const int32_t* tok_seq, const int32_t* tok_pos, int n_tokens, uint8_t* k_pages, uint8_t* v_pages, int n_pages,
    const int32_t* page_table, int max_pages_per_seq, int n_seq, int32_t* seq_lens, cudaStream_t stream, __nv_bfloat16* k_scales,
    __nv_bfloat16* v_meta) {
    PrefillArgs a = {k_new, v_new, tok_seq, tok_pos, n_tokens, ly.pf_r, ly.pf_cb, ly.pf_const, ly.rk_d, ly.rv_d, ly.rk_rows, ly.rv_rows, ly.k_mean_d,
                           ly.v_mean_d, ly.cb_k, ly.cb_v, k_pages, v_pages, k_scales, v_meta, n_pages, page_table, max_pages_per_seq,
                           n_seq, seq_lens, ctx->cfg.n_kv_heads, 1, 1, 1, 0, 0, ctx->wait_clocks, ctx->dev_status, {}, {}};
    if (ctx->cfg.head_dim == 128)
        return v_meta ? launch_prefill_t<128, 2>(ctx, a, stream) : (k_scales ? launch_prefill_t<128, 1>(ctx, a, stream) : launch_prefill_t<128, 0>(ctx, a, stream));
    return v_meta ? launch_prefill_t<64, 2>(ctx, a, stream) : (k_scales ? launch_prefill_t<64, 1>(ctx, a, stream) : launch_prefill_t<64, 0>(ctx, a, stream));
}

// ------------------------------------------------------------------------------------------------
// calibration images of this kernel (host)
// ------------------------------------------------------------------------------------------------
// One (KV head, side): the three bfloat16 slices of R as K-major operands (row = output column, 64-element panels of
// 128-byte rows, 16-byte chunks swizzled by the row), the codebook images, and the constants of error bounds and scaling.
void novakv_build_prefill_image(int d, const float* R /* [d][d] */, const float* mean /* [d] or null */, const float* cb /* [L][256][4] */,
                                uint8_t* r_img, uint8_t* cb_img, float* consts) {
    const int L = d / NOVAKV_G;
    for (int k = 0; k < d; ++k)
        for (int c = 0; c < d; ++c) {
            float rem = R[(size_t)k * d + c];
            for (int s = 0; s < 3; ++s) {
                const __nv_bfloat16 h = __float2bfloat16_rn(rem);
                rem -= __bfloat162float(h);
                const size_t off = (size_t)s * d * d * 2 + (size_t)(k >> 6) * d * 128 + (size_t)c * 128 + ((((k & 63) >> 3) ^ (c & 7)) * 16) + (k & 7) * 2;
                *reinterpret_cast<__nv_bfloat16*>(r_img + off) = h;
            }
        }
    double mn2 = 0.0, fro2 = 0.0, colmax = 0.0;
    for (int k = 0; k < d; ++k) mn2 += mean ? (double)mean[k] * mean[k] : 0.0;
    for (int l = 0; l < L; ++l) {
        double g2 = 0.0;
        for (int c = 4 * l; c < 4 * l + 4; ++c) {
            double m = 0.0, c2 = 0.0;
            for (int k = 0; k < d; ++k) {
                const double v = R[(size_t)k * d + c];
                m += mean ? (double)mean[k] * v : 0.0;
                c2 += v * v;
            }
            consts[c] = (float)m;
            g2 += c2;
            colmax = c2 > colmax ? c2 : colmax;
        }
        fro2 += g2;
        consts[d + l] = (float)(sqrt(g2) * 1.000001);
        // scale of the group: the longest codeword gets a length in [8, 16)
        double cmax2 = 0.0;
        for (int c = 0; c < NOVAKV_C; ++c) {
            double n2 = 0.0;
            for (int i = 0; i < 4; ++i) { const double v = cb[((size_t)l * NOVAKV_C + c) * 4 + i]; n2 += v * v; }
            cmax2 = n2 > cmax2 ? n2 : cmax2;
        }
        int e = 0;
        if (cmax2 > 0.0 && cmax2 < 1e300) { frexp(sqrt(cmax2), &e); e = 4 - e; }
        e = e > 100 ? 100 : (e < -100 ? -100 : e);
        consts[d + L + l] = (float)ldexp(1.0, e);
        uint8_t* g = cb_img + (size_t)l * NOVAKV_PF_GROUP_BYTES;
        for (int n = 0; n < NOVAKV_C; ++n) {
            // column n of the product: packed minima over even / odd columns of 16 make the rows of 8 codewords
            const int reg = n >> 4, half = n & 1, code = (reg * 2 + half) * 8 + ((n & 15) >> 1);
            double pd = 0.0;
            __half v[16];
            for (int i = 0; i < 4; ++i) {
                const float c = (float)ldexp((double)cb[((size_t)l * NOVAKV_C + code) * 4 + i], e);
                pd += 0.5 * (double)c * (double)c;
                const __half h = __float2half_rn(c);
                v[i] = __float2half_rn(-__half2float(h));
                v[8 + i] = v[i];
                v[4 + i] = __float2half_rn(-(c - __half2float(h)));
            }
            v[12] = __float2half_rn((float)pd);
            v[13] = __float2half_rn((float)(pd - (double)__half2float(v[12])));
            v[14] = v[15] = __float2half_rn(1.f);
            for (int kc = 0; kc < 2; ++kc) memcpy(g + kc * 4096 + (n >> 3) * 128 + (n & 7) * 16, v + 8 * kc, 16);
        }
        float* img = reinterpret_cast<float*>(g + 8192);
        for (int code = 0; code < NOVAKV_C; ++code)
            for (int i = 0; i < 4; ++i) img[codeword_offset(code, i)] = cb[((size_t)l * NOVAKV_C + code) * 4 + i];
    }
    consts[d + 2 * L] = (float)(sqrt(mn2) * 1.000001);
    consts[d + 2 * L + 1] = (float)(sqrt(fro2) * 1.000001);
    consts[d + 2 * L + 2] = (float)(sqrt(colmax) * 1.000001);
    consts[d + 2 * L + 3] = 0.f;
}
