// Attention of the tokens of a streaming run, bf16 storage: every token attends over a prefix of its window's list
// (and, in tokens_split_kernel, the first launch of elm_attend's split form: one list per problem)
//   O[t,:] = sum_c w_c exp(<q_t,k_c>/sqrt(d)) v_c / sum_c w_c exp(<q_t,k_c>/sqrt(d)),  c < seen(t)      Eq. (def:att_approx)
//
// Neighbouring tokens see all but a few of the same entries, and a token has one query vector per query head of its KV
// head, so 16 rows of a matrix instruction hold the vectors of 16, 8, 4 or 2 neighbouring tokens (TokenGroups::per_group).
// Both contractions are mma.sync m16n8k16 with fp32 accumulators: Q K^T on the stored bf16 values, P V with each fp32
// probability as the sum of three bf16 values (split3: 24 bits).  How the instruction rounds inside is not documented; against 64 bits it rounds
// toward zero, so its chains are short and their sums go on in fp32 (token_contract has the errors).
// tcgen05 takes 64 rows at least: a single token of four vectors would leave most of them empty, and the accumulators of
// each 32-entry unit (below) would go through tensor memory and back.
//
// The work is cut the same way whatever tokens share a launch: the list in units of k tiles of 32 entries (token_units), a unit's softmax
// by one warp from its own maximum, the units merged in the order of the list.  A row's arithmetic does not depend on
// the other rows, so a token's output is the same bit for bit in every form:
//   cluster  one thread-block cluster per group of neighbouring tokens, one unit per warp; the warps hand their results
//            to the CTA that finishes the slice through distributed shared memory.
//   serial   one CTA per four groups, a group's 16 rows per warp; the tiles come once for all four warps through a ring
//            of asynchronous copies and every warp merges unit after unit in registers.
//
// Bound by the issue of mma.sync: 128 per tile and 16 rows, 32 for the logits and 96 for the values, at the 16 cycles that each
// takes an SM sub-partition (about 2500 cycles per tile with two warps on each; 2250 with the sums of the list left to the instruction).
// With fp32 fma per token and here: a generation of 2496 tokens of 32 query / 8 KV heads, n_out = 256, 1443 -> 490 us; 512 tokens over 6144
// entries 2145 -> 522, over 200 218 -> 65; one token over 6144 entries of 8 KV heads of 4 query heads 16.6 -> 15.2 us, of 8 query heads 22.3 -> 17.3,
// over 200 entries 7.1 -> 7.6; of 1 query head over 4100 entries 10.2 -> 12.5 (its one vector pays for eight), but 8 of them 36.5 -> 14.9.
#include <math.h>

#include <atomic>
#include <type_traits>

#include "elm_attend.cuh"
#include "elm_common.cuh"
#include "elm_sm100.cuh"

namespace elm {
namespace {

using sm100::add2;
using sm100::fma2;
using sm100::mul2;
using sm100::pack2;
using sm100::pack_bf16x2;
using sm100::smem_u32;
using sm100::unpack2;

constexpr int TOK_WARPS = 4;
constexpr int TOK_THREADS = TOK_WARPS * 32;
constexpr int TOK_ROWS = 16;                   // rows of the matrix instruction
constexpr int TOK_TILE = 32;                   // entries per tile
constexpr int TOK_MAX_CLUSTER = 16;
constexpr int TOK_STAGES = 4;                  // ring of the serial form
constexpr int TOK_CTAS = 2;                    // CTAs per SM the kernel is compiled for

struct TokenGroups {
    int32_t cluster;                           // CTAs per group (cluster form)
    TokenCaps caps;                            // most CTAs a list is spread over
    int32_t per_group;                         // neighbouring tokens of a warp: a power of two
    int32_t span;                              // tokens per cluster or CTA: per_group, or four times as many
    int32_t g0[DECODE_MAX_WINDOWS + 1];        // groups of `span` tokens in the windows before
};

// Tiles per unit of a list of n_core entries: at most 4 units per CTA.  Depends on n_core only through the next multiple of
// 128, so that the (at most 64, aligned) tokens of a span agree.
__host__ __device__ __forceinline__ int token_units(int n_core, TokenCaps caps)
{
    const int tiles = (n_core + 127) / 128 * (128 / TOK_TILE), most = TOK_WARPS * (n_core <= TOKENS_SHORT_LIST ? caps.of_short : caps.of_long);
    return (tiles + most - 1) / most;
}

// CTAs of a cluster for lists of n0 .. n1 entries
int tokens_cluster(int n0, int n1, TokenCaps caps)
{
    auto units = [&](int n) { const int k = token_units(n, caps), tiles = (n + TOK_TILE - 1) / TOK_TILE; return (tiles + k - 1) / k; };
    // (where the units grow longer there are fewer of them: the most are at an end, or just below a step)
    int most = units(n1);
    for (int n = (n0 + 127) / 128 * 128; n < n1; n += 128) most = units(n) > most ? units(n) : most;
    int size = 1;
    while (size * TOK_WARPS < most) size *= 2;
    return size;
}

template <int D> struct TokenCfg {
    static constexpr int RB = D * 2;                               // bytes per row
    static constexpr int NC = RB / 16;                             // 16-byte chunks per row
    static constexpr int TILE_BYTES = TOK_TILE * RB;
    static constexpr int MT = D / 16;                              // row tiles of the transposed output
    static constexpr int MAX_UNITS = TOK_WARPS * TOK_MAX_CLUSTER;
    // serial form: [stage][K, V], log2 weights, queries by warp
    static constexpr int S_LW = TOK_STAGES * 2 * TILE_BYTES;
    static constexpr int S_Q = S_LW + TOK_STAGES * TOK_TILE * 4;
    static constexpr int S_TOTAL = S_Q + TOK_WARPS * TOK_ROWS * RB;
    // split form: [warp][K, V], log2 weights, (maximum, denominator) [warp][row], queries by warp
    static constexpr int P_LW = TOK_WARPS * 2 * TILE_BYTES;
    static constexpr int P_ML = P_LW + TOK_WARPS * TOK_TILE * 4;
    static constexpr int P_Q = P_ML + TOK_WARPS * 8 * 8;
    static constexpr int P_TOTAL = P_Q + TOK_WARPS * 8 * RB;
    // cluster form: [warp][K, V], log2 weights; factors of the units, maxima (then factors of the state) and denominators [row][unit];
    // the CTA's slice of every unit's result, [unit][column of the slice][row]
    template <int ROWS> struct Cluster {
        static constexpr int LW = TOK_WARPS * 2 * TILE_BYTES;
        static constexpr int FB = LW + TOK_WARPS * TOK_TILE * 4;
        static constexpr int ML = FB + ROWS * MAX_UNITS * 4;
        static constexpr int RECV = ML + ROWS * MAX_UNITS * 8;
        static constexpr int TOTAL = RECV + TOK_WARPS * D * (ROWS + 2) * 4;
        static_assert(TOK_CTAS * (TOTAL + 1024) <= 228 * 1024, "shared memory for as many CTAs as there are registers for");
    };
};

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void *src, bool live)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// chunk c of row e of a tile lies at chunk c ^ (e mod 8): the eight rows a matrix load reads fall into different banks
template <int NC> __device__ __forceinline__ uint32_t chunk_at(int e, int c) { return (uint32_t)((e * NC + (c ^ (e & 7))) * 16); }

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm2(uint32_t &r0, uint32_t &r1, uint32_t a)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t a)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// the same with c = 0
__device__ __forceinline__ void mma16816_new(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// Two probabilities as sums of three bf16 values each (low halves: p0, high halves: p1).  The first two parts are taken
// just below what they stand for, so that all parts of a positive value are positive: an infinite value of V stays that
// infinity instead of meeting a part that is zero or negative.  So it is for values of 2^-100 and more, whose last bit and with it
// the smallest part is a normal bf16 value; smaller ones do not come here (token_values).
constexpr uint32_t SMALLEST_SPLIT = 27u << 23;                     // the bits of 2^-100
__device__ __forceinline__ void split3(float p0, float p1, uint32_t &hi, uint32_t &mid, uint32_t &lo)
{
    const uint32_t h0 = (max(__float_as_uint(p0), 1u) - 1u) & 0xffff0000u, h1 = (max(__float_as_uint(p1), 1u) - 1u) & 0xffff0000u;
    const float r0 = p0 - __uint_as_float(h0), r1 = p1 - __uint_as_float(h1);
    const uint32_t m0 = (max(__float_as_uint(r0), 1u) - 1u) & 0xffff0000u, m1 = (max(__float_as_uint(r1), 1u) - 1u) & 0xffff0000u;
    hi = __byte_perm(h0, h1, 0x7632);
    mid = __byte_perm(m0, m1, 0x7632);
    lo = pack_bf16x2(r0 - __uint_as_float(m0), r1 - __uint_as_float(m1));
}

// factors of a merge of a unit with maximum m into a state with maximum M
__device__ __forceinline__ void merge_factors(float M, float m, float &Mn, float &a, float &b)
{
    Mn = fmaxf(M, m);
    a = M == -INFINITY ? 0.f : exp2f(M - Mn);
    b = m == -INFINITY ? 0.f : exp2f(m - Mn);
}

// The probabilities P [row][entry] as they leave Q K^T are the B operand of O^T = V^T P^T, whose columns are the query vectors,
// eight at a time: a call of few vectors does not pay for sixteen in the larger of the two products.
//
// A unit's state.  o: of the rows 8 b + 2 (lane % 4) + {0, 1}, b < NB, the columns lane / 4 + 8 k; m, l: of the rows 8 b + lane / 4.
template <int D, int NB> struct TokenUnit {
    float o[D / 16][NB][4];
    float m[NB], l[NB];
    __device__ __forceinline__ void reset()
    {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
#pragma unroll
            for (int j = 0; j < D / 16; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) o[j][b][i] = 0.f;
            m[b] = -INFINITY;
            l[b] = 0.f;
        }
    }
    __device__ __forceinline__ void finish()
    {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            l[b] += __shfl_xor_sync(0xffffffffu, l[b], 1);
            l[b] += __shfl_xor_sync(0xffffffffu, l[b], 2);
        }
    }
};
// what the rows 2 (lane % 4) + {0, 1} of eight have of a value held by row
__device__ __forceinline__ void of_columns(float x, float &x0, float &x1)
{
    const int quad = threadIdx.x & 3;
    x0 = __shfl_sync(0xffffffffu, x, 8 * quad);
    x1 = __shfl_sync(0xffffffffu, x, 8 * quad + 4);
}

// A warp's query vectors, scaled by 1/8 - exactly, and close enough to 1/sqrt(d) that no product is larger than the logit's: as operands
// in registers, or as rows in shared memory that are read again for every tile (where the accumulators need the registers).
template <int D, int NB, bool SHARED> struct TokenQueries;
template <int D, int NB> struct TokenQueries<D, NB, false> {
    uint32_t f[D / 16][4];
    __device__ __forceinline__ void put(int i, int c, int h, uint32_t x) { f[i][2 * c + h] = x; }
    __device__ __forceinline__ void get(int i, uint32_t (&a)[4]) const
    {
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = f[i][k];
    }
};
template <int D, int NB> struct TokenQueries<D, NB, true> {
    static constexpr int BYTES = 8 * NB * D * 2;
    uint32_t at;                                                   // [row][chunk ^ row % 8]
    __device__ __forceinline__ void put(int i, int c, int h, uint32_t x)
    {
        const int lane = threadIdx.x & 31;
        if (h < NB)
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(at + chunk_at<TokenCfg<D>::NC>(8 * h + (lane >> 2), 2 * i + c) + 4 * (lane & 3)), "r"(x) : "memory");
    }
    __device__ __forceinline__ void get(int i, uint32_t (&a)[4]) const
    {
        const int lane = threadIdx.x & 31;
        if constexpr (NB == 2) {
            ldsm4(a, at + chunk_at<TokenCfg<D>::NC>(lane & 15, 2 * i + (lane >> 4)));
        } else {
            ldsm2(a[0], a[2], at + chunk_at<TokenCfg<D>::NC>(lane & 7, 2 * i + ((lane >> 3) & 1)));
            a[1] = a[3] = 0;
        }
    }
};
// The loads and what is made of them, apart: their round trip goes by in between.  row(r): where vector r lies in Q; `rows` of the 8 NB exist.
template <int D, int NB> struct TokenRawQueries { uint32_t x[NB][D / 16][2]; };
template <int D, int NB, typename Row>
__device__ __forceinline__ void load_queries(TokenRawQueries<D, NB> &raw, const __nv_bfloat16 *Q, int rows, Row row)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 0; h < NB; ++h) {
        const int r = 8 * h + (lane >> 2);
        const __nv_bfloat16 *q = Q + (r < rows ? row(r) : 0) + 2 * (lane & 3);
#pragma unroll
        for (int i = 0; i < D / 16; ++i)
#pragma unroll
            for (int c = 0; c < 2; ++c) raw.x[h][i][c] = r < rows ? *reinterpret_cast<const uint32_t *>(q + 16 * i + 8 * c) : 0u;
    }
}
template <int D, int NB, bool SHARED> __device__ __forceinline__ void put_queries(TokenQueries<D, NB, SHARED> &qs, const TokenRawQueries<D, NB> &raw)
{
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < D / 16; ++i)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t x = 0;
                if (h < NB) {
                    const __nv_bfloat162 y = __hmul2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x[h < NB ? h : 0][i][c]), __floats2bfloat162_rn(0.125f, 0.125f));
                    x = *reinterpret_cast<const uint32_t *>(&y);
                }
                qs.put(i, c, h, x);
            }
}

// q k of one tile of 32 entries whose rows lie at kt: s[j][2 b + i], entry 8 j + 2 (lane % 4) + i of row 8 b + lane / 4.  32 dimensions
// at a time by the matrix instruction, their sums by fp32 additions (see token_contract).
template <int D, int NB, bool SHARED>
__device__ __forceinline__ void token_logits(float (&s)[4][4], const TokenQueries<D, NB, SHARED> &qs, uint32_t kt)
{
    constexpr int NC = TokenCfg<D>::NC;
    const int lane = threadIdx.x & 31;
    // The split form leaves this loop one: unrolled, its loads are all moved to the front, where they push accumulators out of the registers
    // (64 problems of 5193 entries 40.0 us, so 32.8; the serial form 258 unrolled, 267 not: 128 tokens over 4100 entries).
    constexpr bool ONE_LOOP = SHARED && NB == 1;
    if constexpr (ONE_LOOP) {
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j][0] = s[j][1] = 0.f;
    }
#pragma unroll(ONE_LOOP ? 1 : D / 32)
    for (int i = 0; i < D / 32; ++i) {
        uint32_t b[4][4], qa[4], qb[4];
        float t[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) ldsm4(b[j], kt + chunk_at<NC>(8 * j + (lane & 7), 4 * i + (lane >> 3)));
        qs.get(2 * i, qa);
        qs.get(2 * i + 1, qb);
#pragma unroll
        for (int j = 0; j < 4; ++j) mma16816_new(t[j], qa, b[j][0], b[j][1]);
#pragma unroll
        for (int j = 0; j < 4; ++j) mma16816(t[j], qb, b[j][2], b[j][3]);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < 2 * NB; k += 2) {
                const uint64_t x = pack2(t[j][k], t[j][k + 1]);
                unpack2(!ONE_LOOP && i == 0 ? x : add2(pack2(s[j][k], s[j][k + 1]), x), s[j][k], s[j][k + 1]);
            }
    }
}

// The tile's softmax: logits to probabilities.  t0 is its first entry, lw its log2 weights; the thread's rows see the entries
// below lim[.], all rows of the group those below `common`.  alpha: by what token_values scales the accumulators of rows
// 8 b + 2 (lane % 4) + {0, 1}, unless the tile is the unit's first.  low: the smallest log2 of the thread's probabilities.
template <int D, int NB>
__device__ __forceinline__ void token_softmax(TokenUnit<D, NB> &u, bool first, float (&s)[4][4], const float *lw, int t0,
                                              const int (&lim)[NB], int common, float scale, uint64_t (&alpha)[NB], float &low)
{
    const int quad = threadIdx.x & 3;
    const bool tail = t0 + TOK_TILE > common;                      // (the same for the whole warp)
    low = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 w2 = *reinterpret_cast<const float2 *>(lw + 8 * j + 2 * quad);
#pragma unroll
        for (int i = 0; i < 2 * NB; ++i) s[j][i] = fmaf(s[j][i], scale, i & 1 ? w2.y : w2.x);
    }
    if (tail) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 2 * NB; ++i)
                if (t0 + 8 * j + 2 * quad + (i & 1) >= lim[i >> 1]) s[j][i] = -INFINITY;
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j) mx = fmaxf(mx, fmaxf(s[j][2 * b], s[j][2 * b + 1]));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        mx = fmaxf(u.m[b], mx);
        const float ref = mx == -INFINITY ? 0.f : mx;
        if (!first) {
            const float f = exp2f(u.m[b] - ref);
            // (rounded on its own: whether a compiler fuses it with the sum below must not depend on the form)
            u.l[b] = __fmul_rn(u.l[b], f);
            float a0, a1;
            of_columns(f, a0, a1);
            alpha[b] = pack2(a0, a1);
        }
        u.m[b] = mx;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float x = s[j][2 * b + i] - ref;
                low = fminf(low, x);
                s[j][2 * b + i] = exp2f(x);
                u.l[b] = __fadd_rn(u.l[b], s[j][2 * b + i]);
            }
    }
}

// The halves of x that are infinite or NaN as masks of ones: an exponent of all ones carries into the sign's place
__device__ __forceinline__ uint32_t not_finite(uint32_t x) { return (((x & 0x7f807f80u) + 0x00800080u) >> 15 & 0x00010001u) * 0xffffu; }
// Probabilities that are too small to be split, and not zero
__device__ __forceinline__ bool too_small(float p) { return __float_as_uint(p) - 1u < SMALLEST_SPLIT - 1u; }

// O^T += V^T P^T of a tile: the unit's accumulators times alpha (not if the tile is the first) plus the tile's products.
// The matrix instruction rounds toward zero, every time by up to a bit of what it has accumulated so far.  So a tile's sums start
// at zero, take the small parts first, and go to the unit's accumulators by fp32 fma (one accumulator through a warp's whole share of a
// list: relative error 5.0e-7 over 5193 entries, 1.9e-6 over 12288; fp32 fma alone 2.1e-7 and 3.6e-7; so 1.8e-7 and 2.3e-7).
// `odd`: entries of which the values that are not finite are taken as zeros, and so are probabilities that cannot be split.
template <int D, int NB, bool ODD, bool SERIAL>
__device__ __forceinline__ void token_contract(TokenUnit<D, NB> &u, bool first, const uint64_t (&alpha)[NB], const float (&s)[4][4],
                                               uint32_t vt, uint32_t odd)
{
    using C = TokenCfg<D>;
    const int lane = threadIdx.x & 31, quad = lane & 3;
    uint32_t p[2][NB][3][2];                                           // [k]: entries 16 k + {0, 8} + 2 (lane % 4) + {0, 1} of row 8 b + lane / 4
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float x = s[2 * k + h][2 * b], y = s[2 * k + h][2 * b + 1];
                if constexpr (ODD) {
                    x = too_small(x) ? 0.f : x;
                    y = too_small(y) ? 0.f : y;
                }
                split3(x, y, p[k][b][0][h], p[k][b][1][h], p[k][b][2][h]);
            }
    // Output tiles at a time: four, or, where eight warps of an SM leave the tensor cores little time between them (serial form), two and two of
    // them on their way while the two before are added (512 tokens over 4100 entries, 4 vectors: 366 us with four, 358 so).
    constexpr int JG = SERIAL ? 2 : 4;
    const int sw = lane & 7, half = (lane >> 3) & 1;
    float t[SERIAL ? 2 : 1][JG][NB][4];
    auto add = [&](int j) {
#pragma unroll
        for (int h = 0; h < JG; ++h)
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                float (&o)[4] = u.o[j + h][b], (&x)[4] = t[SERIAL ? j / JG & 1 : 0][h][b];
#pragma unroll
                for (int i = 0; i < 4; i += 2) {
                    if (first) {
                        o[i] = x[i];
                        o[i + 1] = x[i + 1];
                    } else {
                        unpack2(fma2(pack2(o[i], o[i + 1]), alpha[b], pack2(x[i], x[i + 1])), o[i], o[i + 1]);
                    }
                }
            }
    };
#pragma unroll
    for (int j = 0; j < D / 16; j += JG) {
        uint32_t a[2][JG][4];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            // matrices of a load: entries 16 k + {0, 0, 8, 8} + 0..7, chunks {0, 1, 0, 1} of the 16 columns
            const uint32_t va = vt + (uint32_t)((16 * k + (lane >> 4) * 8 + (lane & 7)) * C::RB);
#pragma unroll
            for (int h = 0; h < JG; ++h) {
                ldsm4_t(a[k][h], va + (uint32_t)(((2 * (j + h) + half) ^ sw) * 16));
                if constexpr (ODD) {
                    auto mask_of = [&](int e) { return (odd >> e & 1 ? 0xffffu : 0u) | (odd >> (e + 1) & 1 ? 0xffff0000u : 0u); };
                    const uint32_t k0 = mask_of(16 * k + 2 * quad), k1 = mask_of(16 * k + 8 + 2 * quad);
                    a[k][h][0] &= ~(not_finite(a[k][h][0]) & k0); a[k][h][1] &= ~(not_finite(a[k][h][1]) & k0);
                    a[k][h][2] &= ~(not_finite(a[k][h][2]) & k1); a[k][h][3] &= ~(not_finite(a[k][h][3]) & k1);
                }
            }
        }
#pragma unroll
        for (int part = 2; part >= 0; --part)
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int h = 0; h < JG; ++h)
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                        if (part == 2 && k == 0) mma16816_new(t[SERIAL ? j / JG & 1 : 0][h][b], a[k][h], p[k][b][part][0], p[k][b][part][1]);
                        else mma16816(t[SERIAL ? j / JG & 1 : 0][h][b], a[k][h], p[k][b][part][0], p[k][b][part][1]);
                    }
        if (!SERIAL) add(j);
        else if (j > 0) add(j - JG);
    }
    if (SERIAL) add(D / 16 - JG);
}

// A tile with entries that do not go through the matrix instruction alone (rare, so on a copy of the accumulators in local memory and
// out of line).  What such an entry needs is added by scalar code: to the rows whose probability is too small to be split all its
// values, to the other rows that see it the values that are not finite.
template <int D, int NB> struct TokenOdd {
    TokenUnit<D, NB> u;
    uint64_t alpha[NB];
    float s[4][4];
    int lim[NB];
};
template <int D, int NB> __device__ __noinline__ void token_values_odd(TokenOdd<D, NB> *x, bool first, const unsigned char *vrows, int t0, uint32_t odd)
{
    using C = TokenCfg<D>;
    const int lane = threadIdx.x & 31, quad = lane & 3;
    token_contract<D, NB, true, false>(x->u, first, x->alpha, x->s, smem_u32(vrows), odd);
    for (uint32_t left = odd; left; left &= left - 1) {
        const int e = __ffs(left) - 1;
        for (int b = 0; b < NB; ++b)
            for (int i = 0; i < 2; ++i) {
                const int from = 8 * quad + 4 * i;                     // the first lane that holds the row's probabilities
                const float pe = __shfl_sync(0xffffffffu, x->s[e >> 3][2 * b + (e & 1)], from + ((e & 7) >> 1));
                const bool sees = t0 + e < __shfl_sync(0xffffffffu, x->lim[b], from), all = too_small(pe);
                for (int j = 0; j < D / 8; ++j) {                      // column lane / 4 + 8 j
                    const uint32_t v = (uint32_t)*reinterpret_cast<const uint16_t *>(vrows + chunk_at<C::NC>(e, j) + 2 * (lane >> 2)) << 16;
                    float &o = x->u.o[j >> 1][b][2 * (j & 1) + i];
                    if (sees && (all || not_finite(v))) o = fmaf(pe, __uint_as_float(v), o);
                }
            }
    }
}

// The tile's values, whose rows lie at vrows; the thread's rows see the entries below lim[.], all rows of the group those
// below `common`, and those below `loaded` are there (what other warps of the CTA see).
template <bool SERIAL, int D, int NB>
__device__ __forceinline__ void token_values(TokenUnit<D, NB> &u, bool first, const uint64_t (&alpha)[NB], float low, const float (&s)[4][4],
                                             const unsigned char *vrows, int t0, const int (&lim)[NB], int common, int loaded)
{
    constexpr int NC = TokenCfg<D>::NC;
    const int lane = threadIdx.x & 31, quad = lane & 3;
    // Entries whose values do not go through the matrix instruction alone.  One that only some rows see, or none, and that holds an infinity
    // or a NaN must not meet the zero probabilities of the others; a probability that three bf16 parts cannot hold (below 2^-100, for
    // which a logit has to lie 69 below the largest of its unit) must meet its values in fp32.  No row's arithmetic depends on another's.
    uint32_t odd = 0;
    const int e0 = common > t0 ? common - t0 : 0, e1 = loaded - t0 < TOK_TILE ? loaded - t0 : TOK_TILE;
    if (e0 < e1) {
        for (int i = lane; i < (e1 - e0) * NC; i += 32) {
            const uint4 x = *reinterpret_cast<const uint4 *>(vrows + chunk_at<NC>(e0 + i / NC, i % NC));
            if (not_finite(x.x) | not_finite(x.y) | not_finite(x.z) | not_finite(x.w)) odd |= 1u << (e0 + i / NC);
        }
        odd = __reduce_or_sync(0xffffffffu, odd);
    }
    if (__any_sync(0xffffffffu, low < -100.f)) {
        uint32_t small = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 2 * NB; ++i)
                if (too_small(s[j][i])) small |= 1u << (8 * j + 2 * quad + (i & 1));
        odd |= __reduce_or_sync(0xffffffffu, small);
    }
    if (odd) {
        TokenOdd<D, NB> x;
        x.u = u;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            x.alpha[b] = first ? 0 : alpha[b];
            x.lim[b] = lim[b];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 2 * NB; ++i) x.s[j][i] = s[j][i];
        token_values_odd(&x, first, vrows, t0, odd);
        u = x.u;
    } else {
        token_contract<D, NB, false, SERIAL>(u, first, alpha, s, smem_u32(vrows), 0);
    }
}

// NB: query vectors of a warp, in eights (the serial form takes two)
template <int D, bool CLUSTER, int NB>
__global__ void __launch_bounds__(TOK_THREADS, TOK_CTAS)
tokens_kernel(const __nv_bfloat16 *__restrict__ Q, const __nv_bfloat16 *__restrict__ K, const __nv_bfloat16 *__restrict__ V,
              const int32_t *__restrict__ idx, const float *__restrict__ w, int64_t n, int64_t list_stride, int q_heads, int kv_heads,
              int per_token, const __grid_constant__ DecodeWindows win, const __grid_constant__ TokenGroups grp,
              __nv_bfloat16 *__restrict__ O, int *__restrict__ status)
{
    using C = TokenCfg<D>;
    using CC = typename C::template Cluster<8 * NB>;
    constexpr int NC = C::NC, MT = C::MT;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, quad = lane & 3;
    // (launched with programmatic stream serialization: nothing is read or written before this point)
    cudaGridDependencySynchronize();
    if constexpr (CLUSTER) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    const int prob = blockIdx.y;
    const int rank = CLUSTER ? (int)blockIdx.x % grp.cluster : 0;
    // (serial form: the longest lists, those of the last tokens, start first)
    const int group = CLUSTER ? (int)blockIdx.x / grp.cluster : (int)(gridDim.x - 1 - blockIdx.x);
#ifndef ELM_BOUNDS_CHECK
    // this path has no bounded waits and (in this build) no row checks: its status word reads 0
    if (tid == 0 && prob == 0 && blockIdx.x == 0) *status = 0;
#endif
    int wi = 0;
    while (wi + 1 < win.n && group >= grp.g0[wi + 1]) ++wi;
    // the tokens of the span see lo + 1 .. lo + span entries, as far as the window has them
    const int lo = ((win.seen0[wi] - 1) / grp.span + (group - grp.g0[wi])) * grp.span;
    const int last_seen = win.seen0[wi] + (win.tok0[wi + 1] - win.tok0[wi]) - 1;
    const int n_span = min(last_seen, lo + grp.span);              // what the last of them sees
    // this warp's group: first entry count that is aligned, first that is in the launch, last
    const int aligned = lo + (CLUSTER ? 0 : warp * grp.per_group) + 1;
    const int first = max(aligned, win.seen0[wi]);
    const int rows = max(min(n_span, aligned + grp.per_group - 1) - first + 1, 0) * per_token;
    const int last = rows ? min(n_span, aligned + grp.per_group - 1) : 0;
    const int b = prob / kv_heads, kvh = prob % kv_heads, rep = q_heads / kv_heads;
    const int32_t *ip = idx + (int64_t)prob * list_stride + win.off[wi];
    const float *wp = w + (int64_t)prob * list_stride + win.off[wi];
    const __nv_bfloat16 *Kp = K + (int64_t)prob * n * D, *Vp = V + (int64_t)prob * n * D;
    // offset of row r in Q and O
    auto q_row = [&](int r) -> int64_t {
        const int64_t z = win.tok0[wi] + (first - win.seen0[wi]) + r / per_token;
        return ((z * (gridDim.y / kv_heads) + b) * q_heads + kvh * rep + r % per_token) * D;
    };
    int lim[NB];
#pragma unroll
    for (int h = 0; h < NB; ++h) lim[h] = 8 * h + (lane >> 2) < rows ? first + (8 * h + (lane >> 2)) / per_token : 0;
    TokenRawQueries<D, NB> raw;
    TokenQueries<D, NB, !CLUSTER> qs;
    const float scale = 8.f * 1.4426950408889634f / sqrtf((float)D);
    const int unit_tiles = token_units(n_span, grp.caps);
    const int tiles = (n_span + TOK_TILE - 1) / TOK_TILE;
    TokenUnit<D, NB> u;

    if constexpr (CLUSTER) {
        // ---- one unit per warp ----
        const int units = (tiles + unit_tiles - 1) / unit_tiles;
        const int unit = rank * TOK_WARPS + warp;
        unsigned char *kt = smem + warp * 2 * C::TILE_BYTES, *vt = kt + C::TILE_BYTES;
        float *lw = reinterpret_cast<float *>(smem + CC::LW) + warp * TOK_TILE;
        int32_t row = 0;
        float wt = 0.f;
        auto fetch_entries = [&](int t) {
            const int e = t * TOK_TILE + lane;
            row = 0;
            wt = 0.f;
            if (e < n_span) {
                row = (int32_t)checked_row(__ldg(ip + e), n, status);
                wt = __ldg(wp + e);
            }
        };
        auto copy_rows = [&](unsigned char *dst, const __nv_bfloat16 *X, int32_t from, int t) {
            const uint32_t d0 = smem_u32(dst);
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                const int e = (lane + 32 * i) / NC, c = lane % NC;
                const int64_t r = __shfl_sync(0xffffffffu, from, e);
                cp_async16_zfill(d0 + chunk_at<NC>(e, c), X + r * D + c * 8, t * TOK_TILE + e < n_span);
            }
            cp_async_commit();
        };
        const int t_end = min((unit + 1) * unit_tiles, tiles);
        int t = unit * unit_tiles;
        u.reset();
        if (t < t_end) fetch_entries(t);
        load_queries(raw, Q, rows, q_row);
        if (t < t_end) {
            copy_rows(kt, Kp, row, t);
            copy_rows(vt, Vp, row, t);
        }
        put_queries(qs, raw);
        for (bool head = true; t < t_end; ++t, head = false) {
            const bool more = t + 1 < t_end;
            float s[4][4];
            uint64_t alpha[NB];
            float low;
            lw[lane] = log2f(wt);
            if (more) fetch_entries(t + 1);
            cp_async_wait<1>();                                        // the keys (the values are the newer group)
            __syncwarp();
            token_logits(s, qs, smem_u32(kt));
            __syncwarp();
            if (more) copy_rows(kt, Kp, row, t + 1);
            token_softmax<D, NB>(u, head, s, lw, t * TOK_TILE, lim, aligned, scale, alpha, low);
            if (more) cp_async_wait<1>();                              // (the next tile's keys may still be on their way)
            else cp_async_wait<0>();
            __syncwarp();
            token_values<false>(u, head, alpha, low, s, vt, t * TOK_TILE, lim, aligned, n_span);
            __syncwarp();
            if (more) copy_rows(vt, Vp, row, t + 1);
        }
        u.finish();
        // ---- to the CTA that finishes the slice: columns of all rows, as many to each of `parts` (a power of two) CTAs ----
        int parts_log = 0;
        while ((1 << parts_log) < (units + TOK_WARPS - 1) / TOK_WARPS) ++parts_log;
        constexpr int D_LOG = D == 64 ? 6 : 7;
        const int cols_log = D_LOG - parts_log;
        // (rows go in pairs, and 18 floats from column to column spread 16 rows over the banks)
        const int col_stride = ((rows + 1) & ~1) + 2, slice = col_stride << cols_log;
        float2 *ml = reinterpret_cast<float2 *>(smem + CC::ML);
        float *fb = reinterpret_cast<float *>(smem + CC::FB), *recv = reinterpret_cast<float *>(smem + CC::RECV);
        auto remote = [&](const void *mine, int to) -> uint32_t {
            uint32_t a;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(mine)), "r"(to));
            return a;
        };
        auto send2 = [&](uint32_t a, float x, float y) {
            asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x), "f"(y) : "memory");
        };
        // every CTA of the cluster is running (its shared memory may be written) once this wait is over
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (unit < units) {
#pragma unroll
            for (int h = 0; h < NB; ++h) {
                const int r = 8 * h + 2 * quad;
                if (r < rows) {
#pragma unroll
                    for (int j = 0; j < 2 * MT; ++j) {
                        const int c = 8 * j + (lane >> 2);
                        send2(remote(recv + unit * slice + (c & ((1 << cols_log) - 1)) * col_stride + r, c >> cols_log), u.o[j >> 1][h][2 * (j & 1)],
                              u.o[j >> 1][h][2 * (j & 1) + 1]);
                    }
                }
                if (8 * h + (lane >> 2) < rows)
                    for (int to = quad; to < 1 << parts_log; to += 4)
                        send2(remote(ml + (8 * h + (lane >> 2)) * C::MAX_UNITS + unit, to), u.m[h], u.l[h]);
            }
        }
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (rank < 1 << parts_log) {
            // factors of the merges: running maxima of the rows' units, by a warp per row or, for short lists, four rows to a warp
            auto factors = [&](auto lanes) {
                constexpr int W = decltype(lanes)::value;
                const int li = lane & (W - 1);
                for (int r = warp * (32 / W) + lane / W; r - lane / W < rows; r += TOK_WARPS * (32 / W)) {
                    float carry = -INFINITY;
                    for (int u0 = 0; u0 < units; u0 += W) {
                        const bool live = r < rows && u0 + li < units;
                        const float m = live ? ml[r * C::MAX_UNITS + u0 + li].x : -INFINITY;
                        float mx = m;
#pragma unroll
                        for (int off = 1; off < W; off <<= 1) {
                            const float y = __shfl_up_sync(0xffffffffu, mx, off, W);
                            if (li >= off) mx = fmaxf(mx, y);
                        }
                        float before = __shfl_up_sync(0xffffffffu, mx, 1, W);
                        before = li == 0 ? carry : fmaxf(before, carry);
                        float Mn, a, b;
                        merge_factors(before, m, Mn, a, b);
                        if (live) {
                            ml[r * C::MAX_UNITS + u0 + li].x = a;
                            fb[r * C::MAX_UNITS + u0 + li] = b;
                        }
                        carry = fmaxf(carry, __shfl_sync(0xffffffffu, mx, W - 1, W));
                    }
                }
            };
            if (units <= 8) factors(std::integral_constant<int, 8>());
            else factors(std::integral_constant<int, 32>());
            __syncthreads();
            const int c0 = rank << cols_log;
            for (int i = tid; i < rows << cols_log; i += TOK_THREADS) {
                const int c = i & ((1 << cols_log) - 1), r = i >> cols_log;
                float den = 0.f, acc = 0.f;
#pragma unroll 4
                for (int k = 0; k < units; ++k) {
                    const float2 f = ml[r * C::MAX_UNITS + k];
                    const float b = fb[r * C::MAX_UNITS + k];
                    den = fmaf(b, f.y, __fmul_rn(den, f.x));
                    acc = fmaf(b, recv[k * slice + c * col_stride + r], __fmul_rn(acc, f.x));
                }
                store_from(O, q_row(r) + c0 + c, acc / den);
            }
        }
    } else {
        // ---- the tiles one after the other, for the four groups of the CTA ----
        qs.at = smem_u32(smem + C::S_Q + warp * TokenQueries<D, NB, true>::BYTES);
        load_queries(raw, Q, rows, q_row);
        put_queries(qs, raw);
        __syncwarp();
        constexpr int RPP = TOK_THREADS / NC, PASSES = TOK_TILE / RPP;
        const int my_row = tid / NC, my_chunk = tid % NC;
        const uint32_t ring = smem_u32(smem);
        float *lw = reinterpret_cast<float *>(smem + C::S_LW);
        int32_t rowno[PASSES];
        float wt = 0.f;
        auto fetch_entries = [&](int t) {
#pragma unroll
            for (int i = 0; i < PASSES; ++i) {
                const int e = t * TOK_TILE + my_row + i * RPP;
                rowno[i] = e < n_span ? (int32_t)checked_row(__ldg(ip + e), n, status) : 0;
            }
            if (tid < TOK_TILE) wt = t * TOK_TILE + tid < n_span ? __ldg(wp + t * TOK_TILE + tid) : 0.f;
        };
        auto fill = [&](int t) {
            if (t < tiles) {
                const int stage = t % TOK_STAGES;
                const uint32_t kd = ring + (uint32_t)(stage * 2 * C::TILE_BYTES), vd = kd + C::TILE_BYTES;
#pragma unroll
                for (int i = 0; i < PASSES; ++i) {
                    const int e = my_row + i * RPP;
                    const bool live = t * TOK_TILE + e < n_span;
                    const int64_t at = (int64_t)rowno[i] * D + my_chunk * 8;
                    cp_async16_zfill(kd + chunk_at<NC>(e, my_chunk), Kp + at, live);
                    cp_async16_zfill(vd + chunk_at<NC>(e, my_chunk), Vp + at, live);
                }
                if (tid < TOK_TILE) lw[stage * TOK_TILE + tid] = log2f(wt);
            }
            cp_async_commit();
        };
#pragma unroll
        for (int t = 0; t < TOK_STAGES - 1; ++t) {
            if (t < tiles) fetch_entries(t);
            fill(t);
        }
        if (TOK_STAGES - 1 < tiles) fetch_entries(TOK_STAGES - 1);
        uint64_t run[MT][NB][2];                                       // pairs of rows
        float M[NB], den[NB];
#pragma unroll
        for (int h = 0; h < NB; ++h) {
            M[h] = -INFINITY;
            den[h] = 0.f;
#pragma unroll
            for (int j = 0; j < MT; ++j) run[j][h][0] = run[j][h][1] = 0;
        }
        int in_unit = 0;
        for (int t = 0; t < tiles; ++t) {
            cp_async_wait<TOK_STAGES - 2>();
            __syncthreads();
            fill(t + TOK_STAGES - 1);                                  // (into the stage of the tile before)
            if (t + TOK_STAGES < tiles) fetch_entries(t + TOK_STAGES);
            const int stage = t % TOK_STAGES;
            const unsigned char *kt = smem + stage * 2 * C::TILE_BYTES;
            if (in_unit == 0) u.reset();
            if (t * TOK_TILE < last) {                                 // (behind what the group sees there is nothing to add)
                float s[4][4];
                uint64_t alpha[NB];
                float low;
                token_logits(s, qs, smem_u32(kt));
                token_softmax<D, NB>(u, in_unit == 0, s, lw + stage * TOK_TILE, t * TOK_TILE, lim, aligned, scale, alpha, low);
                token_values<true>(u, in_unit == 0, alpha, low, s, kt + C::TILE_BYTES, t * TOK_TILE, lim, aligned, n_span);
            }
            if (++in_unit == unit_tiles || t + 1 == tiles) {
                in_unit = 0;
                u.finish();
#pragma unroll
                for (int h = 0; h < NB; ++h) {
                    float fa, fb, x0, x1;
                    merge_factors(M[h], u.m[h], M[h], fa, fb);
                    den[h] = fmaf(fb, u.l[h], __fmul_rn(den[h], fa));
                    of_columns(fa, x0, x1);
                    const uint64_t a2 = pack2(x0, x1);
                    of_columns(fb, x0, x1);
                    const uint64_t b2 = pack2(x0, x1);
#pragma unroll
                    for (int j = 0; j < MT; ++j)
#pragma unroll
                        for (int i = 0; i < 2; ++i)
                            run[j][h][i] = fma2(b2, pack2(u.o[j][h][2 * i], u.o[j][h][2 * i + 1]), mul2(run[j][h][i], a2));
                }
            }
        }
        cp_async_wait<0>();
#pragma unroll
        for (int h = 0; h < NB; ++h) {
            float den2[2];
            of_columns(den[h], den2[0], den2[1]);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = 8 * h + 2 * quad + i;
                if (r >= rows) continue;
                __nv_bfloat16 *o = O + q_row(r) + (lane >> 2);
#pragma unroll
                for (int j = 0; j < 2 * MT; ++j) {
                    float x[2];
                    unpack2(run[j >> 1][h][j & 1], x[0], x[1]);
                    o[8 * j] = __float2bfloat16_rn(x[i] / den2[i]);
                }
            }
        }
    }
}

// elm_attend's lists: CTA (split, problem) takes its split's tiles, a warp every fourth of them, and leaves the merged result of its
// warps in part[problem][split][G][D + 2] (accumulator, maximum, denominator).  Bound by HBM latency and issue: three CTAs to an SM.
template <int D>
__global__ void __launch_bounds__(TOK_THREADS, 3)
tokens_split_kernel(const __nv_bfloat16 *__restrict__ Q, const __nv_bfloat16 *__restrict__ K, const __nv_bfloat16 *__restrict__ V,
                    const int32_t *__restrict__ idx, const float *__restrict__ w, int64_t n, int n_core, int q_heads, int kv_heads,
                    int n_q, int G, float *__restrict__ part, int *__restrict__ status)
{
    using C = TokenCfg<D>;
    constexpr int NC = C::NC;
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, quad = lane & 3;
    // (launched with programmatic stream serialization: nothing is read or written before this point)
    cudaGridDependencySynchronize();
#ifndef ELM_BOUNDS_CHECK
    if (tid == 0 && blockIdx.y == 0 && blockIdx.x == 0) *status = 0;
#endif
    const int prob = blockIdx.y, rep = q_heads / kv_heads, rows = rep * n_q;
    const int b = prob / kv_heads, kvh = prob % kv_heads;
    const int32_t *ip = idx + (int64_t)prob * n_core;
    const float *wp = w + (int64_t)prob * n_core;
    const __nv_bfloat16 *Kp = K + (int64_t)prob * n * D, *Vp = V + (int64_t)prob * n * D;
    const int tiles = (n_core + TOK_TILE - 1) / TOK_TILE, per = (tiles + (int)gridDim.x - 1) / (int)gridDim.x;
    const int t_end = min(((int)blockIdx.x + 1) * per, tiles);
    int t = (int)blockIdx.x * per + warp;
    unsigned char *kt = smem + warp * 2 * C::TILE_BYTES, *vt = kt + C::TILE_BYTES;
    float *lw = reinterpret_cast<float *>(smem + C::P_LW) + warp * TOK_TILE;
    int32_t row = 0;
    float wt = 0.f;
    auto fetch_entries = [&](int tile) {
        const int e = tile * TOK_TILE + lane;
        row = 0;
        wt = 0.f;
        if (e < n_core) {
            row = (int32_t)checked_row(__ldg(ip + e), n, status);
            wt = __ldg(wp + e);
        }
    };
    auto copy_rows = [&](unsigned char *dst, const __nv_bfloat16 *X, int32_t from, int tile) {
        const uint32_t d0 = smem_u32(dst);
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const int e = (lane + 32 * i) / NC, c = lane % NC;
            const int64_t r = __shfl_sync(0xffffffffu, from, e);
            cp_async16_zfill(d0 + chunk_at<NC>(e, c), X + r * D + c * 8, tile * TOK_TILE + e < n_core);
        }
        cp_async_commit();
    };
    TokenUnit<D, 1> u;
    u.reset();
    if (t < t_end) fetch_entries(t);
    TokenRawQueries<D, 1> raw;
    load_queries(raw, Q, rows, [&](int r) -> int64_t { return (((int64_t)b * q_heads + kvh * rep + r / n_q) * n_q + r % n_q) * D; });
    if (t < t_end) {
        copy_rows(kt, Kp, row, t);
        copy_rows(vt, Vp, row, t);
    }
    TokenQueries<D, 1, true> qs;
    qs.at = smem_u32(smem + C::P_Q + warp * TokenQueries<D, 1, true>::BYTES);
    put_queries(qs, raw);
    __syncwarp();
    const float scale = 8.f * 1.4426950408889634f / sqrtf((float)D);
    const int lim[1] = {n_core};
    for (bool head = true; t < t_end; t += TOK_WARPS, head = false) {
        const bool more = t + TOK_WARPS < t_end;
        float s[4][4];
        uint64_t alpha[1];
        float low;
        lw[lane] = log2f(wt);
        if (more) fetch_entries(t + TOK_WARPS);
        cp_async_wait<1>();                                        // the keys (the values are the newer group)
        __syncwarp();
        token_logits(s, qs, smem_u32(kt));
        __syncwarp();
        if (more) copy_rows(kt, Kp, row, t + TOK_WARPS);
        token_softmax<D, 1>(u, head, s, lw, t * TOK_TILE, lim, n_core, scale, alpha, low);
        if (more) cp_async_wait<1>();
        else cp_async_wait<0>();
        __syncwarp();
        token_values<false>(u, head, alpha, low, s, vt, t * TOK_TILE, lim, n_core, n_core);
        __syncwarp();
        if (more) copy_rows(vt, Vp, row, t + TOK_WARPS);
    }
    u.finish();
    // the warps' results over their own tiles, then their merge
    float *po = reinterpret_cast<float *>(kt);
    float2 *ml = reinterpret_cast<float2 *>(smem + C::P_ML);
    if (quad == 0) ml[warp * 8 + (lane >> 2)] = make_float2(u.m[0], u.l[0]);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < D / 8; ++j) po[(2 * quad + i) * D + 8 * j + (lane >> 2)] = u.o[j >> 1][0][2 * (j & 1) + i];
    __syncthreads();
    for (int i = tid; i < rows * D; i += TOK_THREADS) {
        const int g = i / D;
        float M = -INFINITY, acc = 0.f, den = 0.f;
#pragma unroll
        for (int v = 0; v < TOK_WARPS; ++v) M = fmaxf(M, ml[v * 8 + g].x);
#pragma unroll
        for (int v = 0; v < TOK_WARPS; ++v) {
            const float2 x = ml[v * 8 + g];
            const float f = x.x == -INFINITY ? 0.f : exp2f(x.x - M);
            acc = fmaf(f, reinterpret_cast<const float *>(smem + v * 2 * C::TILE_BYTES)[i], acc);
            den = fmaf(f, x.y, den);
        }
        float *out = part + (((int64_t)prob * gridDim.x + blockIdx.x) * G + g) * (D + 2);
        out[i % D] = acc;
        if (i % D == 0) { out[D] = M; out[D + 1] = den; }
    }
}

int tokens_per_group(int per_token)
{
    int t = 1;
    while (2 * t * per_token <= TOK_ROWS) t *= 2;
    return t;
}
// what the last token of window i sees, and the groups of `span` neighbouring tokens that its tokens fall into
int last_seen(const DecodeWindows &win, int i) { return win.seen0[i] + (win.tok0[i + 1] - win.tok0[i]) - 1; }
int token_groups(const DecodeWindows &win, int i, int span) { return (last_seen(win, i) - 1) / span - (win.seen0[i] - 1) / span + 1; }

bool tokens_serial(const DecodeWindows &win, int per_group, int problems, TokenCaps caps)
{
    // The serial form takes as long as one CTA needs for the longest list, 1.9 us a tile (2.5 where two CTAs share an SM), whatever few tokens
    // there are.  Clusters take 0.05 to 0.1 us per CTA, and the larger they are the fewer the device holds at once.  Measured, clusters
    // against serial, us (d = 64 has the same crossings at about 0.7 of the times):
    //   8 problems of 4 vectors, 64 tokens (136 clusters): 200 entries 26 / 27, 1000 61 / 73, 4100 184 / 254, 9000 238 / 540
    //   128 tokens (264 clusters): 200 entries 48 / 31, 1000 116 / 77, 4100 355 / 257, 9000 459 / 541; of 8 vectors (520): 9000 895 / 544
    //   32 problems of 4 vectors, 32 tokens (288 clusters): 1000 entries 113 / 71, 4100 188 / 252; 64 tokens (544): 4100 371 / 333, 9000 543 / 714
    //   32 problems of 1 vector, 64 tokens (160 clusters): 1000 entries 69 / 74; 128 tokens (288): 1000 122 / 78, 4100 206 / 259, 9000 300 / 544
    int longest = 0;
    int64_t clusters = 0;
    for (int i = 0; i < win.n; ++i) {
        const int last = last_seen(win, i);
        longest = last > longest ? last : longest;
        clusters += (int64_t)token_groups(win, i, per_group) * problems;
    }
    const int tiles = (longest + TOK_TILE - 1) / TOK_TILE, cap = longest <= TOKENS_SHORT_LIST ? caps.of_short : caps.of_long;
    // (calls of no more tokens than share a warp would leave three of the CTA's four idle)
    return win.tok0[win.n] > per_group && clusters > 9 * device_sm_count() / 10 + 12 * tiles / cap;
}

template <int D>
int launch_tokens(const void *Q, const void *K, const void *V, const int32_t *idx, const float *w, int64_t list_stride,
                  const DecodeWindows &win, const elm_params *p, void *O, int *status, TokenCaps caps, cudaStream_t st)
{
    using C = TokenCfg<D>;
    const int problems = p->batch * p->kv_heads, per_token = p->q_heads / p->kv_heads;
    TokenGroups grp = {};
    grp.caps = caps;
    grp.per_group = tokens_per_group(per_token);
    auto count = [&](int span) {
        grp.span = span;
        for (int i = 0; i < win.n; ++i) grp.g0[i + 1] = grp.g0[i] + token_groups(win, i, span);
        return grp.g0[win.n];
    };
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(TOK_THREADS);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const bool serial = tokens_serial(win, grp.per_group, problems, caps);
    auto kern = tokens_kernel<D, false, 2>;
    if (serial) {
        grp.cluster = 1;
        cfg.dynamicSmemBytes = C::S_TOTAL;
        cfg.gridDim = dim3((unsigned)count(TOK_WARPS * grp.per_group), (unsigned)problems);
    } else {
        int most = 1;
        count(grp.per_group);
        grp.cluster = 1;
        for (int i = 0; i < win.n; ++i) {
            const int tokens = win.tok0[i + 1] - win.tok0[i], size = tokens_cluster(win.seen0[i], win.seen0[i] + tokens - 1, caps);
            grp.cluster = size > grp.cluster ? size : grp.cluster;
            most = tokens > most ? tokens : most;
        }
        const bool few = (most < grp.per_group ? most : grp.per_group) * per_token <= 8;
        kern = few ? tokens_kernel<D, true, 1> : tokens_kernel<D, true, 2>;
        cfg.dynamicSmemBytes = few ? C::template Cluster<8>::TOTAL : C::template Cluster<16>::TOTAL;
        if (grp.cluster > 8) ELM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)grp.cluster;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
        cfg.gridDim = dim3((unsigned)(grp.g0[win.n] * grp.cluster), (unsigned)problems);
    }
    ELM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes));
    typedef __nv_bfloat16 bf;
    ELM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, (const bf *)Q, (const bf *)K, (const bf *)V, idx, w, (int64_t)p->n_kv, list_stride,
                                    (int)p->q_heads, (int)p->kv_heads, per_token, win, grp, (bf *)O, status));
    count_launches(1);
    return cuda_status(cudaGetLastError());
}

}  // namespace

// Clusters of `size` CTAs that the current device holds at once, asked once per device (0: the size cannot be placed at all)
static int tokens_clusters(int d, int size)
{
    static std::atomic<int> cached[64][2][5];                      // answer + 1 (threads that meet here first find the same)
    int dev = 0, log = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return size == 1 ? 1 : 0;
    while (1 << log < size) ++log;
    std::atomic<int> &slot = cached[dev][d == 64 ? 0 : 1][log];
    int n = slot.load(std::memory_order_relaxed) - 1;
    if (n < 0) {
        n = d == 64 ? resident_clusters(tokens_kernel<64, true, 2>, TOK_THREADS, TokenCfg<64>::Cluster<16>::TOTAL, size)
                    : resident_clusters(tokens_kernel<128, true, 2>, TOK_THREADS, TokenCfg<128>::Cluster<16>::TOTAL, size);
        slot.store(n + 1, std::memory_order_relaxed);
    }
    return n;
}

TokenCaps tokens_caps(int d, int problems, int limit)
{
    // as many CTAs as leave all problems' clusters resident
    int cap = limit < TOK_MAX_CLUSTER ? limit : TOK_MAX_CLUSTER;
    while (cap > 1 && tokens_clusters(d, cap) < problems) cap >>= 1;
    // Up to 4096 entries clusters of 16 gain nothing over 8 with twice the tiles per warp (8 problems of 4 query vectors, one token: 2000 entries
    // 10.3 against 9.2 us, 4000 12.1 / 11.9, 5000 13.7 / 13.4; 8 tokens: 4000 entries 32.8 / 22.5; 8 problems of one vector: 4000 11.1 / 11.6, 5000
    // 12.6 / 13.2; d = 64, 4 vectors: 4000 9.6 / 9.8).
    return {cap < 8 ? cap : 8, cap};
}

bool attend_tokens_serial(const DecodeWindows &win, const elm_params *p, TokenCaps caps)
{
    return tokens_serial(win, tokens_per_group(p->q_heads / p->kv_heads), p->batch * p->kv_heads, caps);
}

int attend_tokens_bf16(const void *Q, const void *K, const void *V, const int32_t *idx, const float *w, int64_t list_stride,
                       const DecodeWindows &win, const elm_params *p, void *O, int *status, TokenCaps caps, cudaStream_t st)
{
    return p->d == 64 ? launch_tokens<64>(Q, K, V, idx, w, list_stride, win, p, O, status, caps, st)
                      : launch_tokens<128>(Q, K, V, idx, w, list_stride, win, p, O, status, caps, st);
}

cudaError_t tokens_split_occupancy(int d, int *ctas_per_sm)
{
    if (d == 64) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, tokens_split_kernel<64>, TOK_THREADS, TokenCfg<64>::P_TOTAL);
    const cudaError_t e = cudaFuncSetAttribute(tokens_split_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, TokenCfg<128>::P_TOTAL);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, tokens_split_kernel<128>, TOK_THREADS, TokenCfg<128>::P_TOTAL);
}

int launch_tokens_split(const void *Q, const void *K, const void *V, const int32_t *idx, const float *w, int n_core, int splits, int G,
                        const elm_params *p, float *part, int *status, cudaStream_t st)
{
    typedef __nv_bfloat16 bf;
    auto kern = p->d == 64 ? tokens_split_kernel<64> : tokens_split_kernel<128>;
    const int smem = p->d == 64 ? TokenCfg<64>::P_TOTAL : TokenCfg<128>::P_TOTAL;
    ELM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    ELM_CUDA_TRY(launch_after(kern, dim3((unsigned)splits, (unsigned)(p->batch * p->kv_heads)), dim3(TOK_THREADS), (size_t)smem, st, (const bf *)Q,
                              (const bf *)K, (const bf *)V, idx, w, (int64_t)p->n_kv, n_core, (int)p->q_heads, (int)p->kv_heads, (int)p->n_q, G,
                              part, status));
    return ELM_OK;
}

}  // namespace elm
