// Weighted attention over a coreset for a few queries per head (decode: one new token, or a handful):
//   O[j,:] = sum_c w_c exp(<q_j,k_c>/sqrt(d)) v_c / sum_c w_c exp(<q_j,k_c>/sqrt(d))      Eq. (def:att_approx)
// With so few queries the work is reading each coreset row of K and V once: HBM-bound, and far too
// small for the tile kernels.  All query heads that share the KV head (and all their query rows: G vectors
// in total, G <= 8) are processed together, so a row is read once for the whole group.  Rows are read through
// the index list straight from K and V (no gathered copy).  fp32 arithmetic on fp32 or bf16 inputs.  On bf16 inputs streaming
// tokens, and lists of three query vectors and more that are not short, go to the kernels of elm_attend_tokens.cu instead.
//
// A warp takes a tile of 32 list entries (16 when a row is 512 bytes, 8 of a short list): the tile's K and V rows come to shared memory
// by asynchronous copies (the next tile's keys are requested as soon as this tile's logits are formed, its values
// behind this tile's), eight lanes share a key row, and their partial dot products are reduced AND distributed in
// one butterfly, so that a lane ends with finished logits of its own - 14 shuffles per 16 entries of four queries
// where a butterfly that leaves every sum in every lane needs 20 per entry.  The softmax of a tile is one entry per
// lane; for the values a lane owns one 16-byte chunk of the row.  The instruction count per entry is what decides
// here: a version with one entry per warp at a time and the softmax repeated in every lane issued about 120
// instructions per entry of four queries, this one about 45.
//
// The list of an attention problem is split over CTAs.  elm_attend: over as many as the SMs can hold, which leave
// partial results (maximum, denominator, accumulator) in the workspace for decode_merge_kernel.  Tokens of a streaming
// run (DecodeWindows: a token sees a prefix of its window's list): each over the CTAs of a thread-block cluster, which
// hand each other their partial results through distributed shared memory, or, once there are tokens enough to fill the
// SMs, by one CTA that walks the parts of the list one after the other - the same parts, tiles and merges in the same
// order as the cluster's, so a token's output is the same bit for bit whichever launch computes it.  How many of a
// token's query vectors go together is free too (decode_form).
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
using sm100::smem_u32;
using sm100::unpack2;

constexpr int DEC_WARPS = 4;
constexpr int DEC_GMAX = 8;
constexpr int DEC_GSTREAM = 4;         // most query vectors a CTA of a streaming token takes
constexpr int DEC_MAX_CLUSTER = 16;
constexpr int DEC_CTAS = 3;                                      // CTAs per SM the kernel is compiled for

// grid (splits, problems); partial results part[problem][split][g][D + 2] = accumulator (D), maximum, denominator
constexpr int DEC_SPLIT = 0;
// grid (tokens x vec_groups x cluster size, problems): rank r of a cluster takes the r-th part of its token's list
constexpr int DEC_CLUSTER = 1;
// grid (tokens x vec_groups, problems): a token's parts one after the other
constexpr int DEC_TOKENS = 2;
// grid (groups, problems): the same for neighbouring tokens whose query vectors fit G together
constexpr int DEC_NEIGHBOURS = 3;

// entries of a warp's tile: 16 when a row is 512 bytes, else 32; 8 for lists so short that the SMs would have nothing else
template <typename Tin, int D> constexpr int DEC_TILE = D * (int)sizeof(Tin) > 256 ? 16 : 32;
constexpr int DEC_SHORT_TILE = 8;

template <typename Tin, int D, int G, int TILE_ = DEC_TILE<Tin, D>> struct DecodeCfg {
    static constexpr int RB = D * (int)sizeof(Tin);              // bytes per row
    static constexpr int EPC = 16 / (int)sizeof(Tin);            // elements per 16-byte chunk
    static constexpr int NC = RB / 16;                           // chunks per row: 8, 16 or 32
    static constexpr int CH = NC / 8;                            // chunks of a key row per lane (eight lanes share a row)
    static constexpr int TILE = TILE_;                           // entries per warp tile
    static constexpr int UB = G == 8 || TILE == DEC_SHORT_TILE ? 2 : 4;      // entries whose dot products a lane forms at a time
    static constexpr int NV = UB * G;                            // partial sums per lane: 4, 8 or 16
    static constexpr int EPI = 32 / NC;                          // entries a warp takes at a time in the value pass
    static constexpr int TILE_BYTES = TILE * RB;
    static_assert(2 * TILE_BYTES >= G * D * 4, "a warp's partial results lie over its tiles");
    // shared memory: per warp a K tile, a V tile and the tile's logits; the scaled queries; what a form needs besides
    static constexpr int OFF_SC = DEC_WARPS * 2 * TILE_BYTES;
    static constexpr int OFF_Q = OFF_SC + DEC_WARPS * 32 * G * 4;
    static constexpr int OFF_ML = OFF_Q + G * D * 4;             // [DEC_WARPS][G][2]
    // DEC_CLUSTER: what the other ranks send, [DEC_MAX_CLUSTER][G][2] and [ranks][slice] with slice = ceil(G D / ranks),
    // at most G D + DEC_MAX_CLUSTER floats.  DEC_TOKENS, DEC_NEIGHBOURS: the running maxima and denominators, [2][G][2].
    static constexpr int OFF_RML = OFF_ML + DEC_WARPS * G * 2 * 4;
    static constexpr int OFF_RECV = OFF_RML + DEC_MAX_CLUSTER * G * 2 * 4;
    template <int MODE> static constexpr int total()
    {
        return MODE == DEC_SPLIT ? OFF_RML : MODE == DEC_CLUSTER ? OFF_RECV + (G * D + DEC_MAX_CLUSTER) * 4 : OFF_RML + 2 * G * 2 * 4;
    }
    // DEC_CTAS to an SM: of its 228 KB the system takes 1 KB per CTA (at G = 8 and D = 128 two CTAs against three cost 1.2
    // times the time, 8 problems x 5193 entries: 24.0 against 20.0 us)
    template <int MODE> static constexpr bool fits = DEC_CTAS * (total<MODE>() + 1024) <= 228 * 1024;
};

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void *src, bool live)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// the elements of a 16-byte chunk as packed pairs of floats
__device__ __forceinline__ void chunk_pairs(const uint4 &x, uint64_t (&f)[4], const __nv_bfloat16 *)
{
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = pack2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
}
__device__ __forceinline__ void chunk_pairs(const uint4 &x, uint64_t (&f)[2], const float *)
{
    f[0] = pack2(__uint_as_float(x.x), __uint_as_float(x.y));
    f[1] = pack2(__uint_as_float(x.z), __uint_as_float(x.w));
}

// folds a part's (maximum, denominator, accumulator) into the running ones
__device__ __forceinline__ void merge_part(float &M, float &den, float &acc, float m, float d, float x)
{
    const float Mn = fmaxf(M, m);
    const float a = M == -INFINITY ? 0.f : exp2f(M - Mn), b = m == -INFINITY ? 0.f : exp2f(m - Mn);
    den = fmaf(b, d, __fmul_rn(den, a));
    acc = fmaf(b, x, __fmul_rn(acc, a));
    M = Mn;
}

// The groups of tokens of a streaming launch, and of a token's query vectors
struct DecodeGroups {
    int32_t cluster;                               // CTAs per group
    int32_t vec_groups;                            // groups a token's query vectors are dealt to, G to each
    int32_t per_group;                             // tokens per group: a power of two, 1 but in DEC_NEIGHBOURS
    int32_t g0[DECODE_MAX_WINDOWS + 1];            // groups of tokens in the windows before
};

// How a list of n_core entries is parted: parts of whole tiles, at least two tiles per warp (with one, a single token over
// 200 entries takes 5.8 us for 6.9, less than the host needs to enqueue it, but a CTA that walks all parts has twice the
// merges: 2000 tokens of 8 KV heads of 4 query heads, n_out = 128, 1010 us for 960; measured on bf16 rows, which took this form then),
// at most `cap` parts.  Depends on n_core only through the next multiple of 128, so that neighbouring tokens share their parts.
__host__ __device__ __forceinline__ void decode_parts(int n_core, int cta_entries, int tile, int cap, int &parts, int &chunk)
{
    const int len = (n_core + 127) / 128 * 128;
    const int t = (len + 2 * cta_entries - 1) / (2 * cta_entries);
    parts = t < 1 ? 1 : (t < cap ? t : cap);
    chunk = ((len + parts - 1) / parts + tile - 1) / tile * tile;
}

template <typename Tin, int D, int G, int MODE, int TILE = DEC_TILE<Tin, D>>
__global__ void __launch_bounds__(DEC_WARPS * 32, DEC_CTAS)
decode_kernel(const Tin *__restrict__ Q, const Tin *__restrict__ K, const Tin *__restrict__ V,
              const int32_t *__restrict__ idx, const float *__restrict__ w, int64_t n, int64_t list_stride, int q_heads,
              int kv_heads, int n_q, int per_token /* query vectors of a token */, const __grid_constant__ DecodeWindows win,
              const __grid_constant__ DecodeGroups grp, int cap, Tin *__restrict__ O, float *__restrict__ part,
              int *__restrict__ status)
{
    using C = DecodeCfg<Tin, D, G, TILE>;
    constexpr int NC = C::NC, CH = C::CH, EPC = C::EPC, UB = C::UB, NV = C::NV, EPI = C::EPI;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char *kt = smem + warp * 2 * C::TILE_BYTES, *vt = kt + C::TILE_BYTES;
    float *sc = reinterpret_cast<float *>(smem + C::OFF_SC) + warp * 32 * G;      // [entry][g] logits, then probabilities
    float *qs = reinterpret_cast<float *>(smem + C::OFF_Q);
    float *ml = reinterpret_cast<float *>(smem + C::OFF_ML);
    float *recv = reinterpret_cast<float *>(smem + C::OFF_RECV), *rml = reinterpret_cast<float *>(smem + C::OFF_RML);
    // (launched with programmatic stream serialization: resident before the kernel in front of it has finished;
    // nothing is read or written before this point)
    cudaGridDependencySynchronize();
    if constexpr (MODE == DEC_CLUSTER) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    constexpr bool SERIAL = MODE == DEC_TOKENS || MODE == DEC_NEIGHBOURS;
    static_assert(C::template fits<MODE>, "shared memory for as many CTAs as there are registers for");
    const int prob = blockIdx.y;
    int group = MODE == DEC_SPLIT ? 0 : (int)blockIdx.x / grp.cluster;
    const int rank = (int)blockIdx.x - group * grp.cluster;
    // the group's query vectors of its token: vec0 .. vec0 + G - 1
    int vec0 = 0;
    if constexpr (MODE == DEC_CLUSTER || MODE == DEC_TOKENS) {
        vec0 = group % grp.vec_groups * G;
        group /= grp.vec_groups;
    }
#ifndef ELM_BOUNDS_CHECK
    // this path has no bounded waits and (in this build) no row checks: its status word reads 0 - written here
    // rather than by a memset of its own
    if (tid == 0 && prob == 0 && blockIdx.x == 0) *status = 0;
#endif
    // the tokens: z0 .. z0 + tokens - 1 of the launch, the first of which sees seen0 entries, the next one more, ...
    int wi = 0, z0 = 0, tokens = 1, seen0 = win.seen0[0];
    if constexpr (MODE != DEC_SPLIT) {
        while (wi + 1 < win.n && group >= grp.g0[wi + 1]) ++wi;
        // group k of a window: the tokens that see (k0 + k) per_group + 1 .. (k0 + k + 1) per_group entries
        const int first = ((win.seen0[wi] - 1) / grp.per_group + (group - grp.g0[wi])) * grp.per_group + 1;
        const int last_seen = win.seen0[wi] + (win.tok0[wi + 1] - win.tok0[wi]) - 1;
        seen0 = first > win.seen0[wi] ? first : win.seen0[wi];
        const int end = first + grp.per_group - 1 < last_seen ? first + grp.per_group - 1 : last_seen;
        tokens = end - seen0 + 1;
        z0 = win.tok0[wi] + (seen0 - win.seen0[wi]);
    }
    const int n_core = seen0 + tokens - 1;                         // what the last token sees
    const int groups = tokens * per_token - vec0;                  // live query vectors (of G, if they are more)
    int parts, chunk;
    if constexpr (MODE == DEC_SPLIT) {
        // whole tiles per part, so that only the end of the list leaves a tile partly filled
        parts = gridDim.x;
        chunk = ((n_core + parts - 1) / parts + TILE - 1) / TILE * TILE;
    } else {
        decode_parts(n_core, DEC_WARPS * TILE, TILE, cap, parts, chunk);
    }
    const int b = prob / kv_heads, kvh = prob % kv_heads, rep = q_heads / kv_heads;
    const int32_t *ip = idx + (int64_t)prob * list_stride + win.off[wi];
    const float *wp = w + (int64_t)prob * list_stride + win.off[wi];
    const Tin *Kp = K + (int64_t)prob * n * D, *Vp = V + (int64_t)prob * n * D;
    // offset of query vector g's row in Q and O: token g / per_token, in it (head within the group) * n_q + row
    auto q_row = [&](int g) -> int64_t {
        const int64_t z = MODE == DEC_NEIGHBOURS ? z0 + g / per_token : z0;
        const int in = MODE == DEC_NEIGHBOURS ? g % per_token : vec0 + g;
        return (((z * (gridDim.y / kv_heads) + b) * q_heads + kvh * rep + in / n_q) * n_q + in % n_q) * D;
    };
    int c0, c1 = 0;                                                // the part being worked on

    // row number and log2 weight of the tile's entry `lane`
    int32_t row = 0, row_next = 0;
    float lw = 0.f, lw_next = 0.f;
    auto fetch_entries = [&](int t0) {
        row_next = 0;
        lw_next = -INFINITY;
        if (lane < TILE && t0 + lane < c1) {
            row_next = (int32_t)checked_row(__ldg(ip + t0 + lane), n, status);
            lw_next = __ldg(wp + t0 + lane);
        }
    };
    // the rows of a tile, chunk by chunk: chunk q = lane + 32 i of the tile lies in entry q / NC.  Entries past the end
    // read as zeros, so that nothing they might hold meets their zero probability.
    auto copy_rows = [&](unsigned char *dst, const Tin *X, int32_t rows, int t0) {
        const uint32_t d0 = smem_u32(dst);
#pragma unroll
        for (int i = 0; i < TILE / EPI; ++i) {
            const int e = lane / NC + i * EPI;
            const int64_t r = __shfl_sync(0xffffffffu, rows, e);
            cp_async16_zfill(d0 + (lane + 32 * i) * 16, X + r * D + (lane % NC) * EPC, t0 + e < c1);
        }
        cp_async_commit();
    };
    // the query vectors, scaled; laid out so that the eight lanes of a key row read
    // 128 contiguous bytes: [g][chunk / 8][16-byte half][chunk % 8][4]
    const float scale = 1.4426950408889634f / sqrtf((float)D);
    for (int i = tid; i < G * D; i += DEC_WARPS * 32) {
        const int g = i / D, dim = i % D, ck = dim / EPC, in = dim % EPC;
        float x = 0.f;
        if (g < groups) x = load_as<float>(Q, q_row(g) + dim) * scale;
        qs[(((g * CH + ck / 8) * (EPC / 4) + in / 4) * 8 + ck % 8) * 4 + in % 4] = x;
    }
    // SERIAL: the running accumulators, element tid + 128 k of [g][D]
    constexpr int EPT = (G * D + DEC_WARPS * 32 - 1) / (DEC_WARPS * 32);
    float run[SERIAL ? EPT : 1];
    if constexpr (SERIAL) {
#pragma unroll
        for (int k = 0; k < EPT; ++k) run[k] = 0.f;
        if (tid < G) { rml[tid * 2] = -INFINITY; rml[tid * 2 + 1] = 0.f; }
    }
    // what query vector g sees of the list: its token's prefix
    auto limit = [&](int g) { return MODE == DEC_NEIGHBOURS ? seen0 + g / per_token : n_core; };
    const int gl = lane >> 3, sub = lane & 7;

    for (int pt = rank; pt < (SERIAL ? parts : rank + 1); ++pt) {
        c0 = pt * chunk < n_core ? pt * chunk : n_core;
        c1 = pt < parts ? (c0 + chunk < n_core ? c0 + chunk : n_core) : c0;
        int t0 = c0 + warp * TILE;
        fetch_entries(t0);
        row = row_next;
        lw = log2f(lw_next);
        // (the queries are laid out / the merge of the part before has read the tiles)
        __syncthreads();
        if (t0 < c1) {
            copy_rows(kt, Kp, row, t0);
            copy_rows(vt, Vp, row, t0);
            fetch_entries(t0 + DEC_WARPS * TILE);
        }
        float m[G], l[G];
        uint64_t o[G][EPC / 2];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            m[g] = -INFINITY;
            l[g] = 0.f;
#pragma unroll
            for (int i = 0; i < EPC / 2; ++i) o[g][i] = 0;
        }
        for (; t0 < c1; t0 += DEC_WARPS * TILE) {
            const bool more = t0 + DEC_WARPS * TILE < c1;
            // ---- logits: entry gl + 4 u of the tile by the eight lanes of group gl ----
            cp_async_wait<1>();                                        // the keys (the values are the newer group)
            __syncwarp();
#pragma unroll
            for (int ub = 0; ub < TILE / 4 / UB; ++ub) {
                uint64_t acc[UB][G];
#pragma unroll
                for (int u = 0; u < UB; ++u)
#pragma unroll
                    for (int g = 0; g < G; ++g) acc[u][g] = 0;
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    uint64_t kf[UB][EPC / 2];
#pragma unroll
                    for (int u = 0; u < UB; ++u) {
                        const int e = gl + 4 * (ub * UB + u);
                        chunk_pairs(*reinterpret_cast<const uint4 *>(kt + (e * NC + c * 8 + sub) * 16), kf[u], (const Tin *)nullptr);
                    }
#pragma unroll
                    for (int g = 0; g < G; ++g) {
#pragma unroll
                        for (int h = 0; h < EPC / 4; ++h) {
                            const float4 q4 = *reinterpret_cast<const float4 *>(qs + (((g * CH + c) * (EPC / 4) + h) * 8 + sub) * 4);
                            const uint64_t qa = pack2(q4.x, q4.y), qb = pack2(q4.z, q4.w);
#pragma unroll
                            for (int u = 0; u < UB; ++u) acc[u][g] = fma2(kf[u][2 * h + 1], qb, fma2(kf[u][2 * h], qa, acc[u][g]));
                        }
                    }
                }
                // reduce over the eight lanes and leave each with its share of the NV sums
                float v[NV];
#pragma unroll
                for (int u = 0; u < UB; ++u)
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        float lo, hi;
                        unpack2(acc[u][g], lo, hi);
                        v[u * G + g] = lo + hi;
                    }
                int base = 0;
                {
                    int cnt = NV;
#pragma unroll
                    for (int off = 4; off > 0; off >>= 1) {
                        if (cnt >= 2) {
                            const bool up = (sub & off) != 0;
                            cnt >>= 1;
#pragma unroll
                            for (int i = 0; i < NV / 2; ++i) {
                                if (i < cnt) {
                                    const float send = up ? v[i] : v[i + cnt], keep = up ? v[i + cnt] : v[i];
                                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                                }
                            }
                            base += up ? cnt : 0;
                        } else {
                            v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
                        }
                    }
                }
                constexpr int LEFT = NV >= 8 ? NV / 8 : 1;             // finished sums in this lane
#pragma unroll
                for (int i = 0; i < LEFT; ++i) {
                    const int j = base + i, u = j / G, g = j % G;
                    sc[(gl + 4 * (ub * UB + u)) * G + g] = v[i];
                }
            }
            __syncwarp();
            const int32_t row_ahead = row_next;
            const float lw_ahead = lw_next;
            if (more) copy_rows(kt, Kp, row_ahead, t0 + DEC_WARPS * TILE);
            // ---- softmax of the tile, one entry per lane ----
            float alpha[G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const bool live = lane < TILE && t0 + lane < (MODE == DEC_NEIGHBOURS ? min(c1, limit(g)) : c1);
                const float s = live ? sc[lane * G + g] + lw : -INFINITY;            // base-2 logit
                float mx = s;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
                mx = fmaxf(m[g], mx);
                const float ref = mx == -INFINITY ? 0.f : mx;
                alpha[g] = exp2f(m[g] - ref);                                        // exp2f(-inf) = 0 on the first tile
                const float pw = live ? exp2f(s - ref) : 0.f;
                l[g] = fmaf(l[g], alpha[g], pw);
                m[g] = mx;
                sc[lane * G + g] = pw;
            }
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const uint64_t a2 = pack2(alpha[g], alpha[g]);
#pragma unroll
                for (int i = 0; i < EPC / 2; ++i) o[g][i] = mul2(o[g][i], a2);
            }
            // ---- values: lane owns chunk lane % NC of a row, EPI entries at a time ----
            if (more) cp_async_wait<1>();                              // (the next tile's keys may still be on their way)
            else cp_async_wait<0>();
            __syncwarp();
            const int filled = c1 - t0 < TILE ? c1 - t0 : TILE;
#pragma unroll 4
            for (int i = 0; i < TILE / EPI; ++i) {
                if (i * EPI >= filled) break;
                const int e = i * EPI + lane / NC;
                uint64_t vf[EPC / 2];
                chunk_pairs(*reinterpret_cast<const uint4 *>(vt + (lane + 32 * i) * 16), vf, (const Tin *)nullptr);
                float pe[G];
                if constexpr (G >= 4) {
#pragma unroll
                    for (int g = 0; g < G; g += 4) {
                        const float4 p4 = *reinterpret_cast<const float4 *>(sc + e * G + g);
                        pe[g] = p4.x; pe[g + 1] = p4.y; pe[g + 2] = p4.z; pe[g + 3] = p4.w;
                    }
                } else {
#pragma unroll
                    for (int g = 0; g < G; ++g) pe[g] = sc[e * G + g];
                }
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    // (an entry behind the token's own must not meet its zero probability: it might be infinite)
                    if (MODE == DEC_NEIGHBOURS && t0 + TILE > seen0 && t0 + e >= limit(g)) continue;
                    const uint64_t p2 = pack2(pe[g], pe[g]);
#pragma unroll
                    for (int j = 0; j < EPC / 2; ++j) o[g][j] = fma2(p2, vf[j], o[g][j]);
                }
            }
            __syncwarp();
            if (more) {
                copy_rows(vt, Vp, row_ahead, t0 + DEC_WARPS * TILE);
                lw = log2f(lw_ahead);
                fetch_entries(t0 + 2 * DEC_WARPS * TILE);
            }
        }

        // ---- the warp's partial result, over its own tiles ----
        float *po = reinterpret_cast<float *>(kt);                     // [g][D]
#pragma unroll
        for (int g = 0; g < G; ++g) {
            float ls = l[g];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, off);
            if (lane == 0) {
                ml[(warp * G + g) * 2] = m[g];
                ml[(warp * G + g) * 2 + 1] = ls;
            }
#pragma unroll
            for (int i = 0; i < EPC / 2; ++i) {
                float x, y;
                unpack2(o[g][i], x, y);
#pragma unroll
                for (int off = NC; off < 32; off <<= 1) {
                    x += __shfl_xor_sync(0xffffffffu, x, off);
                    y += __shfl_xor_sync(0xffffffffu, y, off);
                }
                if (lane < NC) *reinterpret_cast<float2 *>(po + g * D + lane * EPC + 2 * i) = make_float2(x, y);
            }
        }
        __syncthreads();
        // ---- the part's result: to the workspace, to the cluster rank that finishes this slice of the output, or merged
        // into what the parts before left ----
        const int slice = (G * D + parts - 1) / parts;
        // every CTA of the cluster is running (its shared memory may be written) once this wait is over
        if constexpr (MODE == DEC_CLUSTER) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        auto remote = [&](const float *mine, int to) -> uint32_t {
            uint32_t a;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(mine)), "r"(to));
            return a;
        };
        if (pt < parts) {
#pragma unroll
            for (int k = 0; k < EPT; ++k) {
                const int i = tid + k * DEC_WARPS * 32;
                if (i >= G * D) break;
                const int g = i / D;
                float M = -INFINITY;
#pragma unroll
                for (int wv = 0; wv < DEC_WARPS; ++wv) M = fmaxf(M, ml[(wv * G + g) * 2]);
                float acc = 0.f, den = 0.f;
#pragma unroll
                for (int wv = 0; wv < DEC_WARPS; ++wv) {
                    const float mw = ml[(wv * G + g) * 2];
                    const float f = mw == -INFINITY ? 0.f : exp2f(mw - M);
                    acc = fmaf(f, reinterpret_cast<const float *>(smem + wv * 2 * C::TILE_BYTES)[i], acc);
                    den = fmaf(f, ml[(wv * G + g) * 2 + 1], den);
                }
                if constexpr (MODE == DEC_CLUSTER) {
                    const int to = i / slice;
                    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote(recv + rank * slice + i - to * slice, to)), "f"(acc) : "memory");
                    if (i % D < parts) {                               // (parts <= 16 <= D: one thread per (g, rank))
                        const uint32_t a = remote(rml + (rank * G + g) * 2, i % D);
                        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(M) : "memory");
                        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a + 4), "f"(den) : "memory");
                    }
                } else if constexpr (SERIAL) {
                    // (running maximum and denominator in two buffers, part pt reading one and writing the other)
                    const float *was = rml + ((pt & 1) * G + g) * 2;
                    float Mr = was[0], dr = was[1];
                    merge_part(Mr, dr, run[k], M, den, acc);
                    if (i % D == 0) {
                        float *now = rml + (((pt + 1) & 1) * G + g) * 2;
                        now[0] = Mr;
                        now[1] = dr;
                    }
                } else {
                    float *out = part + (((int64_t)prob * gridDim.x + rank) * G + g) * (D + 2);
                    out[i % D] = acc;
                    if (i % D == 0) { out[D] = M; out[D + 1] = den; }
                }
            }
        }
        if constexpr (MODE == DEC_CLUSTER) {
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
            const int i1 = (rank + 1) * slice < G * D ? (rank + 1) * slice : G * D;
            if (rank < parts) {
                for (int i = rank * slice + tid; i < i1; i += DEC_WARPS * 32) {
                    const int g = i / D;
                    if (g >= groups) break;
                    float M = -INFINITY, den = 0.f, acc = 0.f;
                    for (int r = 0; r < parts; ++r)
                        merge_part(M, den, acc, rml[(r * G + g) * 2], rml[(r * G + g) * 2 + 1], recv[r * slice + i - rank * slice]);
                    store_from(O, q_row(g) + i % D, acc / den);
                }
            }
        }
    }
    if constexpr (SERIAL) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
            const int i = tid + k * DEC_WARPS * 32;
            if (i < G * D && i < groups * D) store_from(O, q_row(i / D) + i % D, run[k] / rml[((parts & 1) * G + i / D) * 2 + 1]);
        }
    }
}

// One CTA per (problem, query vector), one thread per dimension.  The splits' maxima and denominators are read
// by one thread each and combined through shared memory, and the accumulators with several loads in flight: the
// kernel is a chain of memory round trips and nothing else, so it is laid out to make that chain three long
// whatever the number of splits (a loop over the splits with one load per turn took 13 us for 37 splits).
constexpr int DEC_MAX_SPLITS = 256;
template <typename Tin, int D, int G>
__global__ void __launch_bounds__(D) decode_merge_kernel(const float *__restrict__ part, int splits, int q_heads, int kv_heads,
                                                         int n_q, Tin *__restrict__ O)
{
    __shared__ float sf[DEC_MAX_SPLITS];
    __shared__ float red[2][D / 32];
    const int prob = blockIdx.y, g = blockIdx.x, d = threadIdx.x;
    const int warp = d >> 5, lane = d & 31;
    const int b = prob / kv_heads, kvh = prob % kv_heads, rep = q_heads / kv_heads;
    const float *p = part + ((int64_t)prob * splits * G + g) * (D + 2);
    // launched with programmatic stream serialization: the CTAs of this kernel are resident while the partial
    // kernel still runs and wait here for its results, so the gap between the two launches is not on the path
    cudaGridDependencySynchronize();
    // thread s (and s + D, ...) fetches split s's maximum and denominator
    float M = -INFINITY;
    float ms[(DEC_MAX_SPLITS + D - 1) / D], ls[(DEC_MAX_SPLITS + D - 1) / D];
#pragma unroll
    for (int i = 0; i < (DEC_MAX_SPLITS + D - 1) / D; ++i) {
        const int sp = d + i * D;
        ms[i] = -INFINITY;
        ls[i] = 0.f;
        if (sp < splits) {
            ms[i] = __ldg(p + (int64_t)sp * G * (D + 2) + D);
            ls[i] = __ldg(p + (int64_t)sp * G * (D + 2) + D + 1);
        }
        M = fmaxf(M, ms[i]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    if (lane == 0) red[0][warp] = M;
    __syncthreads();
    M = red[0][0];
#pragma unroll
    for (int i = 1; i < D / 32; ++i) M = fmaxf(M, red[0][i]);
    float den = 0.f;
#pragma unroll
    for (int i = 0; i < (DEC_MAX_SPLITS + D - 1) / D; ++i) {
        const int sp = d + i * D;
        if (sp < splits) {
            const float f = ms[i] == -INFINITY ? 0.f : exp2f(ms[i] - M);
            sf[sp] = f;
            den += f * ls[i];
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) den += __shfl_xor_sync(0xffffffffu, den, off);
    if (lane == 0) red[1][warp] = den;
    __syncthreads();
    den = 0.f;
#pragma unroll
    for (int i = 0; i < D / 32; ++i) den += red[1][i];
    float acc = 0.f;
    int s0 = 0;
    for (; s0 + 8 <= splits; s0 += 8) {
        float x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = __ldg(p + (int64_t)(s0 + j) * G * (D + 2) + d);
#pragma unroll
        for (int j = 0; j < 8; ++j) acc = fmaf(sf[s0 + j], x[j], acc);
    }
    for (; s0 < splits; ++s0) acc = fmaf(sf[s0], __ldg(p + (int64_t)s0 * G * (D + 2) + d), acc);
    const int h = kvh * rep + g / n_q, r = g % n_q;
    store_from(O, (((int64_t)b * q_heads + h) * n_q + r) * D + d, acc / den);
}

// Calls `f` with the compile-time query count that covers `groups`
template <typename F> auto with_groups(int groups, F f)
{
    if (groups <= 1) return f(std::integral_constant<int, 1>());
    if (groups <= 2) return f(std::integral_constant<int, 2>());
    if (groups <= 4) return f(std::integral_constant<int, 4>());
    return f(std::integral_constant<int, 8>());
}

// The largest cluster (a power of two, at most DEC_MAX_CLUSTER) of which the current device can hold one, asked once per
// device.
std::atomic<int> g_debug_largest_cluster{0};
template <int D> int decode_largest_cluster()
{
    static std::atomic<int> cached[64];                            // (threads that meet here first find the same answer)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
    int largest = cached[dev].load(std::memory_order_relaxed);
    if (largest == 0) {
        using C = DecodeCfg<float, D, DEC_GSTREAM>;
        for (largest = DEC_MAX_CLUSTER; largest > 1; largest >>= 1)
            if (resident_clusters(decode_kernel<float, D, DEC_GSTREAM, DEC_CLUSTER>, DEC_WARPS * 32, C::template total<DEC_CLUSTER>(), largest)) break;
        cached[dev].store(largest, std::memory_order_relaxed);
    }
    const int limit = g_debug_largest_cluster.load(std::memory_order_relaxed);
    return limit && limit < largest ? limit : largest;
}
TokenCaps decode_token_caps(const elm_params *p, int problems)
{
    const int limit = g_debug_largest_cluster.load(std::memory_order_relaxed);
    return tokens_caps(p->d, problems, limit ? limit : DEC_MAX_CLUSTER);
}

// Streaming tokens of `per_token` query vectors: most parts of a list - a power of two, so that the SMs hold one
// token's clusters at once.  A list that would give each CTA of its cluster more than eight rounds of tiles while
// most SMs idle is left to the form with partial results in the workspace, token by token: over as many CTAs as fit the
// device a single token gains (8 KV heads of 4 query heads: fp32, 4500 entries 16.4 us in clusters, 14.5 split, 9000 26.6 and
// 18.3, 24000 57.5 and 43.3; bf16, 9000 17.2 and 14.6, 17000 24.8 and 18.1), but the tokens of a call can then no longer share a launch (32
// tokens together and one by one: fp32, 9000 entries 297 and 563 us; bf16, 17000 177 and 567).
template <int D> int decode_cap(int problems, int per_token, int sms)
{
    const int most = DEC_CTAS * sms / (problems * ((per_token + DEC_GSTREAM - 1) / DEC_GSTREAM));
    int cap = decode_largest_cluster<D>();
    while (cap > 1 && cap > most) cap >>= 1;
    return cap;
}
bool decode_clustered(int n_core, int problems, int cap, int entries)
{
    return n_core <= 8 * entries * cap || problems * cap >= device_sm_count();
}

// The split form of three query vectors and more on bf16 storage is a contraction for the matrix instructions (tokens_split_kernel,
// elm_attend_tokens.cu): both launches, replayed as a graph, 4 vectors, 8 problems of 2048 entries 7.9 -> 6.9 us, 32 of 5193 21.4 -> 16.8 us, 64 of 12288
// 74.8 -> 66.9; 8 vectors, 8 problems of 2048 11.9 -> 7.4, 64 of 12288 136 -> 68.9; d = 64 alike.  One or two vectors would pay for eight.
template <typename Tin, int G> constexpr bool DECODE_MMA = std::is_same<Tin, __nv_bfloat16>::value && G >= 4;
template <typename Tin, int G> constexpr bool DECODE_SHORT = !DECODE_MMA<Tin, G> || G < 8;

// How elm_attend's list is split: CTAs per problem, and whether their warps take short tiles.
struct DecodeSplits {
    int n;
    bool short_tiles;
};
template <typename Tin, int D, int G> DecodeSplits decode_splits(int n_core, int problems, size_t part_room)
{
    const int sms = device_sm_count();
    auto ctas = [](int entries, int tile) { return (entries + DEC_WARPS * tile - 1) / (DEC_WARPS * tile); };
    // A tile is a serial chain (rows, dot products, softmax, values), and a call with few of them is as long as that chain:
    // lists of up to 512 entries take tiles of 8 while that makes no more than two CTAs per SM, or two per problem.
    // 8 problems of 4 query vectors, bf16, d = 128: 32 entries 7.4 -> 5.9 us, 512 entries 7.8 -> 6.5 us, but 1024 entries
    // 7.7 -> 8.0 us; 64 problems: 128 entries 8.0 -> 7.1 us, 200 entries 7.9 -> 8.9 us.
    // (Eight vectors on bf16 storage go to the matrix instructions whatever the length: 8 problems
    // of 130 entries 9.1 -> 6.6 us.)
    const int few = ctas(n_core, DEC_SHORT_TILE);
    DecodeSplits s;
    s.short_tiles = false;
    if constexpr (DECODE_SHORT<Tin, G>) s.short_tiles = few <= 2 || (few <= 16 && few * problems <= 2 * sms);
    // otherwise as many CTAs as are resident at once, but at least one tile per warp; with more problems than that, as many
    // as take the least time in waves of them, a CTA's start and merge counted as 3/4 round of tiles per query vector, on matrix instructions as
    // 3/2 round whatever the vectors (450 problems of 2048 entries, 4 vectors, parts 1 / 2 / 3 / 4: 95.6 / 85.4 / 82.7 / 81.5 us, 8 vectors
    // 98.6 / 89.0 / 87.6 / 86.7; 600 problems 116.8 / 102.1 / 106.0 / 105.0; 300 problems 56.6 / 63.3 / 61.6 / 57.3).
    // 512 problems on 444 CTAs, fp32, d = 128, one query vector: 2048 entries 173 -> 122 us (one CTA per problem: a second
    // wave that is nearly empty), 200 entries 16.9 -> 15.9 us.
    const int resident = DEC_CTAS * sms, wanted = resident / problems;
    s.n = s.short_tiles ? few : ctas(n_core, DEC_TILE<Tin, D>);
    if (!s.short_tiles && wanted < 1) {
        const int most_parts = s.n < 4 ? s.n : 4;
        int64_t least = INT64_MAX;
        for (int n = 1; n <= most_parts; ++n) {
            const int rounds = ctas((n_core + n - 1) / n, DEC_TILE<Tin, D>);
            const int64_t time = (((int64_t)n * problems + resident - 1) / resident) * (4 * rounds + (DECODE_MMA<Tin, G> ? 6 : G == 1 ? 4 : 3 * G));
            if (time < least) { least = time; s.n = n; }
        }
    } else if (!s.short_tiles && s.n > wanted) {
        s.n = wanted;
    }
    // and no more partial results than the workspace has room for
    const size_t most = part_room / ((size_t)problems * G * (D + 2) * sizeof(float));
    if ((size_t)s.n > most) s.n = (int)most;
    if (s.n > DEC_MAX_SPLITS) s.n = DEC_MAX_SPLITS;
    return s;
}

// How a launch of streaming tokens is laid out: query vectors per group, groups they make of a token's, tokens per group,
// CTAs per group's cluster (0: one CTA per group, part after part), most parts of a list.
struct DecodeForm {
    int32_t G, vec_groups, per_group, cluster, cap;
};
template <typename Tin, int D> DecodeForm decode_form(const DecodeWindows &win, int problems, int per_token)
{
    constexpr int TILE = DEC_TILE<Tin, D>;
    const int sms = device_sm_count();
    const int cap = decode_cap<D>(problems, per_token, sms);
    int longest = 0, parts, chunk, size = 1;
    for (int i = 0; i < win.n; ++i) {
        const int last = win.seen0[i] + (win.tok0[i + 1] - win.tok0[i]) - 1;
        longest = last > longest ? last : longest;
    }
    decode_parts(longest, DEC_WARPS * TILE, TILE, cap, parts, chunk);
    while (size < parts) size <<= 1;
    const int64_t tokens = win.tok0[win.n];
    const int whole = (per_token + DEC_GSTREAM - 1) / DEC_GSTREAM;                // groups of DEC_GSTREAM vectors
    // Clusters spread a token over the SMs and are never slower than the tokens one by one (fp32, 6144 entries, 8 KV heads of 4
    // query heads: 2 tokens 25 us, 8 tokens 80 us, one token 20 us).  Walking part after part saves their barriers
    // and merges but takes as long as one CTA needs for a whole list (161 us), so it pays from about one token per SM on
    // (16 tokens of 8 heads: 141 us in clusters, 163 walked; 32 tokens: 264 against 221; 64: 505 against 424), from two
    // on when its CTAs take several tokens (1 query head per KV head: 32 tokens 199 against 307, 64 tokens 379 against
    // 311).  A list of one part needs no merge at all.
    if (tokens > 1) {
        int per_group = 1;
        while (per_group * 2 * per_token <= DEC_GSTREAM) per_group *= 2;
        if (tokens * problems * whole >= (per_group > 1 ? 2 : 1) * sms || (parts == 1 && per_group == 1)) return {DEC_GSTREAM, whole, per_group, 0, cap};
    }
    // The chain of a tile grows with its query vectors, so clusters take as few as leave all their CTAs resident.
    // fp32, 8 KV heads of 8 query heads, vectors one by one, in twos, in fours: 200 entries 6.9 / 7.7 / 9.3 us, 2000 entries 28.7 / 18.9 / 13.0; of 4
    // query heads: 200 entries 6.6 / 7.7 / 9.2, 2000 entries 16.6 / 10.7 / 10.9, 6144 entries 32.7 / 19.9 / 19.7.
    int G = 1;
    while (G < DEC_GSTREAM && G < per_token && tokens * problems * ((per_token + G - 1) / G) * size > DEC_CTAS * sms) G *= 2;
    return {G, (per_token + G - 1) / G, 1, size, cap};
}

template <typename Tin, int D, int G> auto decode_split_kernel(bool short_tiles, int &smem)
{
    auto kern = decode_kernel<Tin, D, G, DEC_SPLIT, DEC_SHORT_TILE>;
    smem = DecodeCfg<Tin, D, G, DEC_SHORT_TILE>::template total<DEC_SPLIT>();
    if constexpr (!DECODE_MMA<Tin, G>) {
        if (!short_tiles) {
            kern = decode_kernel<Tin, D, G, DEC_SPLIT>;
            smem = DecodeCfg<Tin, D, G>::template total<DEC_SPLIT>();
        }
    }
    return kern;
}

// win set: streaming tokens, laid out as `form` says; else the list of elm_attend, n_core entries long
template <typename Tin, int D, int G>
int launch_decode(const Tin *Q, const Tin *K, const Tin *V, const int32_t *idx, const float *w, int64_t list_stride, int n_core,
                  const DecodeWindows *win, DecodeForm form, const elm_params *p, Tin *O, float *part, size_t part_room, int *status,
                  int per_token, cudaStream_t st)
{
    const int problems = p->batch * p->kv_heads;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(DEC_WARPS * 32);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int64_t n_kv = p->n_kv;
    const int q_heads = p->q_heads, kv_heads = p->kv_heads, n_q = p->n_q;
    DecodeGroups grp = {};
    if (win) {
        if constexpr (G <= DEC_GSTREAM && std::is_same<Tin, float>::value) {
            using C = DecodeCfg<Tin, D, G>;
            grp.vec_groups = form.vec_groups;
            grp.per_group = form.per_group;
            for (int i = 0; i < win->n; ++i) {
                const int last = win->seen0[i] + (win->tok0[i + 1] - win->tok0[i]) - 1;
                grp.g0[i + 1] = grp.g0[i] + (last - 1) / grp.per_group - (win->seen0[i] - 1) / grp.per_group + 1;
            }
            auto kern = decode_kernel<Tin, D, G, DEC_CLUSTER>;
            cfg.dynamicSmemBytes = C::template total<DEC_CLUSTER>();
            if constexpr (G == DEC_GSTREAM) {
                if (form.cluster == 0) {
                    kern = form.per_group > 1 ? decode_kernel<Tin, D, G, DEC_NEIGHBOURS> : decode_kernel<Tin, D, G, DEC_TOKENS>;
                    cfg.dynamicSmemBytes = C::template total<DEC_TOKENS>();
                }
            }
            grp.cluster = form.cluster ? form.cluster : 1;
            ELM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes));
            if (grp.cluster > 8) ELM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            attr[1].id = cudaLaunchAttributeClusterDimension;
            attr[1].val.clusterDim.x = (unsigned)grp.cluster;
            attr[1].val.clusterDim.y = 1;
            attr[1].val.clusterDim.z = 1;
            cfg.numAttrs = 2;
            cfg.gridDim = dim3((unsigned)(grp.g0[win->n] * grp.vec_groups * grp.cluster), (unsigned)problems);
            ELM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, Q, K, V, idx, w, n_kv, list_stride, q_heads, kv_heads, n_q, per_token, *win, grp,
                                            form.cap, O, (float *)nullptr, status));
            count_launches(1);
            return cuda_status(cudaGetLastError());
        } else {
            return ELM_ERR_SHAPE;                                  // (decode_form gives no such G; bf16: attend_tokens_bf16)
        }
    }
    DecodeWindows whole = {};
    whole.n = 1;
    whole.tok0[1] = 1;
    whole.seen0[0] = n_core;
    const DecodeSplits sp = decode_splits<Tin, D, G>(n_core, problems, part_room);
    const int splits = sp.n;
    if (splits < 1) return ELM_ERR_WORKSPACE;
    cfg.gridDim = dim3((unsigned)splits, (unsigned)problems);
    if (DECODE_MMA<Tin, G> && !sp.short_tiles) {
        const int rc = launch_tokens_split(Q, K, V, idx, w, n_core, splits, G, p, part, status, st);
        if (rc != ELM_OK) return rc;
    } else if constexpr (DECODE_SHORT<Tin, G>) {
        int smem;
        auto kern = decode_split_kernel<Tin, D, G>(sp.short_tiles, smem);
        cfg.dynamicSmemBytes = (size_t)smem;
        ELM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes));
        ELM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, Q, K, V, idx, w, n_kv, list_stride, q_heads, kv_heads, n_q, per_token, whole, grp, 0, O,
                                        part, status));
    }
    cfg.gridDim = dim3((unsigned)per_token, (unsigned)problems);
    cfg.blockDim = dim3(D);
    cfg.dynamicSmemBytes = 0;
    const float *part_c = part;
    ELM_CUDA_TRY(cudaLaunchKernelEx(&cfg, decode_merge_kernel<Tin, D, G>, part_c, splits, q_heads, kv_heads, n_q, O));
    count_launches(2);
    return cuda_status(cudaGetLastError());
}

template <typename Tin, int D>
int dispatch_decode(const void *Q, const void *K, const void *V, const int32_t *idx, const float *w, int64_t list_stride, int n_core,
                    const DecodeWindows *win, const elm_params *p, void *O, float *part, size_t part_room, int *status, cudaStream_t st)
{
    const int per_token = (p->q_heads / p->kv_heads) * p->n_q;
    DecodeForm form = {per_token, 1, 1, 0, 0};
    if (win) {
        const int problems = p->batch * p->kv_heads;
        if constexpr (std::is_same<Tin, __nv_bfloat16>::value)
            return attend_tokens_bf16(Q, K, V, idx, w, list_stride, *win, p, O, status, decode_token_caps(p, problems), st);
        else
            form = decode_form<Tin, D>(*win, problems, per_token);
    }
    return with_groups(form.G, [&](auto G) {
        return launch_decode<Tin, D, decltype(G)::value>((const Tin *)Q, (const Tin *)K, (const Tin *)V, idx, w, list_stride, n_core, win,
                                                         form, p, (Tin *)O, part, part_room, status, per_token, st);
    });
}
int dispatch_decode(const void *Q, const void *K, const void *V, const int32_t *idx, const float *w, int64_t list_stride, int n_core,
                    const DecodeWindows *win, const elm_params *p, void *O, float *part, size_t part_room, int *status, cudaStream_t st)
{
    if (p->dtype == ELM_F32)
        return p->d == 64 ? dispatch_decode<float, 64>(Q, K, V, idx, w, list_stride, n_core, win, p, O, part, part_room, status, st)
                          : dispatch_decode<float, 128>(Q, K, V, idx, w, list_stride, n_core, win, p, O, part, part_room, status, st);
    return p->d == 64 ? dispatch_decode<__nv_bfloat16, 64>(Q, K, V, idx, w, list_stride, n_core, win, p, O, part, part_room, status, st)
                      : dispatch_decode<__nv_bfloat16, 128>(Q, K, V, idx, w, list_stride, n_core, win, p, O, part, part_room, status, st);
}

}  // namespace

bool attend_decode_applies(const elm_params *p)
{
    if (p->precision != ELM_PREC_FP32) return false;
    const int64_t groups = (int64_t)(p->q_heads / p->kv_heads) * p->n_q;
    return groups <= DEC_GMAX;
}

bool attend_decode_windows_apply(const elm_params *p, int n_core)
{
    if (!attend_decode_applies(p) || p->n_q != 1 || (p->dtype != ELM_F32 && p->dtype != ELM_BF16)) return false;
    const int problems = p->batch * p->kv_heads, per_token = p->q_heads / p->kv_heads;
    if (p->dtype == ELM_F32) {
        const int sms = device_sm_count();
        return p->d == 64 ? decode_clustered(n_core, problems, decode_cap<64>(problems, per_token, sms), DEC_WARPS * DEC_TILE<float, 64>)
                          : decode_clustered(n_core, problems, decode_cap<128>(problems, per_token, sms), DEC_WARPS * DEC_TILE<float, 128>);
    }
    // Clusters cut short because the device cannot hold all problems' longer ones at once leave few SMs idle, although their CTAs may be
    // fewer than the SMs.  16 problems (clusters of 8) of 4 query vectors, 9000 entries: one token 23.6 us for 16.9 token by token, but
    // two 25.0 for 33.2 and 128 554 for 2088; 36 problems (clusters of 4), 4100 entries: 23.4 / 16.7, 24.7 / 32.5, 680 / 2060.
    const int cap = decode_token_caps(p, problems).of_long;
    return decode_clustered(n_core, problems, cap, 128) || cap < decode_token_caps(p, 1).of_long;
}

namespace {
template <typename Tin, int D, int G> int decode_grid(const elm_params *p, int n_core, int32_t *ctas, int32_t *resident)
{
    const AttendLayout L = attend_layout(p, n_core);
    const int problems = p->batch * p->kv_heads;
    const DecodeSplits sp = decode_splits<Tin, D, G>(n_core, problems, L.bias - L.Kc);
    int per_sm = 0;
    if (DECODE_MMA<Tin, G> && !sp.short_tiles) {
        ELM_CUDA_TRY(tokens_split_occupancy(D, &per_sm));
        *ctas = sp.n * problems;
        *resident = per_sm * device_sm_count();
        return ELM_OK;
    }
    if constexpr (DECODE_SHORT<Tin, G>) {
        int smem;
        auto kern = decode_split_kernel<Tin, D, G>(sp.short_tiles, smem);
        ELM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        ELM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, DEC_WARPS * 32, (size_t)smem));
        *ctas = sp.n * problems;
        *resident = per_sm * device_sm_count();
    }
    return ELM_OK;
}
}  // namespace

int attend_decode_windows(const void *Q, const void *K, const void *V, const int32_t *idx, const float *w, int64_t list_stride,
                          const DecodeWindows &win, const elm_params *p, void *O, int *status, cudaStream_t st)
{
    StageTimer t(ELM_STAGE_ATTEND, st, 1);
#ifdef ELM_BOUNDS_CHECK
    ELM_CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(int), st));
#endif
    return dispatch_decode(Q, K, V, idx, w, list_stride, 0, &win, p, O, nullptr, 0, status, st);
}

int attend_decode(const void *Q, const void *K, const void *V, const int32_t *idx, const float *w, int n_core,
                  const elm_params *p, void *O, unsigned char *ws, cudaStream_t st, bool timed)
{
    const AttendLayout L = attend_layout(p, n_core);
    const int problems = p->batch * p->kv_heads;
    // the partial results live where the other paths keep their gathered operands
    float *part = reinterpret_cast<float *>(ws + L.Kc);
    const size_t room = L.bias - L.Kc;
    int *status = reinterpret_cast<int *>(ws + L.flags) + problems;
    StageTimer t(timed ? ELM_STAGE_ATTEND : -1, st, 2);
#ifdef ELM_BOUNDS_CHECK
    // bad row numbers are reported through the status word
    ELM_CUDA_TRY(cudaMemsetAsync(ws + L.flags, 0, sizeof(int) * (size_t)(problems + 1), st));
#endif
    return dispatch_decode(Q, K, V, idx, w, n_core, n_core, nullptr, p, O, part, room, status, st);
}

int debug_set_attend_decode(int32_t what, int64_t value)
{
    if (what != ELM_DEBUG_DECODE_LARGEST_CLUSTER || value < 0 || value > DEC_MAX_CLUSTER || (value & (value - 1))) return ELM_ERR_SHAPE;
    g_debug_largest_cluster.store((int)value);
    return ELM_OK;
}

}  // namespace elm

extern "C" int elm_debug_decode_grid(const elm_params *params, int32_t n_core, int32_t *ctas, int32_t *resident)
{
    using namespace elm;
    if (!params || !ctas || !resident) return ELM_ERR_NULL;
    const int rc = validate_attend_params(params);
    if (rc != ELM_OK) return rc;
    if (n_core < 1 || n_core > params->n_kv || !attend_decode_applies(params)) return ELM_ERR_SHAPE;
    return with_groups((params->q_heads / params->kv_heads) * params->n_q, [&](auto G) {
        constexpr int g = decltype(G)::value;
        if (params->dtype == ELM_F32)
            return params->d == 64 ? decode_grid<float, 64, g>(params, n_core, ctas, resident) : decode_grid<float, 128, g>(params, n_core, ctas, resident);
        return params->d == 64 ? decode_grid<__nv_bfloat16, 64, g>(params, n_core, ctas, resident)
                               : decode_grid<__nv_bfloat16, 128, g>(params, n_core, ctas, resident);
    });
}

extern "C" int elm_debug_stream_form(const elm_params *params, int32_t seen, int32_t tokens, int32_t *form)
{
    using namespace elm;
    if (!params || !form) return ELM_ERR_NULL;
    const int rc = validate_attend_params(params);
    if (rc != ELM_OK) return rc;
    if (seen < 1 || tokens < 1 || (int64_t)seen + tokens - 1 > params->n_kv || params->n_q != 1 || params->dtype != ELM_BF16 ||
        !attend_decode_applies(params))
        return ELM_ERR_SHAPE;
    DecodeWindows win = {};
    win.n = 1;
    win.tok0[1] = tokens;
    win.seen0[0] = seen;
    const TokenCaps caps = decode_token_caps(params, params->batch * params->kv_heads);
    *form = !attend_decode_windows_apply(params, seen + tokens - 1) ? 0 : attend_tokens_serial(win, params, caps) ? 2 : 1;
    return ELM_OK;
}
