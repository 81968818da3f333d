// Kernel evaluation for one Compress2 level on the sm_100a tensor cores (bf16 inputs, fp32 mode).
//
// A CTA produces one 64 x 64 tile of the pair Gram F = P G P^T, i.e. a 128 x 128 tile of
//   G[a,b] = exp(<k_a,k_b>/sqrt(d) - M_pair(b)) * (<v_a,v_b> + v_max^2)                Eq. (katt), shifted
// The 128 row points and 128 column points are gathered through the level's index list straight
// into the 128-byte-swizzled K-major layout tcgen05.mma reads (rows are never copied in HBM).
// Two accumulators in TMEM hold K K^T and V V^T; the epilogue applies the exponential, the
// product and the +/- pair combination F[j,i] = G[2j,2i] - G[2j,2i+1] - G[2j+1,2i] + G[2j+1,2i+1]
// (Algorithm A.1's <f_j, f_i>; of use for j <= i within one Halve call).
#include <math.h>

#include "elm_common.cuh"
#include "elm_compress.cuh"
#include "elm_sm100.cuh"
#include "elm_walk.cuh"

namespace elm {
namespace gramtc {

using namespace sm100;

constexpr int TP = 64;            // pairs per tile side
constexpr int TR = 128;           // points per tile side
constexpr int NTHREADS = 256;
constexpr uint32_t TMEM_COLS = 256;
constexpr int FS_LD = 68;         // row stride of the shared-memory pair Gram of a fused tile (floats)

// Shared memory of the kernel that walks its tiles itself: the tile's keys, its values, its pair Gram.  92 KB (d = 128)
// let two CTAs share an SM.
template <int D> struct Smem {
    static constexpr int KH = D / 64;
    static constexpr int OPERAND = TR * D * 2;                 // one 128-row operand tile, bytes
    static constexpr int OFF_K = 0, OFF_V = OPERAND;
    static constexpr int OFF_MISC = 2 * OPERAND;
    static constexpr int OFF_F = OFF_MISC + 3072;
    // The block walker reads 32 rows and 64 columns from a call's corner whatever the call's size (and ignores what lies
    // outside): from call 3 of 16 pairs on, row 48 + 31, column 48 + 63.
    static constexpr int F_BYTES = ((48 + 31) * FS_LD + 48 + 64) * 4;
    static constexpr int TOTAL = OFF_F + F_BYTES + 1024;       // + alignment slack
};

struct TileMisc {
    float colshift[TP];          // M of each pair column, in log2 units
    float rdec[TP], unif[TP];    // the walk's decay factor and uniform of each pair of the tile
    int32_t rows[TR];
};
struct Misc {
    uint64_t mma_done;
    uint32_t tmem_base;
    uint32_t pad;
    TileMisc tile[2];            // this tile's and the next one's
};
static_assert(sizeof(Misc) <= 3072, "the misc block's share of shared memory");

// Halving walk (Algorithm A.1) of the calls that lie inside one 64-pair tile, on the tile's pair
// Gram in shared memory: warp w walks call w of the tile (P = 16 or 32 pairs per call), one block of the
// warp-cooperative block walker.
__device__ __forceinline__ void walk_in_tile(const float *Fs, const float *rdec, const float *unif, int p,
                                             int64_t JR, int P, int64_t Ptotal, int64_t n,
                                             const int32_t *__restrict__ cur, const WalkArgs &wk, int warp, int lane)
{
    const int calls = TP / P;
    if (warp >= calls) return;
    const int64_t J0 = JR + (int64_t)warp * P;                 // first pair of this call along the level's sequence
    if (J0 >= Ptotal) return;
    const float *Fc = Fs + (warp * P) * FS_LD + warp * P;      // the call's P x P block
    float bmax = 0.f, dn = 0.f;
    const int i = lane;                                        // pair within the call
    const bool live = i < P;
    const float dgn = live ? Fc[i * FS_LD + i] : 0.f;
    const float a = walk_block_thresholds(sqrtf(dgn > 0.f ? dgn : 0.f), live ? rdec[warp * P + i] : 1.f, bmax, wk.logfac, lane);
    // pairs past the end of a short call come after the live ones and decide nothing
    const float d = walk_sign_score(0.f, a, live ? unif[warp * P + i] : 1.f);
    const uint32_t swaps = walk_block_warp(Fc, FS_LD, d, dn, lane);
    if (live) {
        const uint32_t sw = (swaps >> lane) & 1u;
        wk.out[(int64_t)p * wk.out_stride + J0 + i] = cur[(int64_t)p * n + 2 * (J0 + i) + sw];
    }
}

// Gather 128 rows of X (row-major [n][D] bf16) into a swizzled K-major operand tile.
template <int D>
__device__ __forceinline__ void gather_operand(unsigned char *dst, const __nv_bfloat16 *__restrict__ X,
                                               const int32_t *rows, int tid)
{
    constexpr int CHUNKS = D / 8;                              // 16-byte chunks per row
    const uint32_t dst_s = smem_u32(dst);
#pragma unroll
    for (int q = tid; q < TR * CHUNKS; q += NTHREADS) {
        const int r = q / CHUNKS, ch = q % CHUNKS;
        const int kh = ch >> 3, c = ch & 7;
        // asynchronous 16-byte copies: all of a thread's chunks are in flight at once
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst_s + kh * (TR * 128) + (r >> 3) * 1024 +
                                                                        (r & 7) * 128 + ((c ^ (r & 7)) << 4)),
                     "l"(X + (int64_t)rows[r] * D + ch * 8)
                     : "memory");
    }
}

// Levels whose calls are smaller than a tile (P < 64 pairs; a tile holds 64 / P whole calls or the level's last ones):
// row points = column points, and the calls are walked on the tile's pair Gram without it leaving shared memory.
// Persistent, two CTAs per SM, bound by the latency of a tile's stages (row numbers, gather, MMAs, epilogue, walk): the
// row numbers and everything else a tile needs from global memory are fetched while the tile before is multiplied, and
// its rows are gathered while that one's epilogue and walk run.  64 problems x 8192 points, d = 128: 16 pairs a
// call 116 -> 83 us, 32 pairs 57 -> 42 us against one CTA per tile (HBM floor of the first: 41 us).
template <int D>
__global__ void __launch_bounds__(NTHREADS, 2)
gram_walk_kernel(const __nv_bfloat16 *__restrict__ K, const __nv_bfloat16 *__restrict__ V,
                 const int32_t *__restrict__ cur, const float *__restrict__ Mpair,
                 const unsigned *__restrict__ vmax_bits, int64_t n, int P, int64_t Ptotal, int tiles_per_problem, int total_tiles,
                 int *__restrict__ status, WalkArgs wk)
{
    cudaGridDependencySynchronize();           // launched with programmatic stream serialization (launch_after)
    using SM = Smem<D>;
    constexpr int KH = SM::KH;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    Misc *misc = reinterpret_cast<Misc *>(smem + SM::OFF_MISC);
    float *Fs = reinterpret_cast<float *>(smem + SM::OFF_F);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (*reinterpret_cast<volatile int *>(status) != 0) return;
    const float LOG2E = 1.4426950408889634f;
    // what tile `it` needs from global memory besides its rows: row numbers, running shifts, decay factors, uniforms
    auto fetch_misc = [&](int it, TileMisc &m) {
        const int p = it / tiles_per_problem;
        const int64_t JR = (int64_t)(it % tiles_per_problem) * TP;
        if (tid < TR) {
            const int64_t pt = 2 * JR + tid;
            m.rows[tid] = pt < 2 * Ptotal ? __ldg(cur + (int64_t)p * n + pt) : 0;
        } else if (tid < TR + TP) {
            const int i = tid - TR;
            const int64_t jc = JR + i;
            m.colshift[i] = jc < Ptotal ? __ldg(Mpair + (int64_t)p * pair_stride(n) + jc) * LOG2E : 0.f;
            m.rdec[i] = jc < Ptotal ? __ldg(wk.rdecay + (int64_t)p * pair_stride(n) + jc) : 1.f;
        } else {
            const int i = tid - TR - TP;
            const int64_t jc = JR + i;
            uint32_t cgroup, ccode;
            call_counter((int)(jc / P), wk.level, cgroup, ccode);
            m.unif[i] = halving_uniform<float>(wk.seed, (uint32_t)(jc % P), cgroup, ccode, (uint32_t)p + wk.pbase);
        }
    };
    auto gather = [&](int it, const TileMisc &m) {
        const int64_t first = (int64_t)(it / tiles_per_problem) * n * D;
        gather_operand<D>(smem + SM::OFF_K, K + first, m.rows, tid);
        gather_operand<D>(smem + SM::OFF_V, V + first, m.rows, tid);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (tid == 0) {
        mbar_init(&misc->mma_done, 1);
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc(&misc->tmem_base, TMEM_COLS);
    if ((int)blockIdx.x < total_tiles) fetch_misc(blockIdx.x, misc->tile[0]);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = misc->tmem_base;
    if ((int)blockIdx.x < total_tiles) gather(blockIdx.x, misc->tile[0]);

    constexpr uint32_t IDESC = umma_idesc_bf16(TR, TR);
    // (descriptors differ only in the start address, in their low word; see the persistent kernel)
    const uint64_t desc0 = umma_desc_k128(smem_u32(smem));
    const uint32_t d_hi = (uint32_t)(desc0 >> 32), dK = (uint32_t)desc0 + (SM::OFF_K >> 4), dV = (uint32_t)desc0 + (SM::OFF_V >> 4);
    auto desc = [&](uint32_t lo) { uint64_t d; asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(d_hi)); return d; };
    const int r = (warp & 3) * 32 + lane;                     // epilogue: point row in the tile = TMEM lane
    const int ch = warp >> 2;                                 // and column half
    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + ch * 64;
    const float qscale = LOG2E / sqrtf((float)D);
    bool ok = true;
    int k = 0;
    for (int it = blockIdx.x; it < total_tiles; it += gridDim.x, ++k) {
        const TileMisc &m = misc->tile[k & 1];
        const int p = it / tiles_per_problem;
        const int64_t JR = (int64_t)(it % tiles_per_problem) * TP;
        const bool more = it + (int)gridDim.x < total_tiles;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        fence_proxy_async();
        tc_fence_before();
        __syncthreads();                                      // rows gathered; the tile before is walked
        tc_fence_after();
        if (tid == 0) {
#pragma unroll
            for (int op = 0; op < 2; ++op)
#pragma unroll
                for (int kh = 0; kh < KH; ++kh)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        const uint64_t d = desc((op == 0 ? dK : dV) + ((kh * (TR * 128) + ks * 32) >> 4));
                        mma_ss(tmem + op * 128, d, d, IDESC, (kh | ks) != 0);
                    }
            tc_commit(&misc->mma_done);
        }
        if (more) fetch_misc(it + gridDim.x, misc->tile[(k + 1) & 1]);
        const float vm = __uint_as_float(vmax_bits[p]);
        const float vm2 = vm * vm;
        ok = mbar_wait(&misc->mma_done, (uint32_t)k & 1u);
        if (__syncthreads_or(!ok)) { ok = false; break; }     // (and the next tile's row numbers are there)
        tc_fence_after();
        if (more) gather(it + gridDim.x, misc->tile[(k + 1) & 1]);
        float h[32];                                          // G[r,2i] - G[r,2i+1] for the 32 pair columns
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t kk[32], vv[32];
            tmem_ld32(taddr + q * 32, kk);
            tmem_ld32(taddr + 128 + q * 32, vv);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
                const float sh = m.colshift[ch * 32 + q * 16 + (c >> 1)];
                float e0 = fmaf(__uint_as_float(kk[c]), qscale, -sh);
                float e1 = fmaf(__uint_as_float(kk[c + 1]), qscale, -sh);
                float g0 = e0 < -115.f ? 0.f : fast_exp2(e0) * (__uint_as_float(vv[c]) + vm2);
                float g1 = e1 < -115.f ? 0.f : fast_exp2(e1) * (__uint_as_float(vv[c + 1]) + vm2);
                h[q * 16 + (c >> 1)] = g0 - g1;
            }
        }
        // pair rows are adjacent lanes: the even lane finishes pair columns 0..15 of its 32, the odd
        // lane columns 16..31
        const bool odd = lane & 1;
        float *Fr = Fs + (r >> 1) * FS_LD + ch * 32 + (odd ? 16 : 0);
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
            float f[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float send = odd ? h[i + j] : h[i + j + 16];
                const float recv = __shfl_xor_sync(0xffffffffu, send, 1);
                f[j] = odd ? recv - h[i + j + 16] : h[i + j] - recv;
            }
            *reinterpret_cast<float4 *>(Fr + i) = make_float4(f[0], f[1], f[2], f[3]);
        }
        tc_fence_before();
        __syncthreads();
        walk_in_tile(Fs, m.rdec, m.unif, p, JR, P, Ptotal, n, cur, wk, warp, lane);
    }
    if (!ok && lane == 0) atomicExch(status, 4);
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
}

// ---------------------------------------------------------------------------------------------
// Persistent, pipelined variant for levels whose calls span several tiles (P > 64 pairs).
// One CTA per SM walks the level's tile list (tile, problem) round-robin.  Roles:
//   warps 0-3   loaders: gather the tile's row and column points with 16-byte cp.async into a ring
//               of three 64 KB operand buffers -- one "job" for the keys, one for the values of each
//               tile -- and let the copies' completion arrive on the job's mbarrier, so up to three
//               jobs are in flight while earlier ones are multiplied
//   warp 4      issues the tcgen05.mma of each job into one of two TMEM accumulator slots
//               (K K^T | V V^T, 256 columns each); its commits free the operand buffers
//   warps 5-12  epilogue of the previous tile (exp2, product, pair combination, stores) while the
//               next tile is gathered and multiplied
// Bound by the gathers: 128 KB per tile off the diagonal at about 64 bytes per cycle into an SM, and the row numbers
// that queue behind them; about 3500 cycles per tile, of which the MMAs take 1400.  32 problems, d = 128, 128-KB tiles of calls of
// 1024 pairs 67.5 -> 63.2 us per level, of calls of 64 pairs (64 KB from HBM) 128 -> 126, 128 pairs 94 -> 89, 256 pairs 78 -> 71:
// descriptors by adding to one of them (the MMAs' issue took 1175 cycles per operand, now 700), row numbers of the next tile fetched
// behind this tile's copies, pair rows stored as 128 contiguous bytes.
// ---------------------------------------------------------------------------------------------
constexpr int PNS = 3;                       // operand ring depth (jobs)
constexpr int PLOAD = 4;                      // loader warps (8 were slower: 0.76 against 0.71 ms per cfg5 step)
constexpr int PTHREADS = (PLOAD + 1 + 8) * 32;   // loaders, the MMA issuer, 8 epilogue warps
constexpr int PTAB = 256;                    // items of a CTA whose tiles are decoded up front

struct PBarriers {
    uint64_t full[PNS], empty[PNS], accfull[2], accempty[2];
    uint32_t tmem_base;
    uint32_t pad;
};

template <int D> struct PSmem {
    static constexpr int JOB = 2 * TR * D * 2;                // row tile + column tile of one operand type
    static constexpr int OFF_BAR = PNS * JOB;
    static constexpr int TOTAL = OFF_BAR + 1024 + 1024;
};

__device__ __forceinline__ void decode_tile(int tile, int P, int64_t &JR, int64_t &JC)
{
    const int Tg = P / TP, ntri = Tg * (Tg + 1) / 2;
    const int g = tile / ntri, local = tile % ntri;
    int tc = (int)((sqrtf(8.f * (float)local + 1.f) - 1.f) * 0.5f);
    while ((tc + 1) * (tc + 2) / 2 <= local) ++tc;
    while (tc * (tc + 1) / 2 > local) --tc;
    const int tr = local - tc * (tc + 1) / 2;
    JR = (int64_t)g * P + tr * TP;
    JC = (int64_t)g * P + tc * TP;
}

template <int D>
__global__ void __launch_bounds__(PTHREADS, 1)
gram_tc_persistent_kernel(const __nv_bfloat16 *__restrict__ K, const __nv_bfloat16 *__restrict__ V,
                          const int32_t *__restrict__ cur, const float *__restrict__ Mpair,
                          const unsigned *__restrict__ vmax_bits, int64_t n, int P, int tiles_per_problem,
                          int total_items, float *__restrict__ F, int64_t F_stride, int *__restrict__ status)
{
    cudaGridDependencySynchronize();           // launched with programmatic stream serialization (launch_after)
    using SM = PSmem<D>;
    constexpr int KH = D / 64;
    constexpr int CHUNKS = D / 8;                             // 16-byte chunks per row
    extern __shared__ unsigned char smem_dyn[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    PBarriers *bar = reinterpret_cast<PBarriers *>(smem + SM::OFF_BAR);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (*reinterpret_cast<volatile int *>(status) != 0) return;
    // Which tile is item k of this CTA?  Decoding a tile number (two divisions, a square root) costs a lone
    // thread about 900 cycles - a quarter of a tile's time on the MMA issuer - so all threads decode the CTA's
    // items once, in parallel, into a table.
    __shared__ int tab_p[PTAB], tab_jr[PTAB], tab_jc[PTAB];
    for (int i = tid; i < PTAB; i += PTHREADS) {
        const int it = blockIdx.x + i * gridDim.x;
        if (it < total_items) {
            int64_t jr, jc;
            decode_tile(it % tiles_per_problem, P, jr, jc);
            tab_p[i] = it / tiles_per_problem;
            tab_jr[i] = (int)jr;
            tab_jc[i] = (int)jc;
        }
    }
    auto item = [&](int k, int it, int &p, int64_t &JR, int64_t &JC) {
        if (k < PTAB) {
            p = tab_p[k]; JR = tab_jr[k]; JC = tab_jc[k];
        } else {
            p = it / tiles_per_problem;
            decode_tile(it % tiles_per_problem, P, JR, JC);
        }
    };
    if (tid == 0) {
        for (int b = 0; b < PNS; ++b) { mbar_init(&bar->full[b], PLOAD * 32); mbar_init(&bar->empty[b], 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(&bar->accfull[s], 1); mbar_init(&bar->accempty[s], 256); }
        fence_barrier_init();
    }
    if (warp == PLOAD) tmem_alloc(&bar->tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bar->tmem_base;
    bool ok = true;

    if (warp < PLOAD) {
        // ------------------------------ loaders ------------------------------
        // chunk q = tid + NL i of a 128-row tile lies in row tid / CHUNKS + (NL / CHUNKS) i, NL loader threads
        constexpr int NL = PLOAD * 32;
        constexpr int RPT = TR * CHUNKS / NL;                // chunks (= distinct rows) per thread and tile
        int32_t ra[RPT], rb[RPT];
        int p_next = 0;
        bool diagonal_next = false;
        // row numbers of item k: fetched while the copies of the item before are on their way
        auto fetch_rows = [&](int k, int it) {
            int64_t JR, JC;
            item(k, it, p_next, JR, JC);
            diagonal_next = JR == JC;
            const int32_t *curp = cur + (int64_t)p_next * n;
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int r = tid / CHUNKS + (NL / CHUNKS) * i;
                ra[i] = __ldg(curp + 2 * JR + r);
                rb[i] = diagonal_next ? 0 : __ldg(curp + 2 * JC + r);
            }
        };
        int job = 0, lk = 0;
        if ((int)blockIdx.x < total_items) fetch_rows(0, blockIdx.x);
        for (int it = blockIdx.x; it < total_items && ok; it += gridDim.x, ++lk) {
            const int p = p_next;
            const bool diagonal = diagonal_next;
            const int ch = tid % CHUNKS, kh = ch >> 3, c = ch & 7;
            for (int op = 0; op < 2 && ok; ++op, ++job) {     // 0: keys, 1: values
                const int b = job % PNS;
                ok = mbar_wait(&bar->empty[b], ((uint32_t)(job / PNS) & 1u) ^ 1u);
                if (!ok) break;
                const __nv_bfloat16 *X = (op == 0 ? K : V) + (int64_t)p * n * D;
                const uint32_t dstA = smem_u32(smem + b * SM::JOB), dstB = dstA + TR * D * 2;
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const int r = tid / CHUNKS + (NL / CHUNKS) * i;
                    const uint32_t off = kh * (TR * 128) + (r >> 3) * 1024 + (r & 7) * 128 + ((c ^ (r & 7)) << 4);
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dstA + off), "l"(X + (int64_t)ra[i] * D + ch * 8) : "memory");
                    if (!diagonal)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dstB + off), "l"(X + (int64_t)rb[i] * D + ch * 8) : "memory");
                }
                // the job's barrier completes when every loader thread's copies have landed
                asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&bar->full[b])) : "memory");
            }
            if (it + (int)gridDim.x < total_items) fetch_rows(lk + 1, it + gridDim.x);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (!ok && lane == 0) atomicExch(status, 5);
    } else if (warp == PLOAD) {
        // ------------------------------ MMA issuer ------------------------------
        if (lane == 0) {
            constexpr uint32_t IDESC = umma_idesc_bf16(TR, TR);
            // descriptors differ only in the start address (address / 16, in their low word): a lone thread that builds each
            // from its address issues a tile's sixteen MMAs at half the tensor pipe's rate
            const uint64_t d0 = umma_desc_k128(smem_u32(smem));
            const uint32_t d_hi = (uint32_t)(d0 >> 32), d_lo = (uint32_t)d0;
            auto desc = [&](uint32_t lo) { uint64_t d; asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(d_hi)); return d; };
            int job = 0, k = 0;
            for (int it = blockIdx.x; it < total_items && ok; it += gridDim.x, ++k) {
                int p;
                int64_t JR, JC;
                item(k, it, p, JR, JC);
                const bool diagonal = JR == JC;
                const int slot = k & 1;
                ok = mbar_wait(&bar->accempty[slot], ((uint32_t)(k >> 1) & 1u) ^ 1u);
                if (!ok) break;
                tc_fence_after();
                for (int op = 0; op < 2 && ok; ++op, ++job) {
                    const int b = job % PNS;
                    ok = mbar_wait(&bar->full[b], (uint32_t)(job / PNS) & 1u);
                    if (!ok) break;
                    fence_proxy_async();                       // the gathered bytes were written by generic-proxy copies
                    tc_fence_after();
                    const uint32_t dA = d_lo + b * (SM::JOB >> 4), dB = diagonal ? dA : dA + (TR * D * 2 >> 4);
#pragma unroll
                    for (int kh = 0; kh < KH; ++kh)
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            mma_ss(tmem + slot * 256 + op * 128, desc(dA + ((kh * (TR * 128) + ks * 32) >> 4)),
                                   desc(dB + ((kh * (TR * 128) + ks * 32) >> 4)), IDESC, (kh | ks) != 0);
                    tc_commit(&bar->empty[b]);
                }
                if (ok) tc_commit(&bar->accfull[slot]);
            }
            if (!ok) atomicExch(status, 6);
        }
    } else {
        // ------------------------------ epilogue ------------------------------
        const int e = warp - (PLOAD + 1);                     // 0..7
        const int q4 = warp & 3;                              // TMEM lane quarter this warp may access
        const int ch = e >> 2;                                // column half
        const float LOG2E = 1.4426950408889634f;
        const float qscale = LOG2E / sqrtf((float)D);
        int k = 0;
        for (int it = blockIdx.x; it < total_items && ok; it += gridDim.x, ++k) {
            int p;
            int64_t JR, JC;
            item(k, it, p, JR, JC);
            const int slot = k & 1;
            const float vm = __uint_as_float(vmax_bits[p]);
            const float vm2 = vm * vm;
            // running shifts of this thread's 32 pair columns (in log2 units), fetched while the MMAs run
            float sh[32];
            {
                // 32 consecutive floats, 16-byte aligned (the rows' stride is a multiple of 4, JC of 32)
                const float4 *mp = reinterpret_cast<const float4 *>(Mpair + (int64_t)p * pair_stride(n) + JC + ch * 32);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 v = __ldg(mp + i);
                    sh[4 * i] = v.x * LOG2E; sh[4 * i + 1] = v.y * LOG2E; sh[4 * i + 2] = v.z * LOG2E; sh[4 * i + 3] = v.w * LOG2E;
                }
            }
            ok = mbar_wait(&bar->accfull[slot], (uint32_t)(k >> 1) & 1u);
            if (!ok) break;
            tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(q4 * 32) << 16) + slot * 256 + ch * 64;
            float h[32];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t kk[32], vv[32];
                tmem_ld32(taddr + q * 32, kk);
                tmem_ld32(taddr + 128 + q * 32, vv);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 32; c += 2) {
                    const float shc = sh[q * 16 + (c >> 1)];
                    float e0 = fmaf(__uint_as_float(kk[c]), qscale, -shc);
                    float e1 = fmaf(__uint_as_float(kk[c + 1]), qscale, -shc);
                    float g0 = e0 < -115.f ? 0.f : fast_exp2(e0) * (__uint_as_float(vv[c]) + vm2);
                    float g1 = e1 < -115.f ? 0.f : fast_exp2(e1) * (__uint_as_float(vv[c + 1]) + vm2);
                    h[q * 16 + (c >> 1)] = g0 - g1;
                }
            }
            // the accumulator slot is free as soon as its values are in registers
            tc_fence_before();
            mbar_arrive(&bar->accempty[slot]);
            const bool odd = lane & 1;
            float f[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float send = odd ? h[i] : h[i + 16];
                const float recv = __shfl_xor_sync(0xffffffffu, send, 1);
                f[i] = odd ? recv - h[i + 16] : h[i] - recv;
            }
            // A lane pair holds a pair row's 32 columns, 64 bytes each: stored as they are, every 16 bytes of a store instruction
            // would go to a place of their own.  Four lane pairs exchange 16-byte chunks (lane bits 2 and 1 against chunk
            // bits 1 and 0), after which eight lanes hold one pair row per store: 128 contiguous bytes.  On a diagonal tile
            // half of them lie below the diagonal of the call's P x P block, which nothing reads.
#pragma unroll
            for (int s = 1; s <= 2; s *= 2) {
                const bool up = (lane & (2 * s)) != 0;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (c & s) continue;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float got = __shfl_xor_sync(0xffffffffu, up ? f[4 * c + i] : f[4 * (c + s) + i], 2 * s);
                        f[4 * c + i] = up ? got : f[4 * c + i];
                        f[4 * (c + s) + i] = up ? f[4 * (c + s) + i] : got;
                    }
                }
            }
            const int64_t jr0 = JR + (q4 * 32 + (lane & ~7)) / 2;           // the first of the four pair rows
            const int64_t gr = jr0 / P;                                     // (calls begin at multiples of 64 pairs)
            float *Fp = F + (int64_t)p * F_stride + (jr0 - gr) * P + JC + ch * 32 + (odd ? 16 : 0) + 4 * ((lane >> 1) & 3);
#pragma unroll
            for (int b = 0; b < 4; ++b)
                *reinterpret_cast<float4 *>(Fp + (int64_t)b * P) = make_float4(f[4 * b], f[4 * b + 1], f[4 * b + 2], f[4 * b + 3]);
        }
        if (!ok && lane == 0) atomicExch(status, 7);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == PLOAD) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

template <int D>
static int launch(const __nv_bfloat16 *K, const __nv_bfloat16 *V, const elm_params *p, const int32_t *cur,
                  const float *Mpair, const unsigned *vmax_bits, int P, int64_t Ptotal, int groups, float *F,
                  int64_t F_stride, int *status, const WalkArgs &wk, cudaStream_t st)
{
    const int BH = p->batch * p->kv_heads;
    int64_t tiles;
    if (P >= TP) {
        const int Tg = P / TP;
        tiles = (int64_t)groups * (Tg * (Tg + 1) / 2);
    } else {
        tiles = (Ptotal + TP - 1) / TP;
    }
    const int sm_count = device_sm_count();
    const int64_t total = tiles * BH;
    if (total > 0x7fffffff / 2) return ELM_ERR_SHAPE;
    if (!wk.fused) {
        // calls that fill whole tiles: persistent, pipelined kernel, one CTA per SM
        const int grid = (int)(total < sm_count ? total : sm_count);
        auto pk = gram_tc_persistent_kernel<D>;
        ELM_CUDA_TRY(cudaFuncSetAttribute(pk, cudaFuncAttributeMaxDynamicSharedMemorySize, PSmem<D>::TOTAL));
        ELM_CUDA_TRY(launch_after(pk, dim3((unsigned)grid), dim3(PTHREADS), (size_t)PSmem<D>::TOTAL, st, K, V, cur, Mpair, vmax_bits,
                                  p->n_kv, P, (int)tiles, (int)total, F, F_stride, status));
        count_launches(1);
        return cuda_status(cudaGetLastError());
    }
    auto kern = gram_walk_kernel<D>;
    ELM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<D>::TOTAL));
    const int grid = (int)(total < 2 * sm_count ? total : 2 * sm_count);
    ELM_CUDA_TRY(launch_after(kern, dim3((unsigned)grid), dim3(NTHREADS), (size_t)Smem<D>::TOTAL, st, K, V, cur, Mpair, vmax_bits,
                              p->n_kv, P, Ptotal, (int)tiles, (int)total, status, wk));
    count_launches(1);
    return cuda_status(cudaGetLastError());
}

}  // namespace gramtc

int gram_tc(const __nv_bfloat16 *K, const __nv_bfloat16 *V, const elm_params *p, const int32_t *cur,
            const float *Mpair, const unsigned *vmax_bits, int P, int64_t Ptotal, int groups, float *F,
            int64_t F_stride, int *status, const WalkArgs &wk, cudaStream_t st)
{
    if (p->d == 64) return gramtc::launch<64>(K, V, p, cur, Mpair, vmax_bits, P, Ptotal, groups, F, F_stride, status, wk, st);
    return gramtc::launch<128>(K, V, p, cur, Mpair, vmax_bits, P, Ptotal, groups, F, F_stride, status, wk, st);
}

}  // namespace elm
