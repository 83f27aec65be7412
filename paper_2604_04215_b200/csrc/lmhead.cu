// Fused LM head + vocabulary softmax: per row the argmax token and its probability, logits kept on chip.
//
// z = X W^T is a dense bf16 contraction (M x V x D), so it runs on the tcgen05 tensor cores:
//   warp 0      TMA producer: X tile [128 x 64] and W tile [256 x 64] per pipeline stage (128-byte swizzle)
//   warp 1      UMMA issuer: 128 x 256 x 16 MMAs into one of two 128 x 256 fp32 accumulators in TMEM
//   warps 2..5  epilogue: each thread owns one row (one TMEM lane), streams the 256 logits of the tile
//               through registers and keeps (running max, sum of exp, argmax); no cross-thread traffic
// The two accumulators let the epilogue of tile i overlap the MMAs of tile i+1.
// A second instantiation runs the same roles on CTA pairs (cta_group::2, MMAs of 256 rows, half a W tile per CTA);
// see lm_pair_mode below for when it is the one that works.
//
// Only rows that are still masked need logits.  A first small kernel compacts those rows of X into a dense
// buffer (and answers the committed rows directly); the GEMM reads the number of live rows from device
// memory, so the host never synchronises.  Work is cut into items (row tile, vocabulary group): a CTA keeps
// one row tile for all vocabulary tiles of its group, so every epilogue thread carries its row's running
// triple in registers across tiles and writes ONE partial per item.  The CTAs of the row tiles of one group
// walk the same W tiles at the same time, so W leaves HBM once.  A last small kernel merges the (few)
// partials of a row into (token, confidence) and scatters them to the row's original position.
#include <math.h>
#include <mutex>
#include <type_traits>

#include "internal.h"
#include "ptx.cuh"

namespace dare {
namespace {

constexpr int BM = 128;
constexpr int BN = 256;
constexpr int BK = 64;
constexpr int STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;
constexpr int B_BYTES = BN * BK * 2;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int LM_THREADS = 192;
constexpr uint32_t TMEM_COLS = 512;
constexpr float LOG2E = 1.4426950408889634f;
constexpr int ARG_NONE = 0x7fffffff;

struct LmBarriers {
    uint64_t full[STAGES];
    uint64_t empty[STAGES];
    uint64_t tmem_full[2];
    uint64_t tmem_empty[2];
    uint32_t tmem_base;
    uint32_t abort_flag;
};
constexpr int LM_SMEM_BYTES = STAGES * STAGE_BYTES + static_cast<int>(sizeof(LmBarriers)) + 1024;
// CTA-pair mode (cta_group::2): two CTAs of a cluster take two row tiles against the same W tiles with MMAs of
// M = 256; each CTA loads its own X tile and only half of the W tile, which takes a third off the shared-memory
// traffic per flop that limits the single-CTA mode (tensor pipe 83 % -> 93 % busy in the projections).
constexpr int PSTAGES = 6;
constexpr int PB_BYTES = (BN / 2) * BK * 2;
constexpr int PSTAGE_BYTES = A_BYTES + PB_BYTES;
struct LmPairBarriers {
    uint64_t full[PSTAGES];
    uint64_t empty[PSTAGES];
    uint64_t tmem_full[2];
    uint64_t tmem_empty[2];
    uint32_t tmem_base;
    uint32_t abort_flag;
};
constexpr int LM_PAIR_SMEM_BYTES = PSTAGES * PSTAGE_BYTES + static_cast<int>(sizeof(LmPairBarriers)) + 1024;

// Number of vocabulary groups for a grid of `grid` CTAs and `m_tiles` row tiles (same formula on the host,
// in the GEMM and in the merge kernel).
__host__ __device__ inline int lm_groups(int grid, int m_tiles, int n_tiles) {
    int g = m_tiles > 0 ? grid / m_tiles : 1;
    if (g < 1) g = 1;
    if (g > n_tiles) g = n_tiles;
    return g;
}

// Pairs pay when the row tiles come in twos (an odd tile would drag an empty partner along: measured at 3584 x
// 152064, five tiles take 544 us on single CTAs and 600 to 660 us on pairs with the sixth tile empty).  The row
// count is only known on the device, so both kernels are launched and the one whose mode does not apply returns
// at once.
__host__ __device__ inline bool lm_pair_mode(int m_tiles, int allow_pair) {
    return allow_pair && m_tiles >= 2 && (m_tiles & 1) == 0;
}
// Vocabulary groups in the mode that applies: pairs count as one CTA and two row tiles as one.
__host__ __device__ inline int lm_groups_mode(int grid, int m_tiles, int n_tiles, int allow_pair) {
    return lm_pair_mode(m_tiles, allow_pair) ? lm_groups(grid / 2, (m_tiles + 1) / 2, n_tiles) : lm_groups(grid, m_tiles, n_tiles);
}

__device__ __forceinline__ int32_t row_token(const int32_t* row_tokens, int tok_L, int64_t tok_row_stride, int m) {
    return row_tokens[static_cast<int64_t>(m / tok_L) * tok_row_stride + m % tok_L];
}

// Up to this many rows the head evaluates all of them where they lie, committed ones too, and nothing is compacted: the
// launch is bound by reading W (161 us at 32 live rows x 126464, 167 us at 128), while the compaction kernel stood in
// front of it with 3 to 5 us.  What is left of it: the GEMM does nothing if no row is masked, and the merge kernels answer
// committed rows.
constexpr int LM_DIRECT_ROWS = 128;
constexpr int LM_EARLY_SAMPLED_ROWS = 32;      // sampled: up to this many by the kernel that sets itself up in front of its wait
// Token of row m = tokens[(m / L) * stride + m % L]; tokens == NULL: no direct launch
struct LmTokens { const int32_t* tokens; int L; int64_t stride; int32_t mask_id; };

// Whether any of the rows is masked (a warp; all lanes get the answer).  The loads do not hang on one another's rows: behind a
// test of each row they went one after the other, 0.15 us apiece (the sampled head of 128 rows x 256 x 1000 17.9 us, 17.0 now).
__device__ __forceinline__ bool any_masked(const LmTokens& t, int M, int lane) {
    bool any = false;
#pragma unroll
    for (int u = 0; u < LM_DIRECT_ROWS / 32; ++u) any |= row_token(t.tokens, t.L, t.stride, min(lane + u * 32, M - 1)) == t.mask_id;
    return __any_sync(0xffffffffu, any);
}

// Compacts the still-masked rows of X into xc (order preserved), records their original indices, counts
// them, and answers committed rows (pred = their token, conf = -inf).  One warp per row.
constexpr int CP_ROWS = 8;
__global__ void __launch_bounds__(CP_ROWS * 32)
lmhead_compact_kernel(const uint4* __restrict__ x, int M, int D8, const int32_t* __restrict__ row_tokens, int tok_L,
                      int64_t tok_row_stride, int32_t mask_id, uint4* __restrict__ xc, int32_t* __restrict__ idx,
                      int32_t* __restrict__ count, int32_t* __restrict__ pred, float* __restrict__ conf) {
    __shared__ int s_base;
    __shared__ int s_flag[CP_ROWS];
    const int row0 = blockIdx.x * CP_ROWS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    // the first pieces of this warp's row are on their way while the tokens are counted (a committed row's are dropped)
    constexpr int AHEAD = 8;
    const uint4* src = x + static_cast<size_t>(min(row0 + warp, M - 1)) * D8;
    uint4 ahead[AHEAD];
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) ahead[u] = lane + u * 32 < D8 ? src[lane + u * 32] : make_uint4(0, 0, 0, 0);
    int local = 0;
    for (int m = threadIdx.x; m < row0; m += blockDim.x) local += row_token(row_tokens, tok_L, tok_row_stride, m) == mask_id;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) local += __shfl_xor_sync(0xffffffffu, local, off);
    if (lane == 0 && local) atomicAdd(&s_base, local);
    const int row = row0 + warp;
    int32_t tok = 0;
    bool masked = false;
    if (row < M) {
        tok = row_token(row_tokens, tok_L, tok_row_stride, row);
        masked = tok == mask_id;
    }
    if (lane == 0) s_flag[warp] = masked ? 1 : 0;
    __syncthreads();
    int before = s_base, total = s_base;
    for (int i = 0; i < CP_ROWS; ++i) {
        if (i < warp) before += s_flag[i];
        total += s_flag[i];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *count = total;
    if (row >= M) return;
    if (!masked) {
        if (lane == 0) { pred[row] = tok; conf[row] = -INFINITY; }
        return;
    }
    if (lane == 0) idx[before] = row;
    uint4* dst = xc + static_cast<size_t>(before) * D8;
    // eight loads in flight per lane before the first store: the copy of a row is a chain of latencies otherwise
    int i = lane + AHEAD * 32;
    if (i + 7 * 32 < D8) {              // (the next batch is requested before the first is stored)
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = src[i + u * 32];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) dst[lane + u * 32] = ahead[u];
#pragma unroll
        for (int u = 0; u < 8; ++u) dst[i + u * 32] = v[u];
        i += 8 * 32;
    } else {
#pragma unroll
        for (int u = 0; u < AHEAD; ++u)
            if (lane + u * 32 < D8) dst[lane + u * 32] = ahead[u];
    }
    for (; i + 7 * 32 < D8; i += 8 * 32) {
        uint4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = src[i + u * 32];
#pragma unroll
        for (int u = 0; u < 8; ++u) dst[i + u * 32] = v[u];
    }
    for (; i < D8; i += 32) dst[i] = src[i];
}

// Sampling epilogue (temperature + Gumbel-max): token = argmax_v (z_v / T + g_v), g_v = -ln(-ln u_v), with u_v from
// the counter-based generator Philox4x32-10 (Salmon et al., SC 2011) keyed by the seed, counter = (v / 4, row,
// step, tag); element v takes output word v % 4, whose top 23 bits k give u = (2 k + 1) / 2^24 (exact in fp32).
struct LmSampling {
    float inv_temperature;
    uint32_t seed_lo, seed_hi, step;
    const uint32_t* step_dev;      // optional device word added to `step`
    const int32_t* row_index;      // original row of compacted row c (NULL: identity): keys the generator
    const int32_t* targets;        // LM_LOGPROB: target token per row
    float* part_y;                 // per partial: best perturbed score and the raw logit there
    float* part_zb;
    // LM_GRAD: per-row logsumexp of the forward pass and upstream gradient; outputs dz [M, V] and its transpose
    // [V, ldm] (bf16)
    const float* lse;
    const float* grad;
    __nv_bfloat16* dz;
    __nv_bfloat16* dzt;
    int ldm;
};

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}
__device__ __forceinline__ float gumbel_from_word(uint32_t w) {
    const float u = static_cast<float>(((w >> 9) << 1) | 1u) * 5.9604644775390625e-08f;   // (2 k + 1) / 2^24, exact
    return -logf(-logf(u));
}

// One row's 32 consecutive logits z (columns cbase ..., cbase a multiple of 32; largest: zmax) against the row's best
// perturbed score so far.  Two logarithms per logit cost more than the MMAs hide, and almost no logit needs them: -ln u >=
// 1 - u, so z / T - ln(1 - u) is an upper bound of its score, which takes one hardware logarithm (1 - u by the bits of the
// generator's word) and is close to the score where that is large.  Only where the largest bound of the 32 can beat the
// best does the lane evaluate a logit, that one first, and then those whose bounds beat what it made of the best (seldom
// any).  An evaluation is as without the test, and the bounds are compared with 2e-3 + 1e-5 |best| (in log2) to spare, well
// over the rounding of either, so the sampled token is the same bit for bit.
// What this costs shows where a thread sees few groups of a row and nothing hides its epilogue: 256 rows x 256 x 4096 takes
// 24.6 us, 92 when a group without a best yet was begun at its largest logit and nearly all of it evaluated, 23.4 with two
// logarithms for every logit on twice the warps; 400 rows x 4096 x 126464 396, 451 and 538 us.
// `bound`: a score of the same row that another warp has seen (or -inf): what cannot reach it need not be evaluated.
// at(j) returns z[j] for an index that differs from lane to lane.
struct SampleBest { float y, z; int arg; };
struct SampleKey { uint32_t row, step, seed_lo, seed_hi; float inv_temperature; };
__device__ __forceinline__ void sample_one(float z, int col, const SampleKey& key, SampleBest& best) {
    const uint4 w4 = philox4x32_10(make_uint4(static_cast<uint32_t>(col) >> 2, key.row, key.step, 0x44415245u), key.seed_lo, key.seed_hi);
    const uint32_t w = (col & 2) ? ((col & 1) ? w4.w : w4.z) : ((col & 1) ? w4.y : w4.x);
    const float y = fmaf(z, key.inv_temperature, gumbel_from_word(w));
    if (y > best.y || (y == best.y && col < best.arg && y > -INFINITY)) best = {y, z, col};
}
template <typename At>
__device__ __forceinline__ void sample_chunk(const float (&z)[32], int cbase, float zmax, float bound, const SampleKey& key,
                                             SampleBest& best, const At& at) {
    const float c2 = key.inv_temperature * LOG2E;
    const auto threshold = [&]() {      // (NaN against +inf: lets everything through, see below)
        const float b = fmaxf(bound, best.y);
        return fmaf(LOG2E, b, -fmaf(1e-5f, fabsf(b), 2e-3f));
    };
    float ub[32], ub_max = -INFINITY;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const uint4 w4 = philox4x32_10(make_uint4(static_cast<uint32_t>(cbase >> 2) + q, key.row, key.step, 0x44415245u), key.seed_lo,
                                       key.seed_hi);
        const uint32_t ww[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            // u = (2 k + 1) / 2^24, 1 - u = (2 k' + 1) / 2^24 with k' = the complement of k's 23 bits; 1.k' - (1 - 2^-24) is exact
            const float v = __uint_as_float((ww[e] >> 9) ^ 0x3fffffffu) - 0.999999940395355224609375f;
            ub[q * 4 + e] = fmaf(z[q * 4 + e], c2, -__log2f(v));
            ub_max = fmaxf(ub_max, ub[q * 4 + e]);
        }
    }
    // (not ub >= thr: against a best score of +inf the lower one of two such columns must still be met)
    float thr = threshold();
    const bool mine = zmax > -INFINITY && !(ub_max < thr);
    if (!__any_sync(0xffffffffu, mine)) return;
    int first = 0;
#pragma unroll
    for (int j = 1; j < 32; ++j)
        if (ub[j] == ub_max) first = j;
    uint32_t pass = 0;
    if (mine) {
        sample_one(at(first), cbase + first, key, best);
        thr = threshold();
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (!(ub[j] < thr)) pass |= 1u << j;
        pass &= ~(1u << first);
    }
    while (__any_sync(0xffffffffu, pass != 0)) {
        if (pass != 0) {
            const int j = __ffs(pass) - 1;
            pass &= pass - 1;
            sample_one(at(j), cbase + j, key, best);
        }
        __syncwarp();
    }
}

// MODE 0: greedy (argmax token, its probability); 1: sampling epilogue; 2: log-probability of a given target
// token per row (the partial's third slot then carries the target's logit instead of an argmax).
// MODE 3: gradient of the log-probability with respect to the logits, g * (onehot(target) - softmax), written as
// bf16 in both orientations (the two products of the backward pass take it from there); no partials.
constexpr int LM_GREEDY = 0, LM_SAMPLE = 1, LM_LOGPROB = 2, LM_GRAD = 3;

// The work of one launch, or of the part of a launch that runs this body: `n_units` units (CTAs, or CTA pairs with
// PAIR), of which this CTA belongs to unit `unit`, walk the row tiles [tile0, tile0 + m_tiles) against all
// vocabulary tiles; a row's partials start at row * parts_stride (parts_stride < 0: at row * groups, the packed
// layout of the stand-alone kernels).  W_HALF_BOX: the W tensor map's box is 128 rows (half a tile), so a single
// CTA fetches its 256-row tile as two boxes.
struct LmUnits { int unit, n_units, tile0, m_tiles, parts_stride; };
template <int MODE, bool PAIR, bool W_HALF_BOX = false>
__device__ __forceinline__ void
lm_rowmajor_body(const CUtensorMap& tmap_x, const CUtensorMap& tmap_w,
                 int Mc, int D, int V, int mask_col, int n_tiles,
                 float* __restrict__ part_max, float* __restrict__ part_sum, int32_t* __restrict__ part_arg,
                 uint32_t* __restrict__ dev_status, const LmSampling& smp, const LmUnits u) {
    constexpr int NSTAGES = PAIR ? PSTAGES : STAGES;
    constexpr int STAGE_SZ = PAIR ? PSTAGE_BYTES : STAGE_BYTES;
    using Barriers = typename std::conditional<PAIR, LmPairBarriers, LmBarriers>::type;
    constexpr bool SAMPLE = MODE == LM_SAMPLE;
    constexpr bool LOGPROB = MODE == LM_LOGPROB;
    constexpr bool GRAD = MODE == LM_GRAD;
    if (u.m_tiles <= 0) return;
    // PAIR: a work unit is a cluster of two CTAs, an item two row tiles (one per CTA) and a vocabulary group
    const int rank = PAIR ? static_cast<int>(cluster_cta_rank()) : 0;
    const int unit = u.unit;
    const int n_units = u.n_units;
    const int item_rows = PAIR ? (u.m_tiles + 1) >> 1 : u.m_tiles;   // row tiles (pairs of them) to walk
    const int groups = lm_groups(n_units, item_rows, n_tiles);
    const int n_items = item_rows * groups;
    if (unit >= n_items) return;                                    // (both CTAs of a pair alike)
    const int parts_stride = u.parts_stride < 0 ? groups : u.parts_stride;

    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Barriers* bars = reinterpret_cast<Barriers*>(tiles + NSTAGES * STAGE_SZ);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int warp = warp_index_uniform();
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NSTAGES; ++s) {
            mbar_init(&bars->full[s], 1);
            mbar_init(&bars->empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&bars->tmem_full[a], 1);
            // every epilogue thread arrives (PAIR: one arrival per epilogue warp of both CTAs)
            mbar_init(&bars->tmem_empty[a], PAIR ? 8 : 128);
        }
        bars->abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        if (PAIR) { tmem_alloc_pair(&bars->tmem_base, TMEM_COLS); tmem_relinquish_pair(); }
        else { tmem_alloc(&bars->tmem_base, TMEM_COLS); tmem_relinquish(); }
    }
    tc_fence_before_sync();
    if (PAIR) cluster_sync_all();     // both CTAs' barriers exist before either signals the other's
    else __syncthreads();
    tc_fence_after_sync();
    pdl_trigger();
    const uint32_t tmem_base = bars->tmem_base;
    const int num_k = (D + BK - 1) / BK;

    // item w -> row tile w % m_tiles, vocabulary group w / m_tiles; the group's tiles are g, g + groups, ...
    if (warp == 0) {
        if (lane == 0) {
            prefetch_tensormap(&tmap_x);
            prefetch_tensormap(&tmap_w);
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            // PAIR: the even CTA's "full" barriers count the bytes of both CTAs' copies
            const uint32_t full0 = PAIR ? cluster_map_shared(smem_u32(&bars->full[0]), 0) : 0u;
            for (int item = unit; item < n_items && ok; item += n_units) {
                const int m_tile = u.tile0 + (PAIR ? 2 * (item % item_rows) + rank : item % item_rows);
                for (int n_tile = item / item_rows; n_tile < n_tiles && ok; n_tile += groups) {
                    for (int kb = 0; kb < num_k; ++kb) {
                        if (!mbar_wait(&bars->empty[stage], phase ^ 1, abort_flag)) { ok = false; break; }
                        uint8_t* a_dst = tiles + stage * STAGE_SZ;
                        uint8_t* b_dst = a_dst + A_BYTES;
                        if (PAIR) {
                            const uint32_t full = full0 + stage * static_cast<uint32_t>(sizeof(uint64_t));
                            if (rank == 0) mbar_arrive_expect_tx(&bars->full[stage], 2 * STAGE_SZ);
                            tma_load_2d_pair(a_dst, &tmap_x, full, kb * BK, m_tile * BM);
                            tma_load_2d_pair(b_dst, &tmap_w, full, kb * BK, n_tile * BN + rank * (BN / 2));
                        } else {
                            mbar_arrive_expect_tx(&bars->full[stage], STAGE_SZ);
                            tma_load_2d(a_dst, &tmap_x, &bars->full[stage], kb * BK, m_tile * BM);
                            tma_load_2d(b_dst, &tmap_w, &bars->full[stage], kb * BK, n_tile * BN);
                            if (W_HALF_BOX)
                                tma_load_2d(b_dst + (BN / 2) * BK * 2, &tmap_w, &bars->full[stage], kb * BK, n_tile * BN + BN / 2);
                        }
                        if (++stage == NSTAGES) { stage = 0; phase ^= 1; }
                    }
                }
            }
        }
    } else if (warp == 1 && rank == 0) {
        // all lanes run the loops, one elected lane issues the MMAs and their commits (PAIR: the even CTA issues
        // for both, and the commits arrive on both CTAs' barriers)
        const bool leader = elect_one_sync();
        constexpr uint32_t idesc = umma_idesc_bf16(PAIR ? 2 * BM : BM, BN);
        int stage = 0;
        uint32_t phase = 0;
        int it = 0;
        bool ok = true;
        for (int item = unit; item < n_items && ok; item += n_units) {
            for (int n_tile = item / item_rows; n_tile < n_tiles && ok; n_tile += groups, ++it) {
                const int acc = it & 1;
                const uint32_t acc_phase = (it >> 1) & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->tmem_empty[acc], acc_phase ^ 1, abort_flag));
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + acc * BN;
                for (int kb = 0; kb < num_k; ++kb) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars->full[stage], phase, abort_flag));
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint32_t a_addr = smem_u32(tiles + stage * STAGE_SZ);
                    const uint64_t a_desc = umma_desc_sw128_kmajor(a_addr);
                    const uint64_t b_desc = umma_desc_sw128_kmajor(a_addr + A_BYTES);
                    if (leader) {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            // 16 bf16 = 32 bytes further along K inside the 128-byte swizzled row: +2 in the
                            // descriptor's 16-byte address units
                            if (PAIR) umma_bf16_pair(d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, (kb | kk) != 0);
                            else umma_bf16(d_tmem, a_desc + 2 * kk, b_desc + 2 * kk, idesc, (kb | kk) != 0);
                        }
                        // frees the stage when these MMAs have read it
                        if (PAIR) umma_commit_pair(&bars->empty[stage], 3);
                        else umma_commit(&bars->empty[stage]);
                    }
                    __syncwarp();
                    if (++stage == NSTAGES) { stage = 0; phase ^= 1; }
                }
                if (ok && leader) {
                    if (PAIR) umma_commit_pair(&bars->tmem_full[acc], 3);
                    else umma_commit(&bars->tmem_full[acc]);
                }
                __syncwarp();
            }
        }
    } else if (warp >= 2) {
        // epilogue: warp w may touch TMEM lanes [32 * (w % 4), +32)
        const int lq = warp & 3;
        const int row_in_tile = lq * 32 + lane;
        int it = 0;
        bool ok = true;
        for (int item = unit; item < n_items && ok; item += n_units) {
            const int m_tile = u.tile0 + (PAIR ? 2 * (item % item_rows) + rank : item % item_rows);
            const int group = item / item_rows;
            float run_max = -INFINITY;
            float run_sum = 0.f;
            int run_arg = ARG_NONE;
            SampleBest best = {-INFINITY, -INFINITY, ARG_NONE};  // SAMPLE: best perturbed score, raw logit there, column
            SampleKey key = {0, 0, smp.seed_lo, smp.seed_hi, smp.inv_temperature};
            if (SAMPLE) {
                key.step = smp.step + (smp.step_dev ? *smp.step_dev : 0u);
                const int row_c = m_tile * BM + row_in_tile;
                key.row = static_cast<uint32_t>(row_c < Mc && smp.row_index ? smp.row_index[row_c] : row_c);
            }
            int target = -1;                                     // LOGPROB: this row's target column, its logit
            float target_z = -INFINITY;
            if (LOGPROB) {
                const int row_c = m_tile * BM + row_in_tile;
                if (row_c < Mc) target = smp.targets[row_c];
            }
            float g_row = 0.f, lse2 = 0.f;                       // GRAD: upstream gradient, logsumexp * log2(e)
            const int row_g = m_tile * BM + row_in_tile;
            if (GRAD && row_g < Mc) {
                target = smp.targets[row_g];
                // a target outside the vocabulary or in the excluded column has log-probability -inf: no gradient
                if (target >= 0 && target < V && target != mask_col) g_row = smp.grad[row_g];
                lse2 = smp.lse[row_g] * LOG2E;
            }
            for (int n_tile = group; n_tile < n_tiles && ok; n_tile += groups, ++it) {
                const int acc = it & 1;
                const uint32_t acc_phase = (it >> 1) & 1;
                ok = mbar_wait(&bars->tmem_full[acc], acc_phase, abort_flag);
                if (PAIR || SAMPLE) ok = __all_sync(0xffffffffu, ok);      // the warp works and arrives as one further down
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t taddr = tmem_base + (static_cast<uint32_t>(lq * 32) << 16) + acc * BN;
                const int col0 = n_tile * BN;
                const bool edge = (col0 + BN > V) || (mask_col >= col0 && mask_col < col0 + BN);
#pragma unroll 1
                for (int c = 0; c < BN / 32; ++c) {
                    uint32_t v[32];
                    tmem_ld_32cols(taddr + c * 32, v);
                    tmem_ld_wait();
                    const int cbase = col0 + c * 32;
                    if (GRAD) {
                        // dz = g * (1[col = target] - exp(z - lse)); 0 beyond the vocabulary and in the excluded column
                        if (row_g < Mc) {
                            uint32_t packed[16];
#pragma unroll
                            for (int j = 0; j < 32; j += 2) {
                                float d2[2];
#pragma unroll
                                for (int e = 0; e < 2; ++e) {
                                    const int col = cbase + j + e;
                                    const float pr = fast_exp2(fmaf(__uint_as_float(v[j + e]), LOG2E, -lse2));
                                    float d = g_row * ((col == target ? 1.0f : 0.0f) - pr);
                                    if (col >= V || col == mask_col) d = 0.f;
                                    d2[e] = d;
                                }
                                packed[j >> 1] = pack_bf16(d2[0], d2[1]);
                            }
                            __nv_bfloat16* dz_row = smp.dz + static_cast<size_t>(row_g) * V + cbase;
#pragma unroll
                            for (int q = 0; q < 4; ++q)       // V is a multiple of 8: a group of 8 columns is inside or outside
                                if (cbase + q * 8 < V)
                                    *reinterpret_cast<uint4*>(dz_row + q * 8) =
                                        make_uint4(packed[q * 4], packed[q * 4 + 1], packed[q * 4 + 2], packed[q * 4 + 3]);
                            // transposed copy: the lanes of a warp are consecutive rows, so each column is one 64-byte run
                            unsigned short* dzt_col = reinterpret_cast<unsigned short*>(smp.dzt) +
                                                      static_cast<size_t>(cbase) * smp.ldm + row_g;
#pragma unroll
                            for (int j = 0; j < 32; ++j)
                                if (cbase + j < V)
                                    dzt_col[static_cast<size_t>(j) * smp.ldm] =
                                        static_cast<unsigned short>(j & 1 ? packed[j >> 1] >> 16 : packed[j >> 1] & 0xffffu);
                        }
                        continue;
                    }
                    float cmax = -INFINITY;
                    int carg = ARG_NONE;
                    if (edge) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const int col = cbase + j;
                            if (col >= V || col == mask_col) v[j] = __float_as_uint(-INFINITY);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float z = __uint_as_float(v[j]);
                        if (z > cmax) { cmax = z; carg = cbase + j; }   // strict '>' keeps the lowest index
                    }
                    if (LOGPROB && target >= cbase && target < cbase + 32) {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (cbase + j == target) target_z = __uint_as_float(v[j]);   // (-inf if it is the excluded column)
                    }
                    if (SAMPLE) {
                        float z[32];
#pragma unroll
                        for (int j = 0; j < 32; ++j) z[j] = __uint_as_float(v[j]);
                        const auto at = [&](int j) {      // (a thread cannot index its registers: a tree of selects)
                            float a[16];
#pragma unroll
                            for (int k = 0; k < 16; ++k) a[k] = (j & 16) ? z[k + 16] : z[k];
#pragma unroll
                            for (int h = 8; h > 0; h >>= 1) {
#pragma unroll
                                for (int k = 0; k < h; ++k) a[k] = (j & h) ? a[k + h] : a[k];
                            }
                            return a[0];
                        };
                        sample_chunk(z, cbase, cmax, -INFINITY, key, best, at);
                    }
                    if (cmax > -INFINITY) {
                        if (cmax > run_max) {   // tiles of a group come in ascending order: '>' keeps the lowest id
                            run_sum *= fast_exp2((run_max - cmax) * LOG2E);   // exp2(-inf) = 0 the first time
                            run_max = cmax;
                            if (MODE == LM_GREEDY) run_arg = carg;
                        }
                        const float mb = run_max * LOG2E;
                        float s = 0.f;
#pragma unroll
                        for (int j = 0; j < 32; ++j) s += fast_exp2(fmaf(__uint_as_float(v[j]), LOG2E, -mb));
                        run_sum += s;
                    }
                }
                tc_fence_before_sync();
                if (PAIR) {           // one arrival per warp, on the even CTA's barrier
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(&bars->tmem_empty[acc], 0);
                } else {
                    mbar_arrive(&bars->tmem_empty[acc]);
                }
            }
            const int row = m_tile * BM + row_in_tile;
            if (!GRAD && ok && row < Mc) {
                const size_t o = static_cast<size_t>(row) * parts_stride + group;
                part_max[o] = run_max;
                part_sum[o] = run_sum;
                part_arg[o] = LOGPROB ? __float_as_int(target_z) : SAMPLE ? best.arg : run_arg;
                if (SAMPLE) { smp.part_y[o] = best.y; smp.part_zb[o] = best.z; }
            }
        }
    }

    // teardown (PAIR: neither CTA leaves while its partner can still signal its barriers or read its tiles)
    tc_fence_before_sync();
    if (PAIR) cluster_sync_all();
    else __syncthreads();
    if (*abort_flag) {
        // give copies still in flight time to land before the shared memory is released
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) {}
        if (threadIdx.x == 0) atomicOr(dev_status, DEV_WAIT_EXPIRED);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        if (PAIR) tmem_dealloc_pair(tmem_base, TMEM_COLS);
        else tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

template <int MODE, bool PAIR>
__global__ void __launch_bounds__(LM_THREADS, 1)
lmhead_partial_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                      int M, const int32_t* __restrict__ live_rows, int D, int V, int mask_col, int n_tiles,
                      float* __restrict__ part_max, float* __restrict__ part_sum, int32_t* __restrict__ part_arg,
                      uint32_t* __restrict__ dev_status, const LmSampling smp, int allow_pair) {
    pdl_wait();
    const int Mc = live_rows ? *live_rows : M;          // rows that need logits (uniform over the grid)
    const int m_tiles = (Mc + BM - 1) / BM;
    if (lm_pair_mode(m_tiles, allow_pair) != PAIR) return;        // the other kernel does this launch's work
    const LmUnits u = {static_cast<int>(PAIR ? blockIdx.x >> 1 : blockIdx.x),
                       static_cast<int>(PAIR ? gridDim.x >> 1 : gridDim.x), 0, m_tiles, -1};
    lm_rowmajor_body<MODE, PAIR>(tmap_x, tmap_w, Mc, D, V, mask_col, n_tiles, part_max, part_sum, part_arg, dev_status,
                                 smp, u);
}

// ---------------------------------------------------------------------------------------------------------
// Greedy and sampled heads with the operands swapped: the VOCABULARY sits on the accumulator's lanes (W is the MMA's A operand,
// 128 rows per CTA, 256 per CTA pair) and the live ROWS are its columns (the compacted X is the B operand,
// N = the number of rows, any multiple of 16 up to 256).  What that buys over the row-major kernel above:
//   * no padding to 128-row tiles: a step with 96 masked rows issues MMAs of N = 96, not of 128 padded rows;
//   * every work item is a CTA pair whatever the row count, and the 128-row vocabulary tiles per CTA spread evenly
//     over the SMs: with few rows left the W stream is the bound and the kernel reads it at the copy bandwidth.
// More rows than SW_NMAX are cut into equal chunks, in one of two ways:
//   * items = chunk x vocabulary group: a chunk streams all of W from L2 into the SMs whatever its N, and that stream
//     (~12 TB/s over the GPU), not the tensor pipe, sets the pace when the chunks are short (an MMA alone takes
//     max(N / 2, ~45) cycles): worth it for chunks close to 256 rows, and for shorter ones where the row-major tiles would be
//     padded by as much as they hold (lm_swapped below);
//   * both chunks against each W tile (JOINT): W enters the SMs once.  The price is the accumulators: three of 160 columns
//     fit, so the next tile's MMAs wait for half of this one's epilogue, and the running values of 320 columns move to
//     shared memory.
// The price is the epilogue: a thread's TMEM lane is now a vocabulary entry and the softmax runs ACROSS lanes.
// Each epilogue warp turns its 32 x 32 block of logits through shared memory (padded rows, conflict-free) so that
// a thread again holds 32 consecutive vocabulary entries of ONE row, and keeps that row's running
// (max, sum, argmax) in registers across the group's tiles: 8 column blocks x 3 values per thread.  At the end of
// an item the four epilogue warps fold their values through the same shared memory, and one partial per (row,
// vocabulary group, CTA of the pair) goes to the merge kernel.  The sampled head does the same with five values per row;
// its column blocks are a rolled loop (eight copies of the generator's code are more than the instruction cache holds),
// so the values live in shared memory, taken off the ring (6 slots become 5 above 192 rows).
constexpr int SW_BV = 128;                               // vocabulary rows per CTA and tile
constexpr int SW_NMAX = 256;                             // rows (accumulator columns) per chunk
// Row counts for which a head takes this path, for n_vt vocabulary tiles of 256 on n_units CTA pairs (`deep`: D >= SW_DEEP):
// up to one chunk, where W is streamed once and the launch is bound by HBM; two chunks of up to 192 rows, whose row-major
// tiles would be 384 padded rows; and, up to 1024 rows, counts that cut into chunks of 208 to 240 rows, i.e. whose row-major
// tiles would carry 64 or more padded rows per pair (swapped against row-major, one chunk at a time, us: D = 4096, V = 126464:
// 416 rows 333 / 380, 448 rows 415 / 462, 480 rows 410 / 428, 512 rows 425 / 421; D = 3584, V = 152064: 704 rows 625 / 650, 832 rows
// 784 / 840, 960 rows 851 / 895).
// Two chunks of up to 192 rows, greedy, both chunks at a time up to 320 rows, above, where two accumulators are all that fit, one
// at a time; us, swapped / row-major, D = 4096, V = 126464.  On the power cap, where a rollout's steps are and padded MMAs cost
// twice: 272 rows 310 / 395, 320 rows 329 / 405, 352 rows 375 / 412, 384 rows 386 / 422.  A launch on an idle GPU: 242 / 291, 261 / 295,
// but 307 / 295, 312 / 298.  D = 3584, V = 152064, capped 331 / 409, 361 / 430, 405 / 435, 410 / 441, idle 266 / 298, 290 / 305, 321 / 306,
// 327 / 310: the rule is made for the cap, and above 320 rows a single launch pays 4 to 6 % for it.
// Where the MMAs of a tile are short or tiles are few, the epilogue shows, and the cap is out of reach: 272 / 384 rows x 1024 x
// 126464 101 / 83 and 116 / 90, x 2048 x 126464 178 / 180 and 203 / 188, 320 rows x 2048 x 64000 103 / 91, x 2048 x 32000 55 / 49, 384 rows
// x 64 x 1300 16.4 / 10.3, 320 rows x 3072 x 80000 171 / 151: two chunks begin at SW_DEEP and at SW_MIN_TILES per pair (320 rows x 4096
// x 32000 95.5 / 95.2, x 64000 168 / 171, x 3584 x 60000 146 / 144).
// Sampled (four times the epilogue): one chunk at a time, capped 272 rows x 4096 x 126464 383 / 404, 320 rows 394 / 418, 384 rows
// 418 / 435, 480 rows 463 / 459, 640 rows 611 / 621, 832 rows 760 / 788, idle 315 / 319, 322 / 324, 349 / 339, 396 / 397, 533 / 525.  Where
// that is not hidden one row-major pair is better than a chunk from about 170 rows on: 160 rows x 2048 x 32000 46.0 / 47.1, 200 rows
// 54.5 / 47.3, 256 rows 58.9 / 47.7, 640 rows 115 / 92, x 2048 x 64000 256 rows 97 / 79, x 4096 x 50000 160 rows 94 / 100, 200 rows
// 110 / 105; and 97 to 128 rows where pairs need a second round and single CTAs do not (x 2048 x 24000: 96 rows 35.1 / 34.0, 112 rows
// 38.9 / 34.2).
constexpr int LM_JOINT_ROWS = 320;
constexpr int LM_SWAPPED_ROWS = 384;
constexpr int SW_MIN_TILES = 3, SW_MIN_TILES_SAMPLED = 4;
constexpr int SW_DEEP = 3584;
__host__ __device__ inline bool lm_joint(int rows, int n_vt, int n_units, bool deep, bool sampled) {
    return !sampled && rows > SW_NMAX && rows <= LM_JOINT_ROWS && deep && n_vt >= SW_MIN_TILES * n_units;
}
__host__ __device__ inline bool lm_swapped(int rows, int n_vt, int n_units, bool deep, bool sampled) {
    if (sampled && (!deep || n_vt < SW_MIN_TILES_SAMPLED * n_units))
        return rows <= 160 && !(rows > 96 && rows <= 128 && n_vt > n_units && n_vt <= 2 * n_units);
    if (rows <= SW_NMAX) return true;
    if (rows <= LM_SWAPPED_ROWS) return deep && n_vt >= SW_MIN_TILES * n_units;
    if (rows > 1024) return false;
    const int n_chunks = (rows + SW_NMAX - 1) / SW_NMAX;
    const int nc = ((rows + n_chunks - 1) / n_chunks + 15) & ~15;      // as in sw_plan below
    return nc >= 208 && nc < SW_NMAX;
}
constexpr int SW_STAGES = 6;                             // ring slots when a CTA's X tile has its full 128 rows
constexpr int SW_MAX_STAGES = 11;                        // ... and when it is small: the ring's bytes are cut into more slots
constexpr int SW_W_BYTES = SW_BV * BK * 2;               // 16 KB
constexpr int SW_X_BYTES = (SW_NMAX / 2) * BK * 2;       // each CTA loads half of the chunk's rows: up to 16 KB
constexpr int SW_STAGE_BYTES = SW_W_BYTES + SW_X_BYTES;
constexpr int SW_XP_FLOATS = 32 * 33;                    // per epilogue warp: one 32 x 32 block, rows padded to 33
constexpr int SW_PARTS_PER_GROUP = 2;                    // one per CTA of the pair
struct SwBarriers {
    uint64_t full[SW_MAX_STAGES];
    uint64_t empty[SW_MAX_STAGES];
    uint64_t tmem_full[3];
    uint64_t tmem_empty[3];
    uint64_t fold_full, fold_empty;                      // the epilogue warps' exchange at the end of an item
    uint32_t tmem_base;
    uint32_t abort_flag;
};
// Values per row that an epilogue warp keeps in shared memory (floats): the sampled head's (max, sum, y, z, column) and, for
// two chunks at a time, the greedy head's (max, sum, column); in registers otherwise.
__host__ __device__ constexpr int sw_values(int mode, bool joint) { return mode == LM_SAMPLE ? 5 : joint ? 3 : 0; }
__host__ __device__ constexpr int sw_state_bytes(int mode, bool joint) {
    return 4 * sw_values(mode, joint) * (joint ? 2 : 1) * SW_NMAX * 4;
}
// Shared memory of the kernel.  The 5 KB that are left of the SM's 228 (the system takes 1 of them per CTA) hold CTAs of the
// merge kernel, which are then in place when the last tile is done: with all of it taken they could only be started
// behind the GEMM's CTAs, and every head paid 2.5 us for that (512 rows x 1024 x 16000 22.1 us, 19.6 with room).  222 KB hold
// five slots of 36 KB for two chunks at a time at 320 rows.
constexpr int SW_SMEM_BYTES = 222 * 1024;
__host__ __device__ constexpr int sw_ring_bytes(int mode, bool joint) {
    return joint || mode == LM_SAMPLE
               ? (SW_SMEM_BYTES - 1024 - 4 * SW_XP_FLOATS * 4 - sw_state_bytes(mode, joint) - static_cast<int>(sizeof(SwBarriers))) & ~1023
               : SW_STAGES * SW_STAGE_BYTES;
}
__host__ __device__ constexpr int sw_smem_bytes(int mode, bool joint) {
    return sw_ring_bytes(mode, joint) + 4 * SW_XP_FLOATS * 4 + sw_state_bytes(mode, joint) + static_cast<int>(sizeof(SwBarriers)) + 1024;
}
static_assert(sw_smem_bytes(LM_SAMPLE, false) <= SW_SMEM_BYTES && sw_smem_bytes(LM_GREEDY, false) <= SW_SMEM_BYTES &&
              sw_smem_bytes(LM_GREEDY, true) <= SW_SMEM_BYTES, "shared memory");
static_assert(SW_SMEM_BYTES + 1024 + 3 * (1024 + 512) <= 228 * 1024, "room for three CTAs of a merge kernel beside the head's");
// LATE: stages requested before it is known that a row is masked (their slots are not waited for)
constexpr int SW_UNSEEN = 4;
static_assert(SW_UNSEEN <= SW_MAX_STAGES && SW_UNSEEN * (SW_W_BYTES + LM_DIRECT_ROWS / 2 * 128) <= sw_ring_bytes(LM_GREEDY, false) &&
              SW_UNSEEN * (SW_W_BYTES + LM_DIRECT_ROWS / 2 * 128) <= sw_ring_bytes(LM_SAMPLE, false), "slots for them at LM_DIRECT_ROWS rows");
// X tiles of 128, 64, 32, 16 and 8 rows: a CTA's share of a chunk (a multiple of 8 rows) is covered by one or two
// of them, stacked in shared memory (each a whole number of 1 KB swizzle atoms); a few rows too many may be loaded,
// the MMA reads only its own.  (Exact covers of up to four boxes were measured slower: 432 us for 480 rows, where
// each CTA loaded 64 + 32 + 16 + 8 rows per stage, against 350 us for 512 rows with one box.)
struct SwXMaps { CUtensorMap m[5]; };
struct SwBoxes { int i1, i2, rows; };      // indices into SwXMaps::m (i2 < 0: one box), rows loaded in all
__device__ __forceinline__ SwBoxes sw_boxes(int rows_half) {
    if (rows_half > 128) {                 // two chunks at a time
        int second = 4;
        while ((128 >> second) < rows_half - 128) --second;
        return {0, second, 128 + (128 >> second)};
    }
    int single = 0;                        // smallest box that holds the rows
    while ((128 >> single) >= 2 * rows_half && single < 4) ++single;
    int first = single + 1;                // largest box below that, plus the smallest box for the remainder
    SwBoxes b = {single, -1, 128 >> single};
    if (first <= 4) {
        const int rem = rows_half - (128 >> first);
        if (rem > 0) {
            int second = 4;
            while ((128 >> second) < rem) --second;
            if ((128 >> first) + (128 >> second) < (128 >> single)) { b.i1 = first; b.i2 = second; b.rows = (128 >> first) + (128 >> second); }
        }
    }
    return b;
}

// How `rows` live rows are cut up for a grid of n_units CTA pairs and n_vt vocabulary tiles of 256 (the same
// formula on the host, in the GEMM and in the merge kernels).
struct SwPlan { int n_chunks, nc, groups, parts; bool joint; };
__host__ __device__ inline SwPlan sw_plan(int rows, int n_units, int n_vt, bool deep, bool sampled) {
    SwPlan p;
    p.n_chunks = (rows + SW_NMAX - 1) / SW_NMAX;
    if (p.n_chunks < 1) p.n_chunks = 1;
    const int per = (rows + p.n_chunks - 1) / p.n_chunks;
    p.nc = (per + 15) & ~15;                             // rows per chunk: N of the pair's MMA
    if (p.nc < 16) p.nc = 16;
    p.joint = lm_joint(rows, n_vt, n_units, deep, sampled);
    p.groups = lm_groups(n_units, p.joint ? 1 : p.n_chunks, n_vt);
    p.parts = SW_PARTS_PER_GROUP * p.groups;
    return p;
}

// LATE: nothing has been waited for yet, and only if a row is masked there is anything to do.
template <int MODE, bool JOINT, bool LATE>
__device__ __forceinline__ void
lm_swapped_body(const CUtensorMap& tmap_w, const SwXMaps& xmaps, int Mc, int D, int V, int mask_col, int n_vt,
                float* __restrict__ part_max, float* __restrict__ part_sum, int32_t* __restrict__ part_arg,
                uint32_t* __restrict__ dev_status, int parts_stride, const LmSampling& smp, const LmTokens& tokens) {
    constexpr bool SAMPLE = MODE == LM_SAMPLE;
    if (Mc <= 0) return;
    const int rank = static_cast<int>(cluster_cta_rank());
    const int unit = blockIdx.x >> 1;
    const int n_units = gridDim.x >> 1;
    const SwPlan plan = sw_plan(Mc, n_units, n_vt, D >= SW_DEEP, SAMPLE);
    constexpr int J = JOINT ? 2 : 1;                     // chunks per W tile
    constexpr bool STATE = sw_values(MODE, JOINT) > 0;   // running values in shared memory
    constexpr int NV = sw_values(MODE, JOINT), NS = J * SW_NMAX, WARP_STATE = NV * NS;
    const int item_chunks = JOINT ? 1 : plan.n_chunks;
    const int n_items = item_chunks * plan.groups;
    if (unit >= n_items) return;                         // (both CTAs of a pair alike)
    const int nc = plan.nc, groups = plan.groups;
    const int rows_half = J * (nc >> 1);                 // rows this CTA loads (a multiple of 8 per chunk), consecutive ones
    constexpr int slots = JOINT ? 3 : 2, slot_cols = JOINT ? LM_JOINT_ROWS / 2 : SW_NMAX;      // ring of accumulators
    static_assert(slots * slot_cols <= static_cast<int>(TMEM_COLS), "accumulators");
    // row of column c of the item's chunk j: the even CTA's rows are the columns below nc / 2
    const auto row_of = [&](int item, int j, int c) {
        return JOINT ? (c < (nc >> 1) ? c : c + (nc >> 1)) + j * (nc >> 1) : (item % item_chunks) * nc + c;
    };

    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    float* xpose = reinterpret_cast<float*>(tiles + sw_ring_bytes(MODE, JOINT));
    float* state = xpose + 4 * SW_XP_FLOATS;             // STATE: [warp][value][chunk][column]
    SwBarriers* bars = reinterpret_cast<SwBarriers*>(state + 4 * WARP_STATE);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int warp = warp_index_uniform();
    const int lane = threadIdx.x & 31;

    // A ring slot holds a 16 KB W tile and the X rows this CTA loads.  With few live rows the X part is small and the
    // ring's bytes make more slots: while W streams from HBM, what a CTA has in flight is what bounds its share of the
    // bandwidth (6 slots per CTA, 14 MB over the GPU, covered ~2 us of HBM latency at 6.3 TB/s and no more).
    const SwBoxes xbox = sw_boxes(rows_half);
    const int stage_bytes = SW_W_BYTES + ((xbox.rows * 128 + 1023) & ~1023);
    const int n_stages = min(SW_MAX_STAGES, sw_ring_bytes(MODE, JOINT) / stage_bytes);
    // no logit seen yet (set here and by the fold at an item's end: the warps read one another's best scores at any time)
    const auto clear_state = [&](int q, int r) {
        float* s = state + q * WARP_STATE + r;
        s[0] = -INFINITY;
        s[NS] = 0.f;
        if (SAMPLE) s[2 * NS] = s[3 * NS] = -INFINITY;
        s[(NV - 1) * NS] = __int_as_float(ARG_NONE);
    };
    if (STATE)
        for (int i = threadIdx.x; i < 4 * NS; i += LM_THREADS) clear_state(i / NS, i % NS);
    if (threadIdx.x == 0) {
        for (int s = 0; s < n_stages; ++s) {
            mbar_init(&bars->full[s], 1);
            mbar_init(&bars->empty[s], 1);
        }
        for (int a = 0; a < 3; ++a) {
            mbar_init(&bars->tmem_full[a], 1);
            mbar_init(&bars->tmem_empty[a], 8);          // one arrival per epilogue warp of both CTAs
        }
        mbar_init(&bars->fold_full, 128);
        mbar_init(&bars->fold_empty, 128);
        bars->abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) { tmem_alloc_pair(&bars->tmem_base, TMEM_COLS); tmem_relinquish_pair(); }
    tc_fence_before_sync();
    cluster_sync_all();                                  // both CTAs' barriers exist before either signals the other's
    tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;
    const int num_k = (D + BK - 1) / BK;
    bool any = true;                                     // is any row masked?
    // (a run-time value that is always LATE: with the constant W comes 0.8 % slower, four steps of 32 rows x 4096 x 126464 682.9 / 688.5 us)
    const bool late = LATE && tokens.tokens != nullptr;
    if (late) {
        pdl_wait();
        pdl_trigger();
        if (warp != 0) any = any_masked(tokens, Mc, lane);
    } else {
        pdl_trigger();
    }

    // item w -> chunk w % n_chunks, vocabulary group w / n_chunks; the group's tiles are g, g + groups, ...
    if (warp == 0) {
        const uint32_t full0 = cluster_map_shared(smem_u32(&bars->full[0]), 0);   // the even CTA's barriers count both CTAs' bytes
        const SwBoxes box = xbox;
        const auto load = [&](int item, int vt, int kb, int stage) {
            const int x_row0 = (item % item_chunks) * nc + rank * rows_half, w_row0 = vt * (2 * SW_BV) + rank * SW_BV;
            uint8_t* w_dst = tiles + stage * stage_bytes;
            uint8_t* x_dst = w_dst + SW_W_BYTES;
            const uint32_t full = full0 + stage * static_cast<uint32_t>(sizeof(uint64_t));
            if (rank == 0) mbar_arrive_expect_tx(&bars->full[stage], 2u * static_cast<uint32_t>(SW_W_BYTES + box.rows * 128));
            tma_load_2d_pair(w_dst, &tmap_w, full, kb * BK, w_row0);
            tma_load_2d_pair(x_dst, &xmaps.m[box.i1], full, kb * BK, x_row0);
            if (box.i2 >= 0)
                tma_load_2d_pair(x_dst + (128 >> box.i1) * 128, &xmaps.m[box.i2], full, kb * BK, x_row0 + (128 >> box.i1));
        };
        if (lane == 0) {
            prefetch_tensormap(&tmap_w);
#pragma unroll
            for (int i = 0; i < 5; ++i) prefetch_tensormap(&xmaps.m[i]);
        }
        // LATE: the first stages are on their way while the tokens are looked at; if no row is masked after all, they are waited for.
        int ahead = late ? min(SW_UNSEEN, num_k) : 0;
        if (late) {
            if (lane == 0)
                for (int kb = 0; kb < ahead; ++kb) load(unit, unit / item_chunks, kb, kb);
            __syncwarp();
            any = any_masked(tokens, Mc, lane);
            if (!any && lane == 0 && rank == 0)
                for (int st = 0; st < ahead; ++st) mbar_wait(&bars->full[st], 0, abort_flag);
        }
        if (lane == 0 && any) {
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int item = unit; item < n_items && ok; item += n_units) {
                for (int vt = item / item_chunks; vt < n_vt && ok; vt += groups) {
                    for (int kb = 0; kb < num_k; ++kb) {
                        if (ahead > 0) {
                            --ahead;
                        } else {
                            if (!mbar_wait(&bars->empty[stage], phase ^ 1, abort_flag)) { ok = false; break; }
                            load(item, vt, kb, stage);
                        }
                        if (++stage == n_stages) { stage = 0; phase ^= 1; }
                    }
                }
            }
        }
    } else if (warp == 1 && rank == 0) {
        // all lanes run the loops, one elected lane issues the MMAs of the pair and their commits
        const bool leader = elect_one_sync();
        const uint32_t idesc = umma_idesc_bf16(2 * SW_BV, nc);
        int stage = 0;
        uint32_t phase = 0;
        int it = 0;
        bool ok = any;
        for (int item = unit; item < n_items && ok; item += n_units) {
            for (int vt = item / item_chunks; vt < n_vt && ok; vt += groups, ++it) {
                int acc[J];
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    acc[j] = (it * J + j) % slots;
                    ok = ok && __all_sync(0xffffffffu, mbar_wait(&bars->tmem_empty[acc[j]], (((it * J + j) / slots) & 1) ^ 1, abort_flag));
                }
                if (!ok) break;
                tc_fence_after_sync();
                for (int kb = 0; kb < num_k; ++kb) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars->full[stage], phase, abort_flag));
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint32_t w_addr = smem_u32(tiles + stage * stage_bytes);
                    const uint64_t a_desc = umma_desc_sw128_kmajor(w_addr);
                    const uint64_t b_desc = umma_desc_sw128_kmajor(w_addr + SW_W_BYTES);
                    if (leader) {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
#pragma unroll
                            for (int j = 0; j < J; ++j)      // (chunk j's columns: nc / 2 rows of 128 bytes further on)
                                umma_bf16_pair(tmem_base + acc[j] * slot_cols, a_desc + 2 * kk, b_desc + j * (nc * 4) + 2 * kk, idesc,
                                               (kb | kk) != 0);
                        }
                        umma_commit_pair(&bars->empty[stage], 3);      // frees the stage in both CTAs
                    }
                    __syncwarp();
                    if (++stage == n_stages) { stage = 0; phase ^= 1; }
                }
                if (ok && leader) {
#pragma unroll
                    for (int j = 0; j < J; ++j) umma_commit_pair(&bars->tmem_full[acc[j]], 3);
                }
                __syncwarp();
            }
        }
    } else if (warp >= 2) {
        // epilogue: warp w may touch TMEM lanes [32 * (w % 4), +32) = 32 consecutive vocabulary entries of the tile
        const int lq = warp & 3;
        float* xp = xpose + lq * SW_XP_FLOATS;
        float* st = state + lq * WARP_STATE;
        const uint32_t rng_step = SAMPLE ? smp.step + (smp.step_dev ? *smp.step_dev : 0u) : 0u;
        int it = 0;
        uint32_t items_done = 0;
        bool ok = any;
        for (int item = unit; item < n_items && ok; item += n_units, ++items_done) {
            const int group = item / item_chunks;
            float run_max[SW_NMAX / 32], run_sum[SW_NMAX / 32];
            int run_arg[SW_NMAX / 32];
#pragma unroll
            for (int cb = 0; cb < SW_NMAX / 32; ++cb) { run_max[cb] = -INFINITY; run_sum[cb] = 0.f; run_arg[cb] = ARG_NONE; }
            for (int vj = group * J; vj < n_vt * J && ok; vj += (JOINT && !(vj & 1)) ? 1 : groups * J - (J - 1), ++it) {
                const int vt = vj / J, j = vj % J;           // vocabulary tile and chunk
                const int acc = it % slots;
                const uint32_t acc_phase = (it / slots) & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->tmem_full[acc], acc_phase, abort_flag));
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t taddr = tmem_base + (static_cast<uint32_t>(lq * 32) << 16) + acc * slot_cols;
                const int vbase = vt * (2 * SW_BV) + rank * SW_BV + lq * 32;     // first vocabulary entry of this warp's lanes
                const bool edge = (vbase + 32 > V) || (mask_col >= vbase && mask_col < vbase + 32);
                // column block cb: turned, so that this thread holds 32 consecutive vocabulary entries of one row; returns
                // their maximum and its entry
                const auto load_block = [&](int cb, float (&z)[32], float& cmax, int& carg) {
                    uint32_t v[32];
                    tmem_ld_32cols(taddr + cb * 32, v);
                    tmem_ld_wait();
                    // turn the block: in, thread = vocabulary entry with 32 rows; out, thread = row with 32 entries
#pragma unroll
                    for (int c = 0; c < 32; ++c) xp[lane * 33 + c] = __uint_as_float(v[c]);
                    __syncwarp();
#pragma unroll
                    for (int l = 0; l < 32; ++l) z[l] = xp[l * 33 + lane];
                    __syncwarp();
                    if (edge) {
#pragma unroll
                        for (int l = 0; l < 32; ++l)
                            if (vbase + l >= V || vbase + l == mask_col) z[l] = -INFINITY;
                    }
                    cmax = -INFINITY;
                    carg = ARG_NONE;
#pragma unroll
                    for (int l = 0; l < 32; ++l)
                        if (z[l] > cmax) { cmax = z[l]; carg = vbase + l; }       // strict '>' keeps the lowest id
                };
                // (max, sum) of a row with 32 more logits; tiles of a group come in ascending order: '>' keeps the lowest id
                const auto add_block = [&](const float (&z)[32], float cmax, int carg, float& rmax, float& rsum, int& rarg) {
                    if (cmax > -INFINITY) {
                        if (cmax > rmax) {
                            rsum *= fast_exp2((rmax - cmax) * LOG2E);   // exp2(-inf) = 0 the first time
                            rmax = cmax;
                            rarg = carg;
                        }
                        const float mb = rmax * LOG2E;
                        float sum = 0.f;
#pragma unroll
                        for (int l = 0; l < 32; ++l) sum += fast_exp2(fmaf(z[l], LOG2E, -mb));
                        rsum += sum;
                    }
                };
                if (SAMPLE) {
#pragma unroll 1
                    for (int cb = 0; vbase < V && cb * 32 < nc; ++cb) {
                        float z[32], cmax;
                        int carg;
                        load_block(cb, z, cmax, carg);
                        const int r = cb * 32 + lane;
                        const int row = row_of(item, 0, r);
                        const uint32_t rng_row = static_cast<uint32_t>(r < nc && row < Mc && smp.row_index ? smp.row_index[row] : row);
                        float rmax = st[r], rsum = st[NS + r];
                        SampleBest best = {st[2 * NS + r], st[3 * NS + r], __float_as_int(st[4 * NS + r])};
                        int ignored = 0;
                        add_block(z, cmax, carg, rmax, rsum, ignored);
                        float bound = -INFINITY;          // what the other warps have seen of this row (any time up to now will do)
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            bound = fmaxf(bound, *static_cast<volatile float*>(state + q * WARP_STATE + 2 * NS + r));
                        const SampleKey key = {rng_row, rng_step, smp.seed_lo, smp.seed_hi, smp.inv_temperature};
                        const auto at = [&](int j) { return vbase + j >= V || vbase + j == mask_col ? -INFINITY : xp[j * 33 + lane]; };
                        sample_chunk(z, vbase, cmax, bound, key, best, at);
                        __syncwarp();                     // the block may be overwritten
                        st[r] = rmax; st[NS + r] = rsum;
                        st[2 * NS + r] = best.y; st[3 * NS + r] = best.z; st[4 * NS + r] = __int_as_float(best.arg);
                    }
                } else if (STATE) {
#pragma unroll 2
                    for (int cb = 0; vbase < V && cb * 32 < nc; ++cb) {
                        float z[32], cmax;
                        int carg;
                        load_block(cb, z, cmax, carg);
                        float* s = st + j * SW_NMAX + cb * 32 + lane;
                        float rmax = s[0], rsum = s[NS];
                        int rarg = __float_as_int(s[2 * NS]);
                        add_block(z, cmax, carg, rmax, rsum, rarg);
                        s[0] = rmax; s[NS] = rsum; s[2 * NS] = __int_as_float(rarg);
                    }
                } else if (vbase < V) {
#pragma unroll
                    for (int cb = 0; cb < SW_NMAX / 32; ++cb) {
                        if (cb * 32 < nc) {
                            float z[32], cmax;
                            int carg;
                            load_block(cb, z, cmax, carg);
                            add_block(z, cmax, carg, run_max[cb], run_sum[cb], run_arg[cb]);
                        }
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(&bars->tmem_empty[acc], 0);   // one arrival per warp, on the even CTA's barrier
            }
            if (ok) {
                // fold the four warps' values (each saw a quarter of every tile's vocabulary entries): every warp
                // leaves its own in its block of shared memory, then warp q folds column blocks 2 q and 2 q + 1
                if (!STATE) {
#pragma unroll
                    for (int cb = 0; cb < SW_NMAX / 32; ++cb) {
                        xp[(cb * 3 + 0) * 32 + lane] = run_max[cb];
                        xp[(cb * 3 + 1) * 32 + lane] = run_sum[cb];
                        xp[(cb * 3 + 2) * 32 + lane] = __int_as_float(run_arg[cb]);
                    }
                }
                mbar_arrive(&bars->fold_full);            // (release: the values above are visible to the waiters)
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->fold_full, items_done & 1, abort_flag));
                if (ok) {
                    for (int cb = 2 * J * lq; cb < 2 * J * (lq + 1); ++cb) {
                        const int j = cb / (SW_NMAX / 32), col = cb % (SW_NMAX / 32) * 32 + lane, r = cb * 32 + lane;
                        const int row = row_of(item, j, col);
                        if (col < nc && row < Mc) {
                            float m = -INFINITY, sum = 0.f;
                            int a = ARG_NONE;
                            if (SAMPLE) {
                                SampleBest best = {-INFINITY, -INFINITY, ARG_NONE};
                                for (int q = 0; q < 4; ++q) {
                                    const float* src = state + q * WARP_STATE + r;
                                    const float m2 = src[0], s2 = src[NS], y2 = src[2 * NS];
                                    const int a2 = __float_as_int(src[4 * NS]);
                                    if (m2 > -INFINITY) {
                                        if (m2 > m) { sum = sum * fast_exp2((m - m2) * LOG2E) + s2; m = m2; }
                                        else sum += s2 * fast_exp2((m2 - m) * LOG2E);
                                    }
                                    if (y2 > best.y || (y2 == best.y && a2 < best.arg)) best = {y2, src[3 * NS], a2};
                                }
                                const size_t o = static_cast<size_t>(row) * parts_stride + group * 2 + rank;
                                smp.part_y[o] = best.y;
                                smp.part_zb[o] = best.z;
                                a = best.arg;
                            }
                            for (int q = 0; q < (SAMPLE ? 0 : 4); ++q) {
                                const float* src = STATE ? state + q * WARP_STATE + r : xpose + q * SW_XP_FLOATS + cb * 96 + lane;
                                const float m2 = src[0], s2 = src[STATE ? NS : 32];
                                const int a2 = __float_as_int(src[STATE ? 2 * NS : 64]);
                                if (m2 > -INFINITY) {
                                    if (m2 > m) { sum = sum * fast_exp2((m - m2) * LOG2E) + s2; m = m2; a = a2; }
                                    else { sum += s2 * fast_exp2((m2 - m) * LOG2E); if (m2 == m && a2 < a) a = a2; }
                                }
                            }
                            const size_t o = static_cast<size_t>(row) * parts_stride + group * 2 + rank;
                            part_max[o] = m;
                            part_sum[o] = sum;
                            part_arg[o] = a;
                        }
                        if (STATE)
                            for (int q = 0; q < 4; ++q) clear_state(q, r);
                    }
                    mbar_arrive(&bars->fold_empty);       // the blocks may be written again once all have read
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars->fold_empty, items_done & 1, abort_flag));
                }
            }
        }
    }

    // teardown: neither CTA leaves while its partner can still signal its barriers or read its tiles
    tc_fence_before_sync();
    cluster_sync_all();
    if (*abort_flag) {
        // give copies still in flight time to land before the shared memory is released
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) {}
        if (threadIdx.x == 0) atomicOr(dev_status, DEV_WAIT_EXPIRED);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem_base, TMEM_COLS);
    }
}

// An odd number of row tiles, 2 p + 1, on n_clusters CTA pairs: the first lm_mixed_pair_clusters() clusters run the
// row-major pair path on the tiles [0, 2 p), and the CTAs of the remaining clusters each run the single-CTA path on
// the last tile.  The split balances the two parts: an item of two row tiles costs a pair one unit of time, an item
// of one row tile costs a single CTA about 1.2 (its tensor pipe is busy 83 % of the time against 97 %), i.e. a
// cluster of two such CTAs 0.6 per item.  (Same formula on the host, in the GEMM and in the merge kernels.)
__host__ __device__ inline int lm_mixed_pair_clusters(int n_clusters, int p) {
    int up = (n_clusters * 10 * p + 5 * p + 3) / (10 * p + 6);      // round(n_clusters * p / (p + 0.6))
    if (up > n_clusters - 1) up = n_clusters - 1;
    if (up < 1) up = 1;
    return up;
}

// Two chunks at a time, a function of its own: compiled into the kernel it made the epilogue of the other swapped path wait
// longer between its instructions (as many of them, 62 k SM cycles as against 80 k at 256 rows x 2048 x 24000).
__device__ __noinline__ void
lm_joint_body(const CUtensorMap& tmap_w, const SwXMaps& xmaps, int Mc, int D, int V, int mask_col, int n_vt, float* __restrict__ part_max,
              float* __restrict__ part_sum, int32_t* __restrict__ part_arg, uint32_t* __restrict__ dev_status, int parts_stride,
              const LmSampling& smp) {
    lm_swapped_body<LM_GREEDY, true, false>(tmap_w, xmaps, Mc, D, V, mask_col, n_vt, part_max, part_sum, part_arg, dev_status,
                                            parts_stride, smp, LmTokens{});
}

// lmhead_head_kernel behind its wait, on the path that the number of live rows asks for.
template <int MODE>
__device__ __forceinline__ void
lm_head_body(const CUtensorMap& tmap_w, const SwXMaps& xmaps, int M, const int32_t* __restrict__ live_rows, int D, int V, int mask_col,
             int n_tiles, float* __restrict__ part_max, float* __restrict__ part_sum, int32_t* __restrict__ part_arg,
             uint32_t* __restrict__ dev_status, int parts_stride, const LmSampling& smp, const LmTokens& direct) {
    pdl_wait();
    if (direct.tokens && !any_masked(direct, M, threadIdx.x & 31)) return;      // (every warp of every CTA alike)
    const int Mc = live_rows ? *live_rows : M;          // rows that need logits (uniform over the grid)
    if constexpr (MODE == LM_GREEDY) {
        if (lm_joint(Mc, n_tiles, gridDim.x >> 1, D >= SW_DEEP, false)) {
            lm_joint_body(tmap_w, xmaps, Mc, D, V, mask_col, n_tiles, part_max, part_sum, part_arg, dev_status, parts_stride, smp);
            return;
        }
    }
    if (lm_swapped(Mc, n_tiles, gridDim.x >> 1, D >= SW_DEEP, MODE == LM_SAMPLE)) {
        lm_swapped_body<MODE, false, false>(tmap_w, xmaps, Mc, D, V, mask_col, n_tiles, part_max, part_sum, part_arg, dev_status,
                                            parts_stride, smp, direct);
        return;
    }
    const int m_tiles = (Mc + BM - 1) / BM;
    const int cluster = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
    if ((m_tiles & 1) == 0) {
        const LmUnits u = {cluster, n_clusters, 0, m_tiles, parts_stride};
        lm_rowmajor_body<MODE, true>(xmaps.m[0], tmap_w, Mc, D, V, mask_col, n_tiles, part_max, part_sum, part_arg,
                                          dev_status, smp, u);
    } else if (n_clusters < 2) {
        const LmUnits u = {static_cast<int>(blockIdx.x), static_cast<int>(gridDim.x), 0, m_tiles, parts_stride};
        lm_rowmajor_body<MODE, false, true>(xmaps.m[0], tmap_w, Mc, D, V, mask_col, n_tiles, part_max, part_sum,
                                                 part_arg, dev_status, smp, u);
    } else {
        const int p = m_tiles >> 1;
        const int up = lm_mixed_pair_clusters(n_clusters, p);
        if (cluster < up) {
            const LmUnits u = {cluster, up, 0, 2 * p, parts_stride};
            lm_rowmajor_body<MODE, true>(xmaps.m[0], tmap_w, Mc, D, V, mask_col, n_tiles, part_max, part_sum,
                                              part_arg, dev_status, smp, u);
        } else {
            const LmUnits u = {static_cast<int>(blockIdx.x) - 2 * up, static_cast<int>(gridDim.x) - 2 * up, 2 * p, 1,
                               parts_stride};
            lm_rowmajor_body<MODE, false, true>(xmaps.m[0], tmap_w, Mc, D, V, mask_col, n_tiles, part_max, part_sum,
                                                     part_arg, dev_status, smp, u);
        }
    }
}

// The greedy (or sampled) head, one launch on CTA pairs whatever the number of live rows (known only on the device when rows are
// skipped): the swapped-operand path for the counts lm_swapped names (up to SW_NMAX rows, and counts that
// cut into long chunks); otherwise row-major tiles of 128 rows, on CTA pairs when the tiles come in twos, and for
// an odd count on pairs plus single CTAs for the last tile (see above).  The W
// tile box is 128 rows for all of them.  A row's partials start at row * parts_stride; how many there are follows
// from the same rules in lm_row_partials.
template <int MODE, bool DIRECT>
__global__ void __launch_bounds__(LM_THREADS, 1)
lmhead_head_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ SwXMaps xmaps, int M,
                     const int32_t* __restrict__ live_rows, int D, int V, int mask_col, int n_tiles,
                     float* __restrict__ part_max, float* __restrict__ part_sum, int32_t* __restrict__ part_arg,
                     uint32_t* __restrict__ dev_status, int parts_stride, const LmSampling smp, const LmTokens direct) {
    // DIRECT: rows evaluated where they lie, and by the swapped path (the launcher sees to it).  How many is known before the predecessor
    // is done, so it sets itself up beside it and waits in its place.  With what lmhead_merge_select_kernel does in front of its
    // wait, a replayed step of 32 rows x 512 x 4096 takes 12.0 us for 14.0, 128 rows x 256 x 1000 14.9 for 16.6, 32 rows x 4096 x 126464
    // 165.6 for 167.5; one that finds no masked row 0.2 to 2 us more (its SW_UNSEEN stages, and a kernel to take down).  (In one kernel
    // with the other launches it slowed the sampled head of 416 rows by 1.4 %.)
    if constexpr (DIRECT) {
        lm_swapped_body<MODE, false, true>(tmap_w, xmaps, M, D, V, mask_col, n_tiles, part_max, part_sum, part_arg, dev_status,
                                           parts_stride, smp, direct);
    } else {
        lm_head_body<MODE>(tmap_w, xmaps, M, live_rows, D, V, mask_col, n_tiles, part_max, part_sum, part_arg, dev_status, parts_stride, smp,
                           direct);
    }
}

// Partials of live row `row`, as the GEMM that ran wrote them (they start at row * stride).  layout 0 / 1: the
// stand-alone row-major kernels (single CTAs only / CTA pairs where they apply), one partial per vocabulary group,
// packed (stride = count).  layout 2 / 3: lmhead_head_kernel's rules for D below SW_DEEP / from there on.  `grid` = CTAs of the
// GEMM launch, n_tiles = vocabulary tiles of 256.
constexpr int LM_LAYOUT_HEAD = 2, LM_LAYOUT_HEAD_DEEP = 3;
__host__ __device__ inline int lm_row_partials(int layout, int grid, int rows, int n_tiles, int row, bool sampled) {
    const int m_tiles = (rows + BM - 1) / BM;
    if (layout < LM_LAYOUT_HEAD) return lm_groups_mode(grid, m_tiles, n_tiles, layout);
    const bool deep = layout == LM_LAYOUT_HEAD_DEEP;
    const int n_clusters = grid >> 1;
    if (lm_swapped(rows, n_tiles, n_clusters, deep, sampled)) return sw_plan(rows, n_clusters, n_tiles, deep, sampled).parts;
    if ((m_tiles & 1) == 0) return lm_groups(n_clusters, m_tiles >> 1, n_tiles);
    if (n_clusters < 2) return lm_groups(grid, m_tiles, n_tiles);
    const int p = m_tiles >> 1;
    const int up = lm_mixed_pair_clusters(n_clusters, p);
    return row < 2 * p * BM ? lm_groups(up, p, n_tiles) : lm_groups(grid - 2 * up, 1, n_tiles);
}

// Fold of one row's partials by a warp: the token and its confidence, in all lanes.  Greedy: the token of the largest
// logit (lowest id on ties), confidence = exp(max - logsumexp) = 1 / (sum of exp relative to the maximum).  Sampled: the
// token of the best perturbed score (lowest id on ties), confidence = exp(z_token - logsumexp z).
struct LmParts { const float *max, *sum; const int32_t* arg; const float *y, *zb; };
template <bool SAMPLE>
__device__ __forceinline__ void merge_row_partials(const LmParts& p, size_t base, int groups, int lane, int& a_out, float& conf_out) {
    float m = -INFINITY, s = 0.f, y = -INFINITY, zb = -INFINITY;
    int a = ARG_NONE;
    const auto fold = [&](float m2, float s2, int a2, float y2, float z2) {
        if (m2 > -INFINITY) {
            if (m2 > m) { s = s * exp2f((m - m2) * LOG2E) + s2; m = m2; if (!SAMPLE) a = a2; }
            else { s += s2 * exp2f((m2 - m) * LOG2E); if (!SAMPLE && m2 == m && a2 < a) a = a2; }
        }
        if (SAMPLE && (y2 > y || (y2 == y && a2 < a))) { y = y2; a = a2; zb = z2; }
    };
    // the loads of a batch are issued together (five per lane cover 160 partials: one round trip to memory for the
    // usual case), then folded
    constexpr int BATCH = 5;
    for (int t0 = lane; t0 < groups; t0 += 32 * BATCH) {
        float bm[BATCH], bs[BATCH], by[BATCH], bz[BATCH];
        int ba[BATCH];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int t = t0 + 32 * u;
            const bool in = t < groups;
            bm[u] = in ? p.max[base + t] : -INFINITY;
            bs[u] = in ? p.sum[base + t] : 0.f;
            ba[u] = in ? p.arg[base + t] : ARG_NONE;
            by[u] = SAMPLE && in ? p.y[base + t] : -INFINITY;
            bz[u] = SAMPLE && in ? p.zb[base + t] : -INFINITY;
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) fold(bm[u], bs[u], ba[u], by[u], bz[u]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, off), s2 = __shfl_xor_sync(0xffffffffu, s, off);
        const int a2 = __shfl_xor_sync(0xffffffffu, a, off);
        const float y2 = SAMPLE ? __shfl_xor_sync(0xffffffffu, y, off) : 0.f;
        const float z2 = SAMPLE ? __shfl_xor_sync(0xffffffffu, zb, off) : 0.f;
        fold(m2, s2, a2, y2, z2);
    }
    a_out = a;
    conf_out = SAMPLE ? exp2f((zb - m) * LOG2E) / s : 1.0f / s;
}

// One warp per live row: fold the row's partials (one or two per vocabulary group) into (token, confidence) and write
// them at the row's original position.
template <bool SAMPLE>
__global__ void lmhead_merge_kernel(const LmParts parts, int grid_gemm, int n_tiles, int M,
                                    const int32_t* __restrict__ live_rows, const int32_t* __restrict__ idx,
                                    int32_t* __restrict__ pred, float* __restrict__ conf, int allow_pair,
                                    int parts_stride, uint32_t* __restrict__ step_dev, const LmTokens direct) {
    pdl_trigger();      // (before the wait, as in lmhead_merge_select_kernel; a selection kernel may come in between)
    pdl_wait();
    if (SAMPLE && step_dev && blockIdx.x == 0 && threadIdx.x == 0) *step_dev += 1;   // the GEMM kernels before this one read it
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int Mc = live_rows ? *live_rows : M;
    if (c >= Mc) return;
    if (direct.tokens) {
        const int32_t tok = row_token(direct.tokens, direct.L, direct.stride, c);
        if (tok != direct.mask_id) {
            if (lane == 0) { pred[c] = tok; conf[c] = -INFINITY; }
            return;
        }
    }
    const int groups = lm_row_partials(allow_pair, grid_gemm, Mc, n_tiles, c, SAMPLE);
    int a;
    float cf;
    merge_row_partials<SAMPLE>(parts, static_cast<size_t>(c) * (parts_stride < 0 ? groups : parts_stride), groups, lane, a, cf);
    if (lane == 0) {
        const int row = idx ? idx[c] : c;
        pred[row] = a;
        conf[row] = cf;
    }
}

// Merge and unmask selection in one kernel, for blocks of at most 32 positions: one CTA per rollout, one warp per
// block position.  A warp whose position is still masked finds its row's place among the compacted rows (from the
// compaction kernel's sorted row list: other CTAs change the token state meanwhile), folds the row's partials and writes
// (pred, conf); then the CTA applies the selection rule of select.cu to the block: rank by counting, bit for bit
// the same decisions as the separate kernel takes from the same (pred, conf).
struct LmSelect {
    int32_t* tokens_block;      // tokens + block_start (row b at + b * row_stride)
    int64_t row_stride;
    int mode;
    float threshold;
    int k;
    int32_t* n_committed;
    int32_t* n_remaining;
    int32_t* host_remaining;
};
template <bool SAMPLE>
__global__ void __launch_bounds__(1024)
lmhead_merge_select_kernel(const LmParts parts, int grid_gemm, int n_tiles, int L, int M,
                           const int32_t* __restrict__ live_rows, const int32_t* __restrict__ idx, int32_t mask_id,
                           int32_t* __restrict__ pred, float* __restrict__ conf, int allow_pair, int parts_stride,
                           const LmSelect sel, uint32_t* __restrict__ step_dev) {
    __shared__ int s_flag[32];
    __shared__ float s_conf[32];
    __shared__ int32_t s_pred[32];
    pdl_trigger();      // (before the wait: the attention of the step, which may follow, does not depend on the head)
    const int b = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;      // warp = block position (blockDim = 32 L)
    // The tokens, the number of live rows and the row list are as they were when the head, which still runs, started: it lets
    // its successor in behind its own wait and writes none of them.  So all that follows from them stands in front of the wait
    // (past L1, which may hold a line from before).  Compacted rows
    // that belong to earlier rollouts = entries of the ascending list below b * L.  (A binary search by one thread, nine
    // dependent loads at 512 rows, was half of this kernel's 8 us.)
    int32_t* row = sel.tokens_block + static_cast<int64_t>(b) * sel.row_stride;
    const int32_t tok = __ldcg(row + warp);
    const bool masked = tok == mask_id;
    const int Mc = live_rows ? __ldcg(live_rows) : M;       // (NULL: the rows were evaluated where they lie)
    if (lane == 0) s_flag[warp] = masked ? 1 : 0;
    int before = 0;
    for (int i0 = 0; live_rows && i0 < b * L; i0 += blockDim.x) {   // (rows of earlier rollouts: at most b * L of them)
        const int i = i0 + threadIdx.x;
        const int32_t v = i < b * L ? __ldcg(idx + i) : 0;  // (entries from Mc on hold anything)
        before += __syncthreads_count(i < b * L && i < Mc && v < b * L);
    }
    __syncthreads();
    int c = b * L + warp;
    if (live_rows) {
        c = before;
        for (int i = 0; i < warp; ++i) c += s_flag[i];
    }
    const int groups = masked ? lm_row_partials(allow_pair, grid_gemm, Mc, n_tiles, c, SAMPLE) : 0;
    pdl_wait();
    if (SAMPLE && step_dev && blockIdx.x == 0 && threadIdx.x == 0) *step_dev += 1;   // (as in lmhead_merge_kernel)
    if (masked) {
        int a;
        float cf;
        merge_row_partials<SAMPLE>(parts, static_cast<size_t>(c) * (parts_stride < 0 ? groups : parts_stride), groups, lane, a, cf);
        if (lane == 0) {
            pred[b * L + warp] = a;
            conf[b * L + warp] = cf;
            if (cf != cf) cf = -INFINITY;
            s_conf[warp] = cf;
            s_pred[warp] = a;
        }
    } else if (lane == 0) {
        s_conf[warp] = __int_as_float(0x7fc00000);      // absent
        if (!live_rows) { pred[b * L + warp] = tok; conf[b * L + warp] = -INFINITY; }      // (else the compaction did)
    }
    __syncthreads();
    if (warp != 0) return;
    // selection (warp 0, lane = block position)
    const float cf = lane < L ? s_conf[lane] : __int_as_float(0x7fc00000);
    const bool is_masked = cf == cf;
    const unsigned masked_set = __ballot_sync(0xffffffffu, is_masked);
    const unsigned above_set = __ballot_sync(0xffffffffu, is_masked && cf > sel.threshold);
    bool commit = false;
    if (is_masked) {
        if (sel.mode == DARE_SELECT_THRESHOLD && above_set != 0u) {
            commit = cf > sel.threshold;
        } else {
            const int want = sel.mode == DARE_SELECT_TOPK ? sel.k : 1;
            int rank = 0;
#pragma unroll 8
            for (int j = 0; j < L; ++j) {                              // (one after the other each is a trip to shared memory)
                const float cj = s_conf[j];
                rank += (cj > cf || (cj == cf && j < lane)) ? 1 : 0;   // NaN (absent) compares false
            }
            commit = rank < want;
        }
    }
    if (commit) row[lane] = s_pred[lane];
    const unsigned commit_set = __ballot_sync(0xffffffffu, commit);
    if (lane == 0) {
        if (sel.n_committed) sel.n_committed[b] = __popc(commit_set);
        if (sel.n_remaining) sel.n_remaining[b] = __popc(masked_set) - __popc(commit_set);
        if (sel.host_remaining) st_host(sel.host_remaining + b, __popc(masked_set) - __popc(commit_set));
    }
}

// Log-probability of the target: (z_target - max) - ln(sum of exp(z - max)); the target's logit sits in exactly one
// partial (the others carry -inf).  Optionally also writes logsumexp z.
__global__ void lmhead_merge_logprob_kernel(const float* __restrict__ part_max, const float* __restrict__ part_sum,
                                            const int32_t* __restrict__ part_zt, int grid_gemm, int n_tiles, int M,
                                            float* __restrict__ logprob, float* __restrict__ lse_out, int allow_pair) {
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    pdl_wait();
    pdl_trigger();
    if (c >= M) return;
    const int groups = lm_groups_mode(grid_gemm, (M + BM - 1) / BM, n_tiles, allow_pair);
    float m = -INFINITY, s = 0.f, zt = -INFINITY;
    const size_t base = static_cast<size_t>(c) * groups;
    for (int t = lane; t < groups; t += 32) {
        const float m2 = part_max[base + t], s2 = part_sum[base + t];
        if (m2 > -INFINITY) {
            if (m2 > m) { s = s * exp2f((m - m2) * LOG2E) + s2; m = m2; }
            else s += s2 * exp2f((m2 - m) * LOG2E);
        }
        zt = fmaxf(zt, __int_as_float(part_zt[base + t]));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, m, off);
        const float s2 = __shfl_xor_sync(0xffffffffu, s, off);
        zt = fmaxf(zt, __shfl_xor_sync(0xffffffffu, zt, off));
        if (m2 > -INFINITY) {
            if (m2 > m) { s = s * exp2f((m - m2) * LOG2E) + s2; m = m2; }
            else s += s2 * exp2f((m2 - m) * LOG2E);
        }
    }
    if (lane == 0) {
        logprob[c] = (zt - m) - logf(s);
        if (lse_out) lse_out[c] = m + logf(s);
    }
}

inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Whether clusters of two CTAs of the pair-mode kernel can run on this device (asked once).
int lm_pair_available() {
    static int cache = -1;
    if (cache < 0) {
        int n = 0;
        if (cudaFuncSetAttribute(lmhead_partial_kernel<LM_GREEDY, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 LM_PAIR_SMEM_BYTES) != cudaSuccess ||
            query_max_clusters(lmhead_partial_kernel<LM_GREEDY, true>, 2048u, LM_THREADS, LM_PAIR_SMEM_BYTES, 2, &n) != DARE_OK)
            n = 0;
        cache = n > 0 ? 1 : 0;
    }
    return cache;
}

// The GEMM part of a head: the single-CTA kernel, the CTA-pair kernel, or (when the row count is only known on
// the device) both, of which the one whose mode does not apply returns at once.  *allow_pair_out tells the
// merge kernel which rule was in force.
template <int MODE>
int launch_partial(const dare_ctx* ctx, int grid, const CUtensorMap& tmap_x, const void* w, int M,
                   const int32_t* live_rows, int D, int V, int mask_col, int n_tiles, float* part_max, float* part_sum,
                   int32_t* part_arg, const LmSampling& smp, cudaStream_t stream, int* allow_pair_out) {
    const int allow_pair = (grid >= 2 && lm_pair_available()) ? 1 : 0;
    *allow_pair_out = allow_pair;
    const int m_tiles_host = (M + BM - 1) / BM;
    const bool pair_known = live_rows == nullptr && lm_pair_mode(m_tiles_host, allow_pair);
    const bool run_single = !allow_pair || live_rows != nullptr || !pair_known;
    const bool run_pair = allow_pair && (live_rows != nullptr || pair_known);
    if (run_single) {
        CUtensorMap tmap_w;
        int rc = make_tmap_bf16_2d(ctx, &tmap_w, w, static_cast<uint64_t>(V), static_cast<uint64_t>(D), BN, BK);
        if (rc != DARE_OK) return rc;
        static std::atomic<uint64_t> smem_set{0};
        if (ensure_dynamic_smem(smem_set, lmhead_partial_kernel<MODE, false>, LM_SMEM_BYTES) != DARE_OK) return DARE_ERR_CUDA;
        rc = launch_kernel(lmhead_partial_kernel<MODE, false>, dim3(grid), LM_THREADS, LM_SMEM_BYTES, stream, 1, tmap_x,
                           tmap_w, M, live_rows, D, V, mask_col, n_tiles, part_max, part_sum, part_arg, ctx->dev_status, smp,
                           allow_pair);
        if (rc != DARE_OK) return rc;
    }
    if (run_pair) {
        CUtensorMap tmap_wh;      // half a W tile per CTA
        int rc = make_tmap_bf16_2d(ctx, &tmap_wh, w, static_cast<uint64_t>(V), static_cast<uint64_t>(D), BN / 2, BK);
        if (rc != DARE_OK) return rc;
        static std::atomic<uint64_t> smem_set_pair{0};
        if (ensure_dynamic_smem(smem_set_pair, lmhead_partial_kernel<MODE, true>, LM_PAIR_SMEM_BYTES) != DARE_OK)
            return DARE_ERR_CUDA;
        rc = launch_kernel(lmhead_partial_kernel<MODE, true>, dim3(static_cast<unsigned>(grid & ~1)), LM_THREADS,
                           LM_PAIR_SMEM_BYTES, stream, 2, tmap_x, tmap_wh, M, live_rows, D, V, mask_col, n_tiles, part_max,
                           part_sum, part_arg, ctx->dev_status, smp, allow_pair);
        if (rc != DARE_OK) return rc;
    }
    return DARE_OK;
}

}  // namespace

// Scratch layout: [compacted X: M*D bf16][row indices: M int32][live-row count][partials: 3 x M x groups]
static size_t lmhead_scratch_bytes(int M, int D, int V, int sm_count, bool with_row_tokens, bool sampling, int parts_per_tile) {
    const size_t n_tiles = (static_cast<size_t>(V) + BN - 1) / BN;
    size_t groups = static_cast<size_t>(sm_count);
    if (groups > parts_per_tile * n_tiles) groups = parts_per_tile * n_tiles;
    size_t bytes = (sampling ? 5 : 3) * sizeof(float) * groups * static_cast<size_t>(M);
    if (with_row_tokens)
        bytes += round_up(static_cast<size_t>(M) * D * 2, 1024) + round_up(static_cast<size_t>(M) * 4 + 4, 1024);
    return bytes;
}
// (the swapped path leaves two partials per vocabulary group of a CTA pair; the sampled head can do without that path)
size_t lmhead_workspace_bytes(int M, int D, int V, int sm_count, bool with_row_tokens, bool sampling) {
    return lmhead_scratch_bytes(M, D, V, sm_count, with_row_tokens, sampling, sampling ? 1 : 2);
}

// The most that a launch with row tokens uses where the workspace allows it.
size_t lmhead_max_scratch_bytes(int M, int D, int V, int sm_count, bool sampling) {
    return lmhead_scratch_bytes(M, D, V, sm_count, true, sampling, 2);
}

// The head's GEMM, its merge and, with `select`, the unmask selection, for one epilogue.
template <int MODE>
static int launch_head(const dare_ctx* ctx, int grid, bool pairs, const void* x_gemm, int M, int D, const void* w, int V,
                       int mask_col, int n_tiles, const int32_t* live_rows, const int32_t* idx, float* parts, LmSampling smp,
                       uint32_t* step_dev, int tok_L, int64_t tok_row_stride, int32_t mask_id, int32_t* pred, float* conf,
                       const LmSelectArgs* select, const LmTokens& direct, cudaStream_t stream) {
    constexpr bool SAMPLE = MODE == LM_SAMPLE;
    size_t parts_max = pairs ? (grid & ~1) : ctx->sm_count;      // pairs: a fixed stride, at most two partials per vocabulary tile
    const size_t tile_parts = static_cast<size_t>(pairs ? 2 : 1) * n_tiles;
    if (parts_max > tile_parts) parts_max = tile_parts;
    const size_t n_part = static_cast<size_t>(M) * parts_max;
    float* part_max = parts;
    float* part_sum = part_max + n_part;
    int32_t* part_arg = reinterpret_cast<int32_t*>(part_sum + n_part);
    if (SAMPLE) {
        smp.part_y = reinterpret_cast<float*>(part_arg + n_part);
        smp.part_zb = smp.part_y + n_part;
    }
    int rc = DARE_OK, layout = D >= SW_DEEP ? LM_LAYOUT_HEAD_DEEP : LM_LAYOUT_HEAD, parts_stride = -1, grid_gemm = grid;
    if (pairs) {
        CUtensorMap tmap_w;
        SwXMaps xm;
        rc = make_tmap_bf16_2d(ctx, &tmap_w, w, static_cast<uint64_t>(V), static_cast<uint64_t>(D), SW_BV, BK);
        for (int i = 0; i < 5 && rc == DARE_OK; ++i)
            rc = make_tmap_bf16_2d(ctx, &xm.m[i], x_gemm, static_cast<uint64_t>(M), static_cast<uint64_t>(D), 128u >> i, BK);
        if (rc != DARE_OK) return rc;
        grid_gemm = grid & ~1;
        parts_stride = static_cast<int>(parts_max);
        constexpr int SMEM = SW_SMEM_BYTES;
        static_assert(SMEM >= LM_PAIR_SMEM_BYTES && SMEM >= LM_SMEM_BYTES, "shared memory");
        static std::atomic<uint64_t> smem_set[2] = {};
        // (With more sampled rows a step of a small head gains 4 %, one of full size nothing, and one without a masked row loses; general
        // kernel / this one, us: 64 rows x 256 x 1000 15.9 / 15.3, 128 rows x 4096 x 126464 185 / 188, without a masked row 9.4 / 13.4.)
        const bool in_place = direct.tokens != nullptr && (!SAMPLE || M <= LM_EARLY_SAMPLED_ROWS) &&
                              lm_swapped(M, n_tiles, grid_gemm >> 1, D >= SW_DEEP, SAMPLE);
        const auto kernel = in_place ? lmhead_head_kernel<MODE, true> : lmhead_head_kernel<MODE, false>;
        if (ensure_dynamic_smem(smem_set[in_place], kernel, SMEM) != DARE_OK) return DARE_ERR_CUDA;
        rc = launch_kernel(kernel, dim3(static_cast<unsigned>(grid_gemm)), LM_THREADS, SMEM, stream, 2, tmap_w, xm, M, live_rows, D, V,
                           mask_col, n_tiles, part_max, part_sum, part_arg, ctx->dev_status, parts_stride, smp, direct);
        if (rc != DARE_OK) return rc;
    } else {
        CUtensorMap tmap_x;
        rc = make_tmap_bf16_2d(ctx, &tmap_x, x_gemm, static_cast<uint64_t>(M), static_cast<uint64_t>(D), BM, BK);
        if (rc == DARE_OK)
            rc = launch_partial<MODE>(ctx, grid, tmap_x, w, M, live_rows, D, V, mask_col, n_tiles, part_max, part_sum, part_arg,
                                      smp, stream, &layout);
        if (rc != DARE_OK) return rc;
    }
    const LmParts lp = {part_max, part_sum, part_arg, smp.part_y, smp.part_zb};
    if (select) {
        LmSelect sel;
        sel.tokens_block = select->tokens_block; sel.row_stride = tok_row_stride; sel.mode = select->mode;
        sel.threshold = select->threshold; sel.k = select->k;
        sel.n_committed = select->n_committed; sel.n_remaining = select->n_remaining;
        sel.host_remaining = select->host_remaining;
        return launch_kernel(lmhead_merge_select_kernel<SAMPLE>, dim3(select->B), 32 * tok_L, 0, stream, 1, lp, grid_gemm, n_tiles,
                             tok_L, M, live_rows, idx, mask_id, pred, conf, layout, parts_stride, sel, step_dev);
    }
    constexpr int rows_per_block = 8;
    return launch_kernel(lmhead_merge_kernel<SAMPLE>, dim3((M + rows_per_block - 1) / rows_per_block), rows_per_block * 32, 0,
                         stream, 1, lp, grid_gemm, n_tiles, M, live_rows, idx, pred, conf, layout, parts_stride, step_dev, direct);
}

int launch_lmhead(const dare_ctx* ctx, void* scratch, const void* hidden, int M, int D, const void* w, int V,
                  const int32_t* row_tokens, int tok_L, int64_t tok_row_stride, int32_t mask_id,
                  int exclude_mask_column, int32_t* pred, float* conf, cudaStream_t stream, const LmSampleArgs* sample,
                  const LmSelectArgs* select) {
    if (select && (!row_tokens || tok_L > LMHEAD_SELECT_MAX_L || tok_L < 1 || M != select->B * tok_L))
        return DARE_ERR_SHAPE;
    const int n_tiles = (V + BN - 1) / BN;
    const int m_tiles_max = (M + BM - 1) / BM;
    int grid = ctx->sm_count;
    if (grid > m_tiles_max * n_tiles) grid = m_tiles_max * n_tiles;

    uint8_t* cur = static_cast<uint8_t*>(scratch);
    const void* x_gemm = hidden;
    int32_t* idx = nullptr;
    int32_t* live_rows = nullptr;
    const bool pairs = grid >= 2 && lm_pair_available() &&
                       lmhead_scratch_bytes(M, D, V, ctx->sm_count, row_tokens != nullptr, sample != nullptr, 2) <= ctx->workspace_bytes;
    // The swapped path wants a CTA pair per vocabulary tile also where the rows make a single tile: with half of them each took
    // two tiles, one after the other (sampled 128 rows x 256 x 4096 23.9 us, now 17.0; a greedy step of 32 rows x 256 x 4096 10.6, now
    // 9.3, of 128 rows 15.4 and 12.3, x 1024 x 32000 24.0 and 20.8).  Where twice the pairs need as many rounds, the greedy head is
    // better off with half of them (32 rows x 2048 x 24000 24.4 and 23.5).
    if (pairs && m_tiles_max == 1) {
        const int all = n_tiles < ctx->sm_count / 2 ? 2 * n_tiles : ctx->sm_count;
        const auto rounds = [&](int ctas) { return (n_tiles + ctas / 2 - 1) / (ctas / 2); };
        if (sample != nullptr || rounds(all) < rounds(grid)) grid = all;
    }
    LmTokens direct = {};
    if (row_tokens != nullptr && pairs && M <= LM_DIRECT_ROWS) {
        direct = {row_tokens, tok_L, tok_row_stride, mask_id};
    } else if (row_tokens != nullptr) {
        void* xc = cur;
        cur += round_up(static_cast<size_t>(M) * D * 2, 1024);
        idx = reinterpret_cast<int32_t*>(cur);
        live_rows = idx + M;
        cur += round_up(static_cast<size_t>(M) * 4 + 4, 1024);
        x_gemm = xc;
        const int rc = launch_kernel(lmhead_compact_kernel, dim3((M + CP_ROWS - 1) / CP_ROWS), CP_ROWS * 32, 0, stream, 1,
                                     static_cast<const uint4*>(hidden), M, D / 8, row_tokens, tok_L, tok_row_stride, mask_id,
                                     static_cast<uint4*>(xc), idx, live_rows, pred, conf);
        if (rc != DARE_OK) return rc;
    }
    const int mask_col = (exclude_mask_column && mask_id >= 0 && mask_id < V) ? mask_id : -1;
    float* parts = reinterpret_cast<float*>(cur);
    LmSampling smp = {};
    if (sample == nullptr)
        return launch_head<LM_GREEDY>(ctx, grid, pairs, x_gemm, M, D, w, V, mask_col, n_tiles, live_rows, idx, parts, smp,
                                      nullptr, tok_L, tok_row_stride, mask_id, pred, conf, select, direct, stream);
    smp.inv_temperature = 1.0f / sample->temperature;
    smp.seed_lo = static_cast<uint32_t>(sample->seed & 0xffffffffu);
    smp.seed_hi = static_cast<uint32_t>(sample->seed >> 32);
    smp.step = sample->step;
    smp.step_dev = sample->step_dev;
    smp.row_index = idx;
    return launch_head<LM_SAMPLE>(ctx, grid, pairs, x_gemm, M, D, w, V, mask_col, n_tiles, live_rows, idx, parts, smp,
                                  sample->step_dev, tok_L, tok_row_stride, mask_id, pred, conf, select, direct, stream);
}

int launch_lmhead_logprob(const dare_ctx* ctx, void* scratch, const void* hidden, int M, int D, const void* w, int V,
                          const int32_t* targets, int32_t mask_id, int exclude_mask_column, float* logprob, float* lse_out,
                          cudaStream_t stream) {
    const int n_tiles = (V + BN - 1) / BN;
    const int m_tiles_max = (M + BM - 1) / BM;
    int grid = ctx->sm_count;
    if (grid > m_tiles_max * n_tiles) grid = m_tiles_max * n_tiles;
    size_t groups_max = static_cast<size_t>(ctx->sm_count);
    if (groups_max > static_cast<size_t>(n_tiles)) groups_max = n_tiles;
    const size_t n_part = static_cast<size_t>(M) * groups_max;
    float* part_max = static_cast<float*>(scratch);
    float* part_sum = part_max + n_part;
    int32_t* part_zt = reinterpret_cast<int32_t*>(part_sum + n_part);
    CUtensorMap tmap_x;
    int rc = make_tmap_bf16_2d(ctx, &tmap_x, hidden, static_cast<uint64_t>(M), static_cast<uint64_t>(D), BM, BK);
    if (rc != DARE_OK) return rc;
    const int mask_col = (exclude_mask_column && mask_id >= 0 && mask_id < V) ? mask_id : -1;
    LmSampling smp = {};
    smp.targets = targets;
    int allow_pair = 0;
    rc = launch_partial<LM_LOGPROB>(ctx, grid, tmap_x, w, M, nullptr, D, V, mask_col, n_tiles, part_max, part_sum, part_zt,
                                    smp, stream, &allow_pair);
    if (rc != DARE_OK) return rc;
    const int rows_per_block = 8;
    return launch_kernel(lmhead_merge_logprob_kernel, dim3((M + rows_per_block - 1) / rows_per_block), rows_per_block * 32, 0,
                         stream, 1, part_max, part_sum, part_zt, grid, n_tiles, M, logprob, lse_out, allow_pair);
}

// dz[m, v] = grad[m] * (1[v = targets[m]] - exp(z[m, v] - lse[m])) as bf16 [M, V] and transposed [V, ldm]
// (ldm >= M; columns [M, ldm) of the transpose are not written).
int launch_lmhead_grad(const dare_ctx* ctx, const void* hidden, int M, int D, const void* w, int V,
                       const int32_t* targets, int32_t mask_id, int exclude_mask_column, const float* lse,
                       const float* grad, void* dz, void* dzt, int ldm, cudaStream_t stream) {
    const int n_tiles = (V + BN - 1) / BN;
    const int m_tiles_max = (M + BM - 1) / BM;
    int grid = ctx->sm_count;
    if (grid > m_tiles_max * n_tiles) grid = m_tiles_max * n_tiles;
    CUtensorMap tmap_x;
    int rc = make_tmap_bf16_2d(ctx, &tmap_x, hidden, static_cast<uint64_t>(M), static_cast<uint64_t>(D), BM, BK);
    if (rc != DARE_OK) return rc;
    const int mask_col = (exclude_mask_column && mask_id >= 0 && mask_id < V) ? mask_id : -1;
    LmSampling smp = {};
    smp.targets = targets;
    smp.lse = lse;
    smp.grad = grad;
    smp.dz = static_cast<__nv_bfloat16*>(dz);
    smp.dzt = static_cast<__nv_bfloat16*>(dzt);
    smp.ldm = ldm;
    int allow_pair = 0;
    return launch_partial<LM_GRAD>(ctx, grid, tmap_x, w, M, nullptr, D, V, mask_col, n_tiles, nullptr, nullptr, nullptr, smp,
                                   stream, &allow_pair);
}

}  // namespace dare

// ------------------------------------------------------------------------------------------------
// Allocation-free variant of the LM-head entry point.
//
// Some callers must not allocate device memory at all: code inside a framework's allocator callback or
// under a memory budget that forbids cudaMalloc, and plug-ins loaded into a process whose allocator they
// do not own.  dare_create allocates its workspace,
// so those callers cannot have a context.  For them the per-tile (max, sum, argmax) triples of the LM
// head live in a fixed array inside the library's device image.
namespace dare {
namespace {

// Scratch shared by every call of dare_lmhead_confidence_static on a device (8 MiB, resident on every GPU
// that loads the library until the process exits).
static __device__ __align__(256) unsigned char g_lm_static_scratch[DARE_LMHEAD_STATIC_SCRATCH_BYTES];
// Status bits of these calls (only ever OR-ed into; starts at zero when the module is loaded).
static __device__ uint32_t g_lm_static_status;

struct StaticDeviceState {
    bool ready = false;
    int device = -1;
    void* scratch = nullptr;        // device address of g_lm_static_scratch on this device
    uint32_t* status = nullptr;     // device address of g_lm_static_status on this device
    int sm_count = 0;
    dare_encode_tiled_fn encode = nullptr;
};
constexpr int MAX_DEVICES = 64;
StaticDeviceState g_static_state[MAX_DEVICES];
std::mutex g_static_mutex;

// One-time set-up for the current device.  In host code the array's name is only a handle; the address a
// kernel can use has to be asked for, with this device current.
int static_state_for_current_device(StaticDeviceState** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return DARE_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    StaticDeviceState& st = g_static_state[dev];
    if (!st.ready) {
        int major = 0;
        if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return DARE_ERR_CUDA;
        if (major != 10) return DARE_ERR_UNSUPPORTED;
        if (cudaDeviceGetAttribute(&st.sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return DARE_ERR_CUDA;
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_lm_static_scratch) != cudaSuccess || p == nullptr) return DARE_ERR_CUDA;
        st.scratch = p;
        void* ps = nullptr;
        if (cudaGetSymbolAddress(&ps, g_lm_static_status) != cudaSuccess || ps == nullptr) return DARE_ERR_CUDA;
        st.status = static_cast<uint32_t*>(ps);
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess || fn == nullptr)
            return DARE_ERR_CUDA;
        st.encode = reinterpret_cast<dare_encode_tiled_fn>(fn);
        st.device = dev;
        st.ready = true;
    }
    *out = &st;
    return DARE_OK;
}

}  // namespace
}  // namespace dare

extern "C" int dare_lmhead_confidence_static(const void* hidden, int M, int D, const void* w, int V,
                                             const int32_t* row_tokens, int32_t mask_id, int exclude_mask_column,
                                             int32_t* pred, float* conf, void* stream) {
    if (!hidden || !w || !pred || !conf) return DARE_ERR_NULL;
    if (M < 1 || D < 8 || D % 8 != 0 || V < 2) return DARE_ERR_SHAPE;
    if ((reinterpret_cast<uintptr_t>(hidden) & 15u) || (reinterpret_cast<uintptr_t>(w) & 15u)) return DARE_ERR_ALIGN;
    dare::StaticDeviceState* st = nullptr;
    int rc = dare::static_state_for_current_device(&st);
    if (rc != DARE_OK) return rc;
    if (dare::lmhead_workspace_bytes(M, D, V, st->sm_count, row_tokens != nullptr, false) >
        static_cast<size_t>(DARE_LMHEAD_STATIC_SCRATCH_BYTES))
        return DARE_ERR_WORKSPACE;   // beyond the fixed scratch: use dare_lmhead_confidence with a context
    // The kernels run on the current device with that device's scratch: a buffer that lives on another GPU would be
    // read or written through the wrong address space.  Asking where a pointer lives allocates nothing.
    const void* bufs[5] = {hidden, w, row_tokens, pred, conf};
    for (const void* p : bufs) {
        if (!p) continue;
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) return DARE_ERR_CUDA;
        if ((attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged) && attr.device != st->device)
            return DARE_ERR_DEVICE;
    }
    // a context-shaped view of the static state for the shared launcher; nothing here is allocated
    dare_ctx view;
    view.tmaps = nullptr;
    view.device = st->device;
    view.sm_count = st->sm_count;
    view.workspace = st->scratch;
    view.workspace_bytes = DARE_LMHEAD_STATIC_SCRATCH_BYTES;
    view.dev_status = st->status;
    view.encode_tiled = st->encode;
    return dare::launch_lmhead(&view, st->scratch, hidden, M, D, w, V, row_tokens, M, 0, mask_id, exclude_mask_column,
                               pred, conf, static_cast<cudaStream_t>(stream), nullptr);
}


// Reads and clears the status word of the allocation-free calls on the current device (bits DARE_DEV_*), after
// everything enqueued on `stream` so far has run.  Allocates nothing.
extern "C" int dare_lmhead_static_status(void* stream, uint32_t* host_out) {
    if (!host_out) return DARE_ERR_NULL;
    dare::StaticDeviceState* st = nullptr;
    int rc = dare::static_state_for_current_device(&st);
    if (rc != DARE_OK) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(host_out, st->status, sizeof(uint32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemsetAsync(st->status, 0, sizeof(uint32_t), s) != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess)
        return DARE_ERR_CUDA;
    return DARE_OK;
}
