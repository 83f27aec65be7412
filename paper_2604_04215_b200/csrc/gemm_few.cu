// Projections of up to 128 rows: out = epilogue(A W^T), A [M, K], W [N, K] bf16, fp32 accumulation.
//
// With so few rows the work is reading W once, so everything serves that stream (one rollout's block of 32 rows against
// the layers of the LLaDA shape, us per launch, this kernel / row-major tiles of 128 padded rows, weights from HBM: 12288 x 4096
// 19.6 / 29.6, attention-out 4096 x 4096 10.8 / 18.2, gate and up 2 x 12288 x 4096 35.1 / 42.5, down 4096 x 12288 20.9 / 38.9; W alone
// takes 15.4, 5.1, 30.7 and 15.4 at the measured copy bandwidth; of 128 rows 25.7 / 31.0, 16.8 / 18.6, 41.6 / 43.0, 27.3 / 39.9):
//   * operands swapped: 128 W rows are the MMA's A operand (the accumulator's lanes), the rows of A its N columns, so no
//     padded rows are loaded or multiplied and a ring slot is mostly W;
//   * 128-row W tiles are cut along K until the CTAs fill the SMs twice over: two CTAs per SM keep 192 KB of W in flight at 16
//     rows (six slots of 16 KB each), 160 KB at 17 to 48, 96 KB at 128, and one CTA's first and last microseconds lie under
//     the other's stream;
//   * the first ring of W is requested before the kernel waits for its predecessor (w_static: weights, which no kernel
//     of the library writes), so the stream does not stop between kernels;
//   * the CTAs of a tile's K slices form a cluster; each sends the accumulator columns (rows of A) it does not own to their
//     owner through distributed shared memory, the owners add the slices in order and apply the epilogue: a thread holds 8
//     consecutive features of one row (several slices of up to FEW_QUAD_ROWS rows: two features of four rows, so that four rows go in one remote
//     store), which is what SwiGLU (a tile: 64 gate and the matching 64 up rows), RoPE (a tile holds whole heads; channel c
//     and its partner c + d/2 are in the same slab) and coalesced stores want.
//   warp 0 TMA producer, warp 1 MMA issuer, warps 2..5 epilogue (TMEM lane = W row).
#include <math.h>

#include "internal.h"
#include "ptx.cuh"

namespace dare {
namespace {

constexpr int FW = 128;                       // W rows per tile
constexpr int FK = 64;
constexpr int FEW_THREADS = 192;
constexpr int FEW_W_BYTES = FW * FK * 2;
constexpr int FEW_SMEM = 112 * 1024;          // two CTAs per SM
constexpr int FEW_MAX_STAGES = 6;

struct FewBarriers {
    uint64_t full[FEW_MAX_STAGES];
    uint64_t empty[FEW_MAX_STAGES];
    uint64_t tmem_full;
    uint32_t tmem_base;
    uint32_t abort_flag;
};
constexpr int FEW_RING = FEW_SMEM - 1024 - static_cast<int>(sizeof(FewBarriers));

struct FewPlan {
    int nr;          // rows of A, rounded up to 16: the MMA's N
    int wcols;       // output features per tile (128; SwiGLU: 64)
    int splits;      // CTAs along K per tile = cluster size (1, 2, 4 or 8)
    int stages;
    int tiles;
    int slab;        // QUADS: where the slices are added: its offset in the ring, behind the stages in use (0: over them)
    int quads;       // QUADS: groups of four rows of A that a CTA of a cluster finishes, the last CTAs maybe none (0: not QUADS)
};
// Up to this many rows the slices are handed over four rows at a time (QUADS): value by value the stores to the other CTAs were
// 1.25 of the 3.8 us that a small projection of 48 rows takes behind its wait.  A stack of 3 layers of 512 / 1280 values, us, value by
// value / four rows: 16 rows 78.8 / 78.1, 48 rows 88.9 / 85.5, 64 rows 97.2 / 94.0; 64 rows of 2 layers of 256 62.6 / 60.4, 32 rows of 2
// LLaDA-shaped layers 205.0 / 203.9.  More rows are cut into fewer slices, and a CTA's last part is then the longer one, where
// 16 bytes per load and store count: 72 rows 99.0 / 107.7, 128 rows 136 / 155.  So it is with a single slice, which sends nothing
// (48 rows of 4 LLaDA-shaped layers 421.6 with it, 419.3 without).
constexpr int FEW_QUAD_ROWS = 64;

FewPlan few_plan(int epi, int M, int N, int K, int sm_count) {
    FewPlan p;
    p.nr = (M + 15) & ~15;
    p.wcols = epi == GEMM_EPI_SWIGLU ? FW / 2 : FW;
    p.tiles = (N + p.wcols - 1) / p.wcols;
    const int nk = (K + FK - 1) / FK;
    p.splits = 1;
    // as many K slices as the SMs take with two CTAs each, of at least two K blocks, and of more with more than 64 rows, whose
    // exchange takes longer (128 rows, K = 1024, N = 4096: eight slices 13.0 us, two 9.6; K = 512, N = 1280: 6.7 either way)
    const int least = p.nr > 64 ? p.nr / 16 : 2;
    while (p.splits < 8 && 2LL * p.splits * p.tiles <= 2LL * sm_count && nk >= 2 * least * p.splits) p.splits *= 2;
    // (up to four rows all go to one CTA of the cluster, and eight slices of padded groups then take longer to arrive and to add than single
    // values, once the launch fills the SMs: 1 row x 2048 x 2048 4.0 / 4.4 us, x 1024 x 4096 4.7 / 5.0, x 4096 x 4096 6.6 / 6.8; on fewer CTAs
    // 1 row x 1280 x 512 3.4 / 3.0; 8 rows x 2048 x 2048 with a residual 4.3 / 4.1)
    const bool one_owner = M <= 4 && p.splits == 8 && 4LL * p.splits * p.tiles >= 3LL * sm_count;
    p.quads = p.splits > 1 && p.nr <= FEW_QUAD_ROWS && !one_owner ? (p.nr / 4 + p.splits - 1) / p.splits : 0;
    const int stages = FEW_RING / (FEW_W_BYTES + p.nr * FK * 2);
    p.stages = stages > FEW_MAX_STAGES ? FEW_MAX_STAGES : stages;
    // With so few K blocks per CTA that the slab has room behind their stages, the CTAs of a cluster need not wait for one another's
    // last MMAs before they send (48 rows through three layers of 512 / 1280 values 86.7 us, now 84.8).
    const int kbs = (nk + p.splits - 1) / p.splits, used = (kbs < p.stages ? kbs : p.stages) * (FEW_W_BYTES + p.nr * FK * 2);
    p.slab = p.quads > 0 && used + p.splits * p.quads * FW * 16 <= FEW_RING ? used : 0;
    return p;
}

struct FewArgs {
    int M, N, K, ldo;
    FewPlan p;
    __nv_bfloat16* out;
    const __nv_bfloat16* res;
    uint32_t* dev_status;
    int w_static;
    RopeArgs rope;
};

__device__ __forceinline__ float lo_f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_f(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
    return make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
}
__device__ __forceinline__ float round_bf16(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
__device__ __forceinline__ void st_shared_f32(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_shared_cluster_f32(uint32_t addr, uint32_t v) {
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

template <int EPI, bool QUADS>
__global__ void __launch_bounds__(FEW_THREADS, 2)
gemm_few_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_w2,
                const __grid_constant__ CUtensorMap tmap_a, const FewArgs g) {
    const FewPlan& p = g.p;
    const int stage_bytes = FEW_W_BYTES + p.nr * (FK * 2);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    FewBarriers* bars = reinterpret_cast<FewBarriers*>(tiles + FEW_RING);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int warp = warp_index_uniform();
    const int lane = threadIdx.x & 31;
    const int split = p.splits > 1 ? static_cast<int>(cluster_cta_rank()) : 0;
    const int tile = blockIdx.x / p.splits;
    const int nk = (g.K + FK - 1) / FK;
    const int kb_begin = static_cast<int>(static_cast<long long>(nk) * split / p.splits);
    const int kb_end = static_cast<int>(static_cast<long long>(nk) * (split + 1) / p.splits);
    uint32_t tmem_cols = 32;
    while (static_cast<int>(tmem_cols) < p.nr) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(&bars->full[s], 1);
            mbar_init(&bars->empty[s], 1);
        }
        mbar_init(&bars->tmem_full, 1);
        bars->abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(&bars->tmem_base, tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;
    if (QUADS && p.slab) cluster_arrive();               // (waited for before the hand-over: every CTA of the cluster has started)

    if (warp == 0) {
        if (lane == 0) {
            prefetch_tensormap(&tmap_w);
            prefetch_tensormap(&tmap_a);
            const int w_row = tile * p.wcols;
            const auto load_w = [&](int kb, int st) {
                uint8_t* dst = tiles + st * stage_bytes;
                mbar_arrive_expect_tx(&bars->full[st], stage_bytes);
                tma_load_2d(dst, &tmap_w, &bars->full[st], kb * FK, w_row);
                if (EPI == GEMM_EPI_SWIGLU) tma_load_2d(dst + FEW_W_BYTES / 2, &tmap_w2, &bars->full[st], kb * FK, w_row);
            };
            int ahead = g.w_static ? min(p.stages, kb_end - kb_begin) : 0;
            for (int i = 0; i < ahead; ++i) load_w(kb_begin + i, i);
            pdl_wait();
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = kb_begin; kb < kb_end; ++kb) {
                if (ahead > 0) {
                    --ahead;
                } else {
                    if (!mbar_wait(&bars->empty[stage], phase ^ 1, abort_flag)) break;
                    load_w(kb, stage);
                }
                tma_load_2d(tiles + stage * stage_bytes + FEW_W_BYTES, &tmap_a, &bars->full[stage], kb * FK, 0);
                if (++stage == p.stages) { stage = 0; phase ^= 1; }
            }
        }
    } else if (warp == 1) {
        const bool leader = elect_one_sync();
        const uint32_t idesc = umma_idesc_bf16(FW, p.nr);
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int kb = kb_begin; kb < kb_end; ++kb) {
            ok = __all_sync(0xffffffffu, mbar_wait(&bars->full[stage], phase, abort_flag));
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t w_addr = smem_u32(tiles + stage * stage_bytes);
            const uint64_t a_desc = umma_desc_sw128_kmajor(w_addr);
            const uint64_t b_desc = umma_desc_sw128_kmajor(w_addr + FEW_W_BYTES);
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < FK / 16; ++kk)
                    umma_bf16(tmem_base, a_desc + 2 * kk, b_desc + 2 * kk, idesc, (kb > kb_begin) | (kk != 0));
                umma_commit(&bars->empty[stage]);
            }
            __syncwarp();
            if (++stage == p.stages) { stage = 0; phase ^= 1; }
        }
        if (ok && leader) umma_commit(&bars->tmem_full);
        __syncwarp();
    } else {
        pdl_wait();
        mbar_wait(&bars->tmem_full, 0, abort_flag);      // (a wait that gave up leaves the abort flag set)
        tc_fence_after_sync();
        pdl_trigger();
    }
    __syncwarp();

    // Hand-over: the ring of every CTA of the cluster is idle now (or the slab lies behind it).  Slab of the owner:
    // [K slice][row][128 features], or QUADS [K slice][four rows][128 features][row].
    const int per_owner = p.nr / p.splits;               // rows of A that a CTA finishes (nr is a multiple of 16)
    if (QUADS) {
        if (!p.slab) cluster_arrive();
        cluster_wait();
    } else if (p.splits > 1) {
        cluster_sync_all();
    } else {
        __syncthreads();
    }
    if (QUADS && warp >= 2) {
        const int f = (warp & 3) * 32 + lane;            // W row of the tile = TMEM lane
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const uint32_t slab = smem_u32(tiles) + p.slab + (static_cast<uint32_t>(split) * p.quads * FW + f) * 16;
        int owner = 0, q = 0;
        uint32_t addr = cluster_map_shared(slab, 0u);
        for (int c0 = 0; c0 < g.M; c0 += 16) {           // (columns from M on are padding rows: stored, not read)
            uint32_t v[16];
            tmem_ld_16cols(taddr + c0, v);
            tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < 16; c += 4) {
                if (c0 + c < g.M) st_shared_cluster_v4(addr, v[c], v[c + 1], v[c + 2], v[c + 3]);
                addr += FW * 16;
                if (++q == p.quads) {
                    q = 0;
                    if (++owner < p.splits) addr = cluster_map_shared(slab, static_cast<uint32_t>(owner));
                }
            }
        }
    } else if (warp >= 2) {
        // (owner and row are counted, not divided out, and 16 columns are read at a time: with two divisions per column and
        // every 8 columns waited for, each row cost 68 ns, 128 rows 8.6 us)
        const int f = (warp & 3) * 32 + lane;            // W row of the tile = TMEM lane
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const uint32_t slab = smem_u32(tiles) + (static_cast<uint32_t>(split) * per_owner * FW + f) * 4;
        const auto read16 = [&](int c0, uint32_t (&lo)[8], uint32_t (&hi)[8]) {
            tmem_ld_8cols(taddr + c0, lo);
            tmem_ld_8cols(taddr + c0 + 8, hi);
            tmem_ld_wait();
        };
        uint32_t lo[8], hi[8];
        if (p.splits == 1) {
            for (int c0 = 0; c0 < g.M; c0 += 16) {       // (columns from M on are padding rows: stored, not read)
                read16(c0, lo, hi);
#pragma unroll
                for (int c = 0; c < 16; ++c) st_shared_f32(slab + static_cast<uint32_t>(c0 + c) * (FW * 4), c < 8 ? lo[c & 7] : hi[c & 7]);
            }
        } else {
            int owner = 0, r = 0;
            uint32_t addr = cluster_map_shared(slab, 0u);
            for (int c0 = 0; c0 < g.M; c0 += 16) {
                read16(c0, lo, hi);
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    if (c0 + c < g.M) st_shared_cluster_f32(addr, c < 8 ? lo[c & 7] : hi[c & 7]);
                    addr += FW * 4;
                    if (++r == per_owner) {
                        r = 0;
                        if (++owner < p.splits) addr = cluster_map_shared(slab, static_cast<uint32_t>(owner));
                    }
                }
            }
        }
    }
    if (p.splits > 1) cluster_sync_all();
    else __syncthreads();

    // the last part is for all warps (the first two have not waited for the predecessor with all their lanes yet)
    if (warp < 2) pdl_wait();
    if (QUADS && !*abort_flag) {
        const float4* slab = reinterpret_cast<const float4*>(tiles + p.slab);
        // features f and f + 1 of the four rows of group q, the K slices added in order
        const auto sum = [&](int q, int f, float (&s)[2][4]) {
#pragma unroll
            for (int j = 0; j < 4; ++j) s[0][j] = s[1][j] = 0.f;
            for (int k = 0; k < p.splits; ++k) {
                const float4 a = slab[(k * p.quads + q) * FW + f], b = slab[(k * p.quads + q) * FW + f + 1];
                s[0][0] += a.x; s[0][1] += a.y; s[0][2] += a.z; s[0][3] += a.w;
                s[1][0] += b.x; s[1][1] += b.y; s[1][2] += b.z; s[1][3] += b.w;
            }
        };
        const int t = threadIdx.x;
        const int row0 = split * p.quads * 4;
        const int n_rows = min(p.quads * 4, g.M - row0);   // (may be negative: nothing to do)
        const int n_quads = (n_rows + 3) / 4;
        if (EPI == GEMM_EPI_ROPE) {
            const RopeArgs& r = g.rope;
            const int pph = r.d / 4;                     // channel pairs of half a head
            for (int i = t; i < n_quads * (FW / 4); i += FEW_THREADS) {
                const int q = i / (FW / 4), u = i % (FW / 4);
                const int hh = u / pph, c = (u % pph) * 2;
                const int H = tile * (FW / r.d) + hh;
                if (H >= r.Hq + 2 * r.Hkv) continue;
                const bool turns = H < r.Hq + r.Hkv, k = H < r.Hq + r.Hkv;
                int m[4], pos[4], bb[4];
                float4 e[4];                             // (cos, sin) of the two channels
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    m[j] = min(row0 + q * 4 + j, g.M - 1);
                    bb[j] = m[j] / r.length;
                    pos[j] = r.start + m[j] - bb[j] * r.length;
                    if (turns) e[j] = *reinterpret_cast<const float4*>(r.cs + (static_cast<size_t>(pos[j]) * (r.d / 2) + c) * 2);
                }
                float a[2][4], b[2][4];
                sum(q, hh * r.d + c, a);
                sum(q, hh * r.d + r.d / 2 + c, b);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (q * 4 + j >= n_rows) break;
                    __nv_bfloat16* dst;
                    if (H < r.Hq) {
                        dst = static_cast<__nv_bfloat16*>(r.q_out) + (static_cast<size_t>(m[j]) * r.Hq + H) * r.d;
                    } else {
                        const int h = H - r.Hq - (k ? 0 : r.Hkv);
                        dst = static_cast<__nv_bfloat16*>(k ? r.k_cache : r.v_cache) +
                              ((static_cast<size_t>(bb[j]) * r.Hkv + h) * r.cap + pos[j]) * r.d;
                    }
                    if (turns) {                         // (the projection is rounded to bf16 before it turns)
                        const float x1 = round_bf16(a[0][j]), x2 = round_bf16(b[0][j]), y1 = round_bf16(a[1][j]), y2 = round_bf16(b[1][j]);
                        a[0][j] = x1 * e[j].x - x2 * e[j].y;
                        b[0][j] = x2 * e[j].x + x1 * e[j].y;
                        a[1][j] = y1 * e[j].z - y2 * e[j].w;
                        b[1][j] = y2 * e[j].z + y1 * e[j].w;
                    }
                    *reinterpret_cast<uint32_t*>(dst + c) = pack_bf16(a[0][j], a[1][j]);
                    *reinterpret_cast<uint32_t*>(dst + r.d / 2 + c) = pack_bf16(b[0][j], b[1][j]);
                }
            }
        } else {
            constexpr int pairs = (EPI == GEMM_EPI_SWIGLU ? FW / 2 : FW) / 2;
            for (int i = t; i < n_quads * pairs; i += FEW_THREADS) {
                const int q = i / pairs, f = (i % pairs) * 2, col = tile * p.wcols + f;
                if (col >= g.N) continue;                // (N is a multiple of 8)
                const size_t o = static_cast<size_t>(row0 + q * 4) * g.ldo + col;
                uint32_t x[4];
                if (EPI == GEMM_EPI_RESIDUAL) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (q * 4 + j < n_rows) x[j] = *reinterpret_cast<const uint32_t*>(g.res + o + static_cast<size_t>(j) * g.ldo);
                }
                float a[2][4], up[2][4];
                sum(q, f, a);
                if (EPI == GEMM_EPI_SWIGLU) sum(q, FW / 2 + f, up);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (q * 4 + j >= n_rows) break;
                    float y0 = a[0][j], y1 = a[1][j];
                    if (EPI == GEMM_EPI_SWIGLU) {        // silu(gate) * up
                        y0 = __fdividef(y0, 1.0f + __expf(-y0)) * up[0][j];
                        y1 = __fdividef(y1, 1.0f + __expf(-y1)) * up[1][j];
                    } else if (EPI == GEMM_EPI_RESIDUAL) {
                        y0 += lo_f(x[j]);
                        y1 += hi_f(x[j]);
                    }
                    *reinterpret_cast<uint32_t*>(g.out + o + static_cast<size_t>(j) * g.ldo) = pack_bf16(y0, y1);
                }
            }
        }
    } else if (!*abort_flag) {
        const float* slab = reinterpret_cast<const float*>(tiles);
        // 8 features from feature c of row r, the K slices added in order
        const auto sum8 = [&](int r, int c, float (&s)[8]) {
#pragma unroll
            for (int j = 0; j < 8; ++j) s[j] = 0.f;
            for (int k = 0; k < p.splits; ++k) {
                const float4* q = reinterpret_cast<const float4*>(slab + (static_cast<size_t>(k) * per_owner + r) * FW + c);
                const float4 a = q[0], b = q[1];
                s[0] += a.x; s[1] += a.y; s[2] += a.z; s[3] += a.w;
                s[4] += b.x; s[5] += b.y; s[6] += b.z; s[7] += b.w;
            }
        };
        const int t = threadIdx.x;
        const int row0 = split * per_owner;
        const int n_rows = min(per_owner, g.M - row0);   // (may be negative: nothing to do)
        if (EPI == GEMM_EPI_ROPE) {
            const RopeArgs& r = g.rope;
            const int gph = r.d / 16;                    // 8-channel groups of half a head
            for (int i = t; i < n_rows * (FW / 16); i += FEW_THREADS) {
                const int rr = i / (FW / 16), q = i % (FW / 16);
                const int hh = q / gph, c = (q % gph) * 8;
                const int H = tile * (FW / r.d) + hh, m = row0 + rr;
                if (H >= r.Hq + 2 * r.Hkv) continue;
                float a[8], b[8];
                sum8(rr, hh * r.d + c, a);
                sum8(rr, hh * r.d + r.d / 2 + c, b);
                const int bb = m / r.length, pos = r.start + m % r.length;
                __nv_bfloat16* dst;
                if (H < r.Hq) {
                    dst = static_cast<__nv_bfloat16*>(r.q_out) + (static_cast<size_t>(m) * r.Hq + H) * r.d;
                } else {
                    const bool k = H < r.Hq + r.Hkv;
                    const int h = H - r.Hq - (k ? 0 : r.Hkv);
                    dst = static_cast<__nv_bfloat16*>(k ? r.k_cache : r.v_cache) +
                          ((static_cast<size_t>(bb) * r.Hkv + h) * r.cap + pos) * r.d;
                }
                if (H < r.Hq + r.Hkv) {
                    const float2* cs = reinterpret_cast<const float2*>(r.cs) + static_cast<size_t>(pos) * (r.d / 2) + c;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {        // (the projection is rounded to bf16 before it turns)
                        const float x1 = round_bf16(a[j]), x2 = round_bf16(b[j]);
                        const float2 e = cs[j];
                        a[j] = x1 * e.x - x2 * e.y;
                        b[j] = x2 * e.x + x1 * e.y;
                    }
                }
                *reinterpret_cast<uint4*>(dst + c) = pack8(a);
                *reinterpret_cast<uint4*>(dst + r.d / 2 + c) = pack8(b);
            }
        } else {
            constexpr int groups = (EPI == GEMM_EPI_SWIGLU ? FW / 2 : FW) / 8;
            constexpr int BATCH = EPI == GEMM_EPI_RESIDUAL ? 4 : 2;      // items in work at a time (residuals: on their way together)
            for (int i0 = t; i0 < n_rows * groups; i0 += FEW_THREADS * BATCH) {
                uint4 x[BATCH];
                if (EPI == GEMM_EPI_RESIDUAL) {
#pragma unroll
                    for (int u = 0; u < BATCH; ++u) {
                        const int i = i0 + u * FEW_THREADS, col = tile * p.wcols + (i % groups) * 8;
                        if (i < n_rows * groups && col < g.N)
                            x[u] = *reinterpret_cast<const uint4*>(g.res + static_cast<size_t>(row0 + i / groups) * g.ldo + col);
                    }
                }
#pragma unroll
                for (int u = 0; u < BATCH; ++u) {
                    const int i = i0 + u * FEW_THREADS, rr = i / groups, c = (i % groups) * 8;
                    const int col = tile * p.wcols + c;
                    if (i >= n_rows * groups || col >= g.N) continue;      // (N is a multiple of 8)
                    float a[8];
                    sum8(rr, c, a);
                    if (EPI == GEMM_EPI_SWIGLU) {
                        float up[8];
                        sum8(rr, FW / 2 + c, up);
#pragma unroll
                        for (int j = 0; j < 8; ++j) a[j] = __fdividef(a[j], 1.0f + __expf(-a[j])) * up[j];    // silu(gate) * up
                    } else if (EPI == GEMM_EPI_RESIDUAL) {
                        a[0] += lo_f(x[u].x); a[1] += hi_f(x[u].x); a[2] += lo_f(x[u].y); a[3] += hi_f(x[u].y);
                        a[4] += lo_f(x[u].z); a[5] += hi_f(x[u].z); a[6] += lo_f(x[u].w); a[7] += hi_f(x[u].w);
                    }
                    *reinterpret_cast<uint4*>(g.out + static_cast<size_t>(row0 + rr) * g.ldo + col) = pack8(a);
                }
            }
        }
    }

    tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) {}   // let copies in flight land before the shared memory goes away
        if (threadIdx.x == 0) atomicOr(g.dev_status, DEV_WAIT_EXPIRED);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, tmem_cols);
    }
}

template <int EPI>
int launch_few(const CUtensorMap& tw, const CUtensorMap& tw2, const CUtensorMap& ta, const FewArgs& g, cudaStream_t stream) {
    static std::atomic<uint64_t> smem_set[2] = {};
    const bool quad = g.p.quads > 0;
    const auto kernel = quad ? gemm_few_kernel<EPI, true> : gemm_few_kernel<EPI, false>;
    if (ensure_dynamic_smem(smem_set[quad], kernel, FEW_SMEM) != DARE_OK) return DARE_ERR_CUDA;
    const long long ctas = static_cast<long long>(g.p.tiles) * g.p.splits;
    if (ctas > 0x7fffffffLL) return DARE_ERR_SHAPE;
    return launch_kernel(kernel, dim3(static_cast<unsigned>(ctas)), FEW_THREADS, FEW_SMEM, stream, g.p.splits, tw,
                         tw2, ta, g);
}

}  // namespace

int gemm_few_describe(int epi, int M, int N, int K, int sm_count, int* out) {
    const FewPlan p = few_plan(epi, M, N, K, sm_count);
    out[0] = 1; out[1] = FW; out[2] = p.wcols; out[3] = p.splits; out[4] = p.stages; out[5] = 1; out[6] = p.tiles; out[7] = 0;
    return DARE_OK;
}

int launch_gemm_few(const dare_ctx* ctx, int epi, const void* a, int M, int K, const void* w, const void* w2, int N, void* out,
                    const void* res, int ldo, cudaStream_t stream, const RopeArgs* rope, bool w_static) {
    FewArgs g;
    g.M = M; g.N = N; g.K = K; g.ldo = ldo;
    g.p = few_plan(epi, M, N, K, ctx->sm_count);
    g.out = static_cast<__nv_bfloat16*>(out);
    g.res = static_cast<const __nv_bfloat16*>(res);
    g.dev_status = ctx->dev_status;
    g.w_static = w_static;
    g.rope = rope ? *rope : RopeArgs{};
    CUtensorMap ta, tw, tw2;
    int rc = make_tmap_bf16_2d(ctx, &ta, a, static_cast<uint64_t>(M), static_cast<uint64_t>(K), static_cast<uint32_t>(g.p.nr), FK);
    const uint32_t box = static_cast<uint32_t>(g.p.wcols);
    if (rc == DARE_OK) rc = make_tmap_bf16_2d(ctx, &tw, w, static_cast<uint64_t>(N), static_cast<uint64_t>(K), box, FK);
    if (rc == DARE_OK && epi == GEMM_EPI_SWIGLU)
        rc = make_tmap_bf16_2d(ctx, &tw2, w2, static_cast<uint64_t>(N), static_cast<uint64_t>(K), box, FK);
    if (rc != DARE_OK) return rc;
    switch (epi) {
        case GEMM_EPI_STORE: return launch_few<GEMM_EPI_STORE>(tw, tw, ta, g, stream);
        case GEMM_EPI_RESIDUAL: return launch_few<GEMM_EPI_RESIDUAL>(tw, tw, ta, g, stream);
        case GEMM_EPI_SWIGLU: return launch_few<GEMM_EPI_SWIGLU>(tw, tw2, ta, g, stream);
        case GEMM_EPI_ROPE: return launch_few<GEMM_EPI_ROPE>(tw, tw, ta, g, stream);
    }
    return DARE_ERR_RANGE;
}

}  // namespace dare
