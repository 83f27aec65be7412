// Block-bidirectional attention of the current block's queries against the prefix cache, the block's own
// K/V and the optional suffix cache, with GQA.
//
// In every workload of this path the step is bound by reading K/V from HBM (L * Hq/Hkv flops per cache
// byte, at or below the machine's ridge), so the kernel is organised around the K/V stream:
//   * one CTA per (query chunk, batch row x KV head, KV split); the query rows of all Hq/Hkv heads that
//     share a KV head are packed into the same tile so each K/V byte is read once per unit;
//   * a producer warp streams 64-key K and V tiles through a 3-stage shared-memory ring with TMA
//     (128-byte swizzle, full/empty mbarriers); a consumer warp owns 16 query rows and, when few rows
//     share a KV head, a slice of each tile's keys (its running softmax is merged with its peers' at the end);
//   * QK^T and PV run on warp-level tensor-core MMAs (m16n8k16, bf16 -> fp32) straight from the swizzled
//     tiles via ldmatrix; the online softmax lives in registers (quad shuffles for the row max).
// The 128-row tcgen05 tile does not fit these shapes (32 or 4 query rows per KV head in the MHA workloads).
// With KV splits each CTA writes a normalised partial and its log-sum-exp; a small kernel combines them.
#include <math.h>

#include "internal.h"
#include "ptx.cuh"

namespace dare {
namespace {

constexpr int KT_MAX = 64;       // keys per tile of the widest variant (sizes the launch plan)
constexpr int ATT_MAX_STAGES = 4;
constexpr float LOG2E_F = 1.4426950408889634f;
constexpr float LN2_F = 0.6931471805599453f;

struct AttnParams {
    int B, L, Hq, Hkv, g, R;      // R = L * g packed query rows per (row, kv head)
    int prefix_cap, suffix_cap;
    int inplace, has_suffix, splits;
    int uniform_P;                // >= 0: every row's prefix length (used when prefix_len is NULL)
    const int32_t* cu_seqlens;    // packed variable-length mode (tcgen05 kernel): sequence b owns tokens [cu[b], cu[b+1])
    int total_tokens;             // packed mode: rows of q / k / v
    float scale_log2;
    const __nv_bfloat16* q;
    const int32_t* prefix_len;
    const int32_t* suffix_len;
    __nv_bfloat16* out;
    float* lse;
    float* part_o;                // [splits][B*L*Hq][D] fp32, used when splits > 1
    float* part_lse;              // [splits][B*L*Hq]
    uint32_t* dev_status;
    int beside_head;              // inputs are ready although the kernels before this one still run (see enqueue_step)
};

// The CTA that is started last (in a step the attention waits in it for the head, so that what follows in the stream is
// behind both; any other CTA would hold its place on the SM while it waits).
__device__ __forceinline__ bool is_last_cta() {
    return blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1 && blockIdx.z == gridDim.z - 1;
}

struct AttBarriers {
    uint64_t full[ATT_MAX_STAGES];
    uint64_t empty[ATT_MAX_STAGES];
    uint32_t abort_flag;
};

template <int D, int KT>
__host__ __device__ constexpr int att_stage_bytes() { return 2 * KT * D * 2; }
template <int D, int KT, int STAGES>
__host__ __device__ constexpr int att_smem_bytes() { return STAGES * att_stage_bytes<D, KT>() + static_cast<int>(sizeof(AttBarriers)) + 1024; }

// Segment bookkeeping of one (row, kv head) unit: tiles of the prefix, then the block, then the suffix.
struct TileInfo {
    int seg;      // 0 prefix buffer, 1 block buffer, 2 suffix buffer
    int row0;     // first row of the tile in that buffer's 2-D [rows, D] view
    int valid;    // keys of the tile that exist (1..KT)
};

template <int KT>
__device__ __forceinline__ TileInfo tile_info(int t, int n_pre, int n_blk, int len_pre, int len_blk, int len_suf,
                                              int base_pre, int base_blk, int base_suf) {
    TileInfo ti;
    if (t < n_pre) {
        ti.seg = 0; ti.row0 = base_pre + t * KT; ti.valid = min(KT, len_pre - t * KT);
    } else if (t < n_pre + n_blk) {
        t -= n_pre;
        ti.seg = 1; ti.row0 = base_blk + t * KT; ti.valid = min(KT, len_blk - t * KT);
    } else {
        t -= n_pre + n_blk;
        ti.seg = 2; ti.row0 = base_suf + t * KT; ti.valid = min(KT, len_suf - t * KT);
    }
    return ti;
}

// NW row groups of 16 packed query rows; KS warps share a row group and split every 64-key tile between
// them (KT / KS keys each), keeping separate running (max, sum, O) that are merged through shared memory at
// the end.  More warps per SM hide the latency of the ldmatrix -> MMA -> softmax chain.
// KT keys per tile and ATT_STAGES ring slots set the shared memory of a CTA and so how many CTAs an SM holds (CPS).
template <int D, int NW, int KS, int KT, int ATT_STAGES, int CPS>
__global__ void __launch_bounds__((NW * KS + 1) * 32, CPS)
attn_block_kernel(const __grid_constant__ CUtensorMap tm_kpre, const __grid_constant__ CUtensorMap tm_vpre,
                  const __grid_constant__ CUtensorMap tm_kblk, const __grid_constant__ CUtensorMap tm_vblk,
                  const __grid_constant__ CUtensorMap tm_ksuf, const __grid_constant__ CUtensorMap tm_vsuf,
                  const AttnParams p) {
    constexpr int STAGE = att_stage_bytes<D, KT>();
    constexpr int HALF = KT * 128;           // one 64-column half of a tile: KT rows x 128 bytes
    constexpr int NHALF = D / 64;
    constexpr int KV_BYTES = KT * D * 2;
    constexpr int NCW = NW * KS;             // consumer warps
    constexpr int KPW = KT / KS;             // keys per warp per tile
    constexpr int NBK = D / 8 / KS;          // blocks of 8 columns that a warp finishes in the final merge

    extern __shared__ uint8_t smem_raw[];
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    AttBarriers* bars = reinterpret_cast<AttBarriers*>(tiles + ATT_STAGES * STAGE);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int chunk = blockIdx.x;
    const int unit = blockIdx.y;
    const int split = blockIdx.z;
    const int b = unit / p.Hkv;
    const int kvh = unit % p.Hkv;

    // A CTA lives for a handful of tiles, so what it does before its first tile arrives counts.  Nothing below waits
    // for anything else: the row's lengths are requested first (needed only after the barrier below), the producer
    // lane sets up the barriers itself and, where the first tile's place does not depend on the lengths (in-place
    // cache: the prefix segment holds at least the block's L >= 1 keys and starts at the unit's base), sends for that
    // tile at once; the consumers' Q rows are requested beside it.  All of it but the barriers comes behind pdl_wait,
    // except in a step, where the kernels that still run do not write what this one reads.
    if (threadIdx.x == NCW * 32) {
        for (int s = 0; s < ATT_STAGES; ++s) {
            mbar_init(&bars->full[s], 1);
            mbar_init(&bars->empty[s], NCW);
        }
        bars->abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&tm_kpre);
        prefetch_tensormap(&tm_vpre);
    }
    if (!p.beside_head) pdl_wait();
    int P = p.prefix_len ? p.prefix_len[b]
                         : (p.uniform_P >= 0 ? p.uniform_P : (p.inplace ? p.prefix_cap - p.L : p.prefix_cap));
    int S = p.has_suffix ? (p.suffix_len ? p.suffix_len[b] : p.suffix_cap) : 0;
    // (only without a K/V split: a CTA of a split launch may own no tile at all, and a tile sent for must be waited for)
    const bool early_tile = p.inplace && p.splits == 1;     // tile 0 of this CTA is tile 0 of the prefix segment
    if (threadIdx.x == NCW * 32 && early_tile) {
        mbar_arrive_expect_tx(&bars->full[0], 2 * KV_BYTES);
#pragma unroll
        for (int h = 0; h < NHALF; ++h) {
            tma_load_2d(tiles + h * HALF, &tm_kpre, &bars->full[0], h * 64, unit * p.prefix_cap);
            tma_load_2d(tiles + KV_BYTES + h * HALF, &tm_vpre, &bars->full[0], h * 64, unit * p.prefix_cap);
        }
    }

    // per-thread state of the consumers (declared here so that the final merge can see it)
    const int rg = warp % NW;              // row group
    const int ks = warp / NW;              // key slice (NW*KS == producer warp: unused there)
    const int quad = lane >> 2;            // row inside the 16-row tile (and +8)
    const int tq = lane & 3;
    const int rho0 = chunk * (NW * 16) + rg * 16 + quad;
    const int rho1 = rho0 + 8;
    const bool live0 = rho0 < p.R, live1 = rho1 < p.R;
    const int i0 = live0 ? rho0 / p.g : 0, h0 = kvh * p.g + (live0 ? rho0 % p.g : 0);
    const int i1 = live1 ? rho1 / p.g : 0, h1 = kvh * p.g + (live1 ? rho1 % p.g : 0);
    uint32_t qf[D / 16][4];
    if (warp < NCW) {
        const uint32_t* q0 = reinterpret_cast<const uint32_t*>(p.q + ((static_cast<size_t>(b) * p.L + i0) * p.Hq + h0) * D);
        const uint32_t* q1 = reinterpret_cast<const uint32_t*>(p.q + ((static_cast<size_t>(b) * p.L + i1) * p.Hq + h1) * D);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
            qf[kk][0] = live0 ? q0[kk * 8 + tq] : 0u;
            qf[kk][1] = live1 ? q1[kk * 8 + tq] : 0u;
            qf[kk][2] = live0 ? q0[kk * 8 + 4 + tq] : 0u;
            qf[kk][3] = live1 ? q1[kk * 8 + 4 + tq] : 0u;
        }
    }
    __syncthreads();

    // lengths (clamped to capacity; a clamp is reported, never trapped on)
    const int p_max = p.inplace ? p.prefix_cap - p.L : p.prefix_cap;
    if (P < 0 || P > p_max || S < 0 || S > p.suffix_cap) {
        P = max(0, min(P, p_max));
        S = max(0, min(S, p.suffix_cap));
        if (threadIdx.x == 0) atomicOr(p.dev_status, DEV_LEN_CLAMPED);
    }
    const int len_pre = p.inplace ? P + p.L : P;
    const int len_blk = p.inplace ? 0 : p.L;
    const int n_pre = (len_pre + KT - 1) / KT;
    const int n_blk = (len_blk + KT - 1) / KT;
    const int n_suf = (S + KT - 1) / KT;
    const int n_tiles = n_pre + n_blk + n_suf;
    const int t_begin = static_cast<int>(static_cast<long long>(n_tiles) * split / p.splits);
    const int t_end = static_cast<int>(static_cast<long long>(n_tiles) * (split + 1) / p.splits);
    const int base_pre = unit * p.prefix_cap;
    const int base_blk = unit * p.L;
    const int base_suf = unit * p.suffix_cap;

    float oacc[D / 8][4];
#pragma unroll
    for (int n = 0; n < D / 8; ++n) { oacc[n][0] = oacc[n][1] = oacc[n][2] = oacc[n][3] = 0.f; }
    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
    bool ok = true;

    if (warp == NCW) {
        // ---------------- producer
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int t = t_begin;
            if (early_tile) {                         // tile 0 is on its way already (no split: t_begin = 0, t_end = n_tiles >= 1)
                ++t;
                if (++stage == ATT_STAGES) { stage = 0; phase ^= 1; }
            }
            for (; t < t_end; ++t) {
                const TileInfo ti = tile_info<KT>(t, n_pre, n_blk, len_pre, len_blk, S, base_pre, base_blk, base_suf);
                const CUtensorMap* mk = ti.seg == 0 ? &tm_kpre : (ti.seg == 1 ? &tm_kblk : &tm_ksuf);
                const CUtensorMap* mv = ti.seg == 0 ? &tm_vpre : (ti.seg == 1 ? &tm_vblk : &tm_vsuf);
                if (!mbar_wait(&bars->empty[stage], phase ^ 1, abort_flag)) break;
                uint8_t* kdst = tiles + stage * STAGE;
                uint8_t* vdst = kdst + KV_BYTES;
                mbar_arrive_expect_tx(&bars->full[stage], 2 * KV_BYTES);
#pragma unroll
                for (int h = 0; h < NHALF; ++h) {
                    tma_load_2d(kdst + h * HALF, mk, &bars->full[stage], h * 64, ti.row0);
                    tma_load_2d(vdst + h * HALF, mv, &bars->full[stage], h * 64, ti.row0);
                }
                if (++stage == ATT_STAGES) { stage = 0; phase ^= 1; }
            }
        }
    } else {
        // ---------------- consumers
        int stage = 0;
        uint32_t phase = 0;
        const int mi = lane >> 3, rin = lane & 7;
        const int koff = ks * KPW;           // this warp's keys inside a tile: [koff, koff + KPW)
        for (int t = t_begin; t < t_end; ++t) {
            const TileInfo ti = tile_info<KT>(t, n_pre, n_blk, len_pre, len_blk, S, base_pre, base_blk, base_suf);
            if (!mbar_wait(&bars->full[stage], phase, abort_flag)) { ok = false; break; }
            uint8_t* kt = tiles + stage * STAGE;
            uint8_t* vt = kt + KV_BYTES;
            const uint32_t kbase = smem_u32(kt), vbase = smem_u32(vt);

            if (ti.valid < koff + KPW && ti.valid > koff) {
                // rows past the segment's end hold whatever lies behind it in memory: zero this warp's V rows
                // there so that probability 0 times garbage cannot make a NaN (rows are contiguous in a half)
                const int first = ti.valid * 128, count = (koff + KPW - ti.valid) * 128;
#pragma unroll
                for (int h = 0; h < NHALF; ++h)
                    for (int o = lane * 16; o < count; o += 32 * 16)
                        *reinterpret_cast<uint4*>(vt + h * HALF + first + o) = make_uint4(0, 0, 0, 0);
                fence_proxy_async_smem();
                __syncwarp();
            }
            if (ti.valid > koff) {   // (a warp whose key slice lies wholly past the end has nothing to add)
                // S = Q K^T for this warp's keys
                float sacc[KPW / 8][4];
                // (with 32 keys and more a warp's score blocks advance together: one block's eight products after the other's were a
                // chain that two warps per scheduler do not hide, 38.9 -> 38.3 us at 512 units of 12 tiles, 37.3 -> 36.2 at 384; with 16
                // keys 1 % slower)
                if constexpr (KPW >= 32) {
#pragma unroll
                    for (int nb = 0; nb < KPW / 8; ++nb) sacc[nb][0] = sacc[nb][1] = sacc[nb][2] = sacc[nb][3] = 0.f;
#pragma unroll
                    for (int kq = 0; kq < D / 32; ++kq) {
                        uint32_t kf[KPW / 8][4];
#pragma unroll
                        for (int nb = 0; nb < KPW / 8; ++nb) {
                            const int key = koff + nb * 8 + rin, ch = 4 * kq + mi;
                            ldmatrix_x4(kbase + (ch >> 3) * HALF + key * 128 + (((ch & 7) ^ (key & 7)) << 4), kf[nb][0], kf[nb][1], kf[nb][2], kf[nb][3]);
                        }
#pragma unroll
                        for (int nb = 0; nb < KPW / 8; ++nb) mma_bf16_16816(sacc[nb], qf[2 * kq], kf[nb][0], kf[nb][1]);
#pragma unroll
                        for (int nb = 0; nb < KPW / 8; ++nb) mma_bf16_16816(sacc[nb], qf[2 * kq + 1], kf[nb][2], kf[nb][3]);
                    }
                } else {
#pragma unroll
                    for (int nb = 0; nb < KPW / 8; ++nb) {
                        sacc[nb][0] = sacc[nb][1] = sacc[nb][2] = sacc[nb][3] = 0.f;
                        const int key = koff + nb * 8 + rin;
#pragma unroll
                        for (int kq = 0; kq < D / 32; ++kq) {
                            const int ch = 4 * kq + mi;
                            const uint32_t addr = kbase + (ch >> 3) * HALF + key * 128 + (((ch & 7) ^ (key & 7)) << 4);
                            uint32_t r0, r1, r2, r3;
                            ldmatrix_x4(addr, r0, r1, r2, r3);
                            mma_bf16_16816(sacc[nb], qf[2 * kq], r0, r1);
                            mma_bf16_16816(sacc[nb], qf[2 * kq + 1], r2, r3);
                        }
                    }
                }
                // mask keys that do not exist (only a segment's last tile has any), row max.  The scores stay
                // unscaled: the softmax scale (times log2 e) goes into the exponent's multiply-add below, and
                // the running max m0 / m1 is kept in score units until the tiles are done.
                if (ti.valid < koff + KPW) {
#pragma unroll
                    for (int nb = 0; nb < KPW / 8; ++nb) {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (koff + nb * 8 + tq * 2 + (e & 1) >= ti.valid) sacc[nb][e] = -INFINITY;
                    }
                }
                float tmax0 = -INFINITY, tmax1 = -INFINITY;
#pragma unroll
                for (int nb = 0; nb < KPW / 8; ++nb) {
                    tmax0 = fmaxf(tmax0, fmaxf(sacc[nb][0], sacc[nb][1]));
                    tmax1 = fmaxf(tmax1, fmaxf(sacc[nb][2], sacc[nb][3]));
                }
                tmax0 = fmaxf(tmax0, __shfl_xor_sync(0xffffffffu, tmax0, 1));
                tmax0 = fmaxf(tmax0, __shfl_xor_sync(0xffffffffu, tmax0, 2));
                tmax1 = fmaxf(tmax1, __shfl_xor_sync(0xffffffffu, tmax1, 1));
                tmax1 = fmaxf(tmax1, __shfl_xor_sync(0xffffffffu, tmax1, 2));
                const float mn0 = fmaxf(m0, tmax0), mn1 = fmaxf(m1, tmax1);   // finite: the slice has >= 1 key
                const bool moved = __any_sync(0xffffffffu, mn0 != m0 || mn1 != m1);
                const float c = p.scale_log2;
                const float nb0 = -mn0 * c, nb1 = -mn1 * c;
                float ps0 = 0.f, ps1 = 0.f;
                uint32_t pa[KPW / 16][4];
#pragma unroll
                for (int nb = 0; nb < KPW / 8; ++nb) {
                    const float e0 = fast_exp2(fmaf(sacc[nb][0], c, nb0)), e1 = fast_exp2(fmaf(sacc[nb][1], c, nb0));
                    const float e2 = fast_exp2(fmaf(sacc[nb][2], c, nb1)), e3 = fast_exp2(fmaf(sacc[nb][3], c, nb1));
                    ps0 += e0 + e1;
                    ps1 += e2 + e3;
                    pa[nb >> 1][(nb & 1) * 2 + 0] = pack_bf16(e0, e1);
                    pa[nb >> 1][(nb & 1) * 2 + 1] = pack_bf16(e2, e3);
                }
                if (moved) {   // (rare after the first tiles: a row's max over hundreds of keys settles early)
                    const float a0 = fast_exp2((m0 - mn0) * c), a1 = fast_exp2((m1 - mn1) * c);
                    m0 = mn0; m1 = mn1;
                    l0 *= a0;
                    l1 *= a1;
#pragma unroll
                    for (int n = 0; n < D / 8; ++n) {
                        oacc[n][0] *= a0; oacc[n][1] *= a0;
                        oacc[n][2] *= a1; oacc[n][3] *= a1;
                    }
                }
                l0 += ps0;
                l1 += ps1;
                // O += P V
#pragma unroll
                for (int kk = 0; kk < KPW / 16; ++kk) {
                    const int key = koff + kk * 16 + (mi & 1) * 8 + rin;
#pragma unroll
                    for (int nbp = 0; nbp < D / 16; ++nbp) {
                        const int ch = 2 * nbp + (mi >> 1);
                        const uint32_t addr = vbase + (ch >> 3) * HALF + key * 128 + (((ch & 7) ^ (key & 7)) << 4);
                        uint32_t r0, r1, r2, r3;
                        ldmatrix_x4_trans(addr, r0, r1, r2, r3);
                        mma_bf16_16816(oacc[2 * nbp], pa[kk], r0, r1);
                        mma_bf16_16816(oacc[2 * nbp + 1], pa[kk], r2, r3);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->empty[stage]);
            if (++stage == ATT_STAGES) { stage = 0; phase ^= 1; }
        }
        l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
        l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
        l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
        l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
        m0 *= p.scale_log2;      // from here on the max is in the log2 domain (-inf stays -inf: the scale is > 0)
        m1 *= p.scale_log2;
    }

    // ---------------- merge the key slices of a row group (through the now idle tile ring), then write out.  Each of the KS warps
    // finishes its share of the columns and sends the others theirs.  (One warp of the row group adding everything up took 4 k of
    // a CTA's 37 k cycles while the others had left: 40.2 -> 38.9 us at 512 units of 12 tiles, 5.75 -> 5.25 at 6 units of 2.)
    // (The next kernel is let in only now: set up any earlier, the CTAs of a small one pile up on the few SMs that have
    // room beside this kernel's; the row compaction of the next step then took 11 us instead of 6.)
    pdl_trigger();
    __syncthreads();   // every tile has been consumed (or the CTA is aborting): the ring may be reused
    const bool aborted = *abort_flag != 0;
    float4* xch = reinterpret_cast<float4*>(tiles);                    // [finishing slice][slice][row group][block of 8 columns][lane]
    float4* xch_ml = xch + KS * KS * NW * NBK * 32;                    // [slice][row group][lane]: the two rows' max and sum
    if (KS > 1 && !aborted && warp < NCW) {
#pragma unroll
        for (int o = 0; o < KS; ++o) {
            if (o == ks) continue;
#pragma unroll
            for (int i = 0; i < NBK; ++i) {
                const float (&v)[4] = oacc[o * NBK + i];
                xch[(((o * KS + ks) * NW + rg) * NBK + i) * 32 + lane] = make_float4(v[0], v[1], v[2], v[3]);
            }
        }
        xch_ml[(ks * NW + rg) * 32 + lane] = make_float4(m0, m1, l0, l1);
    }
    if (KS > 1) __syncthreads();
    if (!aborted && warp < NCW) {
        float w0[KS], w1[KS];              // what each slice's values count
        if (KS > 1) {
            float4 ml[KS];
            m0 = m1 = -INFINITY;
            l0 = l1 = 0.f;
#pragma unroll
            for (int o = 0; o < KS; ++o) {
                ml[o] = xch_ml[(o * NW + rg) * 32 + lane];
                m0 = fmaxf(m0, ml[o].x);
                m1 = fmaxf(m1, ml[o].y);
            }
#pragma unroll
            for (int o = 0; o < KS; ++o) {
                w0[o] = m0 == -INFINITY ? 0.f : fast_exp2(ml[o].x - m0);
                w1[o] = m1 == -INFINITY ? 0.f : fast_exp2(ml[o].y - m1);
                l0 += ml[o].z * w0[o];
                l1 += ml[o].w * w1[o];
            }
        } else {
            w0[0] = w1[0] = 1.f;
        }
        const float inv0 = l0 > 0.f ? 1.f / l0 : 0.f, inv1 = l1 > 0.f ? 1.f / l1 : 0.f;
        const size_t orow0 = (static_cast<size_t>(b) * p.L + i0) * p.Hq + h0;
        const size_t orow1 = (static_cast<size_t>(b) * p.L + i1) * p.Hq + h1;
        const size_t n_rows = static_cast<size_t>(p.B) * p.L * p.Hq;
        float* po = p.part_o + static_cast<size_t>(split) * n_rows * D;
        const bool whole = p.splits == 1;
#pragma unroll
        for (int o = 0; o < KS; ++o) {
            if (o != ks) continue;         // (a warp runs one of these, with its accumulators in registers)
#pragma unroll
            for (int i = 0; i < NBK; ++i) {
                float (&v)[4] = oacc[o * NBK + i];
                if (KS > 1) { v[0] *= w0[o]; v[1] *= w0[o]; v[2] *= w1[o]; v[3] *= w1[o]; }
#pragma unroll
                for (int q = 0; q < KS; ++q) {
                    if (q == o) continue;
                    const float4 x = xch[(((o * KS + q) * NW + rg) * NBK + i) * 32 + lane];
                    v[0] += x.x * w0[q]; v[1] += x.y * w0[q];
                    v[2] += x.z * w1[q]; v[3] += x.w * w1[q];
                }
                v[0] *= inv0; v[1] *= inv0; v[2] *= inv1; v[3] *= inv1;
            }
            if (whole) {
#pragma unroll
                for (int i = 0; i < NBK; ++i) {
                    const float (&v)[4] = oacc[o * NBK + i];
                    const int col = (o * NBK + i) * 8 + tq * 2;
                    if (live0) *reinterpret_cast<uint32_t*>(p.out + orow0 * D + col) = pack_bf16(v[0], v[1]);
                    if (live1) *reinterpret_cast<uint32_t*>(p.out + orow1 * D + col) = pack_bf16(v[2], v[3]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < NBK; ++i) {
                    const float (&v)[4] = oacc[o * NBK + i];
                    const int col = (o * NBK + i) * 8 + tq * 2;
                    if (live0) *reinterpret_cast<float2*>(po + orow0 * D + col) = make_float2(v[0], v[1]);
                    if (live1) *reinterpret_cast<float2*>(po + orow1 * D + col) = make_float2(v[2], v[3]);
                }
            }
        }
        if (ks == 0 && tq == 0) {
            const float lse0 = l0 > 0.f ? (m0 + log2f(l0)) * LN2_F : -INFINITY;
            const float lse1 = l1 > 0.f ? (m1 + log2f(l1)) * LN2_F : -INFINITY;
            if (p.splits > 1) {
                float* pl = p.part_lse + static_cast<size_t>(split) * n_rows;
                if (live0) pl[orow0] = lse0;
                if (live1) pl[orow1] = lse1;
            } else if (p.lse != nullptr) {
                if (live0) p.lse[(static_cast<size_t>(b) * p.Hq + h0) * p.L + i0] = lse0;
                if (live1) p.lse[(static_cast<size_t>(b) * p.Hq + h1) * p.L + i1] = lse1;
            }
        }
    }
    (void)ok;
    if (aborted) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) {}
        if (threadIdx.x == 0) atomicOr(p.dev_status, DEV_WAIT_EXPIRED);
        __syncthreads();
    }
    if (p.beside_head && is_last_cta()) pdl_wait();
}

// ---------------------------------------------------------------------------------------------------------
// tcgen05 path: used when the query rows that share a KV head fill 128-row tensor-core tiles well (GQA
// groups, long blocks such as the prefill).  A unit of work is one or two tiles of packed query rows of one
// rollout x KV head; the two query tiles share every K/V tile:
//   warp 0        TMA producer: Q tiles, and 64-key K and V tiles through a shared-memory ring; takes the units
//   warps 1, 2    UMMA issuer of query tile 0, 1 (one thread each, so that the order of a tile's MMAs is the order they
//                 run in): S = Q K^T (128 x 64, K-major operands from shared memory) into tensor memory, then
//                 O += P V (128 x D) with P, the A operand, read from TENSOR memory and V, the MN-major B operand,
//                 straight from the TMA tile; O stays in tensor memory over the whole key range
//   warps 4..7    softmax of query tile 0 (warps 8..11: tile 1): one TMEM lane = one query row per thread;
//                 holds a row's 64 scores in registers, keeps the row's reference max and sum, and writes
//                 P as packed bf16 over the columns S came from: P never touches shared memory
// Each query tile has TWO S / P buffers of 64 columns, and S(t + 2) is issued behind P V(t) (it may overwrite P(t)
// because the pipe runs an issuer's MMAs in order), so that a softmax warp finds its next scores ready instead of
// waiting for the chain softmax -> P V -> S.  Two issuers, because one thread takes ~90 cycles for each of the 24 MMAs
// of a step (both query tiles x 64 keys; one issuer 2140 cycles a step, two 1880).
// The kernel is persistent: a CTA that has sent for its unit's last key tile takes over the next unit whose CTA has not
// been started yet (cluster launch control), and the copies of that unit's Q, K and V are under way while the last
// tiles of the current one are worked on; only the write-back of O lies between two units (2.4 k cycles; a CTA per unit
// spent 12 k around its loop).
// What bounds it: on packed batches the power cap (0.81 PFLOP/s at 1.65 GHz and 985 W; 0.63 at 1.91 GHz before), on an
// unthrottled GPU the exponential unit and the waits around it (that unit and the tensor pipe are each busy 45 % of the time).
// Before -> after, us: packed 28 + 4 heads of 128, 32 sequences of 256 to 1024 tokens 333 -> 234 (on the power cap 343 ->
// 270), 16 x 2048 1047 -> 940; 16 x 512 queries x 32 heads 116 -> 80; Dream-shaped step (32 rollouts, 1280 keys) 34.2 -> 30.1.
// 128-key tiles with one S / P buffer, P handed over in halves: 16 x 2048 904 and 16 x 512 77, but 282 on the packed batch
// (its ragged ends) and 30.8 on the step.
// O stays in TMEM, so it cannot be rescaled for free when a row's max grows.  The exponentials are therefore
// taken relative to a reference max that is only moved when the true max has run more than 2^4 ahead of it;
// then (rarely, mostly in the first tiles) the warp waits for the MMAs in flight, multiplies its rows of O by
// the correction factor in place and moves the reference.  The sum uses the same reference, so O / l is exact.
// A tile holds floor(128 / g) block positions x g heads so that a position's heads never straddle two tiles.
constexpr int TC_KT = 64;                 // keys per tile
// log2 units the true max may run ahead of the reference.  The fewer, the oftener a row's largest weight is exactly 1 in bf16.  Distance
// from 64 bits (rel-L2, x 1e-3; 1.5 of it the result's own rounding) for q of standard deviation 1, 2, 4, 8, 16 on 28 + 4 heads of 128:
// 8 units 2.301, 2.223, 2.110, 1.851, 1.525; 4 units 2.300, 2.102, 1.865, 1.707, 1.469; 2 units 2.274, 1.944, 1.761, 1.669, 1.457, but the
// ordinary scores of deviation 1 then move too (7 % on 32 sequences of 256 to 1024 tokens; 8 to 4 units: no difference).
constexpr float TC_RESCALE_GAP = 4.0f;

template <int D, int QT>
struct TcShape {
    static constexpr int Q_BYTES = 128 * D * 2;                        // per query tile
    static constexpr int KV_STAGE = 2 * TC_KT * D * 2;                 // K tile + V tile
    static constexpr int STAGES = D == 128 ? 4 : 8;                    // (a power of two: 128 KB of K/V in flight)
    static constexpr int OUT_BYTES = 32 * 128;                         // per softmax warp: 32 rows x 64 columns of O
    static constexpr int SMEM = QT * Q_BYTES + STAGES * KV_STAGE + 4 * QT * OUT_BYTES + 1024 + 512;
    static constexpr int THREADS = (4 + 4 * QT) * 32;                  // TMA warp, issuing warps (and idle ones), then the softmax warps
    static constexpr uint32_t TMEM_COLS = QT == 2 ? 512 : 256;
    // tensor-memory columns of query tile j: S / P buffers at j * 256 and j * 256 + 64, O at j * 256 + 128
    __host__ __device__ static constexpr uint32_t s_col(int j, int b) { return j * 256 + b * 64; }
    __host__ __device__ static constexpr uint32_t o_col(int j) { return j * 256 + 128; }
};

// The (block position, head) of packed query row r, walked in steps of `step` rows: one division up front.
struct RowWalk {
    int i, h, g, step_i, step_h;
    __device__ __forceinline__ RowWalk(int r, int step, int g_) : i(r / g_), h(r % g_), g(g_), step_i(step / g_), step_h(step % g_) {}
    __device__ __forceinline__ void next() {
        i += step_i;
        h += step_h;
        if (h >= g) { h -= g; ++i; }
    }
};

// A unit of work, as the producer hands it to the other warps.
struct TcUnit {
    int n_tiles;             // key tiles (0: there is no further unit)
    int n_q;                 // query tiles with live rows
    int pos0;                // first block position of the unit
    int token0;              // first token of the rollout / sequence in q and out
    int L_eff;               // block positions of the rollout / sequence
    int b, kvh;
    int len_pre, len_blk, len_suf;
};

template <int STAGES, int QT>
struct TcBarriers {
    uint64_t full[STAGES];
    uint64_t empty[STAGES];
    uint64_t q_full[QT], q_empty[QT];
    uint64_t s_full[QT][2], p_full[QT][2], pv_done[QT][2];     // indexed by the S / P buffer
    uint64_t unit_full[2], unit_empty[2];
    uint64_t turn[2][4];                                       // [query tile][quadrant of tensor-memory lanes]
    uint64_t next_unit;
    TcUnit unit[2];
    alignas(16) uint4 cancelled;                               // cluster launch control's answer
    uint32_t tmem_base;
    uint32_t abort_flag;
};

template <int D, int QT>
__global__ void __launch_bounds__(TcShape<D, QT>::THREADS, 1)
attn_block_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kpre,
                     const __grid_constant__ CUtensorMap tm_vpre, const __grid_constant__ CUtensorMap tm_kblk,
                     const __grid_constant__ CUtensorMap tm_vblk, const __grid_constant__ CUtensorMap tm_ksuf,
                     const __grid_constant__ CUtensorMap tm_vsuf, const AttnParams p) {
    using S = TcShape<D, QT>;
    constexpr int STAGES = S::STAGES;
    constexpr int NHALF = D / 64;
    constexpr int HALF_K = TC_KT * 128;            // one 64-column half of a K or V tile: 64 rows x 128 bytes
    constexpr int KV_BYTES = TC_KT * D * 2;
    constexpr int HALF_Q = 128 * 128;              // one 64-column half of a Q tile: 128 rows x 128 bytes
    static_assert(sizeof(TcBarriers<STAGES, QT>) <= 512, "shared-memory layout");

    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* q_s = base;                                   // [QT][Q_BYTES]
    uint8_t* kv_s = q_s + QT * S::Q_BYTES;                 // [STAGES][KV_STAGE]
    uint8_t* out_s = kv_s + STAGES * S::KV_STAGE;          // [4 * QT][OUT_BYTES]
    TcBarriers<STAGES, QT>* bars = reinterpret_cast<TcBarriers<STAGES, QT>*>(out_s + 4 * QT * S::OUT_BYTES);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int warp = warp_index_uniform();
    const int lane = threadIdx.x & 31;
    const int pos_per_tile = 128 / p.g;            // block positions per query tile
    const int rows_in_tile = pos_per_tile * p.g;
    // Packed variable-length mode: "rollout" b is sequence b of the packed token list; its tokens are both the
    // queries (a block of L_eff positions, no prefix) and, in place, the keys.  K and V are [tokens, Hkv * D].
    const bool packed = p.cu_seqlens != nullptr;
    bool has_last = false;                         // this CTA ran the last unit (thread 0 knows)

    if (warp == 1) {
        tmem_alloc(&bars->tmem_base, S::TMEM_COLS);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&bars->full[s], 1);
            mbar_init(&bars->empty[s], QT);                // released by each query tile's issuer
        }
        for (int j = 0; j < QT; ++j) {
            mbar_init(&bars->q_full[j], 1);
            mbar_init(&bars->q_empty[j], 1);
            for (int i = 0; i < 2; ++i) {
                mbar_init(&bars->s_full[j][i], 1);
                mbar_init(&bars->p_full[j][i], 128);
                mbar_init(&bars->pv_done[j][i], 1);
            }
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars->unit_full[i], 1);
            mbar_init(&bars->unit_empty[i], 5 * QT);       // the issuing warps and the softmax warps
        }
        mbar_init(&bars->next_unit, 1);
        for (int i = 0; i < 8; ++i) mbar_init(&bars->turn[i >> 2][i & 3], 1);
        bars->abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&tm_q);
        prefetch_tensormap(&tm_kpre);
        prefetch_tensormap(&tm_vpre);
    }
    // rows of the Q tiles that no copy writes (128 is not a multiple of every g): zero, once
    for (int o = threadIdx.x; o < (128 - rows_in_tile) * 8 * NHALF * QT; o += S::THREADS) {
        const int piece = o & 7, row = rows_in_tile + (o >> 3) % (128 - rows_in_tile), half = (o >> 3) / (128 - rows_in_tile);
        *reinterpret_cast<uint4*>(q_s + half * HALF_Q + row * 128 + piece * 16) = make_uint4(0, 0, 0, 0);
    }
    fence_proxy_async_smem();
    if (!p.beside_head) pdl_wait();                        // (as in the warp-level kernel)
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;

    if constexpr (QT == 2) {        // 384 threads are launched with 168 registers each = 128 x (56 + 2 x 224)
        if (warp < 4) set_max_regs_dec<56>();
        else set_max_regs_inc<224>();
    }
    if (warp == 0) {
        if (lane == 0) {
            const int p_max = p.inplace ? p.prefix_cap - p.L : p.prefix_cap;
            uint32_t chunk = blockIdx.x, y = blockIdx.y;
            uint32_t n_kv = 0, n_qload[QT] = {}, n_units = 0, n_taken = 0;
            bool ok = true;
            while (ok) {
                has_last = has_last || (chunk == gridDim.x - 1 && y == gridDim.y - 1);
                TcUnit w;
                w.b = static_cast<int>(y) / p.Hkv;
                w.kvh = static_cast<int>(y) % p.Hkv;
                w.pos0 = static_cast<int>(chunk) * QT * pos_per_tile;
                w.token0 = packed ? p.cu_seqlens[w.b] : w.b * p.L;
                w.L_eff = packed ? p.cu_seqlens[w.b + 1] - w.token0 : p.L;
                if (w.pos0 < w.L_eff) {                    // (packed: the grid is cut for the longest sequence)
                    int P = p.prefix_len ? p.prefix_len[w.b]
                                         : (p.uniform_P >= 0 ? p.uniform_P : (p.inplace ? p.prefix_cap - p.L : p.prefix_cap));
                    int Sx = p.has_suffix ? (p.suffix_len ? p.suffix_len[w.b] : p.suffix_cap) : 0;
                    if (!packed && (P < 0 || P > p_max || Sx < 0 || Sx > p.suffix_cap)) {
                        P = max(0, min(P, p_max));
                        Sx = max(0, min(Sx, p.suffix_cap));
                        atomicOr(p.dev_status, DEV_LEN_CLAMPED);
                    }
                    w.len_pre = packed ? w.L_eff : (p.inplace ? P + p.L : P);
                    w.len_blk = (packed || p.inplace) ? 0 : p.L;
                    w.len_suf = Sx;
                    const int n_pre = (w.len_pre + TC_KT - 1) / TC_KT, n_blk = (w.len_blk + TC_KT - 1) / TC_KT;
                    w.n_tiles = n_pre + n_blk + (Sx + TC_KT - 1) / TC_KT;
                    w.n_q = min(QT, (w.L_eff - w.pos0 + pos_per_tile - 1) / pos_per_tile);
                    const int slot = n_units & 1;
                    if (!mbar_wait(&bars->unit_empty[slot], ((n_units >> 1) & 1) ^ 1, abort_flag)) break;
                    bars->unit[slot] = w;
                    mbar_arrive(&bars->unit_full[slot]);
                    ++n_units;
                    const int base_pre = packed ? w.token0 : static_cast<int>(y) * p.prefix_cap;
                    const int base_blk = static_cast<int>(y) * p.L;
                    const int base_suf = static_cast<int>(y) * p.suffix_cap;
                    const int kv_col0 = packed ? w.kvh * D : 0;      // first column of this KV head in the 2-D view of K / V
                    for (int t = 0; t < w.n_tiles; ++t, ++n_kv) {
                        const TileInfo ti = tile_info<TC_KT>(t, n_pre, n_blk, w.len_pre, w.len_blk, Sx, base_pre, base_blk, base_suf);
                        const CUtensorMap* mk = ti.seg == 0 ? &tm_kpre : (ti.seg == 1 ? &tm_kblk : &tm_ksuf);
                        const CUtensorMap* mv = ti.seg == 0 ? &tm_vpre : (ti.seg == 1 ? &tm_vblk : &tm_vsuf);
                        const int stage = n_kv % STAGES;
                        if (!mbar_wait(&bars->empty[stage], ((n_kv / STAGES) & 1) ^ 1, abort_flag)) { ok = false; break; }
                        uint8_t* kdst = kv_s + stage * S::KV_STAGE;
                        uint8_t* vdst = kdst + KV_BYTES;
                        mbar_arrive_expect_tx(&bars->full[stage], 2 * KV_BYTES);
#pragma unroll
                        for (int h = 0; h < NHALF; ++h) {
                            tma_load_2d(kdst + h * HALF_K, mk, &bars->full[stage], kv_col0 + h * 64, ti.row0);
                            tma_load_2d(vdst + h * HALF_K, mv, &bars->full[stage], kv_col0 + h * 64, ti.row0);
                        }
                        if (t != 0) continue;
                        // The Q tiles: rows (position, head of the group), in that order, as one box.  (Positions behind
                        // the rollout's or the sequence's last bring in other rows or zeros; they are not stored.)
#pragma unroll
                        for (int j = 0; j < QT; ++j) {
                            if (j >= w.n_q || !ok) continue;
                            ok = mbar_wait(&bars->q_empty[j], (n_qload[j] & 1) ^ 1, abort_flag);
                            if (!ok) continue;
                            ++n_qload[j];
                            mbar_arrive_expect_tx(&bars->q_full[j], static_cast<uint32_t>(rows_in_tile) * D * 2);
#pragma unroll
                            for (int h = 0; h < NHALF; ++h)
                                tma_load_3d(q_s + j * S::Q_BYTES + h * HALF_Q, &tm_q, &bars->q_full[j], h * 64, w.kvh * p.g,
                                            w.token0 + w.pos0 + j * pos_per_tile);
                        }
                        if (!ok) break;
                    }
                    if (!ok) break;
                }
                // every copy of this unit is under way: take the next one (no earlier, or one CTA would sit on a unit
                // that an idle SM could run)
                mbar_arrive_expect_tx(&bars->next_unit, 16);
                clc_try_cancel(&bars->cancelled, &bars->next_unit);
                if (!mbar_wait(&bars->next_unit, n_taken & 1, abort_flag)) break;
                ++n_taken;
                const bool got = clc_query(&bars->cancelled, chunk, y);
                fence_proxy_async_smem();                  // (read here before the next answer is written there)
                if (!got) {
                    const int slot = n_units & 1;
                    if (!mbar_wait(&bars->unit_empty[slot], ((n_units >> 1) & 1) ^ 1, abort_flag)) break;
                    bars->unit[slot].n_tiles = 0;
                    mbar_arrive(&bars->unit_full[slot]);
                    break;
                }
            }
        }
        __syncwarp();
    } else if (warp < 4) {
      if (warp <= QT) {
        // One issuing warp per query tile.  All 32 lanes run the loops (waits, counters and descriptors stay warp-uniform, in
        // the registers the MMA instruction takes its operands from); one elected lane issues the MMAs and their commits.
        const int j = warp - 1;
        const bool leader = elect_one_sync();
        constexpr uint32_t idesc_s = umma_idesc_bf16(128, TC_KT);
        constexpr uint32_t idesc_o = umma_idesc_bf16(128, D) | UMMA_B_MN_MAJOR;
        // descriptor lower words (address >> 4 [| leading byte offset]); the upper word is a constant
        const uint32_t q_lo = (smem_u32(q_s) + j * S::Q_BYTES) >> 4, kv_lo = smem_u32(kv_s) >> 4;
        const uint32_t v_lbo = static_cast<uint32_t>(HALF_K >> 4) << 16;   // second 64 head-dim columns: one half tile on
        const uint32_t od = tmem_base + S::o_col(j);
        uint32_t n_kv = 0, n_unit = 0, n_q = 0, n_s = 0;   // key tiles of the ring, units, Q tiles and key tiles of query tile j so far
        bool ok = true;
        while (true) {
            const int slot = n_unit & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(&bars->unit_full[slot], (n_unit >> 1) & 1, abort_flag))) break;
            ++n_unit;
            // (through a reduction, whose result the compiler knows to be the same in all lanes)
            const int n_tiles = __reduce_max_sync(0xffffffffu, bars->unit[slot].n_tiles);
            const bool idle = __reduce_max_sync(0xffffffffu, bars->unit[slot].n_q) <= j;
            if (leader) mbar_arrive(&bars->unit_empty[slot]);
            __syncwarp();
            if (n_tiles == 0) break;
            if (idle) {                                    // (no live row in this query tile: the K/V tiles pass by)
                for (int t = 0; t < n_tiles && ok; ++t, ++n_kv) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&bars->full[n_kv % STAGES], (n_kv / STAGES) & 1, abort_flag));
                    if (ok && leader) mbar_arrive(&bars->empty[n_kv % STAGES]);
                    __syncwarp();
                }
                if (!ok) break;
                continue;
            }
            // S(t) = Q K_t^T into the buffer of t's parity (whatever that buffer held has been consumed: the P V
            // product that read it was issued before this, and the pipe keeps the issue order)
            auto issue_s = [&](int t) -> bool {
                const uint32_t n = n_kv + t;
                const int stage = n % STAGES, buf = (n_s + t) & 1;
                if (!__all_sync(0xffffffffu, mbar_wait(&bars->full[stage], (n / STAGES) & 1, abort_flag))) return false;
                tc_fence_after_sync();
                const uint32_t k_lo = kv_lo + stage * (S::KV_STAGE >> 4);
                const uint32_t sd = tmem_base + S::s_col(j, buf);
                if (leader) {
                    umma_bf16_lo<false>(sd, q_lo, k_lo, idesc_s);
#pragma unroll
                    for (int kk = 1; kk < D / 16; ++kk)     // 16 channels = 32 bytes along the swizzled row: +2
                        umma_bf16_lo<true>(sd, q_lo + (kk >> 2) * (HALF_Q >> 4) + 2 * (kk & 3),
                                           k_lo + (kk >> 2) * (HALF_K >> 4) + 2 * (kk & 3), idesc_s);
                    umma_commit(&bars->s_full[j][buf]);
                    if (t == n_tiles - 1) umma_commit(&bars->q_empty[j]);     // the next unit's Q may come
                }
                __syncwarp();
                return true;
            };
            ok = __all_sync(0xffffffffu, mbar_wait(&bars->q_full[j], n_q & 1, abort_flag));
            ++n_q;
            if (ok) ok = issue_s(0);
            if (ok && n_tiles > 1) ok = issue_s(1);
            for (int t = 0; t < n_tiles && ok; ++t) {
                const int stage = (n_kv + t) % STAGES;
                const uint32_t v_lo = (kv_lo + stage * (S::KV_STAGE >> 4) + (KV_BYTES >> 4)) | v_lbo;
                const uint32_t n = n_s + t;
                const int buf = n & 1;
                ok = __all_sync(0xffffffffu, mbar_wait(&bars->p_full[j][buf], (n >> 1) & 1, abort_flag));
                if (!ok) break;
                tc_fence_after_sync();
                // A: P in tensor memory, 16 keys = 8 columns per MMA; B: 16 key rows (2 KB) further down V
                const uint32_t pa = tmem_base + S::s_col(j, buf);
                if (leader) {
                    if (t == 0) umma_bf16_ts_lo<false>(od, pa, v_lo, idesc_o);
                    else umma_bf16_ts_lo<true>(od, pa, v_lo, idesc_o);
#pragma unroll
                    for (int kk = 1; kk < TC_KT / 16; ++kk)
                        umma_bf16_ts_lo<true>(od, pa + 8 * kk, v_lo + kk * (2048 >> 4), idesc_o);
                    umma_commit(&bars->pv_done[j][buf]);       // O holds tiles 0..t
                    umma_commit(&bars->empty[stage]);          // (this query tile is done with this K/V tile)
                }
                __syncwarp();
                if (t + 2 < n_tiles) ok = issue_s(t + 2);
            }
            if (!ok) break;
            n_kv += n_tiles;
            n_s += n_tiles;
        }
        pdl_trigger();                                  // (this late for the reason given in the warp-level kernel)
      }
    } else {
        // ---------------- softmax warps: set j = query tile, thread = packed query row r of that tile = TMEM lane r
        const int j = (warp >> 2) - 1;
        const int r = (warp & 3) * 32 + lane;          // warp w may touch TMEM lanes [32 * (w % 4), +32)
        const int ri = r / p.g, rh = r % p.g;          // block position and head within the tile and the group
        const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const uint32_t tm_o = tmem_base + S::o_col(j) + lane_off;
        const float c2 = p.scale_log2;
        uint8_t* ot = out_s + (warp - 4) * S::OUT_BYTES;
        uint32_t n_kv = 0, n_unit = 0, n_s = 0, n_turn = 0;
        const int quadrant = warp & 3;
        RowWalk out_walk((warp & 3) * 32 + (lane >> 3), 4, p.g);
        while (true) {
            const int slot = n_unit & 1;
            if (!__all_sync(0xffffffffu, mbar_wait(&bars->unit_full[slot], (n_unit >> 1) & 1, abort_flag))) break;
            ++n_unit;
            const TcUnit w = bars->unit[slot];
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->unit_empty[slot]);
            if (w.n_tiles == 0) break;
            if (j >= w.n_q) { n_kv += w.n_tiles; continue; }
            const int n_pre = (w.len_pre + TC_KT - 1) / TC_KT, n_blk = (w.len_blk + TC_KT - 1) / TC_KT;
            // Reference max (log2 domain) and sum of exp2(s - m_ref).  The rows behind a rollout's or a sequence's last position are the
            // next one's queries (see the producer): an infinite reference, all weights 0.  (A flag of their own, alive through
            // the loop, spilled: 243 -> 256 us on 32 sequences of 256 to 1024 tokens.)
            float m_ref = r < rows_in_tile && w.pos0 + j * pos_per_tile + ri < w.L_eff ? -INFINITY : INFINITY, l = 0.f;
            bool ok = true;
            for (int t = 0; t < w.n_tiles; ++t) {
                const int valid = tile_info<TC_KT>(t, n_pre, n_blk, w.len_pre, w.len_blk, w.len_suf, 0, 0, 0).valid;
                const uint32_t n = n_s + t;
                const int buf = n & 1;
                if (!mbar_wait(&bars->s_full[j][buf], (n >> 1) & 1, abort_flag)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t tm_s = tmem_base + S::s_col(j, buf) + lane_off;
                uint32_t s0[32], s1[32];
                tmem_ld_32cols(tm_s, s0);
                tmem_ld_32cols(tm_s + 32, s1);
                tmem_ld_wait();
                if (valid < TC_KT) {                       // (keys past the segment's end do not count)
#pragma unroll
                    for (int k = 0; k < 32; ++k) {
                        if (k >= valid) s0[k] = 0xff800000u;
                        if (k + 32 >= valid) s1[k] = 0xff800000u;
                    }
                }
                float t0 = max3(s0[0], s0[1], s0[2]), t1 = max3(s1[0], s1[1], s1[2]);
                float t2 = max3(s0[3], s0[4], s0[5]), t3 = max3(s1[3], s1[4], s1[5]);
#pragma unroll
                for (int k = 6; k < 30; k += 4) {
                    t0 = max3(__float_as_uint(t0), s0[k], s0[k + 1]);
                    t1 = max3(__float_as_uint(t1), s1[k], s1[k + 1]);
                    t2 = max3(__float_as_uint(t2), s0[k + 2], s0[k + 3]);
                    t3 = max3(__float_as_uint(t3), s1[k + 2], s1[k + 3]);
                }
                t0 = max3(__float_as_uint(t0), s0[30], s0[31]);
                t1 = max3(__float_as_uint(t1), s1[30], s1[31]);
                t0 = fmaxf(t0, t2);
                t1 = fmaxf(t1, t3);
                if (t == 0 && w.n_tiles > 1) {
                    // The first reference is the largest score of 128 keys (the second tile's are on their way already): the oftener a
                    // row's largest weight is 1, the less its rounding to bf16 costs (scores of standard deviation 1 are 0.75 % further from
                    // 64 bits otherwise; it takes 2.5 % of 32 sequences of 256 to 1024 tokens, 5 to 10 of shorter ones).
                    const int valid1 = tile_info<TC_KT>(1, n_pre, n_blk, w.len_pre, w.len_blk, w.len_suf, 0, 0, 0).valid;
                    if (!mbar_wait(&bars->s_full[j][buf ^ 1], ((n + 1) >> 1) & 1, abort_flag)) { ok = false; break; }
                    tc_fence_after_sync();
#pragma unroll 1
                    for (int c = 0; c < TC_KT; c += 16) {
                        uint32_t v[16];
                        tmem_ld_16cols(tmem_base + S::s_col(j, buf ^ 1) + lane_off + c, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            if (c + k < valid1) t0 = fmaxf(t0, __uint_as_float(v[k]));
                    }
                }
                const float tmax = fmaxf(t0, t1) * c2;     // log2 domain (the scale is > 0); finite: every tile has a key
                // move the reference only when the true max has run away from it (decided per warp, so that the
                // TMEM loads and stores below are executed by whole warps; rows that are not live never ask for it, so that
                // nobody's rounding depends on what lies behind the rollout or the sequence)
                if (__any_sync(0xffffffffu, tmax > m_ref + TC_RESCALE_GAP)) {
                    const float m_new = fmaxf(m_ref, tmax);
                    // (0 with a row's first finite score; a row that has seen only -inf stays as it is)
                    const float factor = m_new == -INFINITY ? 1.f : fast_exp2(m_ref - m_new);
                    m_ref = m_new;
                    l *= factor;
                    if (t >= 1) {
                        // every MMA that adds to O must have landed before O is rescaled in place: tile t - 1 is the last
                        if (!mbar_wait(&bars->pv_done[j][(n - 1) & 1], ((n - 1) >> 1) & 1, abort_flag)) { ok = false; break; }
                        tc_fence_after_sync();
#pragma unroll
                        for (int c = 0; c < D / 16; ++c) {
                            uint32_t ov[16];
                            tmem_ld_16cols(tm_o + c * 16, ov);
                            tmem_ld_wait();
#pragma unroll
                            for (int k = 0; k < 16; ++k) ov[k] = __float_as_uint(__uint_as_float(ov[k]) * factor);
                            tmem_st_16cols(tm_o + c * 16, ov);
                        }
                    }
                }
                // The two query tiles' warps of a scheduler take turns at the exponential unit: when both are at it, both
                // take twice as long and then wait for their next scores together, while the unit idles (16 sequences of
                // 2048 tokens 953 -> 908 us; with 64 channels the products are short and turns cost 268 -> 301 us instead).
                const bool turns = QT == 2 && D == 128 && w.n_q == 2;
                if (turns) {
                    if (!mbar_wait(&bars->turn[j][quadrant], (n_turn & 1) ^ (j == 0 ? 1 : 0), abort_flag)) { ok = false; break; }
                    ++n_turn;
                }
                // P = exp2(s - m_ref) as packed bf16 over the columns S came from (all of S is in registers)
                const float nm = m_ref == -INFINITY ? 0.f : -m_ref;      // (every score so far is -inf: all weights 0, not NaN)
                const uint64_t c2c2 = pack_f32x2(c2, c2), nmnm = pack_f32x2(nm, nm);
                uint64_t psum = 0;                           // two partial sums
                uint32_t pk[32];
                uint64_t e[2][4];
#pragma unroll
                for (int g8 = 0; g8 < 9; ++g8) {
                    if (g8 < 8) {
                        const uint32_t (&sv)[32] = g8 < 4 ? s0 : s1;
                        const int k0 = (g8 & 3) * 8;
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            e[g8 & 1][k] = exp2_f32x2(fma_f32x2(pack_b32x2(sv[k0 + 2 * k], sv[k0 + 2 * k + 1]), c2c2, nmnm));
                    }
                    if (g8 > 0) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const uint64_t v = e[(g8 - 1) & 1][k];
                            psum = add_f32x2(psum, v);
                            pk[(g8 - 1) * 4 + k] = pack_bf16(__uint_as_float(static_cast<uint32_t>(v)), __uint_as_float(static_cast<uint32_t>(v >> 32)));
                        }
                    }
                }
                if (turns) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bars->turn[j ^ 1][quadrant]);
                }
                tmem_st_32cols(tm_s, pk);
                tmem_st_wait();
                const float psum0 = __uint_as_float(static_cast<uint32_t>(psum)), psum1 = __uint_as_float(static_cast<uint32_t>(psum >> 32));
                l += psum0 + psum1;
                if (valid < TC_KT) {
                    // V rows past the segment's end hold whatever lies behind it in memory: zero them so that
                    // probability 0 times garbage cannot make a NaN (thread r clears 16-byte pieces of those rows;
                    // both query tiles' warps do it, each before it releases its own second MMA)
                    uint8_t* vt = kv_s + (n_kv + t) % STAGES * S::KV_STAGE + KV_BYTES;
                    const int n_bad = (TC_KT - valid) * 8;          // 16-byte pieces per 64-column half
                    for (int h2 = 0; h2 < NHALF; ++h2)
                        for (int q = r; q < n_bad; q += 128)
                            *reinterpret_cast<uint4*>(vt + h2 * HALF_K + valid * 128 + q * 16) = make_uint4(0, 0, 0, 0);
                    fence_proxy_async_smem();
                }
                tc_fence_before_sync();
                mbar_arrive(&bars->p_full[j][buf]);
            }
            n_kv += w.n_tiles;
            n_s += w.n_tiles;
            if (ok) ok = mbar_wait(&bars->pv_done[j][(n_s - 1) & 1], ((n_s - 1) >> 1) & 1, abort_flag);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after_sync();
            const float inv = l > 0.f ? 1.f / l : 0.f;
            // O rows leave through shared memory so that the global stores are coalesced (a thread holds one whole row,
            // and 32 lanes storing 16 bytes each to 32 different rows cost a request per lane): 64 columns at a time,
            // 16-byte chunk c of row r at c ^ (r & 7).
            const int pos0 = w.pos0 + j * pos_per_tile;
#pragma unroll
            for (int h2 = 0; h2 < NHALF; ++h2) {
                uint32_t oa[32], ob[32];
                tmem_ld_32cols(tm_o + h2 * 64, oa);          // (whole warp, also for rows that are not stored)
                tmem_ld_32cols(tm_o + h2 * 64 + 32, ob);
                tmem_ld_wait();
                if (h2 > 0) __syncwarp();                    // (the first half has been read out of `ot`)
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint32_t (&ov)[32] = k < 4 ? oa : ob;
                    const int k8 = (k & 3) * 8;
                    uint4 o;
                    o.x = pack_bf16(__uint_as_float(ov[k8 + 0]) * inv, __uint_as_float(ov[k8 + 1]) * inv);
                    o.y = pack_bf16(__uint_as_float(ov[k8 + 2]) * inv, __uint_as_float(ov[k8 + 3]) * inv);
                    o.z = pack_bf16(__uint_as_float(ov[k8 + 4]) * inv, __uint_as_float(ov[k8 + 5]) * inv);
                    o.w = pack_bf16(__uint_as_float(ov[k8 + 6]) * inv, __uint_as_float(ov[k8 + 7]) * inv);
                    *reinterpret_cast<uint4*>(ot + lane * 128 + ((k ^ (lane & 7)) << 4)) = o;
                }
                __syncwarp();
                const int c = lane & 7;
                RowWalk rw = out_walk;
                uint4* dst = reinterpret_cast<uint4*>(p.out + ((static_cast<size_t>(w.token0) + pos0) * p.Hq + w.kvh * p.g) * D + h2 * 64) + c;
#pragma unroll
                for (int k = 0; k < 8; ++k, rw.next()) {
                    const int rr = k * 4 + (lane >> 3);
                    if (rw.i < pos_per_tile && pos0 + rw.i < w.L_eff)
                        dst[(static_cast<size_t>(rw.i) * p.Hq + rw.h) * (D / 8)] =
                            *reinterpret_cast<const uint4*>(ot + rr * 128 + ((c ^ (rr & 7)) << 4));
                }
            }
            __syncwarp();
            tc_fence_before_sync();                          // (O has been read: the next unit's first P V may overwrite it)
            if (p.lse != nullptr && r < rows_in_tile && pos0 + ri < w.L_eff) {
                const int i = pos0 + ri, h = w.kvh * p.g + rh;
                p.lse[packed ? static_cast<size_t>(h) * p.total_tokens + w.token0 + i
                             : (static_cast<size_t>(w.b) * p.Hq + h) * p.L + i] = l > 0.f ? (m_ref + log2f(l)) * LN2_F : -INFINITY;
            }
        }
    }

    // teardown
    tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000LL) {}
        if (threadIdx.x == 0) atomicOr(p.dev_status, DEV_WAIT_EXPIRED);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, S::TMEM_COLS);
    }
    if (p.beside_head && has_last) pdl_wait();
}

template <int D, int QT>
int launch_tc(const CUtensorMap& tm_q, const CUtensorMap* tm, const AttnParams& p, int q_tiles, cudaStream_t stream) {
    constexpr int SMEM = TcShape<D, QT>::SMEM;
    static std::atomic<uint64_t> smem_set{0};
    if (ensure_dynamic_smem(smem_set, attn_block_tc_kernel<D, QT>, SMEM) != DARE_OK) return DARE_ERR_CUDA;
    dim3 grid((q_tiles + QT - 1) / QT, p.B * p.Hkv, 1);
    return launch_kernel(attn_block_tc_kernel<D, QT>, grid, TcShape<D, QT>::THREADS, SMEM, stream, 1, tm_q, tm[0], tm[1], tm[2],
                         tm[3], tm[4], tm[5], p);
}

// The tensor-core tile is worth it when a tile's 128 rows are mostly real query rows.
bool use_tc_path(const AttnArgs& a) {
    const int g = a.Hq / a.Hkv;
    if (g > 128) return false;
    const int pos_per_tile = 128 / g;
    const int rows = (a.L < pos_per_tile ? a.L : pos_per_tile) * g;
    return rows >= 96;
}

// Combine KV-split partials: out = sum_s w_s o_s / sum_s w_s with w_s = exp(lse_s - max lse).
template <int D>
__global__ void attn_combine_kernel(const float* __restrict__ part_o, const float* __restrict__ part_lse, int splits,
                                    size_t n_rows, int L, int Hq, __nv_bfloat16* __restrict__ out,
                                    float* __restrict__ lse) {
    const size_t row = static_cast<size_t>(blockIdx.x) * (blockDim.x / (D / 4)) + threadIdx.x / (D / 4);
    const int c4 = threadIdx.x % (D / 4);
    pdl_wait();
    pdl_trigger();
    if (row >= n_rows) return;
    float mx = -INFINITY;
    for (int s = 0; s < splits; ++s) mx = fmaxf(mx, part_lse[s * n_rows + row]);
    float wsum = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = 0; s < splits; ++s) {
        const float ls = part_lse[s * n_rows + row];
        if (ls == -INFINITY) continue;
        const float w = exp2f((ls - mx) * LOG2E_F);
        const float4 o = *reinterpret_cast<const float4*>(part_o + (s * n_rows + row) * D + c4 * 4);
        acc.x += w * o.x; acc.y += w * o.y; acc.z += w * o.z; acc.w += w * o.w;
        wsum += w;
    }
    const float inv = wsum > 0.f ? 1.f / wsum : 0.f;
    uint2 packed;
    packed.x = pack_bf16(acc.x * inv, acc.y * inv);
    packed.y = pack_bf16(acc.z * inv, acc.w * inv);
    *reinterpret_cast<uint2*>(out + row * D + c4 * 4) = packed;
    if (lse != nullptr && c4 == 0) {
        // row = (b * L + i) * Hq + h  ->  lse[b, h, i]
        const size_t h = row % Hq, bi = row / Hq, i = bi % L, bb = bi / L;
        lse[(bb * Hq + h) * L + i] = wsum > 0.f ? mx + logf(wsum) : -INFINITY;
    }
}

template <int D, int NW, int KS, int KT, int STAGES, int CPS>
int launch_one(const CUtensorMap* tm, const AttnParams& p, int chunks, cudaStream_t stream) {
    constexpr int SMEM = att_smem_bytes<D, KT, STAGES>();
    static_assert(KS * NW * (D / 8 + 1) * 512 <= STAGES * att_stage_bytes<D, KT>() && (D / 8) % KS == 0, "merge buffer");
    static_assert(STAGES <= ATT_MAX_STAGES && KT <= KT_MAX && KT % (16 * KS) == 0, "variant");
    static std::atomic<uint64_t> smem_set{0};
    if (ensure_dynamic_smem(smem_set, attn_block_kernel<D, NW, KS, KT, STAGES, CPS>, SMEM) != DARE_OK) return DARE_ERR_CUDA;
    dim3 grid(chunks, p.B * p.Hkv, p.splits);
    return launch_kernel(attn_block_kernel<D, NW, KS, KT, STAGES, CPS>, grid, (NW * KS + 1) * 32, SMEM, stream, 1, tm[0], tm[1],
                         tm[2], tm[3], tm[4], tm[5], p);
}

// The warp-level kernel's variants by the number of packed query rows R per (rollout, KV head):
//   R <= 16   one row group, four key slices of a 64-key tile, 2 CTAs per SM
//   R <= 32   two row groups, two key slices of a 64-key tile, 2 CTAs per SM (32-key tiles with two warps and
//             4 CTAs per SM were measured slower: 58 against 45 us on 16 rollouts x 32 heads x 768 keys)
//   larger    four row groups per 64-row chunk, 64-key tiles, 2 CTAs per SM
struct WarpVariant { int nw, kt, per_sm; };
WarpVariant pick_variant(int R) {
    if (R <= 16) return {1, 64, 2};
    if (R <= 32) return {2, 64, 2};
    return {4, 64, 2};
}

}  // namespace

int attn_plan_splits(const dare_ctx* ctx, const AttnArgs& a) {
    if (use_tc_path(a)) return 1;
    const int g = a.Hq / a.Hkv;
    const int R = a.L * g;
    const WarpVariant var = pick_variant(R);
    const int nw = var.nw;
    const int chunks = (R + nw * 16 - 1) / (nw * 16);
    const long long units = static_cast<long long>(chunks) * a.B * a.Hkv;
    const long long slots = static_cast<long long>(ctx->sm_count) * var.per_sm;
    const int tiles = (a.prefix_cap + (a.k_blk ? a.L : 0) + a.suffix_cap + var.kt - 1) / var.kt;
    // As many K/V splits as keep the launch in one wave.  (As many as fill the slots or more left a second wave of a few CTAs, as
    // long as the first: 32 rows x 32 heads x 733 keys of 2, 4, 6 and 8 rollouts 17.5, 22.9, 27.2 and 30.9 us, now 13.5, 17.3, 19.1 and
    // 21.2; 4 rows x 5120 keys of 1 and 2 rollouts 28.0 and 42.3, now 21.7 and 31.8.  The other side of it is that from half the slots on
    // a unit is not split, and a launch takes as long as its longest one: 5 rollouts x 32 heads, one of 2048 keys and four of 128,
    // 25.1 and 27.7; 12 rollouts x 8 heads x 90 rows of 512 to 2048 keys 46.6 and 54.4.)
    long long s = slots / units;
    if (s > tiles / 2) s = tiles / 2;
    if (s > 32) s = 32;
    if (s < 1) s = 1;
    return static_cast<int>(s);
}

size_t attn_workspace_bytes(const AttnArgs& a, int splits) {
    if (splits <= 1) return 0;
    const size_t n_rows = static_cast<size_t>(a.B) * a.L * a.Hq;
    return static_cast<size_t>(splits) * n_rows * (a.d + 1) * sizeof(float);
}

int launch_attn(const dare_ctx* ctx, const AttnArgs& a, cudaStream_t stream) {
    AttnParams p;
    p.B = a.B; p.L = a.L; p.Hq = a.Hq; p.Hkv = a.Hkv; p.g = a.Hq / a.Hkv; p.R = a.L * p.g;
    p.prefix_cap = a.prefix_cap; p.suffix_cap = a.k_suf ? a.suffix_cap : 0;
    p.inplace = a.k_blk == nullptr; p.has_suffix = a.k_suf != nullptr && a.suffix_cap > 0;
    p.splits = attn_plan_splits(ctx, a);
    p.uniform_P = a.prefix_len_uniform;
    p.cu_seqlens = nullptr; p.total_tokens = 0;
    const float scale = a.scale != 0.f ? a.scale : 1.0f / sqrtf(static_cast<float>(a.d));
    p.scale_log2 = scale * LOG2E_F;
    p.q = static_cast<const __nv_bfloat16*>(a.q);
    p.prefix_len = a.prefix_len; p.suffix_len = a.suffix_len;
    p.out = static_cast<__nv_bfloat16*>(a.out); p.lse = a.lse;
    p.dev_status = ctx->dev_status;
    p.beside_head = a.beside_head;
    const size_t n_rows = static_cast<size_t>(a.B) * a.L * a.Hq;
    p.part_o = static_cast<float*>(a.scratch ? a.scratch : ctx->workspace);
    p.part_lse = p.part_o + static_cast<size_t>(p.splits) * n_rows * a.d;

    CUtensorMap tm[6];
    const uint64_t units = static_cast<uint64_t>(a.B) * a.Hkv;
    const uint32_t KT = static_cast<uint32_t>(use_tc_path(a) ? TC_KT : pick_variant(p.R).kt);   // rows of a K/V tile
    int rc = make_tmap_bf16_2d(ctx, &tm[0], a.k_pre, units * a.prefix_cap, a.d, KT, 64);
    if (rc == DARE_OK) rc = make_tmap_bf16_2d(ctx, &tm[1], a.v_pre, units * a.prefix_cap, a.d, KT, 64);
    if (rc != DARE_OK) return rc;
    if (!p.inplace) {
        rc = make_tmap_bf16_2d(ctx, &tm[2], a.k_blk, units * a.L, a.d, KT, 64);
        if (rc == DARE_OK) rc = make_tmap_bf16_2d(ctx, &tm[3], a.v_blk, units * a.L, a.d, KT, 64);
        if (rc != DARE_OK) return rc;
    } else {
        tm[2] = tm[0]; tm[3] = tm[1];
    }
    if (p.has_suffix) {
        rc = make_tmap_bf16_2d(ctx, &tm[4], a.k_suf, units * a.suffix_cap, a.d, KT, 64);
        if (rc == DARE_OK) rc = make_tmap_bf16_2d(ctx, &tm[5], a.v_suf, units * a.suffix_cap, a.d, KT, 64);
        if (rc != DARE_OK) return rc;
    } else {
        tm[4] = tm[0]; tm[5] = tm[1];
    }

    if (use_tc_path(a)) {
        // two query tiles per CTA halve the K/V traffic, but only pay when the CTAs still fill the SMs
        const int pos_per_tile = 128 / p.g;
        const int q_tiles = (p.L + pos_per_tile - 1) / pos_per_tile;
        CUtensorMap tm_q;
        rc = make_tmap_bf16_3d(ctx, &tm_q, a.q, static_cast<uint64_t>(a.B) * a.L, a.Hq, a.d, pos_per_tile, p.g, 64);
        if (rc != DARE_OK) return rc;
        const long long pairs = static_cast<long long>((q_tiles + 1) / 2) * p.B * p.Hkv;
        if (q_tiles >= 2 && 4 * pairs >= 3LL * ctx->sm_count)
            return a.d == 128 ? launch_tc<128, 2>(tm_q, tm, p, q_tiles, stream) : launch_tc<64, 2>(tm_q, tm, p, q_tiles, stream);
        return a.d == 128 ? launch_tc<128, 1>(tm_q, tm, p, q_tiles, stream) : launch_tc<64, 1>(tm_q, tm, p, q_tiles, stream);
    }
    const int nw = pick_variant(p.R).nw;
    const int chunks = (p.R + nw * 16 - 1) / (nw * 16);
    if (a.d == 128) {
        rc = nw == 1 ? launch_one<128, 1, 4, 64, 3, 2>(tm, p, chunks, stream)
           : nw == 2 ? launch_one<128, 2, 2, 64, 3, 2>(tm, p, chunks, stream)
                     : launch_one<128, 4, 1, 64, 3, 2>(tm, p, chunks, stream);
    } else {
        rc = nw == 1 ? launch_one<64, 1, 4, 64, 3, 2>(tm, p, chunks, stream)
           : nw == 2 ? launch_one<64, 2, 2, 64, 3, 2>(tm, p, chunks, stream)
                     : launch_one<64, 4, 1, 64, 3, 2>(tm, p, chunks, stream);
    }
    if (rc != DARE_OK) return rc;
    if (p.splits > 1) {
        const int tpr = a.d / 4;                    // threads per row
        const int rows_per_block = 256 / tpr;
        const unsigned blocks = static_cast<unsigned>((n_rows + rows_per_block - 1) / rows_per_block);
        return launch_kernel(a.d == 128 ? attn_combine_kernel<128> : attn_combine_kernel<64>, dim3(blocks), 256, 0, stream, 1,
                             p.part_o, p.part_lse, p.splits, n_rows, a.L, a.Hq, p.out, p.lse);
    }
    return DARE_OK;
}

// Packed variable-length bidirectional attention on the tcgen05 kernel: sequence s = "rollout" s, its tokens are the
// queries and, in place, the keys; K and V are 2-D [tokens, Hkv * d] views, a KV head is a column range.
int launch_attn_varlen(const dare_ctx* ctx, int total, int n_seqs, int max_seqlen, int Hq, int Hkv, int d, float scale,
                       const void* q, const void* k, const void* v, const int32_t* cu_seqlens, void* out, float* lse,
                       cudaStream_t stream) {
    AttnParams p = {};
    p.B = n_seqs; p.L = max_seqlen; p.Hq = Hq; p.Hkv = Hkv; p.g = Hq / Hkv; p.R = max_seqlen * p.g;
    p.prefix_cap = 0; p.suffix_cap = 0; p.inplace = 1; p.has_suffix = 0; p.splits = 1; p.uniform_P = 0;
    p.scale_log2 = (scale != 0.f ? scale : 1.0f / sqrtf(static_cast<float>(d))) * LOG2E_F;
    p.q = static_cast<const __nv_bfloat16*>(q);
    p.prefix_len = nullptr; p.suffix_len = nullptr;
    p.out = static_cast<__nv_bfloat16*>(out); p.lse = lse;
    p.part_o = nullptr; p.part_lse = nullptr;
    p.dev_status = ctx->dev_status;
    p.cu_seqlens = cu_seqlens; p.total_tokens = total;
    CUtensorMap tm[6];
    int rc = make_tmap_bf16_2d(ctx, &tm[0], k, static_cast<uint64_t>(total), static_cast<uint64_t>(Hkv) * d, TC_KT, 64);
    if (rc == DARE_OK) rc = make_tmap_bf16_2d(ctx, &tm[1], v, static_cast<uint64_t>(total), static_cast<uint64_t>(Hkv) * d, TC_KT, 64);
    if (rc != DARE_OK) return rc;
    tm[2] = tm[0]; tm[3] = tm[1]; tm[4] = tm[0]; tm[5] = tm[1];
    const int pos_per_tile = 128 / p.g;
    const int q_tiles = (max_seqlen + pos_per_tile - 1) / pos_per_tile;
    CUtensorMap tm_q;
    rc = make_tmap_bf16_3d(ctx, &tm_q, q, static_cast<uint64_t>(total), Hq, d, pos_per_tile, p.g, 64);
    if (rc != DARE_OK) return rc;
    if (q_tiles >= 2) return d == 128 ? launch_tc<128, 2>(tm_q, tm, p, q_tiles, stream) : launch_tc<64, 2>(tm_q, tm, p, q_tiles, stream);
    return d == 128 ? launch_tc<128, 1>(tm_q, tm, p, q_tiles, stream) : launch_tc<64, 1>(tm_q, tm, p, q_tiles, stream);
}

}  // namespace dare
