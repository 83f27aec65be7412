// The bandwidth-bound pieces of the layer stack: embedding gather, RMSNorm, and RoPE with the in-place
// K/V cache write.  Each is one pass over its rows with 128-bit accesses; fp32 inside, bf16 in memory.
#include <math.h>

#include "internal.h"
#include "ptx.cuh"

namespace dare {
namespace {

constexpr int ROWS_PER_BLOCK = 8;   // one warp per row

__device__ __forceinline__ float lo_f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_f(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ float sum_squares(const uint4& v) {
    const float a0 = lo_f(v.x), a1 = hi_f(v.x), a2 = lo_f(v.y), a3 = hi_f(v.y);
    const float a4 = lo_f(v.z), a5 = hi_f(v.z), a6 = lo_f(v.w), a7 = hi_f(v.w);
    return a0 * a0 + a1 * a1 + a2 * a2 + a3 * a3 + a4 * a4 + a5 * a5 + a6 * a6 + a7 * a7;
}
__device__ __forceinline__ uint4 scale_bf16(const uint4& v, float f) {
    return make_uint4(pack_bf16(lo_f(v.x) * f, hi_f(v.x) * f), pack_bf16(lo_f(v.y) * f, hi_f(v.y) * f),
                      pack_bf16(lo_f(v.z) * f, hi_f(v.z) * f), pack_bf16(lo_f(v.w) * f, hi_f(v.w) * f));
}

// x[m, :] = E[tokens[b, start + i], :] for row m = b * length + i.
__global__ void __launch_bounds__(ROWS_PER_BLOCK * 32)
embed_gather_kernel(const uint4* __restrict__ emb, int D8, int V, const int32_t* __restrict__ tokens, int64_t row_stride,
                    int start, int length, int n_rows, uint4* __restrict__ x) {
    const int m = blockIdx.x * ROWS_PER_BLOCK + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    pdl_wait();
    pdl_trigger();
    if (m >= n_rows) return;
    int tok = tokens[static_cast<int64_t>(m / length) * row_stride + start + m % length];
    tok = min(max(tok, 0), V - 1);
    const uint4* src = emb + static_cast<size_t>(tok) * D8;
    uint4* dst = x + static_cast<size_t>(m) * D8;
    for (int i = lane; i < D8; i += 32) dst[i] = src[i];
}

// y = x / sqrt(mean(x^2) + eps), weight 1.  A row's time is one trip to memory and back, so a row gets a whole CTA:
// NORM_THREADS threads read it in one go (NORM_VECS 16-byte pieces each, all in flight together, kept in registers for
// the scaling); longer rows are read a second time.  2.7 us at 512 rows x 4096 between two projections, where one warp
// per row with two passes took 4.2 us.
constexpr int NORM_THREADS = 128;
constexpr int NORM_VECS = 4;
__global__ void __launch_bounds__(NORM_THREADS)
rmsnorm_kernel(const uint4* __restrict__ x, int D8, float eps, uint4* __restrict__ y) {
    __shared__ float s_part[NORM_THREADS / 32];
    const uint4* src = x + static_cast<size_t>(blockIdx.x) * D8;
    uint4* dst = y + static_cast<size_t>(blockIdx.x) * D8;
    pdl_wait();
    pdl_trigger();
    uint4 v[NORM_VECS];
#pragma unroll
    for (int u = 0; u < NORM_VECS; ++u) {
        const int i = threadIdx.x + u * NORM_THREADS;
        v[u] = i < D8 ? src[i] : make_uint4(0, 0, 0, 0);
    }
    float ss = 0.f;
#pragma unroll
    for (int u = 0; u < NORM_VECS; ++u) ss += sum_squares(v[u]);
    for (int i = threadIdx.x + NORM_VECS * NORM_THREADS; i < D8; i += NORM_THREADS) ss += sum_squares(src[i]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = ss;
    __syncthreads();
    ss = 0.f;
#pragma unroll
    for (int w = 0; w < NORM_THREADS / 32; ++w) ss += s_part[w];
    const float inv = rsqrtf(ss / static_cast<float>(D8 * 8) + eps);
#pragma unroll
    for (int u = 0; u < NORM_VECS; ++u) {
        const int i = threadIdx.x + u * NORM_THREADS;
        if (i < D8) dst[i] = scale_bf16(v[u], inv);
    }
    for (int i = threadIdx.x + NORM_VECS * NORM_THREADS; i < D8; i += NORM_THREADS) dst[i] = scale_bf16(src[i], inv);
}

// The same with a warp per row, ROWS_PER_BLOCK rows per CTA, for many short rows (norm_warp_rows below).  Lane l stands for
// the threads l, l + 32, ... of the kernel above and adds in the same order: a row's result does not depend on the number
// of rows beside it.
template <int VECS>
__global__ void __launch_bounds__(ROWS_PER_BLOCK * 32)
rmsnorm_warp_kernel(const uint4* __restrict__ x, int D8, int n_rows, float eps, uint4* __restrict__ y) {
    constexpr int WARPS = NORM_THREADS / 32;
    const int m = blockIdx.x * ROWS_PER_BLOCK + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    pdl_wait();
    pdl_trigger();
    if (m >= n_rows) return;
    const uint4* src = x + static_cast<size_t>(m) * D8;
    uint4* dst = y + static_cast<size_t>(m) * D8;
    uint4 v[VECS];
#pragma unroll
    for (int u = 0; u < VECS; ++u) {
        const int i = lane + u * 32;
        v[u] = i < D8 ? src[i] : make_uint4(0, 0, 0, 0);
    }
    float ss = 0.f;
#pragma unroll
    for (int w = 0; w < (VECS < WARPS ? VECS : WARPS); ++w) {
        float part = 0.f;
#pragma unroll
        for (int u = w; u < VECS; u += WARPS) part += sum_squares(v[u]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
        ss += part;
    }
    const float inv = rsqrtf(ss / static_cast<float>(D8 * 8) + eps);
#pragma unroll
    for (int u = 0; u < VECS; ++u) {
        const int i = lane + u * 32;
        if (i < D8) dst[i] = scale_bf16(v[u], inv);
    }
}

// cs[p, c] = (cos, sin)(p * base^(-2c/d)), c < d/2, evaluated in double precision; cs_t is its transpose.
__global__ void rope_table_kernel(float2* __restrict__ cs, float2* __restrict__ cs_t, int n_pos, int half, double base) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (i >= n_pos * half) return;
    const int p = i / half, c = i % half;
    const double ang = static_cast<double>(p) * pow(base, -static_cast<double>(c) / static_cast<double>(half));
    double s, co;
    sincos(ang, &s, &co);
    cs[i] = make_float2(static_cast<float>(co), static_cast<float>(s));
    cs_t[static_cast<size_t>(c) * n_pos + p] = cs[i];
}

// Row m = (b, i) of the fused QKV projection [n_rows, (Hq + 2 Hkv) d], position p = start + i:
//   q heads  -> q_out[m, h, :] rotated;  k heads -> k_cache[b, h, p, :] rotated;  v heads -> v_cache[b, h, p, :].
// Half-split pairing: channel c turns together with channel c + d/2.  A thread keeps one group of 8 channels of the half head
// and walks the heads, so its 8 angles (a table that nothing writes any more) are in registers before the projection is
// done; what it reads of the projection, it asks for ROPE_BATCH heads at a time.  512 rows of 96 heads of 128 between the
// projection and the attention: 5.4 us, 25 MB through L2; 8.0 with 128 threads that took one head after another and its
// angles with it (256 such threads: 6.5).
// A row has `row_threads` threads (rope_row_threads below; WHOLE: all ROPE_THREADS), a CTA as many rows as ROPE_THREADS hold.
constexpr int ROPE_THREADS = 256;
constexpr int ROPE_BATCH = 2;
template <bool WHOLE>
__global__ void __launch_bounds__(ROPE_THREADS)
rope_kv_write_kernel(const __nv_bfloat16* __restrict__ qkv, int n_rows, int row_threads_, int Hq, int Hkv, int d, int start, int length,
                     const float2* __restrict__ cs, __nv_bfloat16* __restrict__ q_out,
                     __nv_bfloat16* __restrict__ k_cache, __nv_bfloat16* __restrict__ v_cache, int cap) {
    const int row_threads = WHOLE ? ROPE_THREADS : row_threads_, tid = WHOLE ? threadIdx.x : threadIdx.x % row_threads;
    const int m_any = WHOLE ? blockIdx.x : (blockIdx.x * blockDim.x + threadIdx.x) / row_threads;
    const int m = WHOLE ? m_any : min(m_any, n_rows - 1);
    const int b = m / length, i = m % length, p = start + i;
    const int half = d / 2, cpb = half / 8;                 // 8-channel groups per half head (4 or 8)
    const int c0 = tid % cpb * 8, h_step = row_threads / cpb;
    const int n_rot = Hq + Hkv, n_v = Hkv * (d / 8);
    const __nv_bfloat16* row = qkv + static_cast<size_t>(m) * (Hq + 2 * Hkv) * d;
    float2 t[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) t[j] = cs[static_cast<size_t>(p) * half + c0 + j];
    pdl_wait();
    pdl_trigger();
    if (!WHOLE && m_any >= n_rows) return;
    for (int h0 = tid / cpb; h0 < n_rot; h0 += ROPE_BATCH * h_step) {
        uint4 lo[ROPE_BATCH], hi[ROPE_BATCH];
#pragma unroll
        for (int u = 0; u < ROPE_BATCH; ++u) {
            const __nv_bfloat16* src = row + static_cast<size_t>(min(h0 + u * h_step, n_rot - 1)) * d + c0;
            lo[u] = *reinterpret_cast<const uint4*>(src);
            hi[u] = *reinterpret_cast<const uint4*>(src + half);
        }
#pragma unroll
        for (int u = 0; u < ROPE_BATCH; ++u) {
            const int h = h0 + u * h_step;
            if (h >= n_rot) break;
            const uint32_t aw[4] = {lo[u].x, lo[u].y, lo[u].z, lo[u].w}, bw[4] = {hi[u].x, hi[u].y, hi[u].z, hi[u].w};
            uint32_t o1[4], o2[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 t0 = t[2 * j], t1 = t[2 * j + 1];
                const float x10 = lo_f(aw[j]), x11 = hi_f(aw[j]), x20 = lo_f(bw[j]), x21 = hi_f(bw[j]);
                o1[j] = pack_bf16(x10 * t0.x - x20 * t0.y, x11 * t1.x - x21 * t1.y);
                o2[j] = pack_bf16(x20 * t0.x + x10 * t0.y, x21 * t1.x + x11 * t1.y);
            }
            __nv_bfloat16* dst = h < Hq ? q_out + (static_cast<size_t>(m) * Hq + h) * d
                                        : k_cache + ((static_cast<size_t>(b) * Hkv + (h - Hq)) * cap + p) * d;
            *reinterpret_cast<uint4*>(dst + c0) = make_uint4(o1[0], o1[1], o1[2], o1[3]);
            *reinterpret_cast<uint4*>(dst + half + c0) = make_uint4(o2[0], o2[1], o2[2], o2[3]);
        }
    }
#pragma unroll 2
    for (int j = tid; j < n_v; j += row_threads) {
        const int h = j / (d / 8), c = (j % (d / 8)) * 8;
        const uint4 v = *reinterpret_cast<const uint4*>(row + static_cast<size_t>(n_rot + h) * d + c);
        *reinterpret_cast<uint4*>(v_cache + ((static_cast<size_t>(b) * Hkv + h) * cap + p) * d + c) = v;
    }
}

// Shared memory (unused) that a small kernel of `ctas` short CTAs asks for: set up while a projection still runs, its
// CTAs would pile up on the few SMs that the projection leaves idle (sixteen per SM on 8 of 148 at 512 x 12288: the RoPE
// kernel then took 19 us instead of 7.4).  With 44 KB each none fits beside a CTA of the pair kernel, two beside one of the
// few-row kernel's, and SPREAD_CTAS on an SM of their own; more CTAs than that ask for none, all are resident at once then.
constexpr size_t SPREAD_SMEM = 44 * 1024;
constexpr int SPREAD_CTAS = 5;
static_assert(SPREAD_CTAS * (SPREAD_SMEM + 1024 + 128) <= 228 * 1024, "the system takes 1 KB per CTA, RMSNorm 16 bytes");
inline size_t spread_smem(int ctas, int sm_count) { return ctas <= SPREAD_CTAS * sm_count ? SPREAD_SMEM : 0; }

// Rows for which a warp each is the better split.  CTAs start at about one per ns over the GPU, whatever they do: 65536 rows
// of 256 took 68 us with one each and take 9.3, 16384 of 1024 17.5 and 7.0, 4096 of 512 4.7 and 2.4.  Longer rows are bound
// by their bytes, and few of them by one row's trip to memory, which four warps make shorter: 512 of 1024 1.4 us with a CTA
// per row and 1.7 with a warp, 600 of 1024 1.8 and 1.6, 3072 of 2048 4.0 and 4.1, 6144 of 2048 7.1 and 6.5, 4096 of 3072 5.5 and
// 8.2.  (Up to 512 values both take 1.1 to 1.3 us up to 512 rows.)
inline bool norm_warp_rows(int n_rows, int D) { return D <= 2048 && n_rows > (D <= 1024 ? 512 : 4095); }

// Threads per row of the rotary kernel: enough for a batch of heads each, up to a warp also for one piece of v each.  (A whole
// CTA per row, whatever its heads, leaves most threads idle and is bound by how fast CTAs start: 32768 rows of 2 + 1 heads of
// 64 48 us, now 6.9; 2048 rows of 4 + 2 heads of 128 6.3 and 2.8, of 32 + 8 9.0 and 7.4; 48 rows 1.7 to 2.0 either way.)
inline int rope_row_threads(int Hq, int Hkv, int d) {
    const int rot = (Hq + Hkv + ROPE_BATCH - 1) / ROPE_BATCH * (d / 16), v = Hkv * (d / 8);      // (multiples of d / 16)
    const int n = rot >= 32 || rot >= v ? rot : v < 32 ? v : 32;
    return n < ROPE_THREADS ? n : ROPE_THREADS;
}

}  // namespace

int launch_embed(const void* emb, int D, int V, const int32_t* tokens, int64_t row_stride, int start, int length,
                 int n_rows, void* x, cudaStream_t stream) {
    return launch_kernel(embed_gather_kernel, dim3((n_rows + ROWS_PER_BLOCK - 1) / ROWS_PER_BLOCK), ROWS_PER_BLOCK * 32, 0,
                         stream, 1, static_cast<const uint4*>(emb), D / 8, V, tokens, row_stride, start, length, n_rows,
                         static_cast<uint4*>(x));
}

int launch_rmsnorm(const void* x, int D, int n_rows, float eps, void* y, int sm_count, cudaStream_t stream) {
    const uint4* src = static_cast<const uint4*>(x);
    uint4* dst = static_cast<uint4*>(y);
    if (norm_warp_rows(n_rows, D)) {
        const auto kernel = D <= 256 ? rmsnorm_warp_kernel<1> : D <= 512 ? rmsnorm_warp_kernel<2> : D <= 1024 ? rmsnorm_warp_kernel<4>
                            : rmsnorm_warp_kernel<8>;
        return launch_kernel(kernel, dim3((n_rows + ROWS_PER_BLOCK - 1) / ROWS_PER_BLOCK), ROWS_PER_BLOCK * 32, 0, stream, 1, src, D / 8,
                             n_rows, eps, dst);
    }
    return launch_kernel(rmsnorm_kernel, dim3(n_rows), NORM_THREADS, spread_smem(n_rows, sm_count), stream, 1, src, D / 8, eps, dst);
}

int launch_rope_table(float* cs, float* cs_t, int n_pos, int half, double base, cudaStream_t stream) {
    const int n = n_pos * half;
    return launch_kernel(rope_table_kernel, dim3((n + 255) / 256), 256, 0, stream, 1, reinterpret_cast<float2*>(cs),
                         reinterpret_cast<float2*>(cs_t), n_pos, half, base);
}

int launch_rope_kv_write(const void* qkv, int n_rows, int Hq, int Hkv, int d, int start, int length, const float* cs,
                         void* q_out, void* k_cache, void* v_cache, int cap, int sm_count, cudaStream_t stream) {
    const int row_threads = rope_row_threads(Hq, Hkv, d), rows = ROPE_THREADS / row_threads;
    const int ctas = (n_rows + rows - 1) / rows;
    return launch_kernel(row_threads == ROPE_THREADS ? rope_kv_write_kernel<true> : rope_kv_write_kernel<false>, dim3(ctas),
                         rows * row_threads, spread_smem(ctas, sm_count), stream, 1, static_cast<const __nv_bfloat16*>(qkv), n_rows,
                         row_threads, Hq, Hkv, d, start, length, reinterpret_cast<const float2*>(cs),
                         static_cast<__nv_bfloat16*>(q_out), static_cast<__nv_bfloat16*>(k_cache),
                         static_cast<__nv_bfloat16*>(v_cache), cap);
}

}  // namespace dare
