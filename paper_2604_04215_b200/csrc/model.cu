// The end-to-end denoising loop on a decoder-shaped stack (RMSNorm, fused QKV projection, RoPE, block
// attention against the in-place K/V cache, SwiGLU feed-forward, untied LM head): host-side sequencing only.
// Every arithmetic step is a kernel of gemm.cu, layers.cu, attn.cu, lmhead.cu or select.cu.
//
// A forward of the rows [start, start + length) of every rollout writes those rows' post-RoPE K/V into the
// cache at their positions and lets them attend to cache[0, start + length): with start = 0 this is the
// prefill (the prompt is one bidirectional segment); with start = a block's first position it is one
// denoising step's stack, or, once the block holds no mask, the refresh that leaves the block's final K/V in
// the cache before the prefix grows.
//
// A forward may also let its rows see cache[0, kv_len) with kv_len beyond the rows' own end: the positions
// behind the rows are then a cached suffix (whatever an earlier forward wrote there).  That is the dual cache
// of a fully bidirectional model: dare_generate_dual refreshes every position's K/V with one forward of the
// whole sequence before each block and runs the block's steps against prefix + block + suffix.
#include <math.h>
#include <cuda_bf16.h>
#include <new>

#include "internal.h"
#include "ptx.cuh"

struct dare_model {
    dare_ctx* ctx;
    dare_model_desc desc;
    const void* embedding;
    const void* lm_head;
    dare_layer_weights* layers;    // host copy of the caller's array (device pointers inside)
    float *rope_cs, *rope_cs_t;    // [max_positions, d/2] (cos, sin) and its transpose
    void *x, *h, *qkv, *q, *attn, *act;   // activations, max_rows each
    int32_t* host_counts;          // page-locked: remaining masks of the loop's last steps, [COUNT_SLOTS][max_batch]
    int max_batch;
    // sampled head (dare_model_set_sampling): temperature 0 = greedy; the device word counts the steps
    float sample_temperature;
    uint64_t sample_seed;
    uint32_t* step_counter;
};

namespace {

constexpr int COUNT_SLOTS = 4;

__global__ void set_word_kernel(uint32_t* p, uint32_t v) {
    dare::pdl_wait();
    *p = v;
}

// Keys visible to the rows: cache[0, kv_len), start + length <= kv_len <= cap.
int forward_rows(dare_model* m, const int32_t* tokens, int B, int64_t row_stride, int start, int length, int kv_len,
                 void* k_cache, void* v_cache, int cap, void* hidden_out, cudaStream_t s) {
    using namespace dare;
    const dare_model_desc& c = m->desc;
    const int rows = B * length;
    const int nq = c.n_q_heads * c.head_dim, nkv = c.n_kv_heads * c.head_dim;
    int rc = launch_embed(m->embedding, c.hidden, c.vocab, tokens, row_stride, start, length, rows, m->x, s);
    if (rc != DARE_OK) return rc;
    const size_t layer_kv = static_cast<size_t>(B) * c.n_kv_heads * cap * c.head_dim;   // elements per layer
    for (int l = 0; l < c.n_layers; ++l) {
        const dare_layer_weights& w = m->layers[l];
        __nv_bfloat16* kc = static_cast<__nv_bfloat16*>(k_cache) + layer_kv * l;
        __nv_bfloat16* vc = static_cast<__nv_bfloat16*>(v_cache) + layer_kv * l;
        rc = launch_rmsnorm(m->x, c.hidden, rows, c.rms_eps, m->h, m->ctx->sm_count, s);
        if (rc != DARE_OK) return rc;
        if (gemm_takes_rope(rows, nq + 2 * nkv)) {
            const RopeArgs rope = {c.n_q_heads, c.n_kv_heads, c.head_dim, start, length, cap, m->rope_cs, m->rope_cs_t,
                                   c.max_positions, m->q, kc, vc};
            rc = launch_gemm(m->ctx, GEMM_EPI_ROPE, m->h, rows, c.hidden, w.wqkv, nullptr, nq + 2 * nkv, nullptr, nullptr,
                             nq + 2 * nkv, s, &rope, true);
        } else {
            rc = launch_gemm(m->ctx, GEMM_EPI_STORE, m->h, rows, c.hidden, w.wqkv, nullptr, nq + 2 * nkv, m->qkv, nullptr,
                             nq + 2 * nkv, s, nullptr, true);
            if (rc == DARE_OK)
                rc = launch_rope_kv_write(m->qkv, rows, c.n_q_heads, c.n_kv_heads, c.head_dim, start, length, m->rope_cs,
                                          m->q, kc, vc, cap, m->ctx->sm_count, s);
        }
        if (rc != DARE_OK) return rc;
        AttnArgs a;
        a.B = B; a.L = length; a.Hq = c.n_q_heads; a.Hkv = c.n_kv_heads; a.d = c.head_dim;
        a.prefix_cap = cap; a.suffix_cap = 0; a.scale = 0.f;
        a.q = m->q; a.k_pre = kc; a.v_pre = vc; a.prefix_len = nullptr;
        a.prefix_len_uniform = kv_len - length;   // in place: the kernel reads keys [0, this + length) of the cache
        a.k_blk = a.v_blk = a.k_suf = a.v_suf = nullptr; a.suffix_len = nullptr;
        a.out = m->attn; a.lse = nullptr;
        if (attn_workspace_bytes(a, attn_plan_splits(m->ctx, a)) > m->ctx->workspace_bytes) return DARE_ERR_WORKSPACE;
        rc = launch_attn(m->ctx, a, s);
        if (rc != DARE_OK) return rc;
        rc = launch_gemm(m->ctx, GEMM_EPI_RESIDUAL, m->attn, rows, nq, w.wo, nullptr, c.hidden, m->x, m->x, c.hidden, s, nullptr, true);
        if (rc != DARE_OK) return rc;
        rc = launch_rmsnorm(m->x, c.hidden, rows, c.rms_eps, m->h, m->ctx->sm_count, s);
        if (rc != DARE_OK) return rc;
        rc = launch_gemm(m->ctx, GEMM_EPI_SWIGLU, m->h, rows, c.hidden, w.wg, w.wu, c.ffn, m->act, nullptr, c.ffn, s, nullptr, true);
        if (rc != DARE_OK) return rc;
        rc = launch_gemm(m->ctx, GEMM_EPI_RESIDUAL, m->act, rows, c.ffn, w.wd, nullptr, c.hidden, m->x, m->x, c.hidden, s, nullptr, true);
        if (rc != DARE_OK) return rc;
    }
    return launch_rmsnorm(m->x, c.hidden, rows, c.rms_eps, hidden_out ? hidden_out : m->h, m->ctx->sm_count, s);
}

int check_rows(const dare_model* m, const void* tokens, int B, int64_t row_stride, int start, int length, int kv_len,
               const void* k_cache, const void* v_cache, int cap) {
    if (!m || !tokens || !k_cache || !v_cache) return DARE_ERR_NULL;
    if (int rc = dare::check_current_device(m->ctx)) return rc;
    if (B < 1 || length < 1 || B > m->max_batch) return DARE_ERR_SHAPE;
    if (static_cast<long long>(B) * length > m->desc.max_rows) return DARE_ERR_SHAPE;
    if (start < 0 || static_cast<long long>(start) + length > cap || cap > m->desc.max_positions ||
        static_cast<long long>(start) + length > row_stride)
        return DARE_ERR_RANGE;
    if (kv_len < start + length || kv_len > cap) return DARE_ERR_RANGE;
    if ((reinterpret_cast<uintptr_t>(k_cache) & 15u) || (reinterpret_cast<uintptr_t>(v_cache) & 15u)) return DARE_ERR_ALIGN;
    return DARE_OK;
}

int step_rows(dare_model* m, int32_t* tokens, int B, int64_t row_stride, int start, int L, int kv_len, void* k_cache,
              void* v_cache, int cap, int mode, float threshold, int k, int32_t* pred, float* conf, int32_t* n_committed,
              int32_t* n_remaining, cudaStream_t s, int32_t* host_remaining = nullptr) {
    int rc = forward_rows(m, tokens, B, row_stride, start, L, kv_len, k_cache, v_cache, cap, nullptr, s);
    if (rc != DARE_OK) return rc;
    const int M = B * L;
    dare::LmSampleArgs smp;
    const bool sampled = m->sample_temperature > 0.f;
    smp.temperature = m->sample_temperature; smp.seed = m->sample_seed; smp.step = 0; smp.step_dev = m->step_counter;
    if (L <= dare::LMHEAD_SELECT_MAX_L) {      // short blocks: the selection rides on the head's merge kernel
        const dare::LmSelectArgs sel = {tokens + start, B, mode, threshold, k, n_committed, n_remaining,
                                        host_remaining};
        return dare::launch_lmhead(m->ctx, m->ctx->workspace, m->h, M, m->desc.hidden, m->lm_head, m->desc.vocab,
                                   tokens + start, L, row_stride, m->desc.mask_id, 1, pred, conf, s, sampled ? &smp : nullptr,
                                   &sel);
    }
    rc = dare::launch_lmhead(m->ctx, m->ctx->workspace, m->h, M, m->desc.hidden, m->lm_head, m->desc.vocab,
                             tokens + start, L, row_stride, m->desc.mask_id, 1, pred, conf, s, sampled ? &smp : nullptr);
    if (rc != DARE_OK) return rc;
    return dare::launch_unmask_select(tokens, B, row_stride, start, L, pred, conf, m->desc.mask_id, mode, threshold, k,
                                      n_committed, n_remaining, s, host_remaining);
}

int check_step(const dare_model* m, int B, int L, int mode, float threshold, int k, const void* pred, const void* conf) {
    if (!pred || !conf) return DARE_ERR_NULL;
    if (L > 4096) return DARE_ERR_SHAPE;
    if (mode != DARE_SELECT_THRESHOLD && mode != DARE_SELECT_TOPK) return DARE_ERR_RANGE;
    if (mode == DARE_SELECT_THRESHOLD && threshold != threshold) return DARE_ERR_RANGE;
    if (mode == DARE_SELECT_TOPK && k < 1) return DARE_ERR_RANGE;
    if (dare::lmhead_workspace_bytes(B * L, m->desc.hidden, m->desc.vocab, m->ctx->sm_count, true,
                                     m->sample_temperature > 0.f) > m->ctx->workspace_bytes)
        return DARE_ERR_WORKSPACE;
    return DARE_OK;
}

}  // namespace

extern "C" {

int dare_model_create(dare_ctx* ctx, const dare_model_desc* desc, const void* embedding,
                      const dare_layer_weights* layers, const void* lm_head, dare_model** out) {
    if (!ctx || !desc || !embedding || !layers || !lm_head || !out) return DARE_ERR_NULL;
    *out = nullptr;
    const dare_model_desc& c = *desc;
    if (c.n_layers < 1 || c.hidden < 8 || c.hidden % 8 || c.n_q_heads < 1 || c.n_kv_heads < 1 ||
        c.n_q_heads % c.n_kv_heads || (c.head_dim != 64 && c.head_dim != 128) || c.ffn < 8 || c.ffn % 8 || c.vocab < 2 ||
        c.max_positions < 1 || c.max_rows < 1 || c.max_batch < 1)
        return DARE_ERR_SHAPE;
    if (c.mask_id < 0 || c.mask_id >= c.vocab || !(c.rms_eps >= 0.f) || !(c.rope_base > 1.f)) return DARE_ERR_RANGE;
    for (int l = 0; l < c.n_layers; ++l)
        if (!layers[l].wqkv || !layers[l].wo || !layers[l].wg || !layers[l].wu || !layers[l].wd) return DARE_ERR_NULL;
    dare::DeviceScope scope(ctx->device);
    if (!scope.ok()) return DARE_ERR_CUDA;
    dare_model* m = new (std::nothrow) dare_model();
    if (!m) return DARE_ERR_CUDA;
    m->ctx = ctx; m->desc = c; m->embedding = embedding; m->lm_head = lm_head; m->max_batch = c.max_batch;
    m->layers = new (std::nothrow) dare_layer_weights[c.n_layers];
    m->rope_cs = m->rope_cs_t = nullptr; m->x = m->h = m->qkv = m->q = m->attn = m->act = nullptr; m->host_counts = nullptr;
    m->sample_temperature = 0.f; m->sample_seed = 0; m->step_counter = nullptr;
    bool ok = m->layers != nullptr;
    if (ok) for (int l = 0; l < c.n_layers; ++l) m->layers[l] = layers[l];
    const size_t rows = static_cast<size_t>(c.max_rows);
    const size_t nq = static_cast<size_t>(c.n_q_heads) * c.head_dim, nkv = static_cast<size_t>(c.n_kv_heads) * c.head_dim;
    const size_t rope_bytes = sizeof(float) * 2 * static_cast<size_t>(c.max_positions) * (c.head_dim / 2);
    ok = ok && cudaMalloc(&m->rope_cs, rope_bytes) == cudaSuccess;
    ok = ok && cudaMalloc(&m->rope_cs_t, rope_bytes) == cudaSuccess;
    ok = ok && cudaMalloc(&m->x, rows * c.hidden * 2) == cudaSuccess;
    ok = ok && cudaMalloc(&m->h, rows * c.hidden * 2) == cudaSuccess;
    ok = ok && cudaMalloc(&m->qkv, rows * (nq + 2 * nkv) * 2) == cudaSuccess;
    ok = ok && cudaMalloc(&m->q, rows * nq * 2) == cudaSuccess;
    ok = ok && cudaMalloc(&m->attn, rows * nq * 2) == cudaSuccess;
    ok = ok && cudaMalloc(&m->act, rows * c.ffn * 2) == cudaSuccess;
    ok = ok && cudaMalloc(reinterpret_cast<void**>(&m->step_counter), sizeof(uint32_t)) == cudaSuccess;
    ok = ok && cudaMemset(m->step_counter, 0, sizeof(uint32_t)) == cudaSuccess;
    ok = ok && cudaMallocHost(reinterpret_cast<void**>(&m->host_counts), sizeof(int32_t) * COUNT_SLOTS * c.max_batch) == cudaSuccess;
    ok = ok && dare::launch_rope_table(m->rope_cs, m->rope_cs_t, c.max_positions, c.head_dim / 2, static_cast<double>(c.rope_base),
                                       nullptr) == DARE_OK;
    ok = ok && cudaDeviceSynchronize() == cudaSuccess;
    if (!ok) {
        dare_model_destroy(m);
        return DARE_ERR_CUDA;
    }
    *out = m;
    return DARE_OK;
}

int dare_model_destroy(dare_model* m) {
    if (!m) return DARE_ERR_NULL;
    dare::DeviceScope scope(m->ctx->device);
    cudaFree(m->rope_cs); cudaFree(m->rope_cs_t); cudaFree(m->x); cudaFree(m->h); cudaFree(m->qkv); cudaFree(m->q); cudaFree(m->attn);
    cudaFree(m->act);
    cudaFree(m->step_counter);
    if (m->host_counts) cudaFreeHost(m->host_counts);
    delete[] m->layers;
    delete m;
    return DARE_OK;
}

int dare_model_set_sampling(dare_model* m, float temperature, uint64_t seed, uint32_t first_step, void* stream) {
    if (!m) return DARE_ERR_NULL;
    if (int rc = dare::check_current_device(m->ctx)) return rc;
    if (!(temperature >= 0.f) || isinf(temperature)) return DARE_ERR_RANGE;
    m->sample_temperature = temperature;
    m->sample_seed = seed;
    return dare::launch_kernel(set_word_kernel, dim3(1), 1, 0, static_cast<cudaStream_t>(stream), 1, m->step_counter, first_step);
}

int dare_linear(dare_ctx* ctx, int epilogue, const void* a, int M, int K, const void* w, const void* w2, int N, void* out,
                const void* residual, void* stream) {
    if (!ctx || !a || !w || !out) return DARE_ERR_NULL;
    if (int rc = dare::check_current_device(ctx)) return rc;
    if (epilogue == DARE_LINEAR_SWIGLU && !w2) return DARE_ERR_NULL;
    if (epilogue == DARE_LINEAR_RESIDUAL && !residual) return DARE_ERR_NULL;
    if (epilogue < DARE_LINEAR_STORE || epilogue > DARE_LINEAR_SWIGLU) return DARE_ERR_RANGE;
    const uintptr_t bits = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(w2) |
                           reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(residual);
    if (bits & 15u) return DARE_ERR_ALIGN;
    return dare::launch_gemm(ctx, epilogue, a, M, K, w, w2, N, out, residual, N, static_cast<cudaStream_t>(stream));
}

int dare_linear_plan(dare_ctx* ctx, int epilogue, int M, int K, int N, int* plan_out) {
    if (!ctx || !plan_out) return DARE_ERR_NULL;
    if (M < 1 || N < 8 || K < 8 || (N % 8) || (K % 8)) return DARE_ERR_SHAPE;
    if (epilogue < DARE_LINEAR_STORE || epilogue > DARE_LINEAR_SWIGLU) return DARE_ERR_RANGE;
    return dare::gemm_plan_describe(ctx, epilogue, M, N, K, plan_out);
}

int dare_rmsnorm(dare_ctx* ctx, const void* x, int n_rows, int D, float eps, void* y, void* stream) {
    if (!ctx || !x || !y) return DARE_ERR_NULL;
    if (int rc = dare::check_current_device(ctx)) return rc;
    if (n_rows < 1 || D < 8 || D % 8) return DARE_ERR_SHAPE;
    if (!(eps >= 0.f)) return DARE_ERR_RANGE;
    if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15u) return DARE_ERR_ALIGN;
    return dare::launch_rmsnorm(x, D, n_rows, eps, y, ctx->sm_count, static_cast<cudaStream_t>(stream));
}

int dare_rope_kv_write(dare_model* m, const void* qkv, int B, int length, int start, void* q_out, void* k_cache,
                       void* v_cache, int cache_cap, void* stream) {
    if (!m || !qkv || !q_out || !k_cache || !v_cache) return DARE_ERR_NULL;
    if (int rc = dare::check_current_device(m->ctx)) return rc;
    if (B < 1 || length < 1) return DARE_ERR_SHAPE;
    if (start < 0 || static_cast<long long>(start) + length > cache_cap || cache_cap > m->desc.max_positions)
        return DARE_ERR_RANGE;
    const uintptr_t bits = reinterpret_cast<uintptr_t>(qkv) | reinterpret_cast<uintptr_t>(q_out) |
                           reinterpret_cast<uintptr_t>(k_cache) | reinterpret_cast<uintptr_t>(v_cache);
    if (bits & 15u) return DARE_ERR_ALIGN;
    return dare::launch_rope_kv_write(qkv, B * length, m->desc.n_q_heads, m->desc.n_kv_heads, m->desc.head_dim, start,
                                      length, m->rope_cs, q_out, k_cache, v_cache, cache_cap, m->ctx->sm_count,
                                      static_cast<cudaStream_t>(stream));
}

int dare_model_forward_window(dare_model* m, const int32_t* tokens, int B, int64_t row_stride, int start, int length,
                              int kv_len, void* k_cache, void* v_cache, int cache_cap, void* hidden_out, void* stream) {
    int rc = check_rows(m, tokens, B, row_stride, start, length, kv_len, k_cache, v_cache, cache_cap);
    if (rc != DARE_OK) return rc;
    return forward_rows(m, tokens, B, row_stride, start, length, kv_len, k_cache, v_cache, cache_cap, hidden_out,
                        static_cast<cudaStream_t>(stream));
}

int dare_model_forward(dare_model* m, const int32_t* tokens, int B, int64_t row_stride, int start, int length,
                       void* k_cache, void* v_cache, int cache_cap, void* hidden_out, void* stream) {
    return dare_model_forward_window(m, tokens, B, row_stride, start, length, start + length, k_cache, v_cache,
                                     cache_cap, hidden_out, stream);
}

int dare_model_step_window(dare_model* m, int32_t* tokens, int B, int64_t row_stride, int block_start, int L, int kv_len,
                           void* k_cache, void* v_cache, int cache_cap, int mode, float threshold, int k, int32_t* pred,
                           float* conf, int32_t* n_committed, int32_t* n_remaining, void* stream) {
    int rc = check_rows(m, tokens, B, row_stride, block_start, L, kv_len, k_cache, v_cache, cache_cap);
    if (rc == DARE_OK) rc = check_step(m, B, L, mode, threshold, k, pred, conf);
    if (rc != DARE_OK) return rc;
    return step_rows(m, tokens, B, row_stride, block_start, L, kv_len, k_cache, v_cache, cache_cap, mode, threshold, k,
                     pred, conf, n_committed, n_remaining, static_cast<cudaStream_t>(stream));
}

int dare_model_step(dare_model* m, int32_t* tokens, int B, int64_t row_stride, int block_start, int L, void* k_cache,
                    void* v_cache, int cache_cap, int mode, float threshold, int k, int32_t* pred, float* conf,
                    int32_t* n_committed, int32_t* n_remaining, void* stream) {
    return dare_model_step_window(m, tokens, B, row_stride, block_start, L, block_start + L, k_cache, v_cache, cache_cap,
                                  mode, threshold, k, pred, conf, n_committed, n_remaining, stream);
}

}  // extern "C"

namespace {

// Waits until step `slot` has left its counts; *done: no rollout has a mask left.  The kernel that takes the decisions
// writes them straight into page-locked memory (an event behind the step, let alone a copy, would stand between the step
// and the next one, which is already enqueued).
int read_counts(const dare_model* m, int slot, int B, cudaStream_t s, bool* done) {
    const volatile int32_t* c = m->host_counts + slot * m->max_batch;
    *done = true;
    uint32_t spins = 0;
    for (int r = 0; r < B; ++r) {
        while (c[r] < 0) {
            if ((++spins & 0xffff) == 0) {      // now and then: has the stream failed, or ended without writing them?
                const cudaError_t q = cudaStreamQuery(s);
                if (q != cudaErrorNotReady && (q != cudaSuccess || c[r] < 0)) return DARE_ERR_CUDA;
            }
        }
        *done = *done && c[r] == 0;
    }
    return DARE_OK;
}

// All denoising steps of one block.  The host enqueues a step (about thirty launches, 2 us each) while the one before it
// runs; as a CUDA graph per block it cost the GPU 17 us between replays and, on a small model, the capture and the
// instantiation besides (44 us per step of 110 us).
//
// A step whose block holds no mask any more does exactly what the refresh forward of the prefix-cache loop
// must do (the LM head finds no live row, the selection changes nothing, the stack rewrites the block's K/V
// from the committed tokens).  So step t + 1 is enqueued before step t's counts are read: when step t turns
// out to have finished the block, step t + 1 was the refresh, and the GPU never waits for the host.
//
// refresh = false: something else is about to rewrite the block's K/V (the dual-cache loop's forward of the whole
// sequence).  With top-k commits, ceil(L / k) steps leave no mask whatever their counts say, so the extra step is not
// enqueued: 13 instead of 14 steps of 107 us for two blocks of 16 with k = 3 (24 small kernels each).  At one step per
// block the counts that pace the host would never be read: the extra step stays.
int run_block(dare_model* m, int32_t* tokens, int B, int64_t row_stride, int start, int L, int kv_len, void* k_cache,
              void* v_cache, int cap, int mode, float threshold, int k, int32_t* pred, float* conf, int32_t* n_remaining,
              cudaStream_t s, uint32_t* step_no, bool refresh, int* steps_taken) {
    const int enough = mode == DARE_SELECT_TOPK && k < L ? (L + k - 1) / k : 0;
    for (int issued = 0;; ++issued) {
        if (issued > L + 1) return DARE_ERR_CUDA;            // cannot happen: every step commits a token per row
        if (!refresh && enough > 0 && issued == enough) {
            *steps_taken = issued;
            return DARE_OK;
        }
        // The slots go round over the whole loop, not per block: when a slot comes round again, a later step than the one
        // that used it has been read, so nothing writes to it any more.
        const uint32_t n = (*step_no)++;
        int32_t* slot = m->host_counts + (n % COUNT_SLOTS) * m->max_batch;
        for (int r = 0; r < B; ++r) slot[r] = -1;
        int rc = step_rows(m, tokens, B, row_stride, start, L, kv_len, k_cache, v_cache, cap, mode, threshold, k, pred, conf,
                           nullptr, n_remaining, s, slot);
        if (rc != DARE_OK) return rc;
        if (issued == 0) continue;
        bool done = false;
        rc = read_counts(m, (n - 1) % COUNT_SLOTS, B, s, &done);
        if (rc != DARE_OK) return rc;
        if (done) {      // steps 0 .. issued - 1 denoised; the last one issued finds no mask
            *steps_taken = issued;
            return DARE_OK;
        }
    }
}

}  // namespace

extern "C" {

int dare_generate(dare_model* m, int32_t* tokens, int B, int64_t row_stride, int prompt_len, int gen_len, int L,
                  void* k_cache, void* v_cache, int cache_cap, int mode, float threshold, int k, int32_t* pred,
                  float* conf, int32_t* n_remaining, int32_t* steps_per_block, void* stream) {
    if (!n_remaining) return DARE_ERR_NULL;
    if (gen_len < 1 || L < 1 || gen_len % L != 0) return DARE_ERR_SHAPE;
    int rc = check_rows(m, tokens, B, row_stride, 0, prompt_len, prompt_len, k_cache, v_cache, cache_cap);
    if (rc == DARE_OK)
        rc = check_rows(m, tokens, B, row_stride, prompt_len + gen_len - L, L, prompt_len + gen_len, k_cache, v_cache,
                        cache_cap);
    if (rc == DARE_OK) rc = check_step(m, B, L, mode, threshold, k, pred, conf);
    if (rc != DARE_OK) return rc;
    cudaStream_t user = static_cast<cudaStream_t>(stream);
    rc = forward_rows(m, tokens, B, row_stride, 0, prompt_len, prompt_len, k_cache, v_cache, cache_cap, nullptr, user);
    uint32_t step_no = 0;
    for (int b = 0; b < gen_len / L && rc == DARE_OK; ++b) {
        const int start = prompt_len + b * L;
        int taken = -1;
        if (m->sample_temperature > 0.f) {     // step n of block b draws with the counter (b << 16) + n
            rc = dare::launch_kernel(set_word_kernel, dim3(1), 1, 0, user, 1, m->step_counter, static_cast<uint32_t>(b) << 16);
            if (rc != DARE_OK) break;
        }
        rc = run_block(m, tokens, B, row_stride, start, L, start + L, k_cache, v_cache, cache_cap, mode, threshold, k,
                       pred, conf, n_remaining, user, &step_no, true, &taken);
        if (rc == DARE_OK && steps_per_block) steps_per_block[b] = taken;
    }
    const bool synced = cudaStreamSynchronize(user) == cudaSuccess;      // (also after an error: the counts' slots are still in use)
    return rc != DARE_OK ? rc : synced ? DARE_OK : DARE_ERR_CUDA;
}

int dare_generate_dual(dare_model* m, int32_t* tokens, int B, int64_t row_stride, int prompt_len, int gen_len, int L,
                       void* k_cache, void* v_cache, int cache_cap, int mode, float threshold, int k, int32_t* pred,
                       float* conf, int32_t* n_remaining, int32_t* steps_per_block, void* stream) {
    if (!n_remaining) return DARE_ERR_NULL;
    if (prompt_len < 0 || gen_len < 1 || L < 1 || gen_len % L != 0) return DARE_ERR_SHAPE;
    const int T = prompt_len + gen_len;
    int rc = check_rows(m, tokens, B, row_stride, 0, T, T, k_cache, v_cache, cache_cap);   // the refresh: all rows
    if (rc == DARE_OK) rc = check_step(m, B, L, mode, threshold, k, pred, conf);
    if (rc != DARE_OK) return rc;
    cudaStream_t user = static_cast<cudaStream_t>(stream);
    uint32_t step_no = 0;
    for (int b = 0; b < gen_len / L && rc == DARE_OK; ++b) {
        const int start = prompt_len + b * L;
        rc = forward_rows(m, tokens, B, row_stride, 0, T, T, k_cache, v_cache, cache_cap, nullptr, user);
        if (rc != DARE_OK) break;
        int taken = -1;
        if (m->sample_temperature > 0.f) {
            rc = dare::launch_kernel(set_word_kernel, dim3(1), 1, 0, user, 1, m->step_counter, static_cast<uint32_t>(b) << 16);
            if (rc != DARE_OK) break;
        }
        rc = run_block(m, tokens, B, row_stride, start, L, T, k_cache, v_cache, cache_cap, mode, threshold, k, pred, conf,
                       n_remaining, user, &step_no, b + 1 == gen_len / L, &taken);
        if (rc == DARE_OK && steps_per_block) steps_per_block[b] = taken;
    }
    const bool synced = cudaStreamSynchronize(user) == cudaSuccess;      // (also after an error: the counts' slots are still in use)
    return rc != DARE_OK ? rc : synced ? DARE_OK : DARE_ERR_CUDA;
}

}  // extern "C"
