"""GPU tests of kernel variants that the dispatch picks by size, at the sizes where they begin and end."""
import numpy as np
import pytest
import torch

from oracle import dare_sampling_oracle as SO
from paper_2604_04215_b200 import binding as dare
from paper_2604_04215_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = dare.Context(0)
    yield c
    c.close()


def _small_model(ctx, Hq, Hkv, d, rows, batch, positions, hidden=256, ffn=256, vocab=512):
    n = (Hq + 2 * Hkv) * d
    w = {"wqkv": I.normal_bf16(7, 1, (n, hidden), 0.05), "wo": I.normal_bf16(7, 2, (hidden, Hq * d), 0.05),
         "wg": I.normal_bf16(7, 3, (ffn, hidden), 0.05), "wu": I.normal_bf16(7, 4, (ffn, hidden), 0.05),
         "wd": I.normal_bf16(7, 5, (hidden, ffn), 0.05)}
    emb, head = I.normal_bf16(7, 6, (vocab, hidden)), I.normal_bf16(7, 8, (vocab, hidden))
    return dare.Model(ctx, n_layers=1, hidden=hidden, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d, ffn=ffn, vocab=vocab,
                      mask_id=vocab - 1, embedding=emb.cuda(), layers=[{k: v.cuda() for k, v in w.items()}],
                      lm_head=head.cuda(), max_positions=positions, max_rows=rows, max_batch=batch)


# Enough rows for two 256 x 256 tiles of the QKV projection per CTA pair (148 tiles): there rotary embedding rides on
# the projection.  Row counts that are no multiple of a tile, head counts that leave the last column tile part full.
@pytest.mark.parametrize("Hq,Hkv,d,B,length", [(4, 2, 64, 37, 513), (4, 2, 128, 19, 499), (3, 1, 128, 40, 331), (2, 1, 64, 75, 260)])
def test_rope_in_the_projection_matches_the_separate_kernel(ctx, Hq, Hkv, d, B, length):
    start, cap = 3, length + 5
    model = _small_model(ctx, Hq, Hkv, d, B * length, B, cap)
    tok = I.uniform_int(7, 9, (B, cap), 0, 510).cuda()
    hid = torch.empty(B * length, 256, dtype=torch.bfloat16, device="cuda")
    caches = model.new_cache(B, cap)
    dare.dare_model_forward(model, tok, start, length, *caches, hid)
    # the same rollouts a few at a time: too few rows for that
    one = [torch.zeros_like(c) for c in caches]
    hid1 = torch.empty_like(hid)
    for b in range(0, B, 3):
        nb = min(3, B - b)
        part = [c[:, b:b + nb].contiguous() for c in one]
        dare.dare_model_forward(model, tok[b:b + nb].contiguous(), start, length, *part, hid1[b * length:(b + nb) * length])
        for c, p in zip(one, part):
            c[:, b:b + nb] = p
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    # Both round q, k and v to bf16 before the rotation and once after it; the fp32 sums in front may differ in their
    # last bits (another tile shape), which can move a value by one bf16 step (up to 2^-7 of it) before and one after: 2^-6 of
    # the larger of the two channels that turn together, and v by one step, 2^-7.
    k, k1, v, v1 = (t.float() for t in (caches[0], one[0], caches[1], one[1]))
    pair = torch.maximum(k1[..., :d // 2].abs(), k1[..., d // 2:].abs())
    assert ((k - k1).abs() <= 2.0 ** -6 * torch.cat([pair, pair], -1) + 1e-6).all()
    assert ((v - v1).abs() <= 2.0 ** -7 * v1.abs() + 1e-6).all()
    for c in caches:                     # nothing outside the written positions
        assert (c[:, :, :, :start] == 0).all() and (c[:, :, :, start + length:] == 0).all()
    rel = ((hid.float() - hid1.float()).norm() / hid1.float().norm()).item()
    assert rel <= 5e-3                   # one layer: the bar of the stack tests per layer
    model.close()


# RMSNorm: a row per CTA, 4096 values in registers, longer rows read twice.
@pytest.mark.parametrize("rows,D", [(1, 8), (5, 1032), (3, 4088), (3, 4096), (2, 4104), (2, 12296)])
def test_rmsnorm_row_lengths(ctx, rows, D):
    x = I.normal_bf16(3, I.TID_X, (rows, D), 3.0)
    y = dare.dare_rmsnorm(ctx, x.cuda(), 1e-5).float().cpu().double().numpy()
    f = x.double().numpy()
    ref = f / np.sqrt((f * f).mean(1, keepdims=True) + 1e-5)
    assert (np.abs(y - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-6).all()      # one rounding to bf16, fp32 sums


# ... and a warp per row for many short ones: the edges of that rule and of the row lengths a warp holds.  A row's result is
# the same, bit for bit, whichever kernel takes it.
@pytest.mark.parametrize("rows,D", [(1, 256), (9, 264), (31, 504), (7, 512), (512, 520), (513, 520), (514, 1024), (4095, 1032), (4096, 1032),
                                    (4097, 2048), (4096, 2056)])
def test_rmsnorm_of_many_short_rows(ctx, rows, D):
    x = I.normal_bf16(3, I.TID_X, (rows, D), 3.0)
    y = dare.dare_rmsnorm(ctx, x.cuda(), 1e-5)
    f = x.double()
    ref = f / (f.pow(2).mean(1, keepdim=True) + 1e-5).sqrt()
    assert ((y.cpu().double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-6).all()      # one rounding to bf16, fp32 sums
    few = torch.cat([dare.dare_rmsnorm(ctx, x[i:i + 300].cuda(), 1e-5) for i in range(0, rows, 300)])
    assert torch.equal(few, y)


def _us(call, n=40):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(5):
        torch.cuda.synchronize()
        a.record()
        for _ in range(n):
            call()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


def test_many_short_rows_cost_their_bytes(ctx):
    """A CTA per row would take 68 us to start here; a copy of the same bytes, and a warp per row, take about 10."""
    x = torch.randn(65536, 256, device="cuda").bfloat16()
    y = torch.empty_like(x)
    assert _device_us(lambda: dare.dare_rmsnorm(ctx, x, 1e-5, y)) <= 2.5 * max(10.0, _device_us(lambda: y.copy_(x)))


# Projections with so many rows that the tiles are taken in groups of row pairs (32 MB of A per group): one group and a
# row more than that, an uneven last group, K so long that a group is one row pair.
@pytest.mark.parametrize("M,K,N", [(2048, 8192, 264), (2049, 8192, 264), (5000, 8200, 520), (600, 65544, 72)])
def test_linear_in_row_groups(ctx, M, K, N):
    a, w = I.normal_bf16(5, I.TID_X, (M, K)).cuda(), I.normal_bf16(5, I.TID_W, (N, K), 0.05).cuda()
    out = dare.dare_linear(ctx, dare.LINEAR_STORE, a, w).double()
    ref = a.double() @ w.double().T
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    # one rounding to bf16 (2^-8) and fp32 sums of K products: K * 2^-24 of the sum of their magnitudes at most
    bound = 2.0 ** -8 * ref.abs() + K * 2.0 ** -24 * (a.double().abs() @ w.double().abs().T)
    assert ((out - ref).abs() <= bound).all()


# The sampled head takes the same paths as the greedy one: swapped operands up to 256 rows (five ring slots above 192)
# and for rows that cut into chunks of 208 to 240, row-major pairs for an even number of 128-row tiles, pairs and single
# CTAs for an odd one.  V leaves the last vocabulary tile part full.
@pytest.mark.parametrize("M", [1, 16, 17, 33, 192, 193, 255, 256, 257, 300, 400, 420, 512, 520, 900])
@pytest.mark.parametrize("T", [1.0, 0.35])
def test_sampled_head_on_every_path(ctx, M, T):
    D, V, mu, seed, step = 72, 1300, 1290, 0x9876543210 + M, 5
    x, w = I.normal_bf16(M, I.TID_X, (M, D)), I.normal_bf16(3, I.TID_W, (V, D), 0.2)
    ref = SO.lmhead_sample(x.double().numpy(), w.double().numpy(), None, mu, True, T, seed, step)
    pred, conf = dare.dare_lmhead_sample(ctx, x.cuda(), w.cuda(), None, mu, True, T, seed, step)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    pred, conf = pred.cpu().numpy(), conf.cpu().double().numpy()
    # scores are fp32 (sums of 72 products of magnitude ~2: 1e-5) over T plus noise of one ulp: well inside 1e-3
    sure = ref["gap_y"] > 1e-3
    assert (pred[sure] == ref["pred"][sure]).all() and sure.mean() > 0.9
    same = pred == ref["pred"]
    assert np.abs(np.log(conf[same]) - ref["logconf"][same]).max() <= 1e-3


# The test that spares most logits their logarithms must not lose the best one: logits from flat (the noise decides) to steep
# (the logit decides), several tiles per warp, and rows whose best comes early, late or from another warp.
@pytest.mark.parametrize("M", [33, 160, 300, 520])
@pytest.mark.parametrize("sigma,T", [(0.01, 1.0), (0.3, 5.0), (1.0, 0.05), (4.0, 1.0), (4.0, 40.0)])
def test_sampled_head_evaluates_the_best(ctx, M, sigma, T):
    D, V, mu, seed, step = 64, 20_000, 0, 0x1234567890 + M, 9
    x, w = I.normal_bf16(M, I.TID_X, (M, D)), I.normal_bf16(4, I.TID_W, (V, D), sigma / 8)
    ref = SO.lmhead_sample(x.double().numpy(), w.double().numpy(), None, mu, True, T, seed, step)
    pred, _ = dare.dare_lmhead_sample(ctx, x.cuda(), w.cuda(), None, mu, True, T, seed, step)
    torch.cuda.synchronize()
    # scores: fp32 sums of 64 products of magnitude sigma / 8 * 3 (64 * 2^-24 * 64 * that: 1e-4 sigma) over T, noise to an ulp of 20
    sure = ref["gap_y"] > 2e-4 * sigma / T + 1e-5
    assert (pred.cpu().numpy()[sure] == ref["pred"][sure]).all() and sure.mean() > 0.9


# Where a warp sees one or two groups of 32 logits of each row, nothing of a row is known yet when the first group comes: the
# lanes then have to start with their best candidate, or nearly all 32 are evaluated (58 to 95 us here, the greedy head 12 to 18).
@pytest.mark.parametrize("M,D,V", [(128, 256, 4096), (256, 256, 4096), (300, 512, 2048), (640, 256, 2048)])
def test_sampled_head_on_a_small_vocabulary_costs_little_more(ctx, M, D, V):
    x, w = torch.randn(M, D, device="cuda").bfloat16(), torch.randn(V, D, device="cuda").mul(0.02).bfloat16()
    pred, conf = torch.empty(M, dtype=torch.int32, device="cuda"), torch.empty(M, device="cuda")
    greedy = _device_us(lambda: dare.dare_lmhead_confidence(ctx, x, w, None, 3, True, pred, conf))
    assert _device_us(lambda: dare.dare_lmhead_sample(ctx, x, w, None, 3, True, 1.0, 7, 1, pred, conf)) <= 2.5 * greedy


def test_sampled_head_has_a_pair_per_vocabulary_tile(ctx):
    """128 rows are one row tile, 160 two: the launch of the former must not be the smaller one (24 against 19 us it was)."""
    D, V = 256, 4096
    w, us = torch.randn(V, D, device="cuda").mul(0.02).bfloat16(), []
    for M in (128, 160):
        x = torch.randn(M, D, device="cuda").bfloat16()
        pred, conf = torch.empty(M, dtype=torch.int32, device="cuda"), torch.empty(M, device="cuda")
        us.append(_device_us(lambda: dare.dare_lmhead_sample(ctx, x, w, None, 3, True, 1.0, 7, 1, pred, conf)))
    assert us[0] <= 1.1 * us[1]


# Scores that are infinite tie, and the lowest id wins a tie, wherever the columns lie: in one thread's 32 columns, in two
# warps' or two tiles' columns.  (z / T of the columns named is 5e38 and more, beyond fp32; of the others -1e38.)
@pytest.mark.parametrize("M", [1, 40, 300, 420, 700])
@pytest.mark.parametrize("cols", [(3, 9), (3, 40), (7, 64, 999), (100, 101, 130), (515, 1290), (1291,)])
def test_sampled_head_ties_at_infinite_scores(ctx, M, cols):
    D, V, mu, T = 16, 1300, 2, 1e-38
    x, w = torch.zeros(M, D), torch.zeros(V, D)
    x[:, 0], w[:, 0] = 1.0, -1.0
    for n, c in enumerate(cols):
        w[c, 0] = 5.0 + 2 * n                     # (the higher ids have the larger logits)
    pred, conf = dare.dare_lmhead_sample(ctx, x.bfloat16().cuda(), w.bfloat16().cuda(), None, mu, True, T, 11, 3)
    assert (pred.cpu() == cols[0]).all()
    z = w[:, 0].double()
    z[mu] = -float("inf")
    assert torch.allclose(conf.cpu().double(), torch.softmax(z, 0)[cols[0]].expand(M), rtol=1e-5)


def test_sampled_head_with_a_workspace_for_one_partial_per_tile():
    """The swapped path wants room for two partials per vocabulary tile; a context without it takes the other path."""
    M, D, V, mu = 40, 64, 2000, 1999
    need = 20 * M * ((V + 255) // 256)
    c = dare.Context(0, need)
    x, w = I.normal_bf16(1, I.TID_X, (M, D)), I.normal_bf16(2, I.TID_W, (V, D), 0.2)
    ref = SO.lmhead_sample(x.double().numpy(), w.double().numpy(), None, mu, True, 1.0, 4, 1)
    pred, conf = dare.dare_lmhead_sample(c, x.cuda(), w.cuda(), None, mu, True, 1.0, 4, 1)
    torch.cuda.synchronize()
    sure = ref["gap_y"] > 1e-3
    assert (pred.cpu().numpy()[sure] == ref["pred"][sure]).all()
    c.close()


# A step is a chain of kernels in which each may start before its predecessor ends.  With a K/V split the attention's
# partials lie behind the head's scratch; a workspace that does not hold both makes the halves run in sequence.  Steps
# follow one another closely, on inputs that ordinary kernels overwrite in between: each must equal the parts run alone.
@pytest.mark.parametrize("B,L,Hq,Hkv,P,workspace", [(1, 32, 4, 4, 1500, 0), (1, 32, 4, 4, 1500, 800000), (2, 40, 4, 2, 700, 0),
                                                    (40, 4, 8, 8, 300, 0), (3, 32, 28, 4, 500, 0)])
def test_steps_back_to_back_equal_their_parts(ctx, B, L, Hq, Hkv, P, workspace):
    d, D, V, mu = 128, 512, 3000, 2990
    c = dare.Context(0, workspace) if workspace else ctx
    mode, k, n_steps = dare.SELECT_TOPK, 2, 6
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)  # noqa: E731
    w = rnd(V, D) * 0.05
    k_pre, v_pre, plen = rnd(B, Hkv, P, d), rnd(B, Hkv, P, d), torch.full((B,), P - 3, dtype=torch.int32, device="cuda")
    acts = [(rnd(B, L, Hq, d), rnd(B, Hkv, L, d), rnd(B, Hkv, L, d), rnd(B * L, D)) for _ in range(n_steps)]
    bufs = [torch.empty_like(t) for t in acts[0]]
    new = lambda n, t: torch.zeros(n, dtype=t, device="cuda")  # noqa: E731
    tok = torch.full((B, P + L), mu, dtype=torch.int32, device="cuda")
    ref_tok = tok.clone()
    got = []
    for a in acts:
        for dst, src in zip(bufs, a):
            dst.copy_(src)
        out, pred, conf, nc, nr = torch.empty_like(a[0]), new(B * L, torch.int32), new(B * L, torch.float32), new(B, torch.int32), new(B, torch.int32)
        dare.dare_denoise_block(c, bufs[0], k_pre, v_pre, plen, bufs[1], bufs[2], None, None, None, out, None, bufs[3], w, mu,
                                True, tok, P, mode, 0.0, k, pred, conf, nc, nr)
        got.append((out, pred, conf, nc, nr))
    for a, (out, pred, conf, nc, nr) in zip(acts, got):
        ref_out = dare.dare_attn_block(ctx, a[0], k_pre, v_pre, plen, a[1], a[2])
        p2, c2 = dare.dare_lmhead_confidence(ctx, a[3], w, ref_tok[:, P:].contiguous().view(-1), mu, True)
        nc2, nr2 = new(B, torch.int32), new(B, torch.int32)
        dare.dare_unmask_select(ctx, ref_tok, P, L, p2, c2, mu, mode, 0.0, k, nc2, nr2)
        torch.cuda.synchronize()
        for x, y in ((out, ref_out), (pred, p2), (conf, c2), (nc, nc2), (nr, nr2)):
            assert torch.equal(x, y)
    assert torch.equal(tok, ref_tok)
    assert c.device_status() == 0
    if workspace:
        c.close()


# SwiGLU in two rounds of tiles only where they are 208 columns or wider: one round of 352 for gate and up of 256 rows (two of 176
# take 5 to 9 % more), two of 208 and of 256 where one would be 416 or 512.
@pytest.mark.parametrize("M,K,N,w_rows", [(256, 4096, 12288, 352), (768, 12288, 4096, 352), (256, 4096, 14336, 208), (256, 3584, 18944, 256)])
def test_swiglu_tile_width(ctx, M, K, N, w_rows):
    plan = dare.dare_linear_plan(ctx, dare.LINEAR_SWIGLU, M, K, N)
    if plan["resident_clusters"] != 74:
        pytest.skip("the widths are those of 148 SMs")
    assert plan["w_rows"] == w_rows


# Projections of up to 128 rows: one to eight K slices (a cluster), ragged last K block, last W tile part full, every row
# padding; all epilogues.
@pytest.mark.parametrize("M", [1, 15, 16, 17, 47, 96, 127, 128])
@pytest.mark.parametrize("K,N", [(8, 8), (72, 264), (520, 1000), (4096, 136), (1280, 512), (256, 40000)])
def test_linear_of_few_rows(ctx, M, K, N):
    a, w = I.normal_bf16(M, I.TID_X, (M, K)).cuda(), I.normal_bf16(5, I.TID_W, (N, K), 0.05).cuda()
    w2, r = I.normal_bf16(6, I.TID_Q, (N, K), 0.05).cuda(), I.normal_bf16(7, I.TID_Q, (M, N)).cuda()
    store = dare.dare_linear(ctx, dare.LINEAR_STORE, a, w).double()
    resid = dare.dare_linear(ctx, dare.LINEAR_RESIDUAL, a, w, residual=r).double()
    swiglu = dare.dare_linear(ctx, dare.LINEAR_SWIGLU, a, w, w2=w2).double()
    ref, up = a.double() @ w.double().T, a.double() @ w2.double().T
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    # one rounding to bf16 (2^-8) and fp32 sums of K products: K * 2^-24 of the sum of their magnitudes at most
    acc = K * 2.0 ** -24 * (a.double().abs() @ w.double().abs().T)
    acc2 = K * 2.0 ** -24 * (a.double().abs() @ w2.double().abs().T)
    assert ((store - ref).abs() <= 2.0 ** -8 * ref.abs() + acc).all()
    want = ref + r.double()
    assert ((resid - want).abs() <= 2.0 ** -8 * want.abs() + acc).all()
    want = ref * torch.sigmoid(ref) * up                 # |silu'| < 1.1; exp and division to a few ulp
    assert ((swiglu - want).abs() <= 2.0 ** -7.9 * want.abs() + 1.1 * acc * (up.abs() + acc2) + acc2 * ref.abs() + 1e-6).all()


def _device_us(call, n=20):
    """Per call, replayed from a CUDA graph: without the host's share."""
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(n):
            call()
    us = _us(graph.replay, 5) / n
    del graph
    return us


# The way from the accumulator to the output: 128 rows cost 3.5 times what 16 did (10.8 against 3.1 us) when every row's owner was
# divided out and every item's loads were waited for; now 1.9 times.
@pytest.mark.parametrize("epilogue", [dare.LINEAR_STORE, dare.LINEAR_RESIDUAL])
def test_linear_of_few_rows_costs_little_per_row(ctx, epilogue):
    w, us = torch.randn(64, 64, device="cuda").bfloat16(), []
    for M in (16, 128):
        a, r = torch.randn(2, M, 64, device="cuda").bfloat16()
        out = torch.empty_like(r)
        us.append(_device_us(lambda: dare.dare_linear(ctx, epilogue, a, w, residual=r if epilogue else None, out=out)))
    assert us[1] <= 2.6 * us[0]


@pytest.mark.parametrize("Hq,Hkv,d,B,length", [(4, 2, 64, 3, 16), (3, 1, 128, 1, 127), (5, 1, 64, 16, 8), (4, 4, 128, 2, 1)])
def test_rope_in_a_projection_of_few_rows(ctx, Hq, Hkv, d, B, length):
    start, cap = 3, length + 5
    model = _small_model(ctx, Hq, Hkv, d, B * length, B, cap)
    tok = I.uniform_int(7, 9, (B, cap), 0, 510).cuda()
    caches = model.new_cache(B, cap)
    dare.dare_model_forward(model, tok, start, length, *caches)
    # the same projection and the rotation as separate calls
    emb, layers, _ = model._keep
    x = emb[tok[:, start:start + length].reshape(-1).long()].contiguous()
    qkv = dare.dare_linear(ctx, dare.LINEAR_STORE, dare.dare_rmsnorm(ctx, x, 1e-5), layers[0]["wqkv"])
    kc, vc = torch.zeros_like(caches[0]), torch.zeros_like(caches[1])
    q = torch.empty(B * length, Hq, d, dtype=torch.bfloat16, device="cuda")
    dare.dare_rope_kv_write(model, qkv, B, length, start, q, kc[0], vc[0])
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    # the same sums, the same rounding before the rotation; a multiply-add may be contracted differently behind it
    assert torch.equal(caches[1], vc)
    assert ((caches[0].float() - kc.float()).abs() <= 2.0 ** -7 * kc.float().abs() + 1e-6).all()
    model.close()


# Up to 128 rows the head evaluates committed rows too and answers them in its last kernel: the largest such launch and the
# next one, sampled and greedy, with and without the selection on the last kernel, no row and every row masked.
@pytest.mark.parametrize("B,L", [(1, 1), (4, 32), (3, 43), (2, 64)])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
def test_head_with_committed_rows(ctx, B, L, share):
    D, V, mu, M = 64, 1300, 7, B * L
    x, w = I.normal_bf16(M, I.TID_X, (M, D)).cuda(), I.normal_bf16(3, I.TID_W, (V, D), 0.2).cuda()
    tok = I.uniform_int(9, M, (B, L + 5), 8, V - 1)
    masked = torch.rand(B, L, generator=torch.Generator().manual_seed(M)) < share
    tok[:, 5:] = torch.where(masked, torch.full_like(tok[:, 5:], mu), tok[:, 5:])
    tok, flat = tok.cuda(), tok[:, 5:].reshape(-1).cuda()
    for temperature in (0.0, 0.7):
        head = (lambda r: dare.dare_lmhead_sample(ctx, x, w, r, mu, True, temperature, 5, 3)) if temperature else \
               (lambda r: dare.dare_lmhead_confidence(ctx, x, w, r, mu, True))
        p_all, c_all = head(None)                          # every row evaluated
        pred, conf = head(flat)
        m = flat == mu
        assert torch.equal(pred, torch.where(m, p_all, flat))
        # (a row's sums are cut up differently with fewer rows: fp32 rounding of sums of 1300 terms)
        assert torch.allclose(conf[m], c_all[m], rtol=1e-5, atol=0) and torch.isneginf(conf[~m]).all()
        # the step on the same rows
        q, kv = torch.randn(B, L, 1, 64, device="cuda").bfloat16(), torch.randn(B, 1, 40 + L, 64, device="cuda").bfloat16()
        t2, out = tok.clone(), torch.empty_like(q)
        p2, c2 = torch.zeros_like(pred), torch.zeros_like(conf)
        nc, nr = torch.zeros(B, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda")
        args = (ctx, q, kv, kv, torch.full((B,), 40, dtype=torch.int32, device="cuda"), None, None, None, None, None, out, None, x, w,
                mu, True)
        tail = (t2, 5, dare.SELECT_TOPK, 0.0, 2, p2, c2, nc, nr)
        if temperature:
            dare.dare_denoise_block_sampled(*args, temperature, 5, 3, *tail)
        else:
            dare.dare_denoise_block(*args, *tail)
        torch.cuda.synchronize()
        assert torch.equal(p2, pred) and torch.equal(c2, conf)
        n = m.view(B, L).sum(1)
        assert torch.equal(nc.long(), n.clamp(max=2)) and torch.equal(nr.long(), n - n.clamp(max=2))
    assert ctx.device_status() == 0


# Blocks of 8, whose selection rides on the head's last kernel, and of 40, where a kernel of its own takes the decisions and
# writes the counts that pace the host.
LOOP_CASES = [(8, 1), (8, 3), (8, 7), (8, 8), (8, 20), (40, 3), (40, 17), (40, 40)]


@pytest.mark.parametrize("L,k", LOOP_CASES)
@pytest.mark.parametrize("mode", [dare.SELECT_TOPK, dare.SELECT_THRESHOLD])
@pytest.mark.parametrize("temperature", [0.0, 0.7])
def test_dual_loop_equals_its_parts(ctx, temperature, mode, L, k):
    _loop_equals_its_parts(ctx, True, temperature, mode, L, k)


@pytest.mark.parametrize("L,k", LOOP_CASES)
@pytest.mark.parametrize("mode", [dare.SELECT_TOPK, dare.SELECT_THRESHOLD])
@pytest.mark.parametrize("temperature", [0.0, 0.7])
def test_prefix_loop_equals_its_parts(ctx, temperature, mode, L, k):
    _loop_equals_its_parts(ctx, False, temperature, mode, L, k)


def _loop_equals_its_parts(ctx, dual, temperature, mode, L, k):
    """Blocks with some tokens given beforehand (one block whole): whatever the loop leaves out or enqueues ahead, the
    tokens, the steps and all K/V that the last forward of each position wrote are those of the calls it is made of."""
    B, P, G = 2, 5, 4 * L if L == 8 else 2 * L
    T = P + G
    model = _small_model(ctx, 4, 2, 64, B * T, B, T)
    mask_id = 511
    g = torch.Generator().manual_seed(5)
    tok0 = torch.randint(0, 500, (B, T), generator=g, dtype=torch.int32)
    given = torch.rand(B, G, generator=g) < 0.3
    given[:, L:2 * L] = True
    tok0[:, P:][~given] = mask_id
    new = lambda: model.new_cache(B, T)
    pred, conf = torch.empty(B * L, dtype=torch.int32, device="cuda"), torch.empty(B * L, device="cuda")
    nr = torch.zeros(B, dtype=torch.int32, device="cuda")

    tok, (kc, vc), want = tok0.cuda(), new(), []
    if not dual:
        dare.dare_model_forward(model, tok, 0, P, kc, vc)
    for block, start in enumerate(range(P, T, L)):
        if dual:
            dare.dare_model_forward_window(model, tok, 0, T, T, kc, vc)
        dare.dare_model_set_sampling(model, temperature, 99, block << 16)
        n, seen = 0, T if dual else start + L
        while n == 0 or int(nr.sum()) > 0:
            dare.dare_model_step_window(model, tok, start, L, seen, kc, vc, mode, 0.9, k, pred, conf, None, nr)
            n += 1
        want.append(n)
        if not dual:
            dare.dare_model_forward(model, tok, start, L, kc, vc)
    if dual:
        dare.dare_model_forward_window(model, tok, T - L, L, T, kc, vc)

    tok2, (kc2, vc2) = tok0.cuda(), new()
    dare.dare_model_set_sampling(model, temperature, 99, 0)
    loop = dare.dare_generate_dual if dual else dare.dare_generate
    steps = loop(model, tok2, P, G, L, kc2, vc2, mode, 0.9, k, pred, conf, nr)
    assert steps == want
    assert torch.equal(tok2, tok) and torch.equal(kc2, kc) and torch.equal(vc2, vc)
    model.close()


# The step's chain of programmatic launches in a CUDA graph: with the row compaction (more than 128 rows), with a selection kernel
# of its own (blocks of more than 32), with a K/V split and its combination, sampled.  Replayed twice, as the eager call.
@pytest.mark.parametrize("B,L,Hq,Hkv,P", [(5, 32, 4, 4, 300), (2, 40, 4, 2, 300), (5, 40, 28, 4, 100), (1, 32, 4, 4, 1500)])
@pytest.mark.parametrize("temperature", [0.0, 0.7])
def test_step_graphs_equal_the_eager_step(ctx, B, L, Hq, Hkv, P, temperature):
    d, D, V, mu = 128, 512, 3000, 2990
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)  # noqa: E731
    w, x, q = rnd(V, D) * 0.05, rnd(B * L, D), rnd(B, L, Hq, d)
    k_pre, v_pre, plen = rnd(B, Hkv, P, d), rnd(B, Hkv, P, d), torch.full((B,), P - 3, dtype=torch.int32, device="cuda")
    kb, vb = rnd(B, Hkv, L, d), rnd(B, Hkv, L, d)
    new = lambda n, t: torch.zeros(n, dtype=t, device="cuda")  # noqa: E731
    tok0 = torch.full((B, P + L), mu, dtype=torch.int32, device="cuda")
    tok0[:, P::3] = 7
    out = torch.zeros_like(q)
    bufs = [tok0.clone(), out, new(B * L, torch.int32), new(B * L, torch.float32), new(B, torch.int32), new(B, torch.int32)]

    def step():
        tok, out, pred, conf, nc, nr = bufs
        args = (ctx, q, k_pre, v_pre, plen, kb, vb, None, None, None, out, None, x, w, mu, True)
        tail = (tok, P, dare.SELECT_TOPK, 0.0, 2, pred, conf, nc, nr)
        if temperature:
            dare.dare_denoise_block_sampled(*args, temperature, 5, 3, *tail)
        else:
            dare.dare_denoise_block(*args, *tail)

    step()
    torch.cuda.synchronize()
    want = [t.clone() for t in bufs]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    for _ in range(2):
        for t in bufs[1:]:
            t.zero_()
        bufs[0].copy_(tok0)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(bufs, want))
    assert int(want[4].sum()) == 2 * B and ctx.device_status() == 0


# 257 to 384 rows on row-major tiles and, with D = 3584 and 57000 entries, in two chunks: up to 320 rows both against each
# vocabulary tile, above one after the other.  The ranges' edges, tiles of fewer than 256 entries, fewer tiles than CTA
# pairs and enough for every accumulator to come round.
@pytest.mark.parametrize("M", [256, 257, 288, 289, 320, 321, 335, 352, 353, 384, 385])
@pytest.mark.parametrize("D,V", [(72, 100), (72, 1300), (72, 100_000), (3584, 57_001)])
def test_greedy_head_on_two_chunks(ctx, M, D, V):
    mu = V - 3
    x, w = I.normal_bf16(M, I.TID_X, (M, D)).cuda(), I.normal_bf16(V, I.TID_W, (V, D), 1.7 / D ** 0.5).cuda()
    pred, conf = dare.dare_lmhead_confidence(ctx, x, w, None, mu, True)
    torch.cuda.synchronize()
    z = x.double() @ w.double().T
    z[:, mu] = -float("inf")
    best = z.max(1).values
    # an fp32 logit of 72 products is off by up to 72 * 2^-24 * sum |x w| (about 10): 5e-5; of 3584, added 16 at a time to partial
    # sums of a few units, by 224 * 2^-22: 6e-5; the exponentials by less
    assert (best - z.gather(1, pred.long()[:, None])[:, 0] <= 1e-4).all()
    want = torch.exp(best - torch.logsumexp(z, 1))
    assert torch.allclose(conf.double(), want, rtol=2e-4, atol=0)
    assert ctx.device_status() == 0


# Two chunks of rows only at D >= 3584 and three vocabulary tiles of 256 per CTA pair (222 on 148 SMs), four for the sampled head:
# both sides of these lines, at the edges of the row ranges.  A row's answer does not depend on the path: the rows a few at
# a time (row_tokens picks them, the generator is keyed by a row's place) give the same tokens.
@pytest.mark.parametrize("D,V", [(3576, 57_000), (3584, 221 * 256), (3584, 221 * 256 + 1), (3584, 295 * 256), (3584, 295 * 256 + 40)])
def test_heads_at_the_edges_of_the_two_chunk_rules(ctx, D, V):
    mu, big = 5, 512
    g = torch.Generator(device="cuda").manual_seed(V)
    w = torch.randn(V, D, generator=g, device="cuda").mul_(0.05).bfloat16()
    x = torch.randn(big, D, generator=g, device="cuda").bfloat16()
    for M in (97, 112, 128, 160, 161, 256, 257, 272, 320, 321, 352, 384, 385, 400, 480):
        for temperature in (0.0, 0.8):
            head = (lambda r: dare.dare_lmhead_sample(ctx, x[:M], w, r, mu, True, temperature, 5, 3)) if temperature else \
                   (lambda r: dare.dare_lmhead_confidence(ctx, x[:M], w, r, mu, True))
            pred, conf = head(None)
            for lo in range(0, M, 90):
                row = torch.full((M,), 7, dtype=torch.int32, device="cuda")
                row[lo:lo + 90] = mu
                p, c = head(row)
                assert torch.equal(p[lo:lo + 90], pred[lo:lo + 90])
                assert torch.allclose(c[lo:lo + 90], conf[lo:lo + 90], rtol=2e-5, atol=0)      # (sums of 57000 exponentials, cut differently)
        z = x[:M].float() @ w.float().T
        z[:, mu] = -float("inf")
        greedy, conf = dare.dare_lmhead_confidence(ctx, x[:M], w, None, mu, True)
        # fp32 sums of 3584 products of size 0.05: 3584 * 2^-24 * 3584 * 0.03 at the worst, far less in fact
        assert (z.max(1).values - z.gather(1, greedy.long()[:, None])[:, 0] <= 1e-3).all()
        assert torch.allclose(conf, torch.softmax(z, 1).max(1).values, rtol=2e-3, atol=0)
    assert ctx.device_status() == 0


# Where little hides the epilogue, 300 and 384 rows run as three row-major tiles, and cost what 512 rows as four do (18 against 12 us
# here in two chunks).
@pytest.mark.parametrize("D,V", [(512, 2048), (64, 1300)])
def test_greedy_head_of_three_tiles_costs_no_more_than_of_four(ctx, D, V):
    w, us = torch.randn(V, D, device="cuda").mul(0.02).bfloat16(), {}
    for M in (300, 384, 512):
        x = torch.randn(M, D, device="cuda").bfloat16()
        pred, conf = torch.empty(M, dtype=torch.int32, device="cuda"), torch.empty(M, device="cuda")
        us[M] = _device_us(lambda: dare.dare_lmhead_confidence(ctx, x, w, None, 3, True, pred, conf))
    assert us[300] <= 1.2 * us[512] and us[384] <= 1.2 * us[512]


# The rotary kernel on its own: heads that leave the last batch of a thread part full, more heads than one pass takes, and
# fewer than the threads of a CTA.
@pytest.mark.parametrize("Hq,Hkv,d", [(1, 1, 64), (72, 24, 128), (65, 13, 64), (33, 33, 128), (31, 31, 64)])
def test_rope_kernel_head_counts(ctx, Hq, Hkv, d):
    B, length, start, cap = 2, 3, 5, 11
    model = _small_model(ctx, Hq, Hkv, d, B * length, B, cap, hidden=64, ffn=64)
    x = I.normal_bf16(Hq, 3, (B, length, Hq + 2 * Hkv, d)).cuda()
    q = torch.empty(B, length, Hq, d, dtype=torch.bfloat16, device="cuda")
    kc, vc = (torch.zeros(1, B, Hkv, cap, d, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    dare.dare_rope_kv_write(model, x.view(B * length, -1), B, length, start, q, kc, vc)
    torch.cuda.synchronize()
    pos = torch.arange(start, start + length, dtype=torch.float64, device="cuda")
    ang = pos[:, None] * 10000.0 ** (-2.0 * torch.arange(d // 2, dtype=torch.float64, device="cuda") / d)
    c, s = ang.cos()[None, :, None], ang.sin()[None, :, None]
    r = x[:, :, :Hq + Hkv].double()
    lo, hi = r[..., :d // 2], r[..., d // 2:]
    want = torch.cat([lo * c - hi * s, hi * c + lo * s], -1)
    bound = (2.0 ** -8 * want.abs() + 2.0 ** -21 * torch.cat([lo.abs() + hi.abs()] * 2, -1))     # bf16 rounding; fp32 inside
    rows = slice(start, start + length)
    assert ((q.double() - want[:, :, :Hq]).abs() <= bound[:, :, :Hq]).all()
    assert ((kc[0, :, :, rows].transpose(1, 2).double() - want[:, :, Hq:]).abs() <= bound[:, :, Hq:]).all()
    assert torch.equal(vc[0, :, :, rows].transpose(1, 2), x[:, :, Hq + Hkv:])
    assert kc[0, :, :, :start].count_nonzero() == 0 and vc[0, :, :, start + length:].count_nonzero() == 0
    model.close()


# Rows with few heads share a CTA of that kernel: a last CTA with one row, threads that are no power of two, v pieces that take
# more than one pass.  Each row as when it is alone.
@pytest.mark.parametrize("Hq,Hkv,d", [(2, 1, 64), (4, 4, 64), (9, 1, 64), (4, 2, 128), (8, 2, 128), (16, 16, 64), (28, 4, 128), (32, 8, 128)])
def test_rope_kernel_rows_that_share_a_cta(ctx, Hq, Hkv, d):
    B, length, start = 33, 9, 2
    model = _small_model(ctx, Hq, Hkv, d, B * length, B, length + start, hidden=64, ffn=64)
    x = I.normal_bf16(Hq, 3, (B * length, (Hq + 2 * Hkv) * d)).cuda()
    new = lambda *s: torch.zeros(*s, dtype=torch.bfloat16, device="cuda")  # noqa: E731
    q, q1 = new(B * length, Hq, d), new(B * length, Hq, d)
    kc, vc, k1, v1 = (new(B, Hkv, length + start, d) for _ in range(4))
    dare.dare_rope_kv_write(model, x, B, length, start, q, kc, vc)
    for b in range(B):
        for i in range(length):
            r, at = b * length + i, start + i
            row = (new(1, Hkv, length + start, d), new(1, Hkv, length + start, d))
            dare.dare_rope_kv_write(model, x[r:r + 1], 1, 1, at, q1[r:r + 1], *row)
            k1[b, :, at], v1[b, :, at] = row[0][0, :, at], row[1][0, :, at]
    torch.cuda.synchronize()
    assert torch.equal(q, q1) and torch.equal(kc, k1) and torch.equal(vc, v1)
    model.close()


def test_rope_kernel_of_few_heads_costs_its_bytes(ctx):
    """A CTA per row would take 48 us here; a copy of the same bytes and rows that share a CTA take about 10."""
    B, length = 64, 512
    model = _small_model(ctx, 2, 1, 64, B * length, B, length, hidden=64, ffn=64)
    x, y = torch.randn(2, B * length, 256, device="cuda").bfloat16()
    q, kc, vc = torch.empty_like(x[:, :128]).contiguous(), *model.new_cache(B, length)
    us = _device_us(lambda: dare.dare_rope_kv_write(model, x, B, length, 0, q, kc, vc))
    assert us <= 2.5 * max(10.0, _device_us(lambda: y.copy_(x)))
    model.close()
