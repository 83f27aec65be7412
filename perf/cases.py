"""The measured work of this framework: what a rollout, scoring or update program has it do, through the public calls
of paper_2604_04215_b200.binding.

Shapes are those of paper_2604_04215_b200.inputs (LLaDA-, Dream- and SDAR-shaped steps, the 4-layer loop and its small
copies); weights, activations and tokens are random, made on the GPU from the seed.  Where a trained model would be
sure of its answer, the inputs are planted so that the path's decisions (argmax, threshold, top-k) have real margins.

A case is one of
    step      denoising steps of one block (dare_denoise_block or its sampled form) from a given state of the block
    generate  the whole block-by-block loop on a stack of layers (dare_generate / dare_generate_dual)
    forward   a forward of the stack over all rows of a batch (dare_model_forward): the prefill
    score     a Monte-Carlo term of the likelihood bound: masking, forward, log-probabilities, bound
    update    log-probabilities of given tokens and their gradient with respect to hidden states and head weights
    varlen    attention over packed sequences of different lengths
"""
import math
import random

import torch

from paper_2604_04215_b200 import binding as dare
from paper_2604_04215_b200 import inputs

BF16, F32, I32 = torch.bfloat16, torch.float32, torch.int32
TOPK, THRESHOLD = dare.SELECT_TOPK, dare.SELECT_THRESHOLD

# (query heads, KV heads, head dim, hidden, vocabulary, mask id) of the step workloads
HEADS = {n: (w.n_q_heads, w.n_kv_heads, w.head_dim, w.hidden, w.vocab, w.mask_id) for n, w in inputs.WORKLOADS.items()}
# share of the planted confidences (uniform in [0.05, 0.999]) that passes a threshold of 0.9, per step
PASS_SHARE = 0.104


def listed():
    return [
        # The smallest real call: eight iterations of one 32-position block on a tiny head; launches and host time.
        dict(name="tiny_block", kind="step", model="tiny", batch=1, block=32, prefix=64, suffix=0, ragged=False,
             inplace=False, masked=1.0, steps=8, topk=0, threshold=0.9, temperature=0.0),
        # The rollout as the paper runs it (two tokens per step): all 16 steps of one block of 16 rollouts.
        dict(name="llada_block", kind="step", model="llada8b", batch=16, block=32, prefix=608, suffix=0, ragged=False,
             inplace=False, masked=1.0, steps=16, topk=2, threshold=0.0, temperature=0.0),
        # One rollout alone, its block half committed: what an interactive user waits for.
        dict(name="llada_one_rollout", kind="step", model="llada8b", batch=1, block=32, prefix=701, suffix=0,
             ragged=False, inplace=True, masked=0.5, steps=4, topk=2, threshold=0.0, temperature=0.0),
        # GQA, the larger batch and vocabulary, threshold commits, a block that has been worked on for a while.
        dict(name="dream_steps", kind="step", model="dream7b", batch=32, block=32, prefix=1248, suffix=0, ragged=False,
             inplace=False, masked=0.7, steps=4, topk=0, threshold=0.9, temperature=0.0),
        # Block diffusion with short blocks and a cached suffix: long caches of uneven lengths, bound by reading them.
        dict(name="dualcache_steps", kind="step", model="dualcache", batch=64, block=4, prefix=4096, suffix=1024,
             ragged=True, inplace=False, masked=1.0, steps=2, topk=0, threshold=0.95, temperature=0.0),
        # Several different rollouts per prompt: the sampled head.
        dict(name="sampled_steps", kind="step", model="llada8b", batch=16, block=32, prefix=512, suffix=0, ragged=False,
             inplace=False, masked=0.8, steps=4, topk=2, threshold=0.0, temperature=1.0),
        # Prefill of 16 prompts of 512 tokens through the 4-layer stack.
        dict(name="prefill", kind="forward", model="llada_loop", batch=16, prompt=512),
        # A whole generation: 16 prompts of 512, 256 tokens in blocks of 32, two tokens per step.
        dict(name="generate", kind="generate", model="llada_loop", batch=16, prompt=512, gen=256, block=32, topk=2,
             dual=False),
        # A small model with the dual cache: forty short kernels a step.
        dict(name="generate_small", kind="generate", model="loop_small_gqa", batch=3, prompt=40, gen=32, block=16,
             topk=3, dual=True),
        # Likelihood of 8 responses of 256 tokens under one draw of the masking process.
        dict(name="score", kind="score", model="llada_loop", batch=8, prompt=250, gen=256),
        # The actor's update of the head on 2048 response tokens.
        dict(name="update", kind="update", model="llada8b", rows=2048),
        # Training-side attention: 32 packed sequences of 256 to 1024 tokens, GQA.
        dict(name="varlen", kind="varlen", model="dream7b", seqs=32, shortest=256, longest=1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "generate", "forward", "score", "update", "varlen"])
    if kind == "step":
        model = rng.choice(["tiny", "llada8b", "dream7b", "dualcache"])
        dual = model == "dualcache"
        topk = rng.choice([0, 2, 3])
        return dict(kind=kind, model=model, batch=_log_int(rng, 1, 64 if dual else 32),
                    block=rng.choice([4, 8]) if dual else rng.choice([16, 20, 32, 32]),
                    prefix=_log_int(rng, 33, 4096 if dual else 1536), suffix=_log_int(rng, 64, 1024) if dual else 0,
                    ragged=rng.random() < 0.5, inplace=rng.random() < 0.5, masked=round(rng.uniform(0.1, 1.0), 2),
                    steps=rng.randint(1, 4), topk=topk, threshold=0.0 if topk else 0.9,
                    temperature=1.0 if rng.random() < 0.25 else 0.0)
    if kind == "generate":
        model = rng.choice(["llada_loop", "loop_small", "loop_small_gqa", "loop_small_bd4"])
        block = rng.choice([4, 8]) if model == "loop_small_bd4" else rng.choice([16, 32])
        blocks = rng.randint(1, 3)
        return dict(kind=kind, model=model, batch=_log_int(rng, 1, 16), prompt=_log_int(rng, 20, 512),
                    gen=block * blocks, block=block, topk=rng.randint(2, 4), dual=rng.random() < 0.4)
    if kind == "forward":
        return dict(kind=kind, model=rng.choice(["llada_loop", "llada_loop", "loop_small_gqa"]),
                    batch=_log_int(rng, 1, 16), prompt=_log_int(rng, 33, 512))
    if kind == "score":
        return dict(kind=kind, model="llada_loop", batch=_log_int(rng, 1, 8), prompt=_log_int(rng, 20, 512),
                    gen=8 * _log_int(rng, 4, 32))
    if kind == "update":
        return dict(kind=kind, model=rng.choice(["llada8b", "dream7b"]), rows=8 * _log_int(rng, 16, 256))
    shortest = _log_int(rng, 16, 512)
    return dict(kind=kind, model=rng.choice(["llada8b", "dream7b"]), seqs=_log_int(rng, 2, 32), shortest=shortest,
                longest=min(1024, shortest + _log_int(rng, 16, 512)))


# ---------------------------------------------------------------------------------------------- inputs

_CTX = []


def _context():
    """One context per program, as a rollout worker keeps it."""
    if not _CTX:
        _CTX.append(dare.Context(torch.cuda.current_device()))
    return _CTX[0]


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) << 8) + salt)
    return g


def _normal(g, shape, sigma=1.0):
    return torch.randn(shape, generator=g, dtype=BF16, device="cuda").mul_(sigma)


def _ids(g, shape, vocab, mask_id):
    """Token ids that are never the mask id."""
    t = torch.randint(0, vocab - 1, shape, generator=g, device="cuda")
    return torch.where(t >= mask_id, t + 1, t).to(I32)


def _plant(g, x, w, cols):
    """Pushes row m of x towards column cols[m] of the head, to a probability uniform in [0.05, 0.999]."""
    p = 0.05 + 0.949 * torch.rand(x.shape[0], generator=g, dtype=F32, device="cuda")
    a = torch.log(p / (1 - p)) + math.log(w.shape[0]) + 0.02 ** 2 * x.shape[1] / 2
    wc = w[cols.long()].float()
    return (x.float() + a[:, None] * wc / (wc * wc).sum(1, keepdim=True)).to(BF16)


def _lengths(case):
    """Sequence lengths of a packed batch: part of the case's shape, the same for every seed."""
    r = random.Random(case["seqs"] * 7919 + case["longest"])
    return [r.randint(case["shortest"], case["longest"]) for _ in range(case["seqs"])]


def _cache_lengths(case):
    """Visible prefix and suffix length of each rollout."""
    B, P, S = case["batch"], case["prefix"], case["suffix"]
    if not case["ragged"]:
        return [P] * B, [S] * B
    r = random.Random(B * 7919 + P)
    return [r.randint(max(1, P // 4), P) for _ in range(B)], [r.randint(S // 4, S) for _ in range(B)]


def _prepare_step(case, seed):
    Hq, Hkv, d, D, V, mask_id = HEADS[case["model"]]
    B, L, P, S = case["batch"], case["block"], case["prefix"], case["suffix"]
    g = _gen(seed)
    cap = P + L
    s = dict(case=case, ctx=_context(), mask_id=mask_id, w=_normal(g, (V, D), 0.02),
             k_pre=_normal(g, (B, Hkv, cap, d)), v_pre=_normal(g, (B, Hkv, cap, d)), k_suf=None, v_suf=None, slen=None)
    plen, slen = _cache_lengths(case)
    s["plen"] = torch.tensor(plen, dtype=I32, device="cuda")
    if S:
        s["k_suf"], s["v_suf"] = _normal(g, (B, Hkv, S, d)), _normal(g, (B, Hkv, S, d))
        s["slen"] = torch.tensor(slen, dtype=I32, device="cuda")
    # what the layers hand to each step
    s["acts"] = []
    for _ in range(case["steps"]):
        x = _plant(g, _normal(g, (B * L, D)), s["w"], _ids(g, (B * L,), V, mask_id))
        blk = (None, None) if case["inplace"] else (_normal(g, (B, Hkv, L, d)), _normal(g, (B, Hkv, L, d)))
        s["acts"].append((_normal(g, (B, L, Hq, d)), blk[0], blk[1], x))
    # the token state: prompt, then the block, each of its positions still masked with the case's share (one at least)
    tokens = _ids(g, (B, cap), V, mask_id)
    u = torch.rand((B, L), generator=g, device="cuda")
    masked = u <= u.sort(dim=1).values[:, max(1, round(case["masked"] * L)) - 1][:, None]
    tokens[:, P:] = torch.where(masked, torch.full_like(tokens[:, P:], mask_id), tokens[:, P:])
    s["tokens0"], s["tokens"] = tokens, tokens.clone()
    new = lambda shape, dtype: torch.zeros(shape, dtype=dtype, device="cuda")  # noqa: E731
    s["results"] = [(new((B, L, Hq, d), BF16), new(B * L, I32), new(B * L, F32)) for _ in range(case["steps"])]
    s.update(done=new(B, I32), left=new(B, I32), seed=seed)
    return s


def _run_step(s):
    c = s["case"]
    s["tokens"].copy_(s["tokens0"])
    mode, k = (TOPK, c["topk"]) if c["topk"] else (THRESHOLD, 1)
    for n, ((q, kb, vb, x), (out, pred, conf)) in enumerate(zip(s["acts"], s["results"])):
        head = (s["ctx"], q, s["k_pre"], s["v_pre"], s["plen"], kb, vb, s["k_suf"], s["v_suf"], s["slen"], out, None, x,
                s["w"], s["mask_id"], True)
        tail = (s["tokens"], c["prefix"], mode, c["threshold"], k, pred, conf, s["done"], s["left"])
        if c["temperature"] > 0:
            dare.dare_denoise_block_sampled(*head, c["temperature"], s["seed"], n, *tail)
        else:
            dare.dare_denoise_block(*head, *tail)
    return {k: s[k] for k in ("results", "tokens", "done", "left")}


def _work_step(case):
    Hq, Hkv, d, D, V, _ = HEADS[case["model"]]
    B, L = case["batch"], case["block"]
    plen, slen = _cache_lengths(case)
    keys = sum(plen) + sum(slen) + B * L
    masked, live = max(1, round(case["masked"] * L)), 0.0
    for _ in range(case["steps"]):
        live += B * masked
        masked = max(0.0, masked - (case["topk"] or max(1.0, PASS_SHARE * masked)))
    n = case["steps"]
    return {"bytes": n * (2 * V * D + 4 * keys * Hkv * d + 4 * B * L * Hq * d + 8 * B * L) + 2 * live * D,
            "flops": 2 * live * D * V + n * 4 * keys * L * Hq * d}


def _prepare_model(case, seed, rows, cap):
    m = inputs.MODEL_WORKLOADS[case["model"]]
    g = _gen(seed)
    D, F, V = m.hidden, m.ffn, m.vocab
    nq, nk = m.n_q_heads * m.head_dim, m.n_kv_heads * m.head_dim
    emb, head = _normal(g, (V, D), 0.02), _normal(g, (V, D), 0.02)
    layers = [dict(wqkv=_normal(g, (nq + 2 * nk, D), 0.02), wo=_normal(g, (D, nq), 0.02), wg=_normal(g, (F, D), 0.02),
                   wu=_normal(g, (F, D), 0.02), wd=_normal(g, (D, F), 0.02)) for _ in range(m.n_layers)]
    # A trained model has a clear answer for a masked position; random weights have none (every rounding would change
    # the tokens).  The mask token's embedding outweighs what the layers add, and one token's head row follows it.
    u = torch.sign(torch.randn(D, generator=g, device="cuda"))
    emb[m.mask_id] = (16 * u).to(BF16)
    head[1 + seed % 997 % (m.mask_id - 1)] += ((math.log(V) + 2) * u / D).to(BF16)
    model = dare.Model(_context(), n_layers=m.n_layers, hidden=D, n_q_heads=m.n_q_heads, n_kv_heads=m.n_kv_heads,
                       head_dim=m.head_dim, ffn=F, vocab=V, mask_id=m.mask_id, embedding=emb, layers=layers,
                       lm_head=head, max_positions=cap, max_rows=rows, max_batch=case["batch"])
    tokens = _ids(g, (case["batch"], cap), V, m.mask_id)
    return dict(case=case, m=m, model=model, head=head, tokens0=tokens, tokens=tokens.clone(),
                cache=model.new_cache(case["batch"], cap), seed=seed, g=g)


def _prepare_forward(case, seed):
    s = _prepare_model(case, seed, case["batch"] * case["prompt"], case["prompt"])
    s["hidden"] = torch.empty(case["batch"] * case["prompt"], s["m"].hidden, dtype=BF16, device="cuda")
    return s


def _run_forward(s):
    dare.dare_model_forward(s["model"], s["tokens"], 0, s["case"]["prompt"], *s["cache"], s["hidden"])
    return {"hidden": s["hidden"], "k": s["cache"][0], "v": s["cache"][1]}


def _stack_work(m, rows, keys, passes=1):
    """`rows` rows through the stack in all, in `passes` forwards (each reads the weights once); `keys` = (row, visible
    key) pairs of all rows."""
    nq, nk = m.n_q_heads * m.head_dim, m.n_kv_heads * m.head_dim
    weights = (nq + 2 * nk) * m.hidden + m.hidden * nq + 3 * m.ffn * m.hidden
    return {"bytes": m.n_layers * (passes * 2 * weights + rows * 4 * nk) + 4 * rows * m.hidden,
            "flops": m.n_layers * (2 * rows * weights + 4 * keys * nq)}


def _work_forward(case):
    m = inputs.MODEL_WORKLOADS[case["model"]]
    rows = case["batch"] * case["prompt"]
    return _stack_work(m, rows, rows * case["prompt"])


def _prepare_generate(case, seed):
    T, P = case["prompt"] + case["gen"], case["prompt"]
    s = _prepare_model(case, seed, case["batch"] * max(T if case["dual"] else P, case["block"]), T)
    s["tokens0"][:, P:] = s["m"].mask_id
    n = case["batch"] * case["block"]
    s.update(pred=torch.zeros(n, dtype=I32, device="cuda"), conf=torch.zeros(n, dtype=F32, device="cuda"),
             left=torch.zeros(case["batch"], dtype=I32, device="cuda"))
    return s


def _run_generate(s):
    c = s["case"]
    s["tokens"].copy_(s["tokens0"])
    loop = dare.dare_generate_dual if c["dual"] else dare.dare_generate
    steps = loop(s["model"], s["tokens"], c["prompt"], c["gen"], c["block"], *s["cache"], TOPK, 0.0, c["topk"], s["pred"],
                 s["conf"], s["left"])
    return {"tokens": s["tokens"], "k": s["cache"][0], "v": s["cache"][1], "steps": steps}


def _work_generate(case):
    m = inputs.MODEL_WORKLOADS[case["model"]]
    B, P, L, T = case["batch"], case["prompt"], case["block"], case["prompt"] + case["gen"]
    per_block = -(-L // case["topk"])
    rows = keys = passes = 0
    if not case["dual"]:
        rows, keys, passes = B * P, B * P * P, 1
    live, heads = 0, 0
    for b in range(case["gen"] // L):
        seen = T if case["dual"] else P + (b + 1) * L
        if case["dual"]:
            rows, keys, passes = rows + B * T, keys + B * T * T, passes + 1
        n = per_block + (0 if case["dual"] else 1)          # the prefix cache ends a block with a refresh of its K/V
        rows, keys, passes = rows + n * B * L, keys + n * B * L * seen, passes + n
        live += B * sum(max(0, L - case["topk"] * i) for i in range(per_block))
        heads += per_block
    w = _stack_work(m, rows, keys, passes)
    return {"bytes": w["bytes"] + heads * 2 * m.vocab * m.hidden, "flops": w["flops"] + 2 * live * m.hidden * m.vocab}


def _prepare_score(case, seed):
    T = case["prompt"] + case["gen"]
    s = _prepare_model(case, seed, case["batch"] * T, T)
    t = 0.1 + 0.9 * torch.rand(case["batch"], generator=s["g"], device="cuda")       # noise level of each sequence
    s.update(hidden=torch.empty(case["batch"] * T, s["m"].hidden, dtype=BF16, device="cuda"), t=t,
             targets=s["tokens0"][:, case["prompt"]:].reshape(-1).contiguous())
    return s


def _run_score(s):
    c, m, ctx = s["case"], s["m"], s["model"].ctx
    B, P, T = c["batch"], c["prompt"], c["prompt"] + c["gen"]
    s["tokens"].copy_(s["tokens0"])
    xt = dare.dare_forward_mask(ctx, s["tokens0"], P, c["gen"], s["t"], m.mask_id, s["seed"], 0, xt=s["tokens"])
    dare.dare_model_forward_window(s["model"], xt, 0, T, T, *s["cache"], s["hidden"])
    rows = s["hidden"].view(B, T, -1)[:, P:].reshape(B * c["gen"], -1)
    logprob = dare.dare_lmhead_logprob(ctx, rows, s["head"], s["targets"], m.mask_id, True)
    nelbo = dare.dare_masked_nelbo(ctx, logprob, xt, P, c["gen"], m.mask_id, s["t"])
    return {"xt": xt, "logprob": logprob, "nelbo": nelbo}


def _work_score(case):
    m = inputs.MODEL_WORKLOADS[case["model"]]
    T, rows = case["prompt"] + case["gen"], case["batch"] * case["gen"]
    w = _stack_work(m, case["batch"] * T, case["batch"] * T * T)
    return {"bytes": w["bytes"] + 2 * m.vocab * m.hidden, "flops": w["flops"] + 2 * rows * m.hidden * m.vocab}


def _prepare_update(case, seed):
    _, _, _, D, V, mask_id = HEADS[case["model"]]
    M, g = case["rows"], _gen(seed)
    w = _normal(g, (V, D), 0.02)
    targets = _ids(g, (M,), V, mask_id)
    x = _plant(g, _normal(g, (M, D)), w, targets)
    # token-level advantages over the number of tokens, as a policy-gradient loss weighs them
    grad = torch.randn(M, generator=g, device="cuda") / M
    new = lambda *shape: torch.empty(shape, dtype=BF16, device="cuda")  # noqa: E731
    return dict(ctx=_context(), w=w, w_t=dare.dare_transpose_bf16(_context(), w), x=x, targets=targets, grad=grad,
                mask_id=mask_id, logprob=torch.empty(M, device="cuda"), lse=torch.empty(M, device="cuda"), dz=new(M, V),
                dzt=new(V, M), d_x=new(M, D), d_w=new(V, D))


def _run_update(s):
    dare.dare_lmhead_logprob(s["ctx"], s["x"], s["w"], s["targets"], s["mask_id"], True, s["logprob"], s["lse"])
    dare.dare_lmhead_logprob_backward(s["ctx"], s["x"], s["w"], s["w_t"], s["targets"], s["lse"], s["grad"], s["mask_id"],
                                      True, s["dz"], s["dzt"], s["d_x"], s["d_w"])
    return {k: s[k] for k in ("logprob", "lse", "d_x", "d_w")}


def _work_update(case):
    # the logits twice (forward, and recomputed for the gradient), then the two products of the gradient
    _, _, _, D, V, _ = HEADS[case["model"]]
    return {"bytes": 3 * 2 * V * D + 2 * V * D + 4 * 2 * case["rows"] * D, "flops": 4 * 2 * case["rows"] * D * V}


def _prepare_varlen(case, seed):
    Hq, Hkv, d, _, _, _ = HEADS[case["model"]]
    g, lens = _gen(seed), _lengths(case)
    cu = torch.tensor([sum(lens[:i]) for i in range(len(lens) + 1)], dtype=I32, device="cuda")
    n = sum(lens)
    return dict(ctx=_context(), q=_normal(g, (n, Hq, d)), k=_normal(g, (n, Hkv, d)), v=_normal(g, (n, Hkv, d)), cu=cu,
                longest=max(lens), out=torch.empty(n, Hq, d, dtype=BF16, device="cuda"),
                lse=torch.empty(Hq, n, device="cuda"))


def _run_varlen(s):
    dare.dare_attn_varlen(s["ctx"], s["q"], s["k"], s["v"], s["cu"], s["longest"], s["out"], s["lse"])
    return s["out"], s["lse"]


def _work_varlen(case):
    Hq, Hkv, d, _, _, _ = HEADS[case["model"]]
    lens = _lengths(case)
    return {"bytes": sum(lens) * (4 * Hq * d + 4 * Hkv * d + 4 * Hq), "flops": 4 * Hq * d * sum(n * n for n in lens)}


_PREPARE = dict(step=_prepare_step, generate=_prepare_generate, forward=_prepare_forward, score=_prepare_score,
                update=_prepare_update, varlen=_prepare_varlen)
_RUN = dict(step=_run_step, generate=_run_generate, forward=_run_forward, score=_run_score, update=_run_update,
            varlen=_run_varlen)
_WORK = dict(step=_work_step, generate=_work_generate, forward=_work_forward, score=_work_score, update=_work_update,
             varlen=_work_varlen)


def prepare(case, seed):
    s = _PREPARE[case["kind"]](case, seed)
    s["kind"] = case["kind"]
    return s


def run(state):
    return _RUN[state["kind"]](state)


def work(case):
    return _WORK[case["kind"]](case)


def tolerance(case):
    """Each figure is about four times what the path differs by from plain torch at the same precision and rounding
    points (double-precision softmax and attention, fp32 products, the bf16 stores of the stack where it has them)."""
    kind = case["kind"]
    if kind == "step":         # attention output 2.3e-3 (bf16 result), largest 0.011; confidences 1.6e-5
        return {"rel": 0.01, "max": 0.05, "differ": 0.002}
    if kind == "forward":      # hidden states 1.3e-2 behind four layers of bf16 stores, largest 0.074; caches 8e-3
        return {"rel": 0.03, "max": 0.3}
    if kind == "generate":     # caches 8e-3, largest 0.062
        return {"rel": 0.03, "max": 0.25, "differ": 0.002}
    if kind == "score":        # log-probabilities 7e-4, largest 0.0033; the bound 4e-5
        return {"rel": 0.003, "max": 0.015}
    if kind == "update":       # gradients 2.4e-3 (bf16 gradient of the logits), largest 0.066; log-probabilities 2e-5
        return {"rel": 0.01, "max": 0.27}
    return {"rel": 0.01, "max": 0.07}      # varlen: 2.3e-3, largest 0.017
