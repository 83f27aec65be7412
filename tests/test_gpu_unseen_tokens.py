"""The head of up to 128 rows requests its first stages before it has seen the tokens: steps with and without a masked row in
turn, with fewer, as many and more K blocks than those stages, against the head and the selection by themselves; and the head by
itself against the fp64 oracle, with a second vocabulary tile for some CTA pairs, whose stages follow those of the first."""
import numpy as np
import pytest
import torch

from oracle import dare_oracle as O
from oracle import dare_sampling_oracle as SO
from paper_2604_04215_b200 import binding as dare
from paper_2604_04215_b200 import inputs as I

from _util import check_lmhead, f64
from test_gpu_sampling import _check as check_sampled

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L", [(1, 1), (1, 32), (4, 32)])
@pytest.mark.parametrize("D", [64, 256, 264, 1024])
@pytest.mark.parametrize("temperature", [0.0, 0.8])
def test_steps_with_and_without_masked_rows(B, L, D, temperature):
    ctx = dare.Context(0)
    V, d, P, mask = 1500, 64, 40, 1499
    w, x = I.normal_bf16(D, I.TID_W, (V, D), 0.1).cuda(), I.normal_bf16(D, I.TID_X, (B * L, D)).cuda()
    q, k, v = (I.normal_bf16(L, t, s).cuda() for t, s in ((I.TID_Q, (B, L, 2, d)), (I.TID_KPRE, (B, 2, P + L, d)), (I.TID_VPRE, (B, 2, P + L, d))))
    plen = torch.full((B,), P, dtype=torch.int32, device="cuda")
    new = lambda n, t: torch.full((n,), 7, dtype=t, device="cuda")  # noqa: E731
    state, got = [], []
    for n, masked in enumerate((0, 1, 0, 0, B * L, 0)):                  # masked rows, the last ones of the batch
        tok = torch.full((B, P + L), 5, dtype=torch.int32, device="cuda")
        if masked:
            flat = torch.full((B * L,), 5, dtype=torch.int32, device="cuda")
            flat[-masked:] = mask
            tok[:, P:] = flat.view(B, L)
        state.append(tok.clone())
        pred, conf, nc, nr = new(B * L, torch.int32), new(B * L, torch.float32), new(B, torch.int32), new(B, torch.int32)
        head = (ctx, q, k, v, plen, None, None, None, None, None, torch.empty_like(q), None, x, w, mask, True)
        tail = (tok, P, dare.SELECT_TOPK, 0.0, 2, pred, conf, nc, nr)
        if temperature:
            dare.dare_denoise_block_sampled(*head, temperature, 3, n, *tail)
        else:
            dare.dare_denoise_block(*head, *tail)
        got.append((tok, pred, conf, nc, nr))
    for n, (tok, (after, pred, conf, nc, nr)) in enumerate(zip(state, got)):
        rows = tok[:, P:].contiguous().view(-1)
        if temperature:
            p2, c2 = dare.dare_lmhead_sample(ctx, x, w, rows, mask, True, temperature, 3, n)
        else:
            p2, c2 = dare.dare_lmhead_confidence(ctx, x, w, rows, mask, True)
        nc2, nr2 = new(B, torch.int32), new(B, torch.int32)
        dare.dare_unmask_select(ctx, tok, P, L, p2, c2, mask, dare.SELECT_TOPK, 0.0, 2, nc2, nr2)
        torch.cuda.synchronize()
        for a, b in ((after, tok), (pred, p2), (conf, c2), (nc, nc2), (nr, nr2)):
            assert torch.equal(a, b)
    assert ctx.device_status() == 0
    ctx.close()


@pytest.mark.parametrize("M,masked", [(1, 1), (32, 5), (32, 32), (128, 40)])
@pytest.mark.parametrize("D", [200, 264, 1024])
def test_head_in_place_against_the_oracle(M, masked, D):
    ctx = dare.Context(0)
    V, mask = 75 * 256 + 1, 1000
    x, w = I.normal_bf16(D + M, I.TID_X, (M, D)), I.normal_bf16(D, I.TID_W, (V, D), 3.0 / D ** 0.5)
    rows = torch.full((M,), 5, dtype=torch.int32)
    rows[M - masked:] = mask
    args = (x.cuda(), w.cuda(), rows.cuda(), mask, True)
    greedy, sampled = dare.dare_lmhead_confidence(ctx, *args), dare.dare_lmhead_sample(ctx, *args, 0.8, 3, 7)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    check_lmhead(*greedy, O.lmhead_confidence(f64(x), f64(w), rows.numpy(), mask, True), f64(x), f64(w), mask, True, O)
    ref = SO.lmhead_sample(f64(x), f64(w), rows.numpy(), mask, True, 0.8, 3, 7)
    check_sampled(*sampled, ref, f64(x), f64(w), np.arange(M), mask, True, 0.8, 3, 7)
    ctx.close()
