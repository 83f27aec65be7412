"""Heads of up to 128 rows by the number of CTA pairs they get: a pair per vocabulary tile of 256 up to 74 tiles, and where all
pairs save a round; the plan shows in the launches' results only, so these are the counts at which it changes."""
import pytest
import torch

from oracle import dare_oracle as O
from paper_2604_04215_b200 import binding as dare
from paper_2604_04215_b200 import inputs as I

from _util import check_lmhead, f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 33, 128])
@pytest.mark.parametrize("V", [200, 256, 257, 73 * 256, 74 * 256, 74 * 256 + 1, 94 * 256, 125 * 256, 148 * 256 + 3])
def test_head_of_few_rows(M, V):
    ctx = dare.Context(0)
    D = 72
    x, w = I.normal_bf16(M, I.TID_X, (M, D)), I.normal_bf16(V, I.TID_W, (V, D), 0.3)
    ref = O.lmhead_confidence(f64(x), f64(w))
    tok = torch.full((M,), V - 1, dtype=torch.int32, device="cuda")
    a = dare.dare_lmhead_confidence(ctx, x.cuda(), w.cuda())
    b = dare.dare_lmhead_confidence(ctx, x.cuda(), w.cuda(), tok, V - 1, False)      # rows evaluated where they lie
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    check_lmhead(*a, ref)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    ctx.close()
