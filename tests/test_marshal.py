"""The native marshalling of the inner loop's calls leaves every argument that does not fit to the Python checks."""
import pytest
import torch

from paper_2604_04215_b200 import binding as dare
from paper_2604_04215_b200 import inputs as I

WL = I.WORKLOADS["tiny"]
SAMPLED = dict(temperature=1.0, seed=(1 << 64) + 5, step=2)


def _args(device):
    si = I.make_step(WL, step=0, planted=True)
    mv = lambda t: None if t is None else t.to(device)
    z = lambda n, dt: torch.zeros(n, dtype=dt, device=device)
    return dict(q=mv(si.q), k_pre=mv(si.k_pre), v_pre=mv(si.v_pre), prefix_len=mv(si.prefix_len), k_blk=mv(si.k_blk),
                v_blk=mv(si.v_blk), k_suf=mv(si.k_suf), v_suf=mv(si.v_suf), suffix_len=mv(si.suffix_len),
                attn_out=torch.empty_like(si.q, device=device), lse=None, hidden=mv(si.x), w=mv(si.w), mask_id=WL.mask_id,
                exclude_mask_column=True, tokens=mv(si.tokens), block_start=si.block_start, mode=dare.SELECT_TOPK,
                threshold=0.0, k=1, pred=z(WL.M, torch.int32), conf=z(WL.M, torch.float32), n_committed=None, n_remaining=None)


def test_host_tensors_and_short_argument_lists_are_left_to_the_python_checks():
    m = dare._native()
    assert m.denoise_block(0, 0, 0, 0.0, *_args("cpu").values()) is None
    assert m.denoise_block_sampled(0, 0, 0, 0.0, *_args("cpu").values()) is None          # three arguments short
    assert m.attn_varlen(0, 0, 0, 0.0) is None
    assert m.denoise_block(None, 0) is None


@pytest.mark.gpu
@pytest.mark.parametrize("sampled", [False, True])
@pytest.mark.parametrize("name,change", [("w", lambda t: t.float()), ("q", lambda t: t.transpose(1, 2)), ("prefix_len", lambda t: t.cpu()),
                                         ("tokens", lambda t: t.long()), ("n_committed", lambda t: torch.zeros(WL.batch, dtype=torch.int32))])
def test_a_wrong_tensor_raises(name, change, sampled):
    ctx = dare.Context(0)
    a = _args("cuda")
    a[name] = change(a[name])
    with pytest.raises(ValueError):
        dare.dare_denoise_block_sampled(ctx, **a, **SAMPLED) if sampled else dare.dare_denoise_block(ctx, **a)


@pytest.mark.gpu
@pytest.mark.parametrize("sampled", [False, True])
def test_both_ways_to_the_library_give_the_same_step(sampled, monkeypatch):
    class Never:
        denoise_block = denoise_block_sampled = staticmethod(lambda *a: None)

    ctx = dare.Context(0)
    got = []
    for native in (dare._native(), Never):
        monkeypatch.setattr(dare, "_marshal", native)
        a = _args("cuda")
        a["n_remaining"] = torch.zeros(WL.batch, dtype=torch.int32).pin_memory()
        dare.dare_denoise_block_sampled(ctx, **a, **SAMPLED) if sampled else dare.dare_denoise_block(ctx, **a)
        torch.cuda.synchronize()
        got.append([a[k].cpu() for k in ("attn_out", "tokens", "pred", "conf", "n_remaining")])
    assert all(torch.equal(x, y) for x, y in zip(*got))
