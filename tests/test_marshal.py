"""The native marshalling of the inner loop's calls leaves every argument that does not fit to the Python checks."""
import os
import subprocess
import sys
import sysconfig

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


BATCHED = """
import torch
from torch._subclasses import FakeTensorMode
from paper_2604_04215_b200 import binding as dare
m = dare._native()
with FakeTensorMode():
    q = torch.empty(3, 1, 8, 2, 64, dtype=torch.bfloat16, device="cuda:0")
    x = torch.empty(3, 8, 16, dtype=torch.bfloat16, device="cuda:0")
    i = torch.empty(2, dtype=torch.int32, device="cuda:0")
    tok = torch.empty(1, 16, dtype=torch.int32, device="cuda:0")
    k, w, f = q[0], x[0], torch.empty(8, device="cuda:0")
    def varlen(a):
        assert m.attn_varlen(0, 0, 0, 0.0, a[0], k[0], k[0], i, 8, k[0], None) is None
        return a
    def step(a, h):
        for call, more in ((m.denoise_block, ()), (m.denoise_block_sampled, (1.0, 5, 2))):
            for qq, hh in ((a, w), (k, h)):
                assert call(0, 0, 0, 0.0, qq, k, k, None, None, None, None, None, None, k, None, hh, w, 3, True, *more, tok, 0, 0,
                            0.5, 1, i, f, None, None) is None
        return a
    torch.vmap(varlen)(q)
    torch.vmap(step)(q, x)
print("all None")
"""


def test_tensors_without_memory_are_left_to_the_python_checks():
    """Under vmap a tensor has no address: asking for it throws, which must not leave the C++ module (the process would end)."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", BATCHED], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "all None" in r.stdout, r.stderr[-2000:]


def test_the_module_holds_for_one_python_and_one_torch(monkeypatch):
    """With another torch the module that is there is neither up to date nor loaded; the calls then go through ctypes."""
    from paper_2604_04215_b200 import build
    here = build.marshal_path()
    assert os.path.exists(here) and here.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and torch.__version__ in here
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    assert build._stale()
    monkeypatch.setattr(dare, "_marshal", None)
    with pytest.warns(RuntimeWarning, match="marshalling module"):
        m = dare._native()
    assert dare._native() is m                                        # (said once)
    assert m.denoise_block(1, 2) is None and m.denoise_block_sampled(1) is None and m.attn_varlen() is None


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
