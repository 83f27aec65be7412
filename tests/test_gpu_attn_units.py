"""The persistent tcgen05 attention kernel at the edges of its key tiles (64), query tiles (128 rows) and units, and with more
units than CTAs, against the fp64 oracle.  Bars as in the other attention tests (one bf16 result: max-abs 2e-2, rel-L2 5e-3)."""
import numpy as np
import pytest
import torch

from oracle import dare_oracle as O
from paper_2604_04215_b200 import binding as dare
from paper_2604_04215_b200 import inputs as I

from _util import check_attn, f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = dare.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("lens,Hq,Hkv,d", [
    ([1, 63, 64, 65, 127, 128, 129, 255, 256, 257], 2, 2, 128),       # ends of key tiles; one and two live query tiles
    ([191, 192, 193, 320, 449], 2, 1, 64),
    ([35, 36, 37, 54, 55, 72, 73], 7, 1, 128),                        # 18 positions a tile: 126 of 128 rows, 36 a unit
    ([int(n) for n in np.random.default_rng(5).integers(0, 150, 120)], 4, 4, 64),    # 480 units and more: CTAs take over units,
    ([int(n) for n in np.random.default_rng(6).integers(0, 90, 90)], 6, 2, 128),     # empty sequences among them
])
def test_packed_units(ctx, lens, Hq, Hkv, d):
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    T = int(cu[-1])
    q, k, v = (I.normal_bf16(len(lens) + d, t, (T, h, d)) for t, h in ((I.TID_Q, Hq), (I.TID_KPRE, Hkv), (I.TID_VPRE, Hkv)))
    ref, lse_ref = O.attn_varlen(f64(q), f64(k), f64(v), cu)
    lse = torch.full((Hq, T), float("nan"), dtype=torch.float32, device="cuda")
    out = torch.full_like(q, float("nan"), device="cuda")
    dare.dare_attn_varlen(ctx, q.cuda(), k.cuda(), v.cuda(), torch.from_numpy(cu).cuda(), max(lens), out, lse)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    check_attn(out, ref)
    assert np.abs(lse.cpu().double().numpy() - lse_ref).max() < 2e-2


@pytest.mark.parametrize("B,L,Hq,Hkv,d,plens,slens", [
    (3, 32, 14, 2, 128, [1, 64, 129], None),                # GQA group of 7, block apart from the cache
    (2, 100, 2, 2, 128, [0, 65], [63, 1]),                  # no prefix; three segments, each with a ragged end
    (5, 130, 64, 64, 64, [3, 64, 1, 100, 128], None),       # 320 units of two query tiles, the second with two rows
    (90, 20, 14, 2, 128, None, None),                       # 180 units; 20 positions are two query tiles of 18
])
@pytest.mark.parametrize("inplace", [False, True])
def test_block_units(ctx, B, L, Hq, Hkv, d, plens, slens, inplace):
    plens = plens or [int(n) for n in np.random.default_rng(B).integers(0, 140, B)]
    cap = max(plens) + L + 5
    scap = max(slens) + 3 if slens else 0
    q = I.normal_bf16(B, I.TID_Q, (B, L, Hq, d))
    k, v = I.normal_bf16(B, I.TID_KPRE, (B, Hkv, cap, d)), I.normal_bf16(B, I.TID_VPRE, (B, Hkv, cap, d))
    kb, vb = I.normal_bf16(B, I.TID_KBLK, (B, Hkv, L, d)), I.normal_bf16(B, I.TID_VBLK, (B, Hkv, L, d))
    ks = I.normal_bf16(B + 1, I.TID_KPRE, (B, Hkv, scap, d)) if slens else None
    vs = I.normal_bf16(B + 1, I.TID_VPRE, (B, Hkv, scap, d)) if slens else None
    for b, n in enumerate(plens):                             # what lies behind the visible keys must not matter
        if inplace:
            k[b, :, n:n + L], v[b, :, n:n + L] = kb[b], vb[b]
        end = n + L if inplace else n
        k[b, :, end:], v[b, :, end:] = float("nan"), float("nan")
    for b, n in enumerate(slens or []):
        ks[b, :, n:], vs[b, :, n:] = float("nan"), float("nan")
    g = lambda t: None if t is None else t.cuda()  # noqa: E731
    pl = torch.tensor(plens, dtype=torch.int32)
    sl = torch.tensor(slens, dtype=torch.int32) if slens else None
    out = torch.full_like(q, float("nan"), device="cuda")
    dare.dare_attn_block(ctx, g(q), g(k), g(v), g(pl), None if inplace else g(kb), None if inplace else g(vb), g(ks), g(vs),
                         g(sl), out)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    c = lambda t: None if t is None else torch.nan_to_num(t.double(), nan=0.0).numpy()  # noqa: E731
    res = O.attn_block(c(q), c(k), c(v), np.array(plens), c(kb), c(vb), c(ks), c(vs), None if sl is None else np.array(slens))
    check_attn(out, res[0] if isinstance(res, tuple) else res)



# Behind a sequence's or a rollout's last query a tile holds the next one's queries.  With scores this sharp the references of most
# rows lag behind their maxima, so a reference that moves shows in the bits of a row's result.
@pytest.mark.parametrize("n,Hq,Hkv,d", [(300, 2, 2, 128), (129, 4, 2, 64), (37, 7, 1, 128), (250, 1, 1, 64)])
@pytest.mark.parametrize("packed", [True, False])
def test_neighbour_does_not_matter(ctx, n, Hq, Hkv, d, packed):
    P = 200                                                     # block form: cached keys in front of the block
    keys = n if packed else P + n
    q = I.normal_bf16(n, I.TID_Q, (2, n, Hq, d), 5.0)
    k, v = I.normal_bf16(n, I.TID_KPRE, (2, Hkv, keys, d)).cuda(), I.normal_bf16(n, I.TID_VPRE, (2, Hkv, keys, d)).cuda()
    got = []
    for scale in (1.0, 40.0):
        qs = torch.stack((q[0], q[1] * scale)).cuda()
        if packed:
            flat = lambda t: t.transpose(1, 2).reshape(2 * n, Hkv, d).contiguous()  # noqa: E731
            lse = torch.empty(Hq, 2 * n, device="cuda")
            out = dare.dare_attn_varlen(ctx, qs.view(2 * n, Hq, d), flat(k), flat(v),
                                        torch.tensor([0, n, 2 * n], dtype=torch.int32, device="cuda"), n, None, lse)
            got.append((out[:n].clone(), lse[:, :n].clone()))
        else:
            out, lse = torch.empty_like(qs), torch.empty(2, Hq, n, device="cuda")
            dare.dare_attn_block(ctx, qs, k, v, torch.tensor([P, P], dtype=torch.int32, device="cuda"), None, None, None, None, None,
                                 out, lse)
            got.append((out[0].clone(), lse[0].clone()))
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])



# Rows whose first `blind` scores are -inf (the products overflow fp32), in warps whose other rows have finite scores and move
# their references in the first and in later tiles.
@pytest.mark.parametrize("blind", [64, 128, 192])
@pytest.mark.parametrize("d", [64, 128])
def test_rows_that_see_nothing_at_first(ctx, blind, d):
    n, H = 400, 2
    q, k, v = (I.normal_bf16(blind + d, t, (n, H, d), s) for t, s in ((I.TID_Q, 4.0), (I.TID_KPRE, 1.0), (I.TID_VPRE, 1.0)))
    for t in (q, k):
        t[:, :, 0] = 0
    q[::3, :, 0] = 1e30
    k[:blind, :, 0] = -1e30
    k[300:, :, 1:] *= 4                                       # larger scores later on: references move
    ref, lse_ref = O.attn_varlen(f64(q), f64(k), f64(v), np.array([0, n]))
    lse = torch.empty(H, n, device="cuda")
    out = dare.dare_attn_varlen(ctx, q.cuda(), k.cuda(), v.cuda(), torch.tensor([0, n], dtype=torch.int32, device="cuda"), n, None, lse)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    check_attn(out, ref)
    assert np.abs(lse.cpu().double().numpy() - lse_ref).max() < 2e-2



# Sharp rows: a few weights make up the result, and what rounding them to bf16 costs depends on how far a row's reference lags
# behind its maximum.  The result's own rounding is 1.5e-3 of its norm (2^-7 / sqrt(12) of the binade, log-uniform mantissas); a single weight
# rounded like that would double the variance (2.15e-3), one that is exact adds nothing.  The bounds allow the weights half and a third of it.
@pytest.mark.parametrize("sharp,bar", [(4.0, 1.95e-3), (8.0, 1.77e-3)])
@pytest.mark.parametrize("d", [64, 128])
def test_sharp_rows(ctx, sharp, bar, d):
    n, H = 1000, 8
    q, k, v = (I.normal_bf16(d, t, (n, H, d), s).cuda() for t, s in ((I.TID_Q, sharp), (I.TID_KPRE, 1.0), (I.TID_VPRE, 1.0)))
    out = dare.dare_attn_varlen(ctx, q, k, v, torch.tensor([0, n], dtype=torch.int32, device="cuda"), n).double()
    p = torch.softmax(torch.einsum("ihd,jhd->hij", q.double(), k.double()) / d ** 0.5, -1)
    ref = torch.einsum("hij,jhd->ihd", p, v.double())
    assert ((out - ref).norm() / ref.norm()).item() < bar


# The warp-level kernel: rows that share a KV head at the ends of its variants (four, two and one key slices a tile; each slice
# finishes its share of the columns), without and with K/V splits, keys that end inside a slice.
@pytest.mark.parametrize("L,g", [(1, 1), (4, 4), (17, 1), (32, 1), (33, 1), (8, 9), (90, 1)])
@pytest.mark.parametrize("B,Hkv,P", [(1, 1, 900), (2, 160, 37), (3, 32, 70)])
@pytest.mark.parametrize("d", [64, 128])
def test_warp_level_shares(ctx, L, g, B, Hkv, P, d):
    Hq = Hkv * g
    plens = [P - 11 * b for b in range(B)]
    q = I.normal_bf16(L, I.TID_Q, (B, L, Hq, d))
    k, v = I.normal_bf16(L, I.TID_KPRE, (B, Hkv, P + L, d)), I.normal_bf16(L, I.TID_VPRE, (B, Hkv, P + L, d))
    out = torch.full_like(q, float("nan"), device="cuda")
    lse = torch.full((B, Hq, L), float("nan"), device="cuda")
    dare.dare_attn_block(ctx, q.cuda(), k.cuda(), v.cuda(), torch.tensor(plens, dtype=torch.int32).cuda(), None, None, None, None,
                         None, out, lse)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    ref, lse_ref = O.attn_block(f64(q), f64(k), f64(v), np.array(plens))
    check_attn(out, ref)
    assert np.abs(lse.cpu().double().numpy() - lse_ref).max() < 2e-2
