"""Projections of few rows whose K slices are handed over four rows at a time: row counts around groups of four and the last
count that takes this way, one to eight slices, received behind the operand ring (few K blocks per CTA) and over it (as many as
the ring has stages, or more); store, residual and SwiGLU against fp64 products of the bf16 inputs (one bf16 step), rotary embedding
against the projection and the rotation by themselves."""
import pytest
import torch

from paper_2604_04215_b200 import binding as dare
from paper_2604_04215_b200 import inputs as I

from test_gpu_variants import _small_model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = dare.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("M", [1, 3, 4, 5, 16, 31, 33, 48, 63, 64, 65])
@pytest.mark.parametrize("K,N,slices", [(64, 136, 1), (256, 264, 2), (520, 128, 4), (1280, 512, 8), (1288, 72, 8),
                                        (1024, 1792, 8)])     # up to 4 rows: value by value
@pytest.mark.parametrize("epilogue", [dare.LINEAR_STORE, dare.LINEAR_RESIDUAL, dare.LINEAR_SWIGLU])
def test_projection(ctx, M, K, N, slices, epilogue):
    a, w, w2 = I.normal_bf16(M, 1, (M, K)), I.normal_bf16(K, 2, (N, K), 0.05), I.normal_bf16(K, 3, (N, K), 0.05)
    res = I.normal_bf16(M, 4, (M, N))
    if M <= 64:
        assert dare.dare_linear_plan(ctx, epilogue, M, K, N)["k_splits"] == slices
    z = a.double() @ w.double().T
    if epilogue == dare.LINEAR_RESIDUAL:
        z = z + res.double()
    if epilogue == dare.LINEAR_SWIGLU:
        z = z / (1 + torch.exp(-z)) * (a.double() @ w2.double().T)
    out = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    dare.dare_linear(ctx, epilogue, a.cuda(), w.cuda(), w2.cuda() if epilogue == dare.LINEAR_SWIGLU else None,
                     res.cuda() if epilogue == dare.LINEAR_RESIDUAL else None, out)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    # one bf16 rounding (2^-9 of the value, doubled for a sum that lies beside a tie) and fp32 sums of K terms of size ~1
    err = (out.cpu().double() - z).abs()
    assert (err <= z.abs() * 2.0 ** -8 + 2e-5 * K ** 0.5).all()


def _check(ctx, M, K, N, epilogue):
    a, w, w2 = I.normal_bf16(M, 1, (M, K)), I.normal_bf16(K, 2, (N, K), 0.05), I.normal_bf16(K, 3, (N, K), 0.05)
    res = I.normal_bf16(M, 4, (M, N))
    z = a.double() @ w.double().T
    if epilogue == dare.LINEAR_RESIDUAL:
        z = z + res.double()
    if epilogue == dare.LINEAR_SWIGLU:
        z = z / (1 + torch.exp(-z)) * (a.double() @ w2.double().T)
    out = torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    dare.dare_linear(ctx, epilogue, a.cuda(), w.cuda(), w2.cuda() if epilogue == dare.LINEAR_SWIGLU else None,
                     res.cuda() if epilogue == dare.LINEAR_RESIDUAL else None, out)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    err = (out.cpu().double() - z).abs()
    assert (err <= z.abs() * 2.0 ** -8 + 2e-5 * K ** 0.5).all()      # (as above)


def _blocks_and_stages(ctx, epilogue, M, K, N):
    plan = dare.dare_linear_plan(ctx, epilogue, M, K, N)
    assert plan["k_splits"] == 8
    return -(-((K + 63) // 64) // 8), plan["stages"]


@pytest.mark.parametrize("M", [1, 3, 4, 5, 16, 33, 48, 63, 64])
@pytest.mark.parametrize("K,N", [(4096, 136), (4040, 72), (2056, 264)])
@pytest.mark.parametrize("epilogue", [dare.LINEAR_STORE, dare.LINEAR_RESIDUAL, dare.LINEAR_SWIGLU])
def test_projection_over_the_ring(ctx, M, K, N, epilogue):
    blocks, stages = _blocks_and_stages(ctx, epilogue, M, K, N)
    assert K < 4000 or blocks >= stages              # (2056: five blocks; six stages at 16 rows, four at 64)
    _check(ctx, M, K, N, epilogue)


@pytest.mark.parametrize("Hq,Hkv,d,B,length,hidden,over", [(4, 2, 64, 3, 5, 4096, True), (2, 1, 128, 7, 9, 4096, True),
                                                          (2, 1, 128, 1, 33, 2048, None), (4, 2, 64, 1, 2, 2048, False),
                                                          (3, 1, 128, 1, 7, 1088, False)])
def test_rope_of_eight_slices(ctx, Hq, Hkv, d, B, length, hidden, over):
    start, cap, M, n = 3, length + 5, B * length, (Hq + 2 * Hkv) * d
    blocks, stages = _blocks_and_stages(ctx, dare.LINEAR_STORE, M, hidden, n)
    assert over is None or (blocks >= stages) == over
    model = _small_model(ctx, Hq, Hkv, d, M, B, cap, hidden=hidden)
    tok = I.uniform_int(7, 9, (B, cap), 0, 510).cuda()
    caches = model.new_cache(B, cap)
    dare.dare_model_forward(model, tok, start, length, *caches)
    emb, layers, _ = model._keep
    x = emb[tok[:, start:start + length].reshape(-1).long()].contiguous()
    xn = dare.dare_rmsnorm(ctx, x, 1e-5)
    qkv = dare.dare_linear(ctx, dare.LINEAR_STORE, xn, layers[0]["wqkv"])
    z = xn.double() @ layers[0]["wqkv"].double().T
    kc, vc = torch.zeros_like(caches[0]), torch.zeros_like(caches[1])
    q = torch.empty(M, Hq, d, dtype=torch.bfloat16, device="cuda")
    dare.dare_rope_kv_write(model, qkv, B, length, start, q, kc[0], vc[0])
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    assert ((qkv.double() - z).abs() <= z.abs() * 2.0 ** -8 + 2e-5 * hidden ** 0.5).all()
    # the same sums, the same rounding before the rotation; a multiply-add may be contracted differently behind it
    assert torch.equal(caches[1], vc)
    assert ((caches[0].float() - kc.float()).abs() <= 2.0 ** -7 * kc.float().abs() + 1e-6).all()
    model.close()
