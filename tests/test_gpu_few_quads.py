"""Projections of few rows whose K slices are handed over four rows at a time: row counts around groups of four and the last
count that takes this way, one to eight slices, every epilogue, against fp64 products of the bf16 inputs (one bf16 step)."""
import pytest
import torch

from paper_2604_04215_b200 import binding as dare
from paper_2604_04215_b200 import inputs as I

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
