"""The matrix-vector product on matrices with few rows and many columns, in every format
and on both sides of the rule that deals out its tiles: values against the
FP64 product of the stored matrix (the bounds of test_gpu_gemv.py), infinities, and
the time of a wide product, which all SMs must share (2 ms on the CTAs of its
row tiles alone, 0.1 to 0.22 ms on all of them)."""
import numpy as np
import pytest
import torch

from paper_1511_07207_gb300 import binding as B

pytestmark = pytest.mark.gpu

FORMATS = [B.LS_F64_PAIR, B.LS_BF16_IR, B.LS_FP8_IR, B.LS_F32_IR]


def _stored(ctx, gpu, dtype, A):
    """The matrix argument of ls_gemv, the scales, and the stored values in FP64."""
    rows, cols = A.shape
    if dtype == B.LS_F64_PAIR:
        pair = torch.zeros((2 * rows, (cols + 3) // 4 * 4), dtype=torch.float32, device=gpu)
        assert B.ls_split_f64(ctx, A, pair[:, :cols]) == B.LS_OK
        return pair[:rows, :cols], None, A, torch.float64
    tdt = {B.LS_BF16_IR: torch.bfloat16, B.LS_FP8_IR: torch.float8_e4m3fn, B.LS_F32_IR: torch.float32}[dtype]
    raw = {B.LS_BF16_IR: torch.int16, B.LS_FP8_IR: torch.uint8, B.LS_F32_IR: torch.float32}[dtype]
    Q = torch.zeros((rows, (cols + 15) // 16 * 16), dtype=raw, device=gpu)
    s = torch.zeros(rows, dtype=torch.float32, device=gpu) if dtype == B.LS_FP8_IR else None
    assert B.ls_quantize(ctx, dtype, A, Q[:, :cols], s) == B.LS_OK
    D = Q.view(tdt)[:, :cols].double()
    return Q[:, :cols], s, D if s is None else D * s.double()[:, None], torch.float32


@pytest.mark.parametrize("dtype", FORMATS)
@pytest.mark.parametrize("rows,cols", [(1, 70001), (17, 9000), (64, 30000), (65, 15000), (300, 513), (300, 40000),
                                       (4870, 300), (2500, 2500)])
def test_values(ctx, gpu, dtype, rows, cols):
    g = torch.Generator(device=gpu)
    g.manual_seed(rows + cols)
    A = torch.randn(rows, cols, dtype=torch.float64, device=gpu, generator=g)
    M, s, D, vt = _stored(ctx, gpu, dtype, A)
    x = torch.randn(cols, dtype=torch.float64, device=gpu, generator=g).to(vt)
    y = torch.full((rows,), float("nan"), dtype=vt, device=gpu)
    assert B.ls_gemv(ctx, dtype, M, x, y, s) == B.LS_OK
    ref = D @ x.double()
    u = 2.0 ** -45 if dtype == B.LS_F64_PAIR else 2.0 * 2.0 ** -24
    assert torch.all((y.double() - ref).abs() <= (cols + 2) * u * (D.abs() @ x.double().abs()) + 1e-30)


@pytest.mark.parametrize("dtype", [B.LS_BF16_IR, B.LS_F32_IR])
@pytest.mark.parametrize("rows,cols", [(40, 600), (40, 60000)])
def test_infinities(ctx, gpu, dtype, rows, cols):
    """What FP32 additions give: an infinite product stays infinite, two of opposite signs are NaN."""
    A = torch.ones(rows, cols, dtype=torch.float64, device=gpu)
    A[3, cols // 2] = float("inf")
    A[4, 5] = -float("inf")
    A[5, 7] = float("inf")
    A[5, cols - 1] = -float("inf")
    M, s, D, vt = _stored(ctx, gpu, dtype, A)
    y = torch.zeros(rows, dtype=vt, device=gpu)
    assert B.ls_gemv(ctx, dtype, M, torch.ones(cols, dtype=vt, device=gpu), y, s) == B.LS_OK
    assert y[3] == float("inf") and y[4] == -float("inf") and torch.isnan(y[5])
    rest = torch.cat([y[:3], y[6:]])
    assert torch.all(rest == cols)


@pytest.mark.parametrize("dtype", FORMATS)
def test_all_sms_share_a_wide_product(ctx, gpu, dtype):
    rows, cols = 64, 1000000
    A = torch.randn(rows, cols, dtype=torch.float64, device=gpu)
    M, s, D, vt = _stored(ctx, gpu, dtype, A)
    x = torch.ones(cols, dtype=vt, device=gpu)
    y = torch.zeros(rows, dtype=vt, device=gpu)
    st, ms = B.ls_gemv_timed(ctx, dtype, M, x, y, 20, s)
    assert st == B.LS_OK
    assert ms < 0.6
