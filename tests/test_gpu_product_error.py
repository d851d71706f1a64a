"""How far the products in double-single arithmetic are from FP64 ones, as a root
mean square over the rows, for the product from one triangle (exactly symmetric
A) and the general one.

The measure is the same arithmetic formed here in NumPy in its plainest order:
256 accumulators a row, each a chain of ds_fma over column tiles of 256, added
pairwise without settling, the (row tile, column tile) sequence cut into equal pieces
for two CTAs on each of 152 SMs and the pieces of a row added in FP64.  The
kernels' orders have longer chains in places, but their pair sums are settled, so
their error may not exceed that one's by more than the 5 % that two root mean
squares over a thousand rows or more can differ by chance.

The residual of CG with x0 = x and b = fl(A x) is the product's error: the
loop does not start, and info.true_rel_res is formed by the same kernel.
"""
import numpy as np
import pytest
import torch

from paper_1511_07207_gb300 import binding as B
from paper_1511_07207_gb300 import inputs

pytestmark = pytest.mark.gpu
F = np.float32


def _pair(v):
    h = v.astype(F)
    return h, (v - h.astype(np.float64)).astype(F)


def _add(a, b):
    s = a[0] + b[0]
    bv = s - a[0]
    return s, ((a[0] - (s - bv)) + (b[0] - bv)) + (a[1] + b[1])


def _fma(ah, al, xh, xl, acc):
    # fused operations by way of FP64, where a product of two FP32 numbers is exact
    exact = ah.astype(np.float64) * xh.astype(np.float64)
    p = exact.astype(F)
    t = (ah.astype(np.float64) * xl + (exact - p)).astype(F)
    t = (al.astype(np.float64) * xh + t).astype(F)
    s, e = _add((acc[0], F(0)), (p, F(0)))
    return s, acc[1] + (t + e)


def _plain_product(A, x):
    n = len(x)
    ct, rt, grid = -(-n // 256), -(-n // 16), 304
    Ap = np.zeros((rt * 16, ct * 256))
    Ap[:n, :n] = A
    xp = np.zeros(ct * 256)
    xp[:n] = x
    ah, al = _pair(Ap)
    xh, xl = _pair(xp)
    y = np.zeros(rt * 16)
    total = rt * ct
    start = [total * c // grid for c in range(grid + 1)]
    owner = np.searchsorted(start, np.arange(total), side="right") - 1
    for r in range(rt):
        rows = slice(16 * r, 16 * r + 16)
        c = 0
        while c < ct:
            own = owner[r * ct + c]
            acc = (np.zeros((16, 256), F), np.zeros((16, 256), F))
            while c < ct and owner[r * ct + c] == own:
                k = slice(256 * c, 256 * c + 256)
                acc = _fma(ah[rows, k], al[rows, k], xh[k], xl[k], acc)
                c += 1
            while acc[0].shape[1] > 1:
                h = acc[0].shape[1] // 2
                acc = _add((acc[0][:, :h], acc[1][:, :h]), (acc[0][:, h:], acc[1][:, h:]))
            y[rows] += acc[0][:, 0].astype(np.float64) + acc[1][:, 0]
    return y[:n]


def _fp64_product(A, x):
    y = np.zeros(len(x))
    for c in range(0, len(x), 256):
        y += (A[:, c:c + 256] * x[c:c + 256]).sum(axis=1)
    return y


@pytest.mark.parametrize("n", [1024, 1500, 2500, 4000])
def test_error_against_fp64(ctx, gpu, n):
    A = inputs.spd_matrix(n, 0.1, seed=600 + n)
    x = inputs.solution(n, seed=601 + n)
    b = _fp64_product(A, x)
    assert np.array_equal(A, A.T)
    limit = 1.05 * np.linalg.norm(_plain_product(A, x) - b) / np.linalg.norm(b)
    for symmetric in (True, False):
        if not symmetric:
            A[n - 1, 0] = np.nextafter(A[n - 1, 0], 9.0)
        xd = torch.from_numpy(x).to(gpu)
        st, info = B.ls_cg_solve(ctx, torch.from_numpy(A).to(gpu), torch.from_numpy(b).to(gpu), xd,
                                 B.make_opts(rtol=1e-8, x0_given=1, fused=0))
        assert st == B.LS_OK and info["iters"] == 0
        assert (info["bytes_moved"] < 6.0 * n * n) == symmetric     # one product: which kernel
        assert info["true_rel_res"] <= limit, (symmetric, info["true_rel_res"], limit)


# ---- the FP32 formats: y = A x with an FP32 result -------------------------------------
GEO = {B.LS_BF16_IR: (8, 1, 32), B.LS_FP8_IR: (8, 1, 64), B.LS_F32_IR: (4, 2, 16)}   # VEC, WC, TR


def _fma32(a, x, acc):
    return (a.astype(np.float64) * x + acc).astype(F)


def _plain_fp32(dtype, Q, x):
    """The product in plain FP32 chains, equal pieces, the pieces of a row added in FP64."""
    vec, wc, tr = GEO[dtype]
    n = len(x)
    ct, rt, grid = -(-n // 256), -(-n // tr), 304
    Ap = np.zeros((rt * tr, ct * 256), F)
    Ap[:n, :n] = Q
    xp = np.zeros(ct * 256, F)
    xp[:n] = x
    y = np.zeros(rt * tr)
    total = rt * ct
    start = [total * c // grid for c in range(grid + 1)]
    owner = np.searchsorted(start, np.arange(total), side="right") - 1
    for r in range(rt):
        rows = slice(tr * r, tr * r + tr)
        c = 0
        while c < ct:
            own = owner[r * ct + c]
            acc = np.zeros((tr, wc * 32, 2), F)
            while c < ct and owner[r * ct + c] == own:
                a = Ap[rows, 256 * c:256 * c + 256].reshape(tr, wc * 32, vec)
                xc = xp[256 * c:256 * c + 256].reshape(wc * 32, vec)
                for v in range(vec):
                    acc[:, :, v & 1] = _fma32(a[:, :, v], xc[:, v], acc[:, :, v & 1])
                c += 1
            s = (acc[:, :, 0] + acc[:, :, 1]).reshape(tr, wc, 32)
            while s.shape[2] > 1:
                h = s.shape[2] // 2
                s = s[:, :, :h] + s[:, :, h:]
            z = s[:, 0, 0]
            for w in range(1, wc):
                z = z + s[:, w, 0]
            y[rows] += z
    return y[:n].astype(F)


@pytest.mark.parametrize("dtype", [B.LS_BF16_IR, B.LS_FP8_IR, B.LS_F32_IR])
@pytest.mark.parametrize("n", [1024, 2000, 3000, 4000])
def test_error_of_the_fp32_formats(ctx, gpu, oracle, dtype, n):
    A = inputs.nonsym_matrix(n, seed=620 + n)
    raw = {B.LS_BF16_IR: torch.int16, B.LS_FP8_IR: torch.uint8, B.LS_F32_IR: torch.float32}[dtype]
    Q = torch.zeros((n, (n + 15) // 16 * 16), dtype=raw, device=gpu)[:, :n]
    scale = torch.zeros(n, dtype=torch.float32, device=gpu) if dtype == B.LS_FP8_IR else None
    assert B.ls_quantize(ctx, dtype, torch.from_numpy(A).to(gpu), Q, scale) == B.LS_OK
    x = inputs.solution(n, seed=621 + n).astype(F)
    y = torch.zeros(n, dtype=torch.float32, device=gpu)
    assert B.ls_gemv(ctx, dtype, Q, torch.from_numpy(x).to(gpu), y, scale) == B.LS_OK
    q = Q.cpu().numpy()
    if dtype == B.LS_BF16_IR:
        q = oracle.decode_bf16(q.view(np.uint16))
    elif dtype == B.LS_FP8_IR:
        q = oracle.decode_fp8(q)
    s = scale.cpu().numpy() if scale is not None else np.ones(n, F)
    ref = _fp64_product(q.astype(np.float64), x.astype(np.float64)) * s
    plain = np.linalg.norm(_plain_fp32(dtype, q.astype(F), x) * s - ref)
    assert np.linalg.norm(y.cpu().numpy() - ref) <= 1.05 * plain
