"""CG's product from one triangle of an exactly symmetric A (csrc/k_symv.cu).

Iterates at a fixed count, element by element against the oracle, at the
edges of its 128-row blocks and 64-row results (tolerance k kappa sqrt(n) 2^-48
max|x|, as for the other products in double-single arithmetic); one entry
that differs from its mirror image in the last bit, wherever it lies, takes the general
product (seen from the bytes of A per product); BF16 and FP32 storage; x0;
a strided A and a host A; NaN.
"""
import math

import numpy as np
import pytest
import torch

from paper_1511_07207_gb300 import binding as B
from paper_1511_07207_gb300 import inputs

pytestmark = pytest.mark.gpu


def _spd(n, seed, sigma=0.1):
    A = inputs.spd_matrix(n, sigma, seed=seed)
    assert np.array_equal(A, A.T)
    return A


def _cg(ctx, gpu, A, b, x0=None, **kw):
    Ad = torch.from_numpy(A).to(gpu) if isinstance(A, np.ndarray) else A
    xd = torch.from_numpy(np.zeros(len(b)) if x0 is None else x0.copy()).to(gpu)
    o = B.make_opts(fused=0, x0_given=int(x0 is not None), **kw)
    st, info = B.ls_cg_solve(ctx, Ad, torch.from_numpy(b).to(gpu), xd, o)
    return st, info, xd.cpu().numpy()


def _one_triangle(info, n, passes):
    return info["bytes_moved"] == passes * 4.0 * n * (n + 1.0)


@pytest.mark.parametrize("n", [1024, 1025, 1087, 1088, 1089, 1151, 1152, 1153, 1407, 2049])
def test_fixed_count_iterates(ctx, gpu, oracle, n):
    k = 6
    A = _spd(n, 500 + n)
    b = A @ inputs.solution(n, seed=n)
    ev = np.linalg.eigvalsh(A)
    st, info, x = _cg(ctx, gpu, A, b, rtol=1e-300, max_iter=k)
    ref = oracle.cg(A, b, rtol=1e-300, max_iter=k)
    assert st == B.LS_NOT_CONVERGED and info["iters"] == ref["iters"] == k
    assert _one_triangle(info, n, k + 1)
    tol = k * (ev[-1] / ev[0]) * math.sqrt(n) * 2.0 ** -48 * np.max(np.abs(ref["x"]))
    assert np.max(np.abs(x - ref["x"])) <= tol


@pytest.mark.parametrize("i,j", [(1, 0), (0, 1), (1099, 0), (1099, 1098), (64, 63), (127, 128), (1024, 130), (640, 700)])
def test_one_bit_from_symmetric(ctx, gpu, oracle, i, j):
    n = 1100
    A = _spd(n, 520)
    b = A @ inputs.solution(n, seed=521)
    A[i, j] = np.nextafter(A[i, j], 9.0)
    st, info, x = _cg(ctx, gpu, A, b, rtol=1e-10)
    assert st == B.LS_OK
    assert info["bytes_moved"] == (info["iters"] + 1) * 8.0 * n * n
    assert np.linalg.norm(oracle.residual(A, b, x)) <= 1e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("precision", [B.LS_BF16_IR, B.LS_F32_IR])
@pytest.mark.parametrize("n", [1024, 1089, 1500])
@pytest.mark.parametrize("refine", [B.LS_REFINE_FCG, B.LS_REFINE_IR])
def test_stored_formats(ctx, gpu, oracle, n, precision, refine):
    A = _spd(n, 540 + n)
    b = A @ inputs.solution(n, seed=541)
    kw = dict(rtol=1e-10, precision=precision, refine=refine, inner_rtol=1e-2 if refine == B.LS_REFINE_IR else 0.0)
    st, info, x = _cg(ctx, gpu, A, b, **kw)
    A2 = A.copy()
    A2[n - 1, 3] = np.nextafter(A2[n - 1, 3], 9.0)      # the general products
    st2, info2, x2 = _cg(ctx, gpu, A2, b, **kw)
    assert st == st2 == B.LS_OK
    assert info["bytes_moved"] < 0.75 * info2["bytes_moved"]
    assert np.linalg.norm(oracle.residual(A, b, x)) <= 1e-10 * np.linalg.norm(b)
    kap = np.linalg.cond(A)
    assert np.linalg.norm(x - x2) <= 4 * kap * 1e-10 * np.linalg.norm(x2)


def test_x0_strided_and_host_matrix(ctx, gpu, oracle):
    n = 1200
    A = _spd(n, 560)
    b = A @ inputs.solution(n, seed=561)
    st, info, x = _cg(ctx, gpu, A, b, rtol=1e-10)
    big = torch.zeros((n, n + 3), dtype=torch.float64, device=gpu)
    big[:, 1:n + 1] = torch.from_numpy(A).to(gpu)
    st2, info2, x2 = _cg(ctx, gpu, big[:, 1:n + 1], b, rtol=1e-10)
    xh = np.zeros(n)
    st3, info3 = B.ls_cg_solve(ctx, A, b, xh, B.make_opts(fused=0, rtol=1e-10))
    assert st == st2 == st3 == B.LS_OK
    assert np.array_equal(x, x2) and np.array_equal(x, xh)
    assert _one_triangle(info2, n, info2["iters"] + 1)
    x0 = inputs.solution(n, seed=561) + 1e-4
    st4, info4, x4 = _cg(ctx, gpu, A, b, x0=x0, rtol=1e-10)
    assert st4 == B.LS_OK and info4["iters"] < info["iters"]
    assert np.linalg.norm(oracle.residual(A, b, x4)) <= 1e-10 * np.linalg.norm(b)


def test_nan_and_indefinite(ctx, gpu):
    n = 1100
    A = _spd(n, 580)
    b = A @ inputs.solution(n, seed=581)
    N = A.copy()
    N[700, 20] = N[20, 700] = np.nan
    st, _, _ = _cg(ctx, gpu, N, b, rtol=1e-10)
    M = N.copy()
    M[700, 21] = np.nextafter(M[700, 21], 9.0)          # the general product's answer
    assert st == _cg(ctx, gpu, M, b, rtol=1e-10)[0]
    st, info, _ = _cg(ctx, gpu, -A, b, rtol=1e-10)
    assert st == B.LS_BREAKDOWN
