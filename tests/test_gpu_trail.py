"""The direct methods' trailing update forms its products on the integer pipes
(csrc/ls_rank.cuh).  Factors bit for bit against the oracle where that can
go wrong: edges of the 32 x 32 tiles, products that are exact ties, zeros and
exponents outside the integer form's range (a tile of them, or one element of
a tile)."""
import numpy as np
import pytest
import torch

from paper_1511_07207_gb300 import binding as B
from paper_1511_07207_gb300 import inputs

pytestmark = pytest.mark.gpu


def _odd27(r, shape):
    """Odd integers of 27 bits: the product of two has 53 or 54 bits, and with 54 its rounding is a tie."""
    return (r.integers(1 << 25, 1 << 26, shape) * 2 + 1).astype(np.float64)


def _matrix(n, kind):
    r = np.random.default_rng(1000 + n)
    A = inputs.nonsym_matrix(n, seed=300 + n, shift=0.0, scale=1.0)
    if kind == "ties":            # step 0: pivot 1, l_i0 = odd 2^-28, u_0j = odd 2^-20
        A[:, 0] = _odd27(r, n) * 2.0 ** -28
        A[0, :] = _odd27(r, n) * 2.0 ** -20
        A[0, 0] = 1.0
    elif kind == "zeros":
        A[r.random((n, n)) < 0.3] = 0.0
        A[np.diag_indices(n)] += 4.0
    elif kind == "range":         # rows and columns of very different scales
        A *= 2.0 ** r.integers(-400, 401, n)[:, None]
        A *= 2.0 ** r.integers(-400, 401, n)[None, :]
    elif kind == "one":           # a subnormal and a zero among ordinary entries
        A[n - 1, n - 1] = 5e-310
        A[n // 2, n - 2] = 0.0
        A[3, n - 1] = 1e-200
    return A


@pytest.mark.parametrize("kind", ["plain", "ties", "zeros", "range", "one"])
@pytest.mark.parametrize("n", [33, 63, 64, 65, 96, 97, 131, 300])
def test_lu_trailing_update_bits(ctx, gpu, oracle, n, kind):
    A = _matrix(n, kind)
    b = inputs.solution(n, seed=n)
    LU = torch.zeros((n, n), dtype=torch.float64, device=gpu)
    ipiv = torch.zeros(n, dtype=torch.int32, device=gpu)
    y = torch.zeros(n, dtype=torch.float64, device=gpu)
    st = B.ls_lu_factor(ctx, torch.from_numpy(A).to(gpu), torch.from_numpy(b).to(gpu), LU, ipiv, y)
    LUr, ipr, yr, str_ = oracle.ge_factor(A, b)
    assert st == str_ == B.LS_OK
    assert np.array_equal(ipiv.cpu().numpy(), ipr)
    assert np.array_equal(LU.cpu().numpy().view(np.uint64), LUr.view(np.uint64))
    assert np.array_equal(y.cpu().numpy().view(np.uint64), yr.view(np.uint64))


@pytest.mark.parametrize("kind", ["plain", "ties", "zeros", "range"])
@pytest.mark.parametrize("n", [33, 63, 64, 65, 96, 97, 131, 300])
def test_cholesky_trailing_update_bits(ctx, gpu, oracle, n, kind):
    r = np.random.default_rng(2000 + n)
    A = inputs.spd_matrix(n, 0.1, seed=310 + n)
    if kind == "ties":            # step 0: pivot 1, so l_i0 l_j0 = odd odd 2^-64
        A[np.diag_indices(n)] += 4.0
        A[:, 0] = _odd27(r, n) * 2.0 ** -32
        A[0, :] = A[:, 0]
        A[0, 0] = 1.0
    elif kind == "zeros":
        M = np.triu(r.random((n, n)) < 0.3, 1)
        A[M | M.T] = 0.0
        A[np.diag_indices(n)] += 4.0 + n / 16.0
    elif kind == "range":
        d = 2.0 ** r.integers(-300, 301, n)
        A = A * d[:, None] * d[None, :]
    b = inputs.solution(n, seed=n)
    L = torch.zeros((n, n), dtype=torch.float64, device=gpu)
    y = torch.zeros(n, dtype=torch.float64, device=gpu)
    st, step = B.ls_chol_factor(ctx, torch.from_numpy(A).to(gpu), torch.from_numpy(b).to(gpu), L, y)
    Lr, str_ = oracle.chol_factor(A)[:2]
    assert st == str_ == B.LS_OK and step == -1
    assert np.array_equal(L.cpu().numpy().view(np.uint64), Lr.view(np.uint64))
    assert np.array_equal(y.cpu().numpy().view(np.uint64), oracle.chol_forward(Lr, b).view(np.uint64))
