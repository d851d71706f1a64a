"""The direct methods' panel kernels where they can go wrong: rows spread over one
and several CTAs (64 rows each below n = 3073), pivots far from their row, columns
with no comparable candidate (NaN), a zero pivot inside a panel,
and a short last panel.  Bit for bit against the oracle."""
import numpy as np
import pytest
import torch

from paper_1511_07207_gb300 import binding as B
from paper_1511_07207_gb300 import inputs

pytestmark = pytest.mark.gpu


def _lu(ctx, gpu, A, b):
    n = A.shape[0]
    LU = torch.zeros((n, n), dtype=torch.float64, device=gpu)
    ipiv = torch.zeros(n, dtype=torch.int32, device=gpu)
    y = torch.zeros(n, dtype=torch.float64, device=gpu)
    st = B.ls_lu_factor(ctx, torch.from_numpy(np.ascontiguousarray(A)).to(gpu), torch.from_numpy(b).to(gpu), LU, ipiv, y)
    return st, LU.cpu().numpy(), ipiv.cpu().numpy(), y.cpu().numpy()


@pytest.mark.parametrize("n", [31, 32, 64, 65, 129, 200, 513])
def test_lu_pivots_far_away(ctx, gpu, oracle, n):
    A = inputs.nonsym_matrix(n, seed=400 + n, shift=0.0, scale=1.0)
    A *= np.linspace(1.0, 50.0, n)[:, None]        # the last rows win
    b = inputs.solution(n, seed=401 + n)
    st, LU, ipiv, y = _lu(ctx, gpu, A, b)
    LUr, ipr, yr, str_ = oracle.ge_factor(A, b)
    assert st == str_ == B.LS_OK
    assert np.array_equal(ipiv, ipr) and np.array_equal(LU, LUr) and np.array_equal(y, yr)


@pytest.mark.parametrize("col", [0, 5, 33, 69])
def test_lu_columns_without_a_finite_candidate(ctx, gpu, oracle, col):
    n = 70
    A = inputs.nonsym_matrix(n, seed=410, shift=0.0, scale=1.0)
    A[:, col] = np.nan
    b = inputs.solution(n, seed=411)
    st, LU, ipiv, y = _lu(ctx, gpu, A, b)
    LUr, ipr, yr, str_ = oracle.ge_factor(A, b)
    assert st == str_
    assert np.array_equal(ipiv, ipr)
    np.testing.assert_array_equal(LU, LUr)
    np.testing.assert_array_equal(y, yr)


def test_lu_zero_pivot_then_a_good_system(ctx, gpu, oracle):
    n = 150
    A = inputs.nonsym_matrix(n, seed=420, shift=0.0, scale=1.0)
    b = inputs.solution(n, seed=421)
    S = A.copy()
    S[:, 40] = 0.0                                  # singular at step 40, inside the second panel
    assert _lu(ctx, gpu, S, b)[0] == B.LS_BREAKDOWN == oracle.ge_factor(S, b)[3]
    st, LU, ipiv, y = _lu(ctx, gpu, A, b)
    LUr, ipr, yr, _ = oracle.ge_factor(A, b)
    assert st == B.LS_OK
    assert np.array_equal(ipiv, ipr) and np.array_equal(LU, LUr) and np.array_equal(y, yr)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 40, 41, 1215, 1250])
def test_cholesky_rows_per_cta(ctx, gpu, oracle, n):
    """8 rows a CTA up to 152 of them (n + 1 - 32 = 1216 rows), then more."""
    A = inputs.spd_matrix(n, 0.1, seed=430 + n)
    b = inputs.solution(n, seed=431 + n)
    L = torch.zeros((n, n), dtype=torch.float64, device=gpu)
    y = torch.zeros(n, dtype=torch.float64, device=gpu)
    st, _ = B.ls_chol_factor(ctx, torch.from_numpy(A).to(gpu), torch.from_numpy(b).to(gpu), L, y)
    Lr, str_ = oracle.chol_factor(A)
    assert st == str_ == B.LS_OK
    assert np.array_equal(L.cpu().numpy(), Lr) and np.array_equal(y.cpu().numpy(), oracle.chol_forward(Lr, b))
