"""The two Gram-Schmidt passes of the general GMRES form exchange their partial
sums through slots of their own: repeated solves of a fixed number of steps
give the same bits, and the oracle's iterate, on one, several and all CTAs."""
import numpy as np
import pytest
import torch

from paper_1511_07207_gb300 import binding as B
from paper_1511_07207_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reorth", [0, 1])
@pytest.mark.parametrize("n", [30, 65, 2001, 5000])
def test_second_pass_is_deterministic(ctx, gpu, oracle, n, reorth):
    A = inputs.nonsym_matrix(n, seed=500 + n)
    b = A @ inputs.solution(n, seed=501 + n)
    Ad, bd = torch.from_numpy(A).to(gpu), torch.from_numpy(b).to(gpu)
    opts = B.make_opts(rtol=0.0, max_iter=10, restart=30, reorth=reorth, fused=0)
    first = None
    for _ in range(200):
        x = torch.full((n,), np.nan, dtype=torch.float64, device=gpu)
        st, info = B.ls_gmres_solve(ctx, Ad, bd, x, opts)
        assert st == B.LS_NOT_CONVERGED and info["iters"] == 10
        if first is None:
            first = x
        assert torch.equal(x, first)
    ref = oracle.gmres(A, b, m=30, rtol=0.0, max_iter=10)
    # both are the minimiser over the same Krylov space
    assert np.linalg.norm(first.cpu().numpy() - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])


@pytest.mark.parametrize("n", [64, 2000])
def test_zero_right_side_with_x0_makes_no_product(ctx, gpu, n):
    """b = 0 is solved by x = 0 whatever A holds: an infinity or a NaN in A is not looked at."""
    A = inputs.nonsym_matrix(n, seed=510)
    A[3, 5], A[n - 1, 0] = np.inf, np.nan
    x = torch.from_numpy(inputs.solution(n, seed=511)).to(gpu)
    st, info = B.ls_gmres_solve(ctx, torch.from_numpy(A).to(gpu), torch.zeros(n, dtype=torch.float64, device=gpu), x,
                                B.make_opts(x0_given=1, fused=0))
    assert st == B.LS_OK and info["iters"] == 0 and info["true_rel_res"] == 0.0
    assert not x.any()
    assert info["bytes_moved"] == 0.0


@pytest.mark.parametrize("rtol", [1e-10, 1e-3])
def test_cycles_from_x0(ctx, gpu, oracle, rtol):
    """Several cycles from a given x0, and an x0 that already passes."""
    n = 300
    A = inputs.restart_matrix(n, seed=512)
    xs = inputs.solution(n, seed=513)
    b = A @ xs
    x0 = xs + (1e-6 if rtol > 1e-6 else 0.5) * inputs.solution(n, seed=514)
    x = torch.from_numpy(x0).to(gpu)
    st, info = B.ls_gmres_solve(ctx, torch.from_numpy(A).to(gpu), torch.from_numpy(b).to(gpu), x,
                                B.make_opts(x0_given=1, fused=0, rtol=rtol, restart=5, max_iter=20000))
    ref = oracle.gmres(A, b, m=5, rtol=rtol, max_iter=20000, x0=x0)
    assert st == B.LS_OK == ref["status"]
    assert np.linalg.norm(oracle.residual(A, b, x.cpu().numpy())) <= rtol * np.linalg.norm(b)
    assert abs(info["iters"] - ref["iters"]) <= 0.1 * ref["iters"] + 3
    if rtol > 1e-6:
        assert info["iters"] == 0 and np.array_equal(x.cpu().numpy(), x0)
