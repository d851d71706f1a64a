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
