"""What a context keeps between calls, seen from outside: alternating between an
exactly symmetric A and one that differs from it in the last bit builds no graph
again, and the device time of a call that builds one does not contain the building."""
import time

import numpy as np
import pytest
import torch

from paper_1511_07207_gb300 import binding as B
from paper_1511_07207_gb300 import inputs

pytestmark = pytest.mark.gpu


def _median(f, reps=31):
    f()
    f()
    t = []
    for _ in range(reps):
        t0 = time.perf_counter()
        f()
        t.append(time.perf_counter() - t0)
    return sorted(t)[reps // 2]


@pytest.mark.parametrize("precision", [B.LS_F64, B.LS_BF16_IR])
def test_alternating_symmetry(ctx, gpu, precision):
    """Building a graph takes more than a call of one step; both orders make the same two calls."""
    n = 1024
    S = inputs.spd_matrix(n, 0.1, seed=650)
    N = S.copy()
    N[3, 0] = np.nextafter(N[3, 0], 9.0)
    b = torch.from_numpy(S @ inputs.solution(n, seed=651)).to(gpu)
    x = torch.zeros(n, dtype=torch.float64, device=gpu)
    o = B.make_opts(rtol=1e-10, max_iter=1, fused=0, precision=precision, inner_iters=1)
    mats = [torch.from_numpy(S).to(gpu), torch.from_numpy(N).to(gpu)]

    def call(A):
        assert B.ls_cg_solve(ctx, A, b, x, o)[0] == B.LS_NOT_CONVERGED

    apart = _median(lambda: call(mats[0])) + _median(lambda: call(mats[1]))

    def both():
        call(mats[0])
        call(mats[1])

    assert _median(both) <= 1.3 * apart
