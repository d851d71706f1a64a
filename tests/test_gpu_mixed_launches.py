"""info.launches of the mixed-precision solver counts every kernel: the same solve of a
symmetric A, and of one that differs from it in one bit, takes the same kernels but for the
packing that found the difference (packed twice, or packed, quantised and split)."""
import numpy as np
import pytest
import torch

from paper_1511_07207_gb300 import binding as B
from paper_1511_07207_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,extra", [(1023, 0), (1024, 1), (1100, 1)])
@pytest.mark.parametrize("precision", [B.LS_BF16_IR, B.LS_F32_IR])
def test_packing_is_counted(ctx, gpu, n, extra, precision):
    S = inputs.spd_matrix(n, 0.1, seed=670 + n)
    N = S.copy()
    N[n - 1, 0] = np.nextafter(N[n - 1, 0], 9.0)
    b = torch.from_numpy(S @ inputs.solution(n, seed=671)).to(gpu)
    o = B.make_opts(rtol=0.0, max_iter=2, precision=precision)
    count = []
    for A in (S, N):
        x = torch.zeros(n, dtype=torch.float64, device=gpu)
        total = B.ls_kernel_launches(ctx)
        st, info = B.ls_cg_solve(ctx, torch.from_numpy(A).to(gpu), b, x, o)
        assert st == B.LS_NOT_CONVERGED
        assert B.ls_kernel_launches(ctx) - total == info["launches"]
        count.append(info["launches"])
    assert count[1] == count[0] + extra
