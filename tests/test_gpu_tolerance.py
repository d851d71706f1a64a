"""One context, one system, another tolerance in every call: the loops that a context
keeps between calls hold no tolerance of an earlier call."""
import numpy as np
import pytest
import torch

from paper_1511_07207_gb300 import binding as B
from paper_1511_07207_gb300 import inputs

pytestmark = pytest.mark.gpu

CASES = {
    "cg": ("spd", B.ls_cg_solve, {"fused": 0}, 300),
    "cg_one_triangle": ("spd", B.ls_cg_solve, {"fused": 0}, 1100),
    "cg_native": ("spd", B.ls_cg_solve, {"f64_matvec": 1}, 300),
    "cg_fused": ("spd", B.ls_cg_solve, {}, 300),
    "gmres": ("nonsym", B.ls_gmres_solve, {"fused": 0}, 300),
    "gmres_fused": ("nonsym", B.ls_gmres_solve, {}, 300),
    "bicgstab": ("nonsym", B.ls_bicgstab_solve, {}, 300),
    "jacobi": ("nonsym", B.ls_jacobi_solve, {}, 300),
    "gauss_seidel": ("nonsym", B.ls_gauss_seidel_solve, {}, 300),
    "mixed_fcg": ("spd", B.ls_cg_solve, {"precision": B.LS_BF16_IR}, 300),
    "mixed_ir": ("spd", B.ls_cg_solve, {"precision": B.LS_F32_IR, "refine": B.LS_REFINE_IR}, 300),
    "block_cg": ("spd", B.ls_block_cg_solve, {}, 300),
    "block_cg_oleary": ("spd", B.ls_block_cg_solve, {"deflate": 0}, 300),
    "block_gmres": ("nonsym", B.ls_block_gmres_solve, {"restart": 20}, 300),
}


@pytest.mark.parametrize("name", list(CASES))
def test_each_call_has_its_own_tolerance(ctx, gpu, name):
    kind, solve, kw, n = CASES[name]
    A = inputs.spd_matrix(n, 0.1, seed=640) if kind == "spd" else inputs.nonsym_matrix(n, seed=641)
    s = 3 if "block" in name else 1
    Bm = A @ inputs.solution(n, seed=642, nrhs=s).reshape(n, s)
    Ad = torch.from_numpy(A).to(gpu)
    bd = torch.from_numpy(Bm.T.copy()).to(gpu).t() if s > 1 else torch.from_numpy(Bm[:, 0].copy()).to(gpu)
    seen = []
    for rtol in (1e-2, 1e-10, 1e-2):
        x = torch.zeros((s, n), dtype=torch.float64, device=gpu).t() if s > 1 else torch.zeros(n, dtype=torch.float64, device=gpu)
        st, info = solve(ctx, Ad, bd, x, B.make_opts(rtol=rtol, **kw))
        assert st == B.LS_OK
        R = Bm - A @ x.cpu().numpy().reshape(n, s)
        assert np.all(np.linalg.norm(R, axis=0) <= rtol * np.linalg.norm(Bm, axis=0))
        seen.append(info["iters"])
    assert seen[0] == seen[2] < seen[1]
