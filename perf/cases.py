"""The work that users of this library have it do, as cases that can be timed.

Each case is one pass through the public entry points of
``paper_1511_07207_gb300.binding`` on matrices that are resident in device
memory, as a program that keeps its systems on the GPU calls them.  The
matrices are the families of ``paper_1511_07207_gb300.inputs`` (SPD
G G^T/n + sigma I, nonsymmetric 2 I + G/(2 sqrt n), x* ~ U[-1, 1], b = A x*),
made on the GPU from the case's seed: the FP32 product G G^T is mirrored,
widened and scaled on both sides by FP64 factors near 1, so that A is exactly
symmetric and its entries have full FP64 mantissas.

Well-conditioned systems (sigma = 0.1, and the nonsymmetric family) are solved
to a relative residual of 1e-10; those with condition number about 4e3
(sigma = 1e-3) to 1e-12, where the residual also fixes the solution to about
1e-10.
"""
from __future__ import annotations

import math
import time

import torch

from paper_1511_07207_gb300 import binding as B

DEV = "cuda:0"

_SOLVE = {"cg": "ls_cg_solve", "mixed": "ls_cg_solve", "gmres": "ls_gmres_solve", "bicgstab": "ls_bicgstab_solve",
          "jacobi": "ls_jacobi_solve", "gauss_seidel": "ls_gauss_seidel_solve", "lu": "ls_lu_solve",
          "chol": "ls_chol_solve"}
_BLOCK = {"block_cg": "ls_block_cg_solve", "block_gmres": "ls_block_gmres_solve"}
_PRECISION = {"f64": B.LS_F64, "bf16": B.LS_BF16_IR, "f32": B.LS_F32_IR}
_SPD = ("cg", "mixed", "chol", "block_cg")


def listed():
    return [
        # a small system in a latency-bound loop (the smallest configuration: n = 512, cond about 40)
        {"name": "cg_512", "kind": "cg", "n": 512, "sigma": 0.1, "rtol": 1e-10},
        # the ordinary sizes of the paper's tables (n = 2000 ... 20000)
        {"name": "cg_4000", "kind": "cg", "n": 4000, "sigma": 0.1, "rtol": 1e-10},
        {"name": "gmres35_2000", "kind": "gmres", "n": 2000, "restart": 35, "rtol": 1e-10},
        {"name": "gauss_seidel_8000", "kind": "gauss_seidel", "n": 8000, "rtol": 1e-10},
        # the headline systems: A of 2 GiB, CG at cond about 4e3 to the accuracy gate and GMRES(50)
        {"name": "cg_16384", "kind": "cg", "n": 16384, "sigma": 1e-3, "rtol": 1e-12},
        {"name": "gmres50_16384", "kind": "gmres", "n": 16384, "restart": 50, "rtol": 1e-10},
        # mixed precision: BF16 storage of an 8 GiB matrix inside the FP64 flexible CG
        {"name": "mixed_bf16_32768", "kind": "mixed", "n": 32768, "sigma": 1e-3, "precision": "bf16", "rtol": 1e-12},
        # many independent systems at once: n log-uniform in [64, 2048], half SPD, 1..32 right-hand sides
        {"name": "batch_512", "kind": "batch", "count": 512, "lo": 64, "hi": 2048, "max_rhs": 32, "rtol": 1e-10},
        # a burst of requests on resident matrices, n log-uniform in [128, 8192], 1..8 right-hand sides
        {"name": "serve_96", "kind": "serve", "count": 96, "pool": 16, "lo": 128, "hi": 8192, "max_rhs": 8,
         "rtol": 1e-10},
        # several right-hand sides of one large system
        {"name": "block_cg_8192x8", "kind": "block_cg", "n": 8192, "s": 8, "sigma": 1e-3, "rtol": 1e-12},
        # the direct methods: LU as one solve of a large system, Cholesky as a factorization that is kept
        {"name": "lu_8192", "kind": "lu", "n": 8192},
        {"name": "chol_factor_3500", "kind": "chol", "n": 3500, "sigma": 0.1, "factor": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cg", "cg", "gmres", "gmres", "bicgstab", "jacobi", "gauss_seidel", "mixed", "block_cg",
                       "block_gmres", "batch", "serve", "lu", "chol"])
    if kind == "batch":
        hi = _log_int(rng, 128, 2048)
        return {"kind": kind, "count": _log_int(rng, 4, 512), "lo": 64, "hi": hi, "max_rhs": rng.randint(1, 32),
                "rtol": 1e-10}
    if kind == "serve":
        return {"kind": kind, "count": _log_int(rng, 8, 96), "pool": rng.randint(4, 16), "lo": 128,
                "hi": _log_int(rng, 512, 8192), "max_rhs": rng.randint(1, 8), "rtol": 1e-10}
    if kind in ("lu", "chol"):
        case = {"kind": kind, "n": _log_int(rng, 500, 8192 if kind == "chol" else 7000), "factor": rng.random() < 0.5}
        if kind == "chol":
            case["sigma"] = 0.1
        return case
    if kind in ("block_cg", "block_gmres"):
        case = {"kind": kind, "n": _log_int(rng, 500, 8192), "s": rng.randint(2, 16), "rtol": 1e-10}
        if kind == "block_cg":
            case["sigma"] = 0.1
        else:
            case["restart"] = 10
        return case
    if kind == "mixed":
        return {"kind": kind, "n": _log_int(rng, 2000, 32768), "sigma": 1e-3,
                "precision": rng.choice(["bf16", "bf16", "f32"]), "rtol": 1e-12}
    n = _log_int(rng, 100, 16384)
    if kind == "cg":
        sigma = rng.choice([0.1, 1e-3])
        return {"kind": kind, "n": n, "sigma": sigma, "rtol": 1e-10 if sigma == 0.1 else 1e-12,
                "f64_matvec": rng.random() < 0.15}
    if kind == "gmres":
        return {"kind": kind, "n": n, "restart": rng.choice([10, 30, 35, 50]), "rtol": 1e-10,
                "f64_matvec": rng.random() < 0.15}
    return {"kind": kind, "n": n, "rtol": 1e-10}


# ---- inputs ---------------------------------------------------------------

def _spd(n, sigma, g):
    G = torch.randn(n, n, dtype=torch.float32, device=DEV, generator=g)
    S = G @ G.t()
    del G
    S = torch.triu(S) + torch.triu(S, 1).t()
    A = S.double()
    del S
    d = 1.0 + 0.01 * torch.rand(n, dtype=torch.float64, device=DEV, generator=g)
    A.mul_(torch.outer(d, d)).div_(n)
    A.diagonal().add_(sigma)
    return A


def _nonsym(n, g):
    A = torch.randn(n, n, dtype=torch.float64, device=DEV, generator=g)
    A.mul_(0.5 / math.sqrt(n))
    A.diagonal().add_(2.0)
    return A


def _columns(n, s):
    """n x s FP64, each column contiguous."""
    return torch.zeros(s, n, dtype=torch.float64, device=DEV).t()


def _rhs(A, s, g):
    X = 2.0 * torch.rand(s, A.shape[0], dtype=torch.float64, device=DEV, generator=g).t() - 1.0
    return (X.t() @ A.t()).contiguous().t()


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _systems(case, seed):
    """The systems of a batch or a burst: [(kind, A, B)].  The sizes are a
    fixed low-discrepancy sequence over the range, so that the work does not
    depend on the seed."""
    g = _generator(seed)
    lo, hi, count = case["lo"], case["hi"], case["count"]

    def size(i, of):
        u = (0.5 + i * 0.6180339887498949) % 1.0 if of > 1 else 0.5
        return int(round(lo * (hi / lo) ** u))

    def rhs_count(i):
        return 1 + int(case["max_rhs"] * ((0.25 + i * 0.7548776662466927) % 1.0))

    pool = case.get("pool", count)
    mats = []
    for i in range(pool):
        n = size(i, pool)
        mats.append(("spd", _spd(n, 0.1, g)) if i % 2 == 0 else ("nonsym", _nonsym(n, g)))
    got = []
    for i in range(count):
        kind, A = mats[(i * 5 + i // pool) % pool if pool < count else i]
        got.append((kind, A, _rhs(A, rhs_count(i), g)))
    return got


class _State:
    """One user's handle on the library with its resident inputs and outputs."""

    def __init__(self, case):
        self.case = case
        self.srv = None
        self.ctx = B.ls_create(0, torch.cuda.current_stream(torch.device(DEV)))

    def close(self):
        if self.srv is not None:
            B.ls_server_stop(self.srv)
            self.srv = None
        if self.ctx is not None:
            B.ls_destroy(self.ctx)
            self.ctx = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def _single(case, seed):
    """A and the right-hand side (a vector, or an n x s block) of a case with one matrix."""
    g = _generator(seed)
    A = _spd(case["n"], case["sigma"], g) if case["kind"] in _SPD else _nonsym(case["n"], g)
    Bm = _rhs(A, case.get("s", 1), g)
    return A, (Bm if "s" in case else Bm[:, 0].contiguous())


def prepare(case, seed):
    st = _State(case)
    kind = case["kind"]
    if kind in ("batch", "serve"):
        st.systems = []
        parts = _systems(case, seed)
        sizes = [b.numel() for _, _, b in parts]
        # one buffer for all solutions, each system's block column-major in it
        st.out = torch.zeros(sum(sizes), dtype=torch.float64, device=DEV)
        at = 0
        for (what, A, b), size in zip(parts, sizes):
            X = st.out[at:at + size].view(b.shape[1], b.shape[0]).t()
            at += size
            opts = B.make_opts(rtol=case["rtol"], restart=30)
            st.systems.append(B.make_system(B.LS_METHOD_CG if what == "spd" else B.LS_METHOD_GMRES, A, b, X, opts))
        if kind == "serve":
            st.srv = B.ls_server_start(st.ctx, 24 << 30, max_slots=64, step_iters=8)
        return st
    st.A, st.b = _single(case, seed)
    st.opts = B.make_opts(rtol=case.get("rtol"), restart=case.get("restart"),
                          precision=_PRECISION[case.get("precision", "f64")],
                          f64_matvec=int(case.get("f64_matvec", False)))
    n = case["n"]
    st.x = _columns(n, case["s"]) if "s" in case else torch.zeros(n, dtype=torch.float64, device=DEV)
    if case.get("factor"):
        st.F = torch.zeros(n, n, dtype=torch.float64, device=DEV)
        st.ipiv = torch.zeros(n, dtype=torch.int32, device=DEV)
    return st


def _burst(st):
    """Submit every request, then wait for the tickets."""
    open_, worst = [], 0
    for s in st.systems:
        status, ticket = B.ls_server_submit(st.srv, s)
        if status != B.LS_OK:
            raise RuntimeError(B.ls_strerror(status))
        open_.append(ticket)
    while open_:
        still = []
        for t in open_:
            status, done, info = B.ls_server_poll(st.srv, t)
            if status < 0:
                raise RuntimeError(B.ls_strerror(status))
            if done:
                worst = max(worst, abs(info["status"]))
            else:
                still.append(t)
        open_ = still
        if open_:
            time.sleep(20e-6)
    return worst


def run(state):
    kind = state.case["kind"]
    if kind == "batch":
        status, _ = B.ls_batch_solve(state.ctx, state.systems)
        return {"status": status, "x": state.out}
    if kind == "serve":
        return {"status": _burst(state), "x": state.out}
    if state.case.get("factor"):
        if kind == "lu":
            status = B.ls_lu_factor(state.ctx, state.A, state.b, state.F, state.ipiv, state.x)
            return {"status": status, "lu": state.F, "ipiv": state.ipiv, "y": state.x}
        status, _ = B.ls_chol_factor(state.ctx, state.A, state.b, state.F, state.x)
        return {"status": status, "l": state.F, "y": state.x}
    solve = getattr(B, _BLOCK.get(kind) or _SOLVE[kind])
    status, _ = solve(state.ctx, state.A, state.b, state.x, state.opts)
    return {"status": status, "x": state.x}


# ---- work and exact results -------------------------------------------------

def _steps(case):
    """About how many products with A the method cannot do without at this condition and tolerance."""
    kind, rtol = case["kind"], case.get("rtol", 1e-10)
    if kind in _SPD:
        return max(1.0, 0.5 * math.sqrt(4.0 / case["sigma"] + 1.0) * math.log(2.0 / rtol) * 0.8)
    return max(1.0, math.log(1.0 / rtol) / math.log(4.0))


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        lo, hi = math.log(case["lo"]), math.log(case["hi"])
        n2 = (math.exp(2 * hi) - math.exp(2 * lo)) / (2 * (hi - lo)) if hi > lo else math.exp(2 * lo)
        s = (1 + case["max_rhs"]) / 2
        steps = (_steps({"kind": "cg", "sigma": 0.1}) + _steps({"kind": "gmres"})) / 2
        mats = min(case["count"], case.get("pool", case["count"]))
        return {"bytes": 8.0 * n2 * mats, "flops": 2.0 * n2 * case["count"] * s * steps}
    n = case["n"]
    if kind == "lu":
        return {"bytes": 8.0 * n * n * (2 if case.get("factor") else 1), "flops": 2.0 * n ** 3 / 3}
    if kind == "chol":
        return {"bytes": (12.0 if case.get("factor") else 4.0) * n * n, "flops": n ** 3 / 3.0}
    s = case.get("s", 1)
    return {"bytes": 8.0 * n * n + 16.0 * n * s, "flops": 2.0 * n * n * s * _steps(case)}


def _exact_solve(A, b):
    """x = A^-1 b by LAPACK-style elimination in FP64 and one step of refinement."""
    lu, piv = torch.linalg.lu_factor(A)
    b2 = b if b.dim() == 2 else b[:, None]
    x = torch.linalg.lu_solve(lu, piv, b2)
    x = x + torch.linalg.lu_solve(lu, piv, b2 - A @ x)
    return x if b.dim() == 2 else x[:, 0]


def _exact_spd(A, b):
    """x = A^-1 b by conjugate gradients in FP64 down to rounding (too large to factor)."""
    x = torch.zeros_like(b)
    tiny = 1e-15 * float(b.norm())
    for _ in range(3):
        r = b - A @ x
        p, rho = r.clone(), float(r @ r)
        for _ in range(2000):
            if math.sqrt(rho) <= tiny:
                break
            q = A @ p
            alpha = rho / float(p @ q)
            x = x + alpha * p
            r = r - alpha * q
            new = float(r @ r)
            p = r + (new / rho) * p
            rho = new
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        parts = []
        for _, A, b in _systems(case, seed):
            parts.append(_exact_solve(A, b).t().reshape(-1))
        return {"status": 0, "x": torch.cat(parts)}
    A, b = _single(case, seed)
    if case.get("factor"):
        if kind == "chol":
            L = torch.linalg.cholesky(A)
            return {"status": 0, "l": L, "y": torch.linalg.solve_triangular(L, b[:, None], upper=False)[:, 0]}
        lu, piv = torch.linalg.lu_factor(A)
        pb = torch.linalg.lu(A)[0].t() @ b
        y = torch.linalg.solve_triangular(lu, pb[:, None], upper=False, unitriangular=True)[:, 0]
        return {"status": 0, "lu": lu, "ipiv": (piv - 1).to(torch.int32), "y": y}
    if case["n"] > 20000:
        return {"status": 0, "x": _exact_spd(A, b)}
    return {"status": 0, "x": _exact_solve(A, b)}
