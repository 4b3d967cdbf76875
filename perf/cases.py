"""The workloads whose speed this repository tracks.

Each case is one call, or one pair of calls, that a program linked against the
solver makes: generating a system, factoring it, refining with factors it
keeps, solving a batch of small systems, checking a residual.  Systems are
n x n fp64, uniform in (-0.5, 0.5) with the diagonal of a strictly row
diagonally dominant matrix, the class the method is defined on.

Kinds:
  generate   api.generate: the matrix and right-hand sides on the device
  factor     api.Solver.factor: cast and low-precision LU without pivoting
  refine     api.Solver.solve: GMRES-IR with factors that the program keeps
  solve      api.Solver.__call__: factor and refine in one call
  batch      api.factor_batched + api.solve_ir_batched over uneven systems
  residual   capi.hpmxp_residual_vector: r = b - A x in fp64
"""
from __future__ import annotations

import math
import random

import torch

from paper_2509_19618_gb300 import api, capi

DEV = "cuda"
PRECS = {"bf16": capi.BF16, "fp16": capi.FP16, "fp8": capi.FP8_E4M3, "bf16_trail32": capi.BF16_TRAIL32}


def listed():
    return [
        # A benchmark run builds its system on the device first.
        {"name": "generate_16384", "kind": "generate", "n": 16384, "nrhs": 1, "diag": capi.DIAG_DOMINANT},
        # A small dense system, not a multiple of the block: all launches and the diagonal-block chain.
        {"name": "factor_small_ragged", "kind": "factor", "n": 1000, "prec": "bf16", "nb": 128},
        # A mid-size system at the middle update depth, odd order, IEEE half factors.
        {"name": "factor_mid_fp16", "kind": "factor", "n": 5001, "prec": "fp16", "nb": 256},
        # The headline size: BF16 factors, deepest update.
        {"name": "factor_large_bf16", "kind": "factor", "n": 32768, "prec": "bf16", "nb": 512},
        # The E4M3 trailing update with per-tile scales.
        {"name": "factor_fp8", "kind": "factor", "n": 16384, "prec": "fp8", "nb": 512},
        # The smallest refinement: one right-hand side, fp32 preconditioner; latency of every step counts.
        {"name": "refine_small", "kind": "refine", "n": 1024, "nrhs": 1, "prec": "bf16", "nb": 128, "fp32": 1},
        # A request with the most right-hand sides that one call takes.
        {"name": "refine_multi", "kind": "refine", "n": 8192, "nrhs": 8, "prec": "bf16", "nb": 256, "fp32": 1},
        # The headline refinement: fp32 preconditioner, fp64 products.
        {"name": "refine_large", "kind": "refine", "n": 32768, "nrhs": 1, "prec": "bf16", "nb": 512, "fp32": 1},
        # The library's defaults: every operator of the refinement in fp64, two right-hand sides.
        {"name": "refine_fp64", "kind": "refine", "n": 4096, "nrhs": 2, "prec": "bf16", "nb": 256, "fp32": 0},
        # A whole solve with balancing, three right-hand sides, odd order, FP16 factors.
        {"name": "solve_balanced", "kind": "solve", "n": 9001, "nrhs": 3, "prec": "fp16", "nb": 256, "fp32": 1,
         "balance": True},
        # One batch of the serving path: uneven systems, 1 to 8 right-hand sides each.
        {"name": "batch_serving", "kind": "batch", "count": 24, "lo": 256, "hi": 4096, "mix": 7, "prec": "bf16",
         "fp32": 1},
        # Checking solutions computed elsewhere: the fp64 residual of a few vectors.
        {"name": "residual_16384", "kind": "residual", "n": 16384, "nrhs": 4},
    ]


def _log_uniform(rng: random.Random, lo: float, hi: float) -> int:
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng: random.Random):
    kind = rng.choice(["generate", "factor", "factor", "refine", "refine", "refine", "solve", "batch", "residual"])
    if kind == "generate":
        return {"kind": kind, "n": _log_uniform(rng, 256, 24000), "nrhs": rng.randint(1, 8),
                "diag": rng.choice([capi.DIAG_DOMINANT, capi.DIAG_SQRTN, capi.DIAG_DOMINANT])}
    if kind == "factor":
        nb = rng.choice([128, 256, 512])
        return {"kind": kind, "n": _log_uniform(rng, 256, 24000), "prec": rng.choice(list(PRECS)), "nb": nb}
    if kind == "refine":
        return {"kind": kind, "n": _log_uniform(rng, 256, 20000), "nrhs": rng.randint(1, 8),
                "prec": rng.choice(["bf16", "fp16", "fp8"]), "nb": rng.choice([128, 256, 512]),
                "fp32": rng.choice([1, 1, 0])}
    if kind == "solve":
        return {"kind": kind, "n": _log_uniform(rng, 256, 20000), "nrhs": rng.randint(1, 8),
                "prec": rng.choice(["bf16", "fp16", "bf16_trail32"]), "nb": rng.choice([128, 256, 512]),
                "fp32": rng.choice([1, 1, 0]), "balance": rng.random() < 0.4}
    if kind == "batch":
        lo = _log_uniform(rng, 200, 900)
        return {"kind": kind, "count": rng.randint(4, 30), "lo": lo, "hi": lo * rng.randint(2, 5),
                "mix": rng.randint(1, 10**6), "prec": rng.choice(["bf16", "fp16"]), "fp32": 1}
    return {"kind": kind, "n": _log_uniform(rng, 256, 30000), "nrhs": rng.randint(1, 8)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rng(seed: int) -> torch.Generator:
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _dominant(n: int, g: torch.Generator) -> torch.Tensor:
    """Column major n x n as a (columns, ld) tensor: entry (i, j) at [j, i]."""
    s = torch.empty((n, api._round_up(n, 8)), dtype=torch.float64, device=DEV)
    s.uniform_(-0.5, 0.5, generator=g)
    v = s[:, :n]
    rows = torch.zeros(n, dtype=torch.float64, device=DEV)
    for j0 in range(0, n, 4096):   # in slabs: no second matrix-sized array
        rows += v[j0:j0 + 4096].abs().sum(dim=0)
    d = v.diagonal()
    d.copy_(rows - d.abs() + 1.0)
    return s


def _vectors(n: int, k: int, g: torch.Generator) -> torch.Tensor:
    s = torch.empty((k, api._round_up(n, 8)), dtype=torch.float64, device=DEV)
    s.uniform_(-0.5, 0.5, generator=g)
    return s


def _sizes(case):
    r = random.Random(case["mix"])
    return [(_log_uniform(r, case["lo"], case["hi"]), r.randint(1, 8)) for _ in range(case["count"])]


def _params(case):
    # an fp32 preconditioner gains nothing past its own accuracy in one cycle: inner tolerance 1e-5
    return api.ir_params(precond_fp32=1, inner_tol=1e-5) if case["fp32"] else api.ir_params()


def prepare(case, seed):
    kind = case["kind"]
    g = _rng(seed)
    if kind == "generate":
        return {"case": case, "seed": int(seed)}
    if kind == "batch":
        As, bs = [], []
        for n, k in _sizes(case):
            As.append(api.ColMajor(_dominant(n, g), n, n))
            bs.append(api.ColMajor(_vectors(n, k, g), n, k))
        dt = api.factor_storage_dtype(PRECS[case["prec"]])
        return {"case": case, "A": As, "b": bs, "LU": [api.ColMajor.empty(A.rows, A.rows, dt, DEV) for A in As],
                "x": [api.ColMajor.empty(b.rows, b.cols, torch.float64, DEV) for b in bs], "params": _params(case)}
    n = case["n"]
    A = api.ColMajor(_dominant(n, g), n, n)
    if kind == "residual":
        k = case["nrhs"]
        return {"case": case, "A": A, "x": api.ColMajor(_vectors(n, k, g), n, k),
                "b": api.ColMajor(_vectors(n, k, g), n, k), "r": api.ColMajor.empty(n, k, torch.float64, DEV),
                "ws": api.workspace(capi.hpmxp_residual_workspace(n, k), DEV)}
    k = case.get("nrhs", 1)
    params = _params(case) if "fp32" in case else None
    solver = api.Solver(n, k, PRECS[case["prec"]], case["nb"], DEV, params, balance=bool(case.get("balance", False)))
    st = {"case": case, "A": A, "solver": solver}
    if kind != "factor":
        st["b"] = api.ColMajor(_vectors(n, k, g), n, k)
    if kind == "refine":
        solver.factor(A)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "generate":
        A, b = api.generate(case["n"], seed=state["seed"], diag=case["diag"], nrhs=case["nrhs"], device=DEV)
        return {"A": A.storage[:, : A.rows], "b": b.storage[:, : b.rows]}
    if kind == "batch":
        prec = PRECS[case["prec"]]
        api.factor_batched(state["A"], prec, state["LU"])
        api.solve_ir_batched(state["A"], state["LU"], state["b"], prec, state["params"], state["x"])
        return {"LU": [m.storage[:, : m.rows] for m in state["LU"]], "x": [m.storage[:, : m.rows] for m in state["x"]]}
    if kind == "residual":
        A, x, b, r, ws = (state[k] for k in ("A", "x", "b", "r", "ws"))
        capi.hpmxp_residual_vector(A.rows, A.ptr, A.ld, x.ptr, x.ld, b.ptr, b.ld, x.cols, r.ptr, r.ld, ws.data_ptr(),
                                   ws.numel(), api.stream_handle())
        return {"r": r.storage[:, : r.rows]}
    solver, A = state["solver"], state["A"]
    if kind == "factor":
        LU = solver.factor(A)
        return {"LU": LU.storage[:, : LU.rows]}
    if kind == "refine":
        x, _, _ = solver.solve(A, state["b"])
        return {"x": x.storage[:, : x.rows]}
    x, _, _ = solver(A, state["b"])
    return {"LU": solver.LU.storage[:, : A.rows], "x": x.storage[:, : x.rows]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _factor_work(n):
    return 10.0 * n * n, 2.0 / 3.0 * n**3           # A read, factors written


def _refine_work(n, k):
    return 10.0 * n * n + 16.0 * n * k, 4.0 * n * n * k   # A and factors read; one solve and one residual


def work(case):
    kind = case["kind"]
    if kind == "generate":
        n = case["n"]
        return {"bytes": 8.0 * n * n + 8.0 * n * case["nrhs"], "flops": 0.0}
    if kind == "batch":
        w = [tuple(map(sum, zip(_factor_work(n), _refine_work(n, k)))) for n, k in _sizes(case)]
        return {"bytes": sum(b for b, _ in w), "flops": sum(f for _, f in w)}
    n, k = case["n"], case.get("nrhs", 1)
    if kind == "residual":
        return {"bytes": 8.0 * n * n + 24.0 * n * k, "flops": 2.0 * n * n * k}
    if kind == "factor":
        b, f = _factor_work(n)
    elif kind == "refine":
        b, f = _refine_work(n, k)
    else:
        (b, f), (b2, f2) = _factor_work(n), _refine_work(n, k)
        b, f = b + b2, f + f2
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from torch alone
# ---------------------------------------------------------------------------
_MUL, _INC, _M64 = 6364136223846793005, 1442695040888963407, (1 << 64) - 1


def _signed(v: int) -> int:
    v &= _M64
    return v - (1 << 64) if v >> 63 else v


def _draws(seed: int, first: int, count: int) -> torch.Tensor:
    """Odd integers q of draws first .. first + count - 1 of the generator's LCG stream (value q 2^-53)."""
    def jump(k):
        a, c, pa, pc = 1, 0, _MUL, _INC
        while k:
            if k & 1:
                a, c = a * pa & _M64, (c * pa + pc) & _M64
            pa, pc = pa * pa & _M64, (pa + 1) * pc & _M64
            k >>= 1
        return a, c

    a, c = jump(first + 1)
    s = torch.empty(count, dtype=torch.int64, device=DEV)
    s[0] = _signed(a * (seed & _M64) + c)
    have = 1
    while have < count:   # int64 arithmetic wraps modulo 2^64
        m = min(have, count - have)
        a, c = jump(have)
        s[have:have + m] = s[:m] * _signed(a) + _signed(c)
        have += m
    u = (s >> 12) & ((1 << 52) - 1)
    return 2 * u + 1 - (1 << 52)


def _exact_generate(case, seed):
    n, k = case["n"], case["nrhs"]
    q = _draws(seed, 0, n * n).view(n, n)             # [j, i]
    A = q.to(torch.float64) * 2.0**-53
    d = A.diagonal()
    if case["diag"] == capi.DIAG_DOMINANT:
        m = q.abs()
        m.diagonal().zero_()
        hi, lo = (m >> 26).sum(dim=0), (m & ((1 << 26) - 1)).sum(dim=0)
        s = hi.to(torch.float64) * 2.0**26 + lo.to(torch.float64)   # both terms exact: one rounding
        d.copy_(s * 2.0**-53 + 1.0)
    else:
        d.copy_(d + torch.sign(d) * math.sqrt(n))
    b = _draws(seed, n * n, n * k).view(k, n).to(torch.float64) * 2.0**-53
    return {"A": A, "b": b}


def _lu64(A: torch.Tensor) -> torch.Tensor:
    """LU without pivoting of A (fp64), blocked, in place."""
    n, w = A.shape[0], 256
    eye = torch.eye(w, dtype=torch.float64, device=A.device)
    for k in range(0, n, w):
        e = min(k + w, n)
        D = A[k:e, k:e]
        for p in range(e - k - 1):
            D[p + 1:, p] /= D[p, p]
            D[p + 1:, p + 1:] -= torch.outer(D[p + 1:, p], D[p, p + 1:])
        if e == n:
            break
        Linv = torch.linalg.solve_triangular(D, eye[:e - k, :e - k], upper=False, unitriangular=True)
        Uinv = torch.linalg.solve_triangular(D.triu(), eye[:e - k, :e - k], upper=True)
        A[k:e, e:] = Linv @ A[k:e, e:]
        A[e:, k:e] = A[e:, k:e] @ Uinv
        A[e:, e:] -= A[e:, k:e] @ A[k:e, e:]
    return A


_EXACT_MAX = 12000   # fp64 elimination of larger systems takes too long to be a check


def exact(case, seed):
    kind = case["kind"]
    if kind == "generate":
        return _exact_generate(case, seed)
    g = _rng(seed)
    if kind == "batch":
        LUs, xs = [], []
        for n, k in _sizes(case):
            A = _dominant(n, g)[:, :n]
            b = _vectors(n, k, g)[:, :n]
            xs.append(torch.linalg.solve(A.t(), b.t()).t())
            LUs.append(_lu64(A.t().contiguous()).t() if n <= 1500 else None)
        return {"LU": LUs, "x": xs}
    n, k = case["n"], case.get("nrhs", 1)
    if kind == "residual":
        A = _dominant(n, g)[:, :n]
        x, b = _vectors(n, k, g)[:, :n], _vectors(n, k, g)[:, :n]
        return {"r": b - x @ A}
    if n > _EXACT_MAX:
        return None
    A = _dominant(n, g)[:, :n]
    out = {}
    if kind in ("refine", "solve"):
        b = _vectors(n, k, g)[:, :n]
        out["x"] = torch.linalg.solve(A.t(), b.t()).t()
    if kind == "factor" or (kind == "solve" and not case.get("balance", False)):
        out["LU"] = _lu64(A.t().contiguous()).t()
    elif kind == "solve":
        out["LU"] = None   # factors of the balanced matrix
    return out
