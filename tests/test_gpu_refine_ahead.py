"""The refinement issued ahead of the host's knowledge (the first cycle before the
first check, a cycle's first Arnoldi step before its start) against the same
solve decided step by step (the order used while the kernel timers are on):
the decisions are the device's either way, so x and the report are the same bits."""
import numpy as np
import pytest
import torch

from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _solve(A, LU, b, params, timers):
    capi.hpmxp_prof_enable(timers)
    try:
        x, infos, st = api.solve_ir(A, LU, b, capi.BF16, params)
        torch.cuda.synchronize()
    finally:
        capi.hpmxp_prof_enable(0)
    return x.view().cpu().numpy(), infos, st


@pytest.mark.parametrize("n,k", [(1, 1), (300, 3), (1024, 1), (5000, 2)])
@pytest.mark.parametrize("kw", [{}, {"max_iters": 0}, {"max_iters": 1}, {"restart": 1, "accept": 1e-3, "max_iters": 7},
                                {"restart": 2, "accept": 1e-3, "max_iters": 9}, {"accept": 1e30},
                                {"precond_fp32": 1, "inner_tol": 1e-5}, {"precond_fp32": 1, "matvec_fp32": 1}])
def test_ahead_equals_step_by_step(n, k, kw):
    A, b = api.generate(n, seed=n, nrhs=k, device=DEV)
    LU = api.factor(A, capi.BF16, 128)
    p = api.ir_params(**kw)
    x1, i1, s1 = _solve(A, LU, b, p, 0)
    x2, i2, s2 = _solve(A, LU, b, p, 1)
    assert s1 == s2 and i1 == i2
    assert np.array_equal(x1, x2)


def test_breakdown_and_early_columns():
    n, k = 700, 3
    A, b = api.generate(n, seed=5, nrhs=k, device=DEV)
    LU = api.factor(A, capi.BF16, 128)
    bv = b.view()
    bv[:, 1] = 0.0            # solved by x0
    bv[3, 2] = float("nan")   # breaks down at the first check
    out = [_solve(A, LU, b, api.ir_params(), t) for t in (0, 1)]
    (x1, i1, s1), (x2, i2, s2) = out
    assert s1 == s2 != capi.OK
    assert repr(i1) == repr(i2)
    assert np.array_equal(x1, x2, equal_nan=True)


def test_batched_ahead_equals_alone():
    sizes = [(64, 1), (700, 3), (1024, 8), (300, 2)]
    As, bs = zip(*[api.generate(n, seed=n, nrhs=k, device=DEV) for n, k in sizes])
    LUs = [api.factor(A, capi.BF16, 128) for A in As]
    for kw in ({}, {"max_iters": 0}, {"restart": 1, "accept": 1e-3, "max_iters": 5}, {"accept": 1e30}):
        p = api.ir_params(**kw)
        res = []
        for timers in (0, 1):
            capi.hpmxp_prof_enable(timers)
            try:
                xs, infos, st = api.solve_ir_batched(list(As), LUs, list(bs), capi.BF16, p)
                torch.cuda.synchronize()
            finally:
                capi.hpmxp_prof_enable(0)
            res.append(([x.view().cpu().numpy() for x in xs], infos, st))
        assert res[0][1:] == res[1][1:]
        assert all(np.array_equal(a, c) for a, c in zip(res[0][0], res[1][0]))
