"""The tensor-core fp64 product when its pipeline waits run out (a short wait
budget: nothing is missing and nothing faults).  The kernel then reads whatever
its stages hold, so shared memory is filled beforehand with patterns that decode
as huge entries and exponents, at orders whose last 64-column block and last
512-row tile are partial.  It must end with its copies and tensor-core work
drained: the calls after it, on the same stream, give the right products."""
import numpy as np
import pytest
import torch

from paper_2509_19618_gb300 import api, capi
from test_gpu_gemv_tc import _inputs, _residual
from test_gpu_timeout import short_budget

pytestmark = pytest.mark.gpu


def _close(got, A, X, B):
    # the tolerance of the products' own test: 2^-48 of the row's largest term and 2^-51 of their sum
    rows = np.arange(0, A.shape[0], 41)
    for r in range(X.shape[1]):
        terms = A[rows].astype(np.longdouble) * X[:, r].astype(np.longdouble)
        tol = 2.0**-48 * np.abs(terms).max(axis=1) + 2.0**-51 * (np.abs(terms).sum(axis=1) + np.abs(B[rows, r]))
        assert np.all(np.abs(got[rows, r] - (B[rows, r] - terms.sum(axis=1))) <= tol)


@pytest.mark.parametrize("pattern", [0x7F7F7F7F, 0xFFFFFFFF, 0x40404040])
@pytest.mark.parametrize("n,k", [(4097, 1), (2112, 2), (2305, 8)])
def test_wait_runs_out_then_recovers(n, k, pattern):
    A, X = _inputs("dominant", n, k)
    B = np.random.default_rng(n).standard_normal((n, k))
    with short_budget():
        for _ in range(3):
            assert capi.hpmxp_test_fill_smem(pattern, api.stream_handle()) == capi.OK
            _residual(A, X, B)
    for _ in range(2):
        _close(_residual(A, X, B), A, X, B)


def test_solve_reports_timeout_then_recovers():
    n = 4096
    A, b = api.generate(n, seed=12)
    s = api.Solver(n, 1, capi.BF16, nb=256)
    s.factor(A)
    with short_budget():
        with pytest.raises(capi.HpmxpError) as e:
            s.solve(A, b)
        assert e.value.status == capi.ETIMEOUT
    x, info, st = s.solve(A, b)
    torch.cuda.synchronize()
    assert st == capi.OK and api.residual(A, x, b)[0] < 16.0
