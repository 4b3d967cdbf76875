"""The tensor-core fp64 product where it takes fp64 FMAs from its own stages:
rows without an exponent yet (zero blocks), columns of X that have little in
common, entries and x at the ends of the range, non-finite x against zero
entries; against extended precision and the IEEE rules."""
import numpy as np
import pytest
import torch

from paper_2509_19618_gb300 import api, capi
from test_gpu_gemv_tc import _residual

pytestmark = pytest.mark.gpu


def _inputs(kind, n, k):
    g = np.random.default_rng(n + k)
    A, X = g.standard_normal((n, n)), g.standard_normal((n, k))
    if kind == "lower":
        A = np.tril(A)
    elif kind == "upper":
        A = np.triu(A)
    elif kind == "band":
        A = np.triu(np.tril(A, 70), -70)
    elif kind == "unlike":      # every column of A large for one right-hand side only
        X *= np.where(np.arange(n)[:, None] % k == np.arange(k)[None, :], 1.0, 2.0**-30)
    elif kind == "decaying":    # x below 2^-400 of its largest, rows that see only such x
        X *= np.exp2(-np.arange(n) * 0.5)[:, None]
        A = np.triu(A)
    elif kind == "subnormal":   # rows whose first blocks hold subnormal entries only
        A[:, : n // 2] *= 2.0**-1060
    return A, X


@pytest.mark.parametrize("kind", ["lower", "upper", "band", "unlike", "decaying", "subnormal"])
@pytest.mark.parametrize("n,k", [(4100, 1), (2050, 2), (1101, 8)])
def test_fp64_blocks_against_extended_precision(n, k, kind):
    A, X = _inputs(kind, n, k)
    got = -_residual(A, X, np.zeros((n, k)), n % 2)
    rows = np.unique(np.concatenate([np.arange(0, n, 61), [0, 63, 64, 511, 512, n - 1]]))
    for r in range(k):
        terms = A[rows].astype(np.longdouble) * X[:, r].astype(np.longdouble)
        # the digits' share (2^-50 of the row's largest product, random signs over the columns) and
        # fp64 sums of at most 64-column blocks and as many pieces
        tol = 2.0**-48 * np.abs(terms).max(axis=1) + 2.0**-48 * np.abs(terms).sum(axis=1) + np.longdouble(2.0)**-1074 * n
        assert np.all(np.abs(got[rows, r] - terms.sum(axis=1)) <= tol), r


def test_non_finite_x_meets_zero_entries():
    n, k = 2048, 3
    A, X = _inputs("lower", n, k)
    X[1500, 0] = np.inf           # rows above 1500 multiply it by zero
    X[700, 2] = np.nan
    got = _residual(A, X, np.ones((n, k)))
    assert np.isnan(got[:1500, 0]).all() and not np.isfinite(got[1500:, 0]).any()
    assert np.isfinite(got[:, 1]).all()
    assert np.isnan(got[:, 2]).all()


def test_infinite_row_sums_over_unlike_columns():
    # the first residual of a solve also estimates ||A||_inf (fp32, 20 bits of each entry); x0, whose
    # residual is far above rounding, is accepted
    n, k = 2304, 2
    A, X = _inputs("unlike", n, k)
    A += np.diag(np.abs(A).sum(axis=1))
    dA = api.ColMajor.from_tensor(torch.from_numpy(A), "cuda")
    LU = api.factor(dA, capi.BF16, 128)
    b = api.ColMajor.from_tensor(torch.from_numpy(A @ X), "cuda")
    x, infos, st = api.solve_ir(dA, LU, b, capi.BF16, api.ir_params(accept=1e30))
    torch.cuda.synchronize()
    assert st == capi.OK
    exact = api.residual(dA, x, b)
    for i, e in zip(infos, exact):
        assert abs(i["scaled_resid"] - e) <= 1e-5 * e
