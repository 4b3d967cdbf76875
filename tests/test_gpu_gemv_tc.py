"""The fp64 products on the tensor cores (exact digit products) against extended
precision, row by row: ordinary, graded, lone large and non-finite entries,
right-hand sides of different sizes and supports, ragged orders, odd leading
dimensions.

Tolerance, per entry of A x: the digits drop at most 2^-55 of the row block's
largest |a_ij x_jr| per column (2^-49 of it over 64 columns if all rounded the
same way, a factor 8 less with signs), the right-hand sides of one column may
differ by 2^6 before a block falls back to fp64, and the sums round at 2^-53:
2^-48 times the row's largest |a_ij x_jr|, plus 2^-51 sum_j |a_ij x_jr|.  A
plain fp64 sum only guarantees n 2^-53 times that sum."""
import numpy as np
import pytest
import torch

from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu


def _inputs(kind, n, k):
    g = np.random.default_rng(n + k)
    A = g.uniform(-0.5, 0.5, size=(n, n))
    X = g.standard_normal((n, k))
    if kind == "dominant":
        A[np.arange(n), np.arange(n)] = np.abs(A).sum(axis=1)
    elif kind == "graded":       # columns of A and x graded against each other, rows of A too
        s = np.exp2(g.integers(-40, 41, n))
        A = A * s * np.exp2(g.integers(-300, 301, n))[:, None]
        X = X / s[:, None]
    elif kind == "supports":     # unit vectors and zero columns, on columns of very different sizes
        A = A * np.exp2(g.integers(-30, 31, n))
        X[:] = 0.0
        X[g.integers(0, n, k), np.arange(k)] = g.uniform(1, 2, k)
        if k > 2:
            X[:, 2] = 0.0
    elif kind == "scales":       # right-hand sides of very different norms
        X = X * np.exp2(np.linspace(-400, 400, k)) if k > 1 else X * 2.0**500
    elif kind == "lone":         # single large entries scattered over the rows; zero rows
        A[np.arange(n), g.integers(0, n, n)] *= 2.0**30
        A[::17] = 0.0
    elif kind == "tiny":         # entries around the bottom of the range
        A = A * 2.0**-1020
        A[:, ::5] = 0.0
    return np.asfortranarray(A), np.asfortranarray(X)


def _residual(A, X, B, lda_pad=0):
    n, k = X.shape
    dA = api.ColMajor.empty(n, n, torch.float64, "cuda", ld=n + lda_pad)
    dA.view().copy_(torch.from_numpy(A))
    dX, dB = (api.ColMajor.from_tensor(torch.from_numpy(m), "cuda") for m in (X, B))
    R = api.ColMajor.empty(n, k, torch.float64, "cuda")
    ws = api.workspace(capi.hpmxp_residual_workspace(n, k), "cuda")
    st = capi.hpmxp_residual_vector(n, dA.ptr, dA.ld, dX.ptr, dX.ld, dB.ptr, dB.ld, k, R.ptr, R.ld, ws.data_ptr(),
                                    ws.numel(), api.stream_handle())
    assert st == capi.OK
    torch.cuda.synchronize()
    return R.view().cpu().numpy()


@pytest.mark.parametrize("kind", ["plain", "dominant", "graded", "supports", "scales", "lone", "tiny"])
@pytest.mark.parametrize("n,k,pad", [(2048, 8, 0), (4097, 1, 0), (2112, 2, 0), (2111, 2, 1), (2500, 3, 3), (4225, 5, 0),
                                     (2300, 8, 5)])
def test_product_against_extended_precision(n, k, pad, kind):
    A, X = _inputs(kind, n, k)
    got = -_residual(A, X, np.zeros((n, k)), pad)
    rows = np.unique(np.concatenate([np.arange(0, n, 97), [0, 63, 64, 127, 128, n - 1]]))
    for r in range(k):
        terms = A[rows].astype(np.longdouble) * X[:, r].astype(np.longdouble)
        want, mag, big = terms.sum(axis=1), np.abs(terms).sum(axis=1), np.abs(terms).max(axis=1)
        tol = 2.0**-48 * big + 2.0**-51 * mag + np.longdouble(2.0) ** -1074 * n
        err = np.abs(got[rows, r].astype(np.longdouble) - want)
        assert np.all(err <= tol), (r, rows[np.argmax(err - tol)], float(err.max()))


def test_digit_sums_are_exact_at_their_largest():
    # every digit at its largest magnitude: all entries 1 - 2^-53, x just below one:
    # each fp32 sum of a block reaches 64 * 7 * 255 * 127
    n = 2048
    A = np.full((n, n), 1.0 - 2.0**-53, order="F")
    X = np.full((n, 8), 1.0 - 2.0**-53)
    X[:, 1::2] *= -1.0
    got = -_residual(A, X, np.zeros((n, 8)))
    want = n * (1.0 - 2.0**-52)      # (1 - 2^-53)^2 n to within n 2^-106
    assert np.all(np.abs(np.abs(got) - want) <= 2.0**-52 * want)
    assert np.all(np.sign(got[:, 0]) == 1) and np.all(np.sign(got[:, 1]) == -1)


def test_non_finite_entries_reach_their_rows_only():
    n, k = 2200, 3
    A, X = _inputs("plain", n, k)
    A[5, 100] = np.inf
    A[700, 2100] = np.nan
    B = np.ones((n, k))
    got = _residual(A, X, B)
    clean = np.ones(n, bool)
    clean[[5, 700]] = False
    assert np.all(np.isnan(got[700])) and np.all(np.isinf(got[5]))
    assert np.all(np.isfinite(got[clean]))
    X[9, 1] = np.inf
    got = _residual(A, X, B)
    assert not np.isfinite(got[clean][:, 1]).any() and np.all(np.isfinite(got[clean][:, [0, 2]]))
