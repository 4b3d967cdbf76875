"""The digit products are no less accurate than the fp64 FMAs they replace: both
routes of hpmxp_residual_vector (an odd leading dimension takes the FMAs)
against extended precision, rms over rows, for inputs that cost digits: full
53-bit entries, a right-hand side 2^5 below its own maximum and the other in most
columns, dominant diagonals, rows whose largest products cancel, graded rows."""
import numpy as np
import pytest
import torch

from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _inputs(kind, n, k):
    g = np.random.default_rng(n + k)
    A, X = g.standard_normal((n, n)), g.standard_normal((n, k))
    if kind == "low":
        X[:, k - 1] *= 2.0**-5
        X[g.integers(0, n, n // 50), k - 1] *= 2.0**5
    elif kind == "dominant":
        A[np.arange(n), np.arange(n)] = np.abs(A).sum(axis=1)
    elif kind == "cancel":      # two large products in the row's first columns, 2^-30 apart
        A[:, 3], A[:, 5] = 2.0**20, -(2.0**20)
        X[5] = X[3] * (1.0 + 2.0**-30 * g.uniform(-1, 1, k))
    elif kind == "graded":
        A *= np.exp2(g.integers(-20, 1, (n, n)))
    return A, X


def _product(A, X, ld):
    n, k = X.shape
    dA = api.ColMajor.empty(n, n, torch.float64, DEV, ld=ld)
    dA.view().copy_(torch.from_numpy(A))
    dX = api.ColMajor.from_tensor(torch.from_numpy(X), DEV)
    B, R = (api.ColMajor.empty(n, k, torch.float64, DEV) for _ in range(2))
    B.storage.zero_()
    ws = api.workspace(capi.hpmxp_residual_workspace(n, k), DEV)
    st = capi.hpmxp_residual_vector(n, dA.ptr, dA.ld, dX.ptr, dX.ld, B.ptr, B.ld, k, R.ptr, R.ld, ws.data_ptr(),
                                    ws.numel(), api.stream_handle())
    torch.cuda.synchronize()
    assert st == capi.OK
    return -R.view().cpu().numpy()


@pytest.mark.parametrize("kind", ["full", "low", "dominant", "cancel", "graded"])
@pytest.mark.parametrize("n,k", [(2048, 2), (2048, 5), (4098, 1), (1026, 8)])
def test_no_less_accurate_than_the_plain_sums(n, k, kind):
    A, X = _inputs(kind, n, k)
    rows = np.arange(0, n, 13)
    digits, plain = (_product(A, X, n + pad)[rows] for pad in (0, 1))
    for r in range(k):
        want = (A[rows].astype(np.longdouble) * X[:, r].astype(np.longdouble)).sum(axis=1)
        rms = [float(np.sqrt(((p[:, r].astype(np.longdouble) - want) ** 2).mean())) for p in (digits, plain)]
        assert rms[0] <= rms[1], (r, rms)
