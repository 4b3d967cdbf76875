"""Right-hand sides that share one tensor-core fp64 product but must not affect
each other: a zero one, and those whose refinement has ended (their Krylov
vectors are then unwritten workspace)."""
import numpy as np
import pytest
import torch

from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _fill(ws, pattern):
    g = torch.Generator(device=DEV).manual_seed(5)
    if pattern == "zeros":
        ws.zero_()
    elif pattern == "nan":
        ws.fill_(255)
    elif pattern == "bytes":
        ws.random_(0, 256, generator=g)
    else:                       # vectors as they could have been left there
        ws[: ws.numel() // 8 * 8].view(torch.float64).normal_(generator=g)


def _solve(A, LU, b, pattern, params):
    n, k = A.rows, b.cols
    x = api.ColMajor.empty(n, k, torch.float64, DEV)
    ws = api.workspace(capi.hpmxp_solve_workspace(n, k, params.restart), DEV)
    _fill(ws, pattern)
    info = (capi.IRInfo * k)()
    st = capi.hpmxp_solve_ir(n, A.ptr, A.ld, LU.ptr, LU.ld, capi.BF16, b.ptr, b.ld, x.ptr, x.ld, k, params, info,
                             ws.data_ptr(), ws.numel(), api.stream_handle())
    torch.cuda.synchronize()
    return x.view().cpu().numpy(), [(i.iters, i.outer, i.status, repr(i.scaled_resid)) for i in info], st


@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("n,k", [(2304, 2), (2111, 4), (1100, 7)])
def test_ended_and_zero_columns_leave_the_others_alone(n, k, fp32):
    A, b = api.generate(n, seed=n, diag=capi.DIAG_SQRTN, nrhs=k, device=DEV)
    Av, bv = A.view(), b.view()
    p = n // 3
    Av[p, :] = 0.0
    Av[:, p] = 0.0
    Av[p, p] = 1.0
    bv[p, :] = 0.0
    bv[:, 1] = 0.0
    bv[p, 1] = 1.0              # x0 is the solution: ended at the first check
    if k > 3:
        bv[:, 3] = 0.0
    # the diagonal's factors: many Arnoldi steps, whose products reach x in full
    D = api.ColMajor.empty(n, n, torch.float64, DEV)
    D.storage.zero_()
    D.view().diagonal().copy_(Av.diagonal())
    LU = api.factor(D, capi.BF16, 128)
    prm = api.ir_params(precond_fp32=fp32, max_iters=24, restart=10)
    out = [_solve(A, LU, b, pattern, prm) for pattern in ("zeros", "nan", "bytes", "vectors")]
    for x, info, st in out[1:]:
        assert st == out[0][2] and info == out[0][1]
        assert np.array_equal(x, out[0][0], equal_nan=True)


def test_zero_column_does_not_change_the_sums_of_the_others():
    n = 2600
    g = torch.Generator(device=DEV).manual_seed(3)
    A, X = (api.ColMajor.empty(n, c, torch.float64, DEV) for c in (n, 3))
    for m in (A, X):
        m.storage.uniform_(-0.5, 0.5, generator=g)
    X.view()[:, 1] = 0.0

    def product(cols):
        k = len(cols)
        x, b, r = (api.ColMajor.empty(n, k, torch.float64, DEV) for _ in range(3))
        x.view().copy_(X.view()[:, cols])
        b.storage.zero_()
        ws = api.workspace(capi.hpmxp_residual_workspace(n, k), DEV)
        st = capi.hpmxp_residual_vector(n, A.ptr, A.ld, x.ptr, x.ld, b.ptr, b.ld, k, r.ptr, r.ld, ws.data_ptr(),
                                        ws.numel(), api.stream_handle())
        torch.cuda.synchronize()
        assert st == capi.OK
        return r.view()

    with_zero, without = product([0, 1, 2]), product([0, 2])
    assert torch.equal(with_zero[:, [0, 2]], without)
    assert bool((with_zero[:, 1] == 0).all())
