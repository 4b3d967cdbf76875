"""Which products take the tensor cores, seen by the launches of a residual (two of
the FMA product, five of the digit product): from the orders where they pay on,
and at those smallest orders the digits fit into the scratch."""
import pytest
import torch

from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,k,pad,launches", [(1023, 8, 1, 2), (1024, 5, 0, 2), (1024, 6, 0, 5), (1024, 8, 0, 5), (1057, 7, 1, 5),
                                              (1088, 8, 0, 5), (1088, 8, 1, 2), (2047, 2, 1, 2), (2048, 2, 0, 5),
                                              (4095, 1, 1, 2), (4096, 1, 0, 5), (17920, 1, 0, 5)])
def test_route(n, k, pad, launches):
    A = api.ColMajor.empty(n, n, torch.float64, DEV, ld=n + pad)
    X, B, R = (api.ColMajor.empty(n, k, torch.float64, DEV) for _ in range(3))
    g = torch.Generator(device=DEV).manual_seed(n)
    for m in (A, X, B):
        m.storage.uniform_(-0.5, 0.5, generator=g)
    ws = api.workspace(capi.hpmxp_residual_workspace(n, k), DEV)
    before = capi.hpmxp_launch_count()
    st = capi.hpmxp_residual_vector(n, A.ptr, A.ld, X.ptr, X.ld, B.ptr, B.ld, k, R.ptr, R.ld, ws.data_ptr(), ws.numel(),
                                    api.stream_handle())
    torch.cuda.synchronize()
    assert st == capi.OK and capi.hpmxp_launch_count() - before == launches
    bound = 0.1 * n * 2.0**-53 * (A.view().abs() @ X.view().abs() + B.view().abs())
    assert bool(((R.view() - (B.view() - A.view() @ X.view())).abs() <= bound).all())
