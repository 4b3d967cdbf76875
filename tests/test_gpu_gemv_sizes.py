"""Orders and right-hand side counts whose column chunks of the fp64 FMA product do
not divide evenly into its staging buffer: the residual check, the fp32 operator's
product and an odd leading dimension take that product, and no size is refused."""
import pytest
import torch

from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _system(n, k, pad=0):
    g = torch.Generator(device=DEV).manual_seed(n + k)
    A = api.ColMajor.empty(n, n, torch.float64, DEV, ld=n + pad)
    X, B = (api.ColMajor.empty(n, k, torch.float64, DEV) for _ in range(2))
    for m in (A, X, B):
        m.storage.uniform_(-0.5, 0.5, generator=g)
    return A, X, B


def test_chunks_fit_for_every_size():
    """The chunk count (restated) never gives a chunk above the staging buffer, and
    never more chunks than the workspace holds (those of eight right-hand sides)."""
    def chunks(n, k):
        spread = min(-(-1216 // -(-n // 512)), -(-n // 32))
        return max(1, min(max(-(-n // (4096 // k)), spread), -(-n // 8)))

    for k in range(1, 9):
        for n in list(range(1, 5000)) + list(range(19000, 131073, 7)) + [32768, 65536, 98304, 131072]:
            c = chunks(n, k)
            assert -(-n // c) * k <= 4096 and c <= chunks(n, 8)


@pytest.mark.parametrize("n,k", [(19116, 7), (20480, 7), (32768, 3), (32768, 6)])
def test_residual_check(n, k):
    A, X, B = _system(n, k)
    r = B.view() - A.view() @ X.view()
    want = r.abs().amax(0) / ((A.view().abs().sum(1).max() * X.view().abs().amax(0) + B.view().abs().amax(0)) * n * 2.0**-53)
    got = api.residual(A, X, B)
    for c in range(k):
        assert abs(got[c] - float(want[c])) <= 1e-9 * float(want[c])


def test_odd_leading_dimension():
    n, k = 20480, 7
    A, X, B = _system(n, k, 1)
    R = api.ColMajor.empty(n, k, torch.float64, DEV)
    ws = api.workspace(capi.hpmxp_residual_workspace(n, k), DEV)
    st = capi.hpmxp_residual_vector(n, A.ptr, A.ld, X.ptr, X.ld, B.ptr, B.ld, k, R.ptr, R.ld, ws.data_ptr(), ws.numel(),
                                    api.stream_handle())
    torch.cuda.synchronize()
    assert st == capi.OK
    bound = 0.1 * n * 2.0**-53 * (A.view().abs() @ X.view().abs() + B.view().abs())
    assert bool(((R.view() - (B.view() - A.view() @ X.view())).abs() <= bound).all())


def test_fp32_operator():
    n, k = 20480, 7
    A, b = api.generate(n, seed=3, nrhs=k, device=DEV)
    LU = api.factor(A, capi.BF16, 512)
    x, infos, st = api.solve_ir(A, LU, b, capi.BF16, api.ir_params(precond_fp32=1, matvec_fp32=1, inner_tol=1e-5))
    torch.cuda.synchronize()
    assert st == capi.OK and max(api.residual(A, x, b)) < 16.0
