"""The tensor-core fp64 product when its pipeline waits run out (a short wait
budget: nothing is missing and nothing faults).  The kernel then reads whatever
its stages hold, so shared memory is filled beforehand with patterns that decode
as huge entries and exponents.  It must end with its copies and tensor-core work
drained: the calls after it, on the same stream, give the right products.

At small orders the loads are there in time and no wait runs out; at 24001 with
eight right-hand sides one does in every call, at 16400 with one in some."""
import pytest
import torch

from paper_2509_19618_gb300 import api, capi
from test_gpu_timeout import short_budget

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


class _System:
    def __init__(self, n, k, seed=1):
        g = torch.Generator(device=DEV).manual_seed(seed)
        self.n, self.k = n, k
        self.A, self.X, self.B, self.R = (api.ColMajor.empty(n, c, torch.float64, DEV) for c in (n, k, k, k))
        for m in (self.A, self.X, self.B):
            m.storage.uniform_(-0.5, 0.5, generator=g)
        self.ws = api.workspace(capi.hpmxp_residual_workspace(n, k), DEV)
        A, X, B = self.A.view(), self.X.view(), self.B.view()
        self.want = B - A @ X
        # fp64 sums in any order: n 2^-53 of the terms' sum, taken at a tenth (both sides round)
        self.tol = 0.1 * n * 2.0**-53 * (A.abs() @ X.abs() + B.abs())

    def residual(self):
        """(r, whether a wait ran out: the status word heads the workspace)"""
        st = capi.hpmxp_residual_vector(self.n, self.A.ptr, self.A.ld, self.X.ptr, self.X.ld, self.B.ptr, self.B.ld,
                                        self.k, self.R.ptr, self.R.ld, self.ws.data_ptr(), self.ws.numel(),
                                        api.stream_handle())
        assert st == capi.OK
        torch.cuda.synchronize()
        return self.R.view(), bool(self.ws[:4].view(torch.int32).item() & 1)

    def right(self, r):
        return bool(((r - self.want).abs() <= self.tol).all())


# At both orders the last 64-column block and the last 512-row tile are partial.
@pytest.mark.parametrize("n,k", [(16400, 1), (24001, 8)])
def test_product_is_right_when_a_wait_runs_out(n, k):
    # hpmxp_residual_vector returns before its work is done and cannot report a timeout, so the
    # vector itself has to be right
    s = _System(n, k)
    r, out = s.residual()
    assert not out and s.right(r)
    clean = r.clone()
    hits = 0
    for t in range(24):
        with short_budget():
            assert capi.hpmxp_test_fill_smem([0x7F7F7F7F, 0xFFFFFFFF, 0x40404040][t % 3], api.stream_handle()) == capi.OK
            r, out = s.residual()
        assert s.right(r)
        hits += out
        r, out = s.residual()
        assert not out and torch.equal(r, clean)
    assert hits > 0 or k == 1, "no wait ran out: the path was not taken"


def test_solve_reports_timeout_then_recovers():
    n = 16400
    A, b = api.generate(n, seed=12, device=DEV)
    s = api.Solver(n, 1, capi.BF16, nb=256, device=DEV)
    s.factor(A)
    with short_budget():
        with pytest.raises(capi.HpmxpError) as e:
            s.solve(A, b)
        assert e.value.status == capi.ETIMEOUT
    x, info, st = s.solve(A, b)
    torch.cuda.synchronize()
    assert st == capi.OK and api.residual(A, x, b)[0] < 16.0
