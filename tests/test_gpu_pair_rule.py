"""Which products of depth 512 take pairs of CTAs: the launch's grid is not
visible, so both sides of the rule (128 to 1152 columns, odd and even tile counts,
tile counts at the number of SMs) are compared with the 128-row tiles bit for
bit, and a panel's product of 128 columns must not take longer than one of the
same rows and 256 columns (with pairs the two cost the same work)."""
import pytest
import torch

from paper_2509_19618_gb300 import api, capi
from test_gpu_gemm_pairs import STORE, SUB, _product

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("mode", [SUB, STORE])
@pytest.mark.parametrize("M,N", [(20000, 128), (20000, 129), (12000, 384), (9000, 640), (6000, 896), (5000, 1025),
                                 (38 * 256, 512), (38 * 256 + 1, 512)])
def test_both_sides_equal_single_ctas(M, N, mode):
    st, word, C, R = _product(M, N, 512, mode, 0)
    assert st == capi.OK and word == 0
    st, word, C1, R1 = _product(M, N, 512, mode, 128)
    assert st == capi.OK and word == 0
    assert torch.equal(C, C1) and torch.equal(R, R1)


def _time(M, N):
    A, B = torch.randn(M, 512, device=DEV).bfloat16(), torch.randn(N, 512, device=DEV).bfloat16()
    C, R = torch.zeros(N, M, device=DEV).bfloat16(), torch.zeros(M, N, device=DEV).bfloat16()
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    ts = []
    for _ in range(30):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        capi.hpmxp_test_gemm(M, N, 512, A.data_ptr(), 512, B.data_ptr(), 512, C.data_ptr(), M, R.data_ptr(), N, STORE,
                             1.0, 0, 0, None, 0, None, 0, 0, status.data_ptr(), api.stream_handle())
        e1.record()
        torch.cuda.synchronize()
        ts.append(e0.elapsed_time(e1))
    return sorted(ts)[10]


def test_a_panel_does_not_pay_for_an_empty_half():
    M = 96 * 1024               # 384 row tiles, more than one wave either way
    one, two = _time(M, 128), _time(M, 256)
    assert one <= 0.85 * two, (one, two)
