"""Large products of depth 512 run on pairs of CTAs: against the 128-row tiles on
single CTAs, which add the same products in the same order, bit for bit, at
ragged sizes (the last pair's second CTA partly or wholly outside, odd tile
counts), on few SMs, with the row-major copy; and a wait that runs out."""
import pytest
import torch

from paper_2509_19618_gb300 import api, capi
from test_gpu_timeout import short_budget

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
BF16, SUB, STORE = 0, 0, 1


def _product(M, N, K, mode, tile, budget=0):
    g = torch.Generator(device=DEV).manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, device=DEV).bfloat16()
    B = torch.randn(N, K, generator=g, device=DEV).bfloat16()
    ld = -(-M // 8) * 8
    C = torch.randn(N, ld, generator=g, device=DEV).bfloat16()
    R = torch.zeros(M, N, dtype=torch.bfloat16, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    assert capi.hpmxp_set_tuning(tile, 0, 0, budget) == capi.OK
    try:
        st = capi.hpmxp_test_gemm(M, N, K, A.data_ptr(), K, B.data_ptr(), K, C.data_ptr(), ld,
                                  R.data_ptr() if mode == STORE else None, N if mode == STORE else 0, mode, 1.0, BF16,
                                  0, None, 0, None, 0, 0, status.data_ptr(), api.stream_handle())
    finally:
        assert capi.hpmxp_set_tuning(0, 0, 0, 0) == capi.OK
    torch.cuda.synchronize()
    return st, int(status.item()), C, R


@pytest.mark.parametrize("mode", [SUB, STORE])
@pytest.mark.parametrize("M,N,K,budget", [(2304, 2304, 512, 0), (2500, 2433, 512, 0), (2305, 2177, 512, 0),
                                          (9000, 1030, 1024, 0), (2600, 2700, 512, 2), (2600, 2700, 512, 7),
                                          (2600, 2700, 512, 1)])
def test_pairs_equal_single_ctas(M, N, K, mode, budget):
    st, word, C, R = _product(M, N, K, mode, 0, budget)
    assert st == capi.OK and word == 0
    st, word, C1, R1 = _product(M, N, K, mode, 128)
    assert st == capi.OK and word == 0
    assert torch.equal(C, C1) and torch.equal(R, R1)


def test_pair_wait_runs_out_then_recovers():
    with short_budget():
        st, word, _, _ = _product(2500, 2433, 512, SUB, 0)
    assert st == capi.OK and word == 1        # the timeout bit, nothing else
    st, word, C, _ = _product(2500, 2433, 512, SUB, 0)
    assert st == capi.OK and word == 0
    _, _, C1, _ = _product(2500, 2433, 512, SUB, 128)
    assert torch.equal(C, C1)
