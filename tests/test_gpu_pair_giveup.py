"""Pairs of CTAs whose waits run out at different points (budgets of 1 to a few
hundred polls): the ranks' producers have then loaded different numbers of stages,
and the pair must still see every copy land before it ends.  Each call returns at
once (a copy that was never seen to land would cost the drain's full 2 s), sets
nothing but the timeout bit, and the next one gives the right bits."""
import time

import pytest
import torch

from paper_2509_19618_gb300 import capi
from test_gpu_gemm_pairs import STORE, SUB, _product

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,mode", [(2500, 2433, 512, SUB), (9000, 1030, 1024, STORE), (6000, 6100, 512, SUB)])
def test_waits_run_out_anywhere(M, N, K, mode):
    _, _, want, want_r = _product(M, N, K, mode, 128)
    words = []
    for polls in (1, 2, 3, 5, 8, 13, 21, 34, 55, 89, 144, 233):
        assert capi.hpmxp_test_set_wait_budget(polls, 0) == capi.OK
        try:
            t = time.perf_counter()
            st, word, C, R = _product(M, N, K, mode, 0)
            t = time.perf_counter() - t
        finally:
            assert capi.hpmxp_test_set_wait_budget(0, 0) == capi.OK
        assert st == capi.OK and word in (0, 1) and t < 1.5
        if word == 0:
            assert torch.equal(C, want) and torch.equal(R, want_r)
        words.append(word)
        st, word, C, R = _product(M, N, K, mode, 0)
        assert st == capi.OK and word == 0 and torch.equal(C, want) and torch.equal(R, want_r)
    assert words[0] == 1
