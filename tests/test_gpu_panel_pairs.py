"""The row and column panels of a step share a launch, and the rows below a
diagonal block are packed beside its LU: ragged orders around the 128-wide
tiles, every update depth, the plain and the look-ahead schedule, the batched
factorization.

The schedules give the same bits.  Tolerance of L U against the rounded matrix:
an entry is rounded to 16 bits once per 128 columns to its left at most, by half
an ulp (2^-9 for bf16, 2^-12 for fp16) of values no larger than the diagonal's,
and both factors once more: (n / 128 + 4) half ulps of the largest entry."""
import numpy as np
import pytest
import torch

from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("prec,ulp", [(capi.BF16, 2.0**-9), (capi.FP16, 2.0**-12)])
@pytest.mark.parametrize("nb", [128, 256, 512])
@pytest.mark.parametrize("n", [129, 256, 257, 383, 513, 641, 1025, 1281, 1700])
def test_schedules_agree(n, nb, prec, ulp):
    A, _ = api.generate(n, seed=n, device=DEV)
    outs = []
    for overlap in (0, 128):   # 0: plain at these orders; 128: look-ahead
        assert capi.hpmxp_set_tuning(0, 0, overlap) == capi.OK
        try:
            outs.append(api.factor(A, prec, nb).view().double().cpu().numpy())
        finally:
            assert capi.hpmxp_set_tuning(0, 0, 0) == capi.OK
    if nb == 128:
        dt = api.factor_storage_dtype(prec)
        LU = api.ColMajor.empty(n, n, dt, DEV)
        api.factor_batched([A], prec, [LU])
        outs.append(LU.view().double().cpu().numpy())
    torch.cuda.synchronize()
    for o in outs[1:]:
        assert np.array_equal(outs[0], o)
    L, U = np.tril(outs[0], -1) + np.eye(n), np.triu(outs[0])
    a = A.view().cpu().numpy()
    assert np.abs(L @ U - a).max() <= (n / 128 + 4) * ulp * np.abs(a).max()
