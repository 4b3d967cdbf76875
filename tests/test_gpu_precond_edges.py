"""The preconditioner at orders that are not a multiple of 8, its factors without
meaningful padding: rows n .. ldlu - 1 of every column, and what follows the array,
hold NaN, and the result equals the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from inputs import vectors
from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("n", [1, 7, 63, 65, 129, 250, 387])
def test_last_rows_without_padding(n, fp32):
    A_o, _ = oracle.generate(n, n)
    LU_o, _ = oracle.factor(A_o, oracle.BF16, 128)
    ld = -(-n // 8) * 8
    buf = torch.full(((n + 2) * ld,), float("nan"), dtype=torch.bfloat16, device=DEV)
    buf[: n * ld].view(n, ld)[:, :n] = torch.from_numpy(np.ascontiguousarray(LU_o.T)).to(DEV, torch.bfloat16)
    V = vectors(n, 2, 3)
    v = api.ColMajor.from_tensor(torch.from_numpy(V), DEV)
    z = api.ColMajor.empty(n, 2, torch.float64, DEV)
    ws = api.workspace(capi.hpmxp_solve_workspace(n, 2, 1), DEV)
    st = capi.hpmxp_test_precond(n, buf.data_ptr(), ld, capi.BF16, v.ptr, v.ld, z.ptr, z.ld, 2, fp32, ws.data_ptr(),
                                 ws.numel(), api.stream_handle())
    torch.cuda.synchronize()
    assert st == capi.OK
    for c in range(2):
        want = oracle.precond(LU_o, V[:, c], prec=fp32)
        assert np.abs(z.view().cpu().numpy()[:, c] - want).max() <= (1e-5 if fp32 else 1e-13) * np.abs(want).max()
