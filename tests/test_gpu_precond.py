"""The preconditioner at the edges of its blocks (128 rows in fp32, 64 in fp64;
terms beyond the two blocks next to the diagonal from the fourth block on),
with every count of right-hand sides, both factor formats, few CTAs, and
factors whose columns are not 16-byte aligned.

Tolerance against fp64 substitution by the oracle: a sum has at most 64 terms
per thread and about as many additions as there are blocks after that, in both
sweeps, with the rows of the diagonally dominant factors summing to at most
about one: 4 (64 + blocks) roundings of the largest |z|, plus the oracle's own
n roundings at 2^-53."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_19618_gb300 import api, capi
from inputs import vectors

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
BLOCK = {1: 128, 0: 64}


def _apply(LU, n, ld, prec, V, fp32, offset=0):
    """z for the factors laid out with leading dimension ld, `offset` entries into their buffer."""
    k = V.shape[1]
    dt = torch.bfloat16 if prec == capi.BF16 else torch.float16
    buf = torch.full((offset + ld * n,), float("nan"), dtype=dt, device=DEV)
    buf[offset:].view(n, ld)[:, :n] = torch.from_numpy(np.ascontiguousarray(LU.T)).to(dt)
    v = api.ColMajor.from_tensor(torch.from_numpy(V), DEV)
    z = api.ColMajor.empty(n, k, torch.float64, DEV)
    ws = api.workspace(capi.hpmxp_solve_workspace(n, k, 1), DEV)
    st = capi.hpmxp_test_precond(n, buf.data_ptr() + 2 * offset, ld, prec, v.ptr, v.ld, z.ptr, z.ld, k, fp32,
                                 ws.data_ptr(), ws.numel(), api.stream_handle())
    torch.cuda.synchronize()
    return st, z.view().cpu().numpy()


def _check(z, LU, V, n, fp32):
    blocks = -(-n // BLOCK[fp32])
    tol = 4 * (64 + blocks) * 2.0 ** (-24 if fp32 else -53) + n * 2.0**-53
    for c in range(V.shape[1]):
        want = oracle.precond(LU, V[:, c], prec=0)
        assert np.abs(z[:, c] - want).max() <= tol * np.abs(want).max()


@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("prec", [capi.BF16, capi.FP16])
@pytest.mark.parametrize("blocks,extra,k", [(1, -1, 1), (1, 0, 2), (1, 1, 3), (2, 0, 4), (3, -1, 5), (3, 0, 6),
                                            (3, 1, 7), (4, 0, 8), (4, 1, 1), (5, -7, 2), (9, 5, 8), (17, 0, 1)])
def test_block_edges(blocks, extra, k, prec, fp32):
    n = blocks * BLOCK[fp32] + extra
    A, _ = oracle.generate(n, 9)
    LU, _ = oracle.factor(A, oracle.BF16 if prec == capi.BF16 else oracle.FP16, 128)
    V = vectors(n, k, n + k)
    outs = []
    for budget in (0, 3):
        assert capi.hpmxp_set_tuning(0, 0, 0, budget) == capi.OK
        try:
            st, z = _apply(LU, n, -(-n // 8) * 8, prec, V, fp32)
        finally:
            assert capi.hpmxp_set_tuning(0, 0, 0, 0) == capi.OK
        assert st == capi.OK
        outs.append(z)
    _check(outs[0], LU, V, n, fp32)
    assert np.array_equal(outs[0], outs[1])


@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("n,ld,offset", [(1, 1, 1), (63, 63, 0), (100, 101, 3), (128, 128, 1), (127, 128, 4)])
def test_one_block_of_unaligned_factors(n, ld, offset, fp32):
    A, _ = oracle.generate(n, 9)
    LU, _ = oracle.factor(A, oracle.BF16, 128)
    V = vectors(n, 2, n)
    st, z = _apply(LU, n, ld, capi.BF16, V, fp32, offset)
    assert st == capi.OK
    _check(z, LU, V, n, fp32)


def test_unaligned_factors_of_more_blocks_are_refused():
    n = 300
    st, _ = _apply(np.eye(n), n, 301, capi.BF16, vectors(n, 1, 1), 1)
    assert st == capi.EINVAL
