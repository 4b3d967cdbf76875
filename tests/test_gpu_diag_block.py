"""Diagonal-block kernels on blocks that leave the branch-free division's range
(zeros, -0, pivots and entries below 2^-60), against the oracle bit for bit on
the SIMT engine; 200 and 300 also run the inverses
(they feed the panels) on full and ragged blocks."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu


def _matrix(n, kind):
    g = np.random.default_rng(100 + n)
    A = g.uniform(-0.5, 0.5, size=(n, n))
    A[np.arange(n), np.arange(n)] = n * (1.0 + g.random(n))
    if kind == "zeros":          # structural zeros of both signs
        A[g.random((n, n)) < 0.3] = 0.0
        A[g.random((n, n)) < 0.1] = -0.0
        A[np.arange(n), np.arange(n)] = n
    elif kind == "tiny":         # every entry and pivot below the range
        A *= 2.0**-75
    elif kind == "graded":       # some rows below the range, some pivots tiny
        A *= np.where(np.arange(n) % 7 == 3, 2.0**-66, 1.0)[:, None]
    elif kind == "ones":         # pivots start at BF16's all-ones significand; lower triangular
        A[np.arange(n), np.arange(n)] = 255.0 * 2.0**-7
        A -= np.triu(A, 1) + np.tril(A, -1) * (1 - 2.0**-9)
    elif kind == "below_pow2":   # pivots one fp32 ulp below a power of two
        A = np.abs(A) * 0.5
        A[np.arange(n), np.arange(n)] = 2048.0
    return np.asfortranarray(A)


@pytest.mark.parametrize("kind", ["plain", "zeros", "tiny", "graded", "ones", "below_pow2"])
@pytest.mark.parametrize("n", [1, 16, 17, 40, 128, 200, 300])
def test_diagonal_block_bit_exact(n, kind, monkeypatch):
    A_o = _matrix(n, kind)
    monkeypatch.setenv("HPMXP_GEMM_ENGINE", "simt")
    LU = api.factor(api.ColMajor.from_tensor(torch.from_numpy(A_o), "cuda"), capi.BF16, 128)
    torch.cuda.synchronize()
    got = LU.view().double().cpu().numpy()
    want, rc = oracle.factor(A_o, oracle.BF16, 128)
    assert rc == 0
    assert np.array_equal(got, want), np.argwhere(got != want)[:5]
    if n <= 128:   # one block: the signs of zeros too
        assert np.array_equal(np.signbit(got), np.signbit(want))
