"""Products of depth 128, whose tiles are short: ragged sizes against the SIMT
engine bit for bit up to rounding order (small integers, so every sum is exact),
stored, subtracted and with the row-major copy; and a stored product, which moves
half the bytes of a subtracted one, takes clearly less time."""
import pytest
import torch

from paper_2509_19618_gb300 import api, capi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
SUB, STORE = 0, 1


def _call(M, N, A, B, C, R, mode, engine, status):
    st = capi.hpmxp_test_gemm(M, N, 128, A.data_ptr(), 128, B.data_ptr(), 128, None if C is None else C.data_ptr(),
                              0 if C is None else C.shape[1], None if R is None else R.data_ptr(), N if R is not None else 0,
                              mode, 1.0, 0, 0, None, 0, None, 0, engine, status.data_ptr(), api.stream_handle())
    assert st == capi.OK


@pytest.mark.parametrize("M,N", [(1, 1), (127, 129), (128, 20000), (20001, 128), (2500, 2433), (129, 64 * 152 + 1)])
@pytest.mark.parametrize("mode,with_c,with_r", [(SUB, True, False), (STORE, True, False), (STORE, True, True), (STORE, False, True)])
def test_ragged(M, N, mode, with_c, with_r):
    g = torch.Generator(device=DEV).manual_seed(M + N)
    A, B = (torch.randint(-3, 4, (m, 128), generator=g, device=DEV).bfloat16() for m in (M, N))
    C0 = torch.randint(-99, 100, (N, -(-M // 8) * 8), generator=g, device=DEV).bfloat16()
    out = []
    for engine in (0, 1):
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        C = C0.clone() if with_c else None
        R = torch.zeros(M, N, device=DEV).bfloat16() if with_r else None
        _call(M, N, A, B, C, R, mode, engine, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        out.append((None if C is None else C[:, :M], R))   # rows past M are padding
    for x, y in zip(*out):
        assert x is None or torch.equal(x, y)


def test_stores_are_not_held_up():
    n = 16384
    A, B = (torch.randn(n, 128, device=DEV).bfloat16() for _ in range(2))
    C = torch.zeros(n, n, device=DEV).bfloat16()
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    t = {}
    for mode in (SUB, STORE):
        ts = []
        for _ in range(20):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            _call(n, n, A, B, C, None, mode, 0, status)
            e1.record()
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        t[mode] = sorted(ts)[8]
    assert t[STORE] <= 0.82 * t[SUB], t
