"""Workspace of the repeatable backward: what its passes use and no more (sizes
only, no launch)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def N():
    from paper_2408_11988_gb300.build import build
    from paper_2408_11988_gb300 import _native as N
    build()
    N.lib()
    return N


def _size(N, n, nnzA, nnzB, d, mode):
    # the boolean semiring reserves nothing for the autotuner's trials
    A, B = N.CsrDesc(n, n, nnzA, 8, 8, None), N.CsrDesc(n, d, nnzB, 8, 8, None)
    h, f, sz = ctypes.c_void_p(), N.Tuning.from_dict({"dB_mode": mode}), ctypes.c_size_t()
    assert N.lib().ts_plan_create(ctypes.byref(A), ctypes.byref(B), 1, ctypes.byref(f), ctypes.byref(h)) == N.TS_OK
    assert N.lib().ts_workspace_size(h, ctypes.byref(sz)) == N.TS_OK
    assert N.lib().ts_plan_destroy(h) == N.TS_OK
    return sz.value


@pytest.mark.parametrize("n,nnzA,nnzB,d", [(10**7, 10**6, 10**6, 64), (10**5, 10**7, 10**6, 200), (1000, 8000, 9000, 40),
                                           (10, 1, 1, 8)])
def test_repeatable_backward_regions(N, n, nnzA, nnzB, d):
    extra = _size(N, n, nnzA, nnzB, d, 2) - _size(N, n, nnzA, nnzB, d, 1)
    tiles = -(-nnzA // 8704)
    # rows, two keys and two payloads per entry of A; 1024 counters a tile of the sort and their scan; one column
    # pointer a row; the long columns' sums; 256 bytes of alignment each
    counters = 8 * 1024 * tiles
    need = 5 * 4 * nnzA + counters + 8 * (1024 * tiles // 4096 + 2) + 8 * (n + 1) + 4 * (nnzB + d * (nnzA // 512 + 1))
    assert need <= extra + 16 and extra <= need + 9 * 256
