"""msbfs_search: arguments that are refused on the host, before any launch."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2408_11988_gb300.build import build
    from paper_2408_11988_gb300 import _native as N
    build()
    return N.lib()


P = ctypes.c_void_p(256)  # non-NULL and aligned, never dereferenced


def search(lib, n=10, ncols=None, nnz=30, d=8, src=P, levels=P, start=0, max_steps=4, nnz_out=True, steps=True, ws=P,
           ws_bytes=None):
    from paper_2408_11988_gb300 import _native as N
    A = N.CsrDesc(n, n if ncols is None else ncols, nnz, 8, 8, None)
    out, done = (ctypes.c_int64 * 4)(), ctypes.c_int64()
    need = ctypes.c_size_t()
    if ws_bytes is None:
        assert lib.msbfs_search_workspace_size(n, nnz, max(1, min(d, 256)), ctypes.byref(need)) == N.TS_OK
        ws_bytes = need.value - 1  # a call that gets as far as the workspace stops there
    return lib.msbfs_search(ctypes.byref(A), d, src, levels, None, start, max_steps, out if nnz_out else None,
                            ctypes.byref(done) if steps else None, ws, ws_bytes, None)


def test_search_workspace_size(lib):
    from paper_2408_11988_gb300 import _native as N
    sz = ctypes.c_size_t()
    assert lib.msbfs_search_workspace_size(10, 30, 256, ctypes.byref(sz)) == N.TS_OK and sz.value > 0
    assert lib.msbfs_search_workspace_size(10, 30, 257, ctypes.byref(sz)) == N.TS_ERR_UNSUPPORTED
    for bad in ((-1, 30, 8), (10, -1, 8), (10, 30, 0)):
        assert lib.msbfs_search_workspace_size(*bad, ctypes.byref(sz)) == N.TS_ERR_INVALID_ARG
    assert lib.msbfs_search_workspace_size(10, 30, 8, None) == N.TS_ERR_INVALID_ARG


def test_search_arguments(lib):
    from paper_2408_11988_gb300 import _native as N
    for bad in ({"d": 0}, {"src": None}, {"levels": None}, {"start": -1}, {"max_steps": -1}, {"steps": False},
                {"nnz_out": False}, {"ncols": 9}):
        assert search(lib, **bad) == N.TS_ERR_INVALID_ARG, bad
    assert search(lib, d=257) == N.TS_ERR_UNSUPPORTED
    assert search(lib) == N.TS_ERR_WORKSPACE_TOO_SMALL
    assert search(lib, ws=None, ws_bytes=1 << 30) == N.TS_ERR_WORKSPACE_TOO_SMALL
    assert search(lib, ws=ctypes.c_void_p(264), ws_bytes=1 << 30) == N.TS_ERR_INVALID_ARG
    # no steps asked for: the counts may be NULL
    assert search(lib, max_steps=0, nnz_out=False) == N.TS_ERR_WORKSPACE_TOO_SMALL


@pytest.mark.parametrize("start,max_steps", [(2**31 - 1, 1), (0, 2**31), (2**31, 0), (2**62, 2**62), (2**63 - 1, 1),
                                             (1, 2**63 - 1), (2**63 - 1, 2**63 - 1)])
def test_levels_are_32_bit(lib, start, max_steps):
    from paper_2408_11988_gb300 import _native as N
    assert search(lib, start=start, max_steps=max_steps) == N.TS_ERR_OVERFLOW
