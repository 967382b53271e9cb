"""The pull form of the multi-source BFS at the row lengths where its paths
meet: a lane per row, a warp per row (64 or 128 entries a step), blocks of 4096
entries.  Integers: bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR, TSError
from paper_2408_11988_gb300.msbfs import msbfs

LENGTHS = [0, 1, 3, 15, 16, 17, 31, 33, 63, 64, 65, 127, 128, 129, 255, 257, 2047, 2048, 2049, 4095, 4096, 4097, 8193]


def _graph(n, seed, copies=3):
    """Directed: `copies` rows of every length among n vertices, the others with 0 to 4 entries."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 5, n)
    at = rng.permutation(n)[:copies * len(LENGTHS)]
    lens[at] = np.tile([min(x, n) for x in LENGTHS], copies)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rowptr[1:])
    col = np.concatenate([np.sort(rng.choice(n, m, replace=False)) for m in lens] or [[]]).astype(np.int32)
    return CSR(n, n, rowptr, col), at


@pytest.mark.parametrize("d", [1, 32, 33, 65, 128, 129, 256])
@pytest.mark.parametrize("n", [9001, 30016])
def test_row_lengths(n, d):
    A, _ = _graph(n, n + d)
    src = np.random.default_rng(d).choice(n, d, replace=False).astype(np.int32)
    r = msbfs(DeviceCSR.from_host(A, with_values=False), torch.as_tensor(src), parents=True)
    lev, par, prods, fnnz = oracle.msbfs_parents(A, src)
    np.testing.assert_array_equal(r.levels.cpu().numpy(), lev)
    np.testing.assert_array_equal(r.parents.cpu().numpy(), par)
    assert r.products == prods and list(r.frontier_nnz) == list(fnnz)
    q = msbfs(DeviceCSR.from_host(A, with_values=False), torch.as_tensor(src))
    np.testing.assert_array_equal(q.levels.cpu().numpy(), lev)
    assert q.products == prods and list(q.frontier_nnz) == list(fnnz)


@pytest.mark.parametrize("length", [1, 16, 17, 129, 2049, 8193])
@pytest.mark.parametrize("bad", [-1, 9001])
def test_bad_column_is_reported(length, bad):
    # wherever it stands, also in a row whose sources were all found before it
    A, at = _graph(9001, 5)
    row = at[LENGTHS.index(length)]
    col = A.col.copy()
    col[(A.rowptr[row] if bad < 0 else A.rowptr[row + 1] - 1)] = bad
    with pytest.raises(TSError):
        msbfs(DeviceCSR.from_host(CSR(A.nrows, A.ncols, A.rowptr, col), with_values=False),
              torch.as_tensor(np.array([row, 3], dtype=np.int32)))


@pytest.mark.parametrize("d", [3, 40])
def test_long_search_and_max_levels(d):
    # a path of 600 vertices: more levels than one call of the library makes, and a search cut short
    n = 600
    rowptr = np.zeros(n + 1, dtype=np.int64)
    lens = np.full(n, 2)
    lens[[0, -1]] = 1
    np.cumsum(lens, out=rowptr[1:])
    col = np.concatenate([[v for v in (i - 1, i + 1) if 0 <= v < n] for i in range(n)]).astype(np.int32)
    A = CSR(n, n, rowptr, col)
    src = np.arange(d, dtype=np.int32)
    lev, par, prods, fnnz = oracle.msbfs_parents(A, src)
    Ad = DeviceCSR.from_host(A, with_values=False)
    r = msbfs(Ad, torch.as_tensor(src), parents=True)
    np.testing.assert_array_equal(r.levels.cpu().numpy(), lev)
    np.testing.assert_array_equal(r.parents.cpu().numpy(), par)
    assert r.products == prods and list(r.frontier_nnz) == list(fnnz)
    for most in (0, 1, 5, 256, 300):
        q = msbfs(Ad, torch.as_tensor(src), max_levels=most)
        np.testing.assert_array_equal(q.levels.cpu().numpy(), np.where(lev <= most, lev, -1))
        assert q.products == most and list(q.frontier_nnz) == list(fnnz[:most + 1])


def test_steps_agree_with_the_search():
    # msbfs_step and msbfs_step_parents, level by level, on the rows of test_row_lengths
    import ctypes

    from paper_2408_11988_gb300 import _native as N
    from paper_2408_11988_gb300.ops import _ptr, _stream
    for n, d in ((9001, 40), (9001, 200), (9001, 300)):
        A, _ = _graph(n, 7)
        src = np.random.default_rng(d).choice(n, d, replace=False).astype(np.int32)
        lev, prods, fnnz = oracle.msbfs(A, src)
        Ad = DeviceCSR.from_host(A, with_values=False)
        sd = torch.as_tensor(src).cuda()
        sz = ctypes.c_size_t()
        N.call("msbfs_workspace_size", n, A.nnz, d, ctypes.byref(sz))
        ws = torch.empty(int(sz.value), dtype=torch.uint8, device="cuda")
        S = torch.empty(n * ((d + 31) // 32), dtype=torch.int32, device="cuda")
        levels = torch.empty(n * d, dtype=torch.int32, device="cuda")
        par = torch.empty(n * d, dtype=torch.int32, device="cuda")
        F, G = (DeviceCSR(n, d, torch.empty(n + 1, dtype=torch.int64, device="cuda"),
                          torch.empty(n * d, dtype=torch.int32, device="cuda")) for _ in range(2))
        f = F.desc()
        N.call("msbfs_init", n, d, _ptr(sd), _ptr(S), _ptr(levels), ctypes.byref(f), _stream())
        if d <= 256:
            N.call("msbfs_init_parents", n, d, _ptr(sd), _ptr(par), _stream())
        F.nnz_, sizes = d, [d]
        while F.nnz:
            a, f, g, nnz = Ad.desc(), F.desc(), G.desc(), ctypes.c_int64()
            tail = (len(sizes), ctypes.byref(g), n * d, ctypes.byref(nnz), _ptr(ws), ws.numel(), _stream())
            if d <= 256:
                N.call("msbfs_step_parents", ctypes.byref(a), ctypes.byref(f), _ptr(S), _ptr(levels), _ptr(par), *tail)
            else:
                N.call("msbfs_step", ctypes.byref(a), ctypes.byref(f), _ptr(S), _ptr(levels), *tail)
            G.nnz_ = nnz.value
            sizes.append(G.nnz)
            F, G = G, F
        np.testing.assert_array_equal(levels.cpu().numpy().reshape(n, d), lev)
        assert sizes == list(fnnz)
        if d <= 256:
            np.testing.assert_array_equal(par.cpu().numpy().reshape(n, d), oracle.msbfs_parents(A, src)[1])
