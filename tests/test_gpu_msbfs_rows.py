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
