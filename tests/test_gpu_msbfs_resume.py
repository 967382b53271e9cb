"""msbfs_search call by call: no level at all, and searches resumed after any
number of levels."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR
from paper_2408_11988_gb300 import _native as N
from paper_2408_11988_gb300.msbfs import msbfs


def test_search_of_no_levels_waits_for_its_stream():
    # the workspace is freed when the call returns, on another stream than its own
    G = synth.rmat(10, 8, 1, symmetrize=True)
    src = synth.sources(G, 40, 2)
    A = DeviceCSR.from_host(G, with_values=False)
    st = torch.cuda.Stream()
    msbfs(A, torch.as_tensor(src), stream=st)
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        torch.cuda._sleep(200_000_000)
    r = msbfs(A, torch.as_tensor(src), max_levels=0, stream=st, parents=True)
    assert st.query(), "work of the search is still queued"
    lev, par = r.levels.cpu().numpy(), r.parents.cpu().numpy()
    want = np.full_like(lev, -1)
    want[src, np.arange(40)] = 0
    np.testing.assert_array_equal(lev, want)
    assert r.products == 0 and r.frontier_nnz == [40]
    assert np.array_equal(par[src, np.arange(40)], src) and int((par >= 0).sum()) == 40


def _graph_with_tail(seed, tail=30):
    """An R-MAT graph with a path of `tail` vertices hanging from vertex 0, and one of another component."""
    G = synth.rmat(9, 6, seed, symmetrize=True)
    n = G.nrows + tail + 5
    edges = {(int(i), int(j)) for i in range(G.nrows) for j in G.col[G.rowptr[i]:G.rowptr[i + 1]]}
    path = [0] + list(range(G.nrows, G.nrows + tail))
    for a, b in zip(path, path[1:]):
        edges |= {(a, b), (b, a)}
    rows = sorted(edges)
    rp = np.zeros(n + 1, dtype=np.int64)
    for i, _ in rows:
        rp[i + 1] += 1
    return CSR(n, n, np.cumsum(rp), np.array([j for _, j in rows], dtype=np.int32))


@pytest.mark.parametrize("steps", [[1], [2], [3], [5, 1, 7, 2], [6, 0, 3], [9, 4]])
@pytest.mark.parametrize("d", [3, 50, 130])
def test_search_resumed_after_any_number_of_levels(d, steps):
    G = _graph_with_tail(d)
    src = synth.sources(G, d, 4)
    lev, par, products, _ = oracle.msbfs_parents(G, src)
    assert products > 20
    A = DeviceCSR.from_host(G, with_values=False)
    whole = msbfs(A, torch.as_tensor(src), parents=True)
    n = G.nrows
    sz, done = ctypes.c_size_t(), ctypes.c_int64()
    N.call("msbfs_search_workspace_size", n, A.nnz, d, ctypes.byref(sz))
    ws = torch.empty(sz.value, dtype=torch.uint8, device="cuda")
    s = torch.as_tensor(src).to("cuda", torch.int32)
    levels, parents = (torch.empty(n * d, dtype=torch.int32, device="cuda") for _ in range(2))
    sizes, calls = [], 0
    while True:
        m = steps[calls % len(steps)]
        calls += 1
        out = (ctypes.c_int64 * max(m, 1))()
        a = A.desc()
        N.call("msbfs_search", ctypes.byref(a), d, s.data_ptr(), levels.data_ptr(), parents.data_ptr(), len(sizes), m,
               out, ctypes.byref(done), ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
        assert done.value <= m
        sizes += out[:done.value]
        if sizes and sizes[-1] == 0:
            break
        assert done.value == m and calls < 200
    assert [d] + sizes == whole.frontier_nnz and len(sizes) == whole.products == products
    np.testing.assert_array_equal(levels.view(n, d).cpu().numpy(), lev)
    np.testing.assert_array_equal(parents.view(n, d).cpu().numpy(), par)
