"""The BFS pull where a warp owns 16 and 32 rows, a half and a whole word of the
bits of non-empty frontier rows (from 38,912 and 77,824 vertices on a chip of 152
SMs): searches and single steps, levels and parents bit for bit."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from test_gpu_msbfs_rows import _graph

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR
from paper_2408_11988_gb300 import _native as N
from paper_2408_11988_gb300.msbfs import msbfs
from paper_2408_11988_gb300.ops import _ptr, _stream


@pytest.mark.parametrize("d", [20, 64, 128, 200])
@pytest.mark.parametrize("n", [40_000, 80_001])
def test_rows_per_warp(n, d):
    A, _ = _graph(n, n + d)
    src = np.random.default_rng(d).choice(n, d, replace=False).astype(np.int32)
    lev, par, prods, fnnz = oracle.msbfs_parents(A, src)
    Ad = DeviceCSR.from_host(A, with_values=False)
    for parents in (True, False):
        r = msbfs(Ad, torch.as_tensor(src), parents=parents)
        np.testing.assert_array_equal(r.levels.cpu().numpy(), lev)
        assert r.products == prods and list(r.frontier_nnz) == list(fnnz)
        if parents:
            np.testing.assert_array_equal(r.parents.cpu().numpy(), par)
    # the same, step by step
    sd, sz = torch.as_tensor(src).cuda(), ctypes.c_size_t()
    N.call("msbfs_workspace_size", n, A.nnz, d, ctypes.byref(sz))
    ws = torch.empty(int(sz.value), dtype=torch.uint8, device="cuda")
    S = torch.empty(n * ((d + 31) // 32), dtype=torch.int32, device="cuda")
    levels, parent = (torch.empty(n * d, dtype=torch.int32, device="cuda") for _ in range(2))
    F, G = (DeviceCSR(n, d, torch.empty(n + 1, dtype=torch.int64, device="cuda"),
                      torch.empty(n * d, dtype=torch.int32, device="cuda")) for _ in range(2))
    f = F.desc()
    N.call("msbfs_init", n, d, _ptr(sd), _ptr(S), _ptr(levels), ctypes.byref(f), _stream())
    N.call("msbfs_init_parents", n, d, _ptr(sd), _ptr(parent), _stream())
    F.nnz_, sizes = d, [d]
    while F.nnz:
        a, f, g, nnz = Ad.desc(), F.desc(), G.desc(), ctypes.c_int64()
        N.call("msbfs_step_parents", ctypes.byref(a), ctypes.byref(f), _ptr(S), _ptr(levels), _ptr(parent), len(sizes),
               ctypes.byref(g), n * d, ctypes.byref(nnz), _ptr(ws), ws.numel(), _stream())
        G.nnz_ = nnz.value
        sizes.append(G.nnz)
        F, G = G, F
    assert sizes == list(fnnz)
    np.testing.assert_array_equal(levels.cpu().numpy().reshape(n, d), lev)
    np.testing.assert_array_equal(parent.cpu().numpy().reshape(n, d), par)
