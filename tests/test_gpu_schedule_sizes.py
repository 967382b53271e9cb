"""Row counts at the edges of the schedule's and the scan's launches: one tile,
clusters of two, four and eight tiles (4096 rows each), separate passes, and
one or eight rows a thread in the ordering of the rows."""
import numpy as np
import pytest

import synth
from _cmp import compare_full
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR, Plan


@pytest.mark.parametrize("n", [1, 255, 257, 4095, 4096, 4097, 8192, 8193, 12289, 16384, 16385, 32767, 32768, 32769,
                               (1 << 18) - 1, 1 << 18])
@pytest.mark.parametrize("d", [40, 600])
def test_rows(n, d):
    rng = np.random.default_rng(n + d)
    lens = rng.integers(0, 4, n)
    lens[rng.integers(0, n, 3)] = min(n, 1100)  # some rows cut into parts
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rowptr[1:])
    first = rng.integers(0, n, n)
    col = np.concatenate([np.sort((first[i] + np.arange(m) * max(1, n // max(m, 1))) % n) if m <= 4 else
                          np.sort(rng.choice(n, m, replace=False)) for i, m in enumerate(lens)]).astype(np.int32)
    A = CSR(n, n, rowptr, col)
    A.val = synth.uniform(A.nnz, n + 1)
    B = synth.tall_skinny(n, d, 3.0 / d, n + 2)
    B.val = synth.normal(B.nnz, n + 3)
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    plan = Plan(Ad, Bd)
    for _ in range(2):  # the second pass on a used workspace
        C = plan.forward(Ad, Bd)
        plan.check()
        compare_full(C, A, B)
