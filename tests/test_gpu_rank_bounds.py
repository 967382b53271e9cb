"""Ranked columns (4096 < d <= 32768): a row's class comes from the products
counted by the symbolic pass, the columns from what the numeric pass walks.  A
row of B that grew in between (its pattern rewritten in place, the sizes as
before) must be reported, at more columns than a warp's row holds values
(1024) as below that, and leave every other row and the next product right."""
import numpy as np
import pytest
import torch

import oracle
import synth
from _cmp import assert_values_close, compare_full
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import OR_SELECT2ND, PLUS_TIMES, DeviceCSR, Plan, TSError


def _b(lens, d, seed):
    rng = np.random.default_rng(seed)
    rp = np.zeros(len(lens) + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    B = CSR(len(lens), d, rp, np.concatenate([np.sort(rng.choice(d, m, replace=False)) for m in lens]).astype(np.int32))
    B.val = synth.normal(B.nnz, seed + 1)
    return B


@pytest.mark.parametrize("semiring", [PLUS_TIMES, OR_SELECT2ND])
@pytest.mark.parametrize("grown", [900, 1023, 1024, 1025, 3000, 8000])
def test_row_of_b_grown_after_the_symbolic_pass(grown, semiring):
    n, d, k0 = 2500, 8192, 5
    # A: row i holds column i alone; rows 0..299 hold k0 as well
    rows = [[i] if i >= 300 or i == k0 else sorted({i, k0}) for i in range(n)]
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum([len(r) for r in rows], out=rp[1:])
    A = CSR(n, n, rp, np.concatenate(rows).astype(np.int32))
    A.val = synth.uniform(A.nnz, 1)
    lens = np.full(n, 4)
    lens[k0] = 100
    B = _b(lens, d, 2)
    wide = lens.copy()  # the same number of entries, k0's row longer, rows from 1000 on empty or shorter
    wide[k0] = grown
    at = n
    while wide.sum() > lens.sum():
        at -= 1
        wide[at] -= min(wide[at], wide.sum() - lens.sum())
    assert at >= 300 and wide.sum() == lens.sum()
    B2 = _b(wide, d, 3)
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    plan = Plan(Ad, Bd, semiring)
    C = plan.forward(Ad, Bd)
    plan.check()
    compare_full(C, A, B, semiring)
    rowptr, nnz = plan.symbolic(Ad, Bd)
    C = plan.alloc_c(rowptr, nnz)
    for t, h in ((Bd.rowptr, B2.rowptr), (Bd.col, B2.col), (Bd.val, B2.val)):
        t.copy_(torch.as_tensor(h).to(t.dtype))
    plan.numeric(Ad, Bd, C)
    with pytest.raises(TSError):
        plan.check()
    # rows that do not meet a changed length are whole
    grp, col, val = C.to_host()
    Cp, Ci, Cx, Cb = oracle.spgemm(A, B2, semiring=semiring)
    for i in range(300, at):
        assert np.array_equal(col[grp[i]:grp[i + 1]], Ci[Cp[i]:Cp[i + 1]]), i
        if semiring == PLUS_TIMES:
            assert_values_close(val[grp[i]:grp[i + 1]], Cx[Cp[i]:Cp[i + 1]], Cb[Cp[i]:Cp[i + 1]])
    C = plan.forward(Ad, Bd)  # the product of what is there now
    plan.check()
    compare_full(C, A, B2, semiring)
