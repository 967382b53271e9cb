"""Products of more than 4096 columns with the chosen accumulator (ranked
columns up to 32768, hashing above), at the lines between rows in registers,
warp rows and block rows, and rows of more columns than a block holds values."""
import numpy as np
import pytest

import oracle
import synth
from _cmp import compare_full
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import OR_SELECT2ND, PLUS_TIMES, DeviceCSR, Plan


@pytest.mark.parametrize("semiring", [PLUS_TIMES, OR_SELECT2ND])
@pytest.mark.parametrize("d", [4097, 8191, 20000, 32768, 32769])
@pytest.mark.parametrize("per_row", [4, 16])
def test_many_columns(d, per_row, semiring):
    n = 2600
    rng = np.random.default_rng(d + per_row)
    lens = rng.integers(0, 7, n)
    # products = entries * per_row: 28 .. 32, 1020 .. 1028, then block rows of
    # both kernels, one with almost every row of B
    want = np.array([28, 32, 36, 1020, 1024, 1028, 1280, 8192, 9600, 16380, 16384, 16400, 33000]) // per_row
    lens[rng.permutation(n)[:want.size]] = np.minimum(want, n)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rowptr[1:])
    A = CSR(n, n, rowptr, np.concatenate([np.sort(rng.choice(n, m, replace=False)) for m in lens]).astype(np.int32))
    A.val = synth.uniform(A.nnz, 1)
    B = synth.tall_skinny(n, d, per_row / d, 2)
    lose = rng.random(n) < 0.1  # some empty rows of B
    keep = np.repeat(~lose, B.row_lengths())
    B = CSR(n, d, np.concatenate([[0], np.cumsum(np.where(lose, 0, B.row_lengths()))]).astype(np.int64), B.col[keep])
    B.val = synth.normal(B.nnz, 3)
    plan = Plan(DeviceCSR.from_host(A), DeviceCSR.from_host(B), semiring)
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    for _ in range(2):
        C = plan.forward(Ad, Bd)
    plan.check()
    compare_full(C, A, B, semiring)
