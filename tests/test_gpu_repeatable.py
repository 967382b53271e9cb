"""The repeatable dB (dB_mode = 2): bit for bit the same on every call, against
the oracle, over the widths of B's rows (8, 16 and 32 lanes), of C's bitmaps,
with and without room for these (binary search), columns at the chunk's line,
and sizes at the lines of the sort's digits and tiles."""
import numpy as np
import pytest
import torch

import oracle
import synth
from _cmp import REL
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR, Plan


def _check(A, B, tuning):
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    plan = Plan(Ad, Bd, tuning=dict(tuning, dB_mode=2))
    C = plan.forward(Ad, Bd)
    dC = torch.as_tensor(synth.grad_output(C.nnz, 7), device="cuda")
    dA, dB = plan.backward(Ad, Bd, C, dC)
    plan.check()
    for _ in range(2):
        assert torch.equal(plan.backward(Ad, Bd, C, dC)[1], dB)
    plan.forward(Ad, Bd)
    rp, col, _ = C.to_host()
    rA, bA, rB, bB = oracle.backward(A, B, rp, col, dC.double().cpu().numpy())
    assert np.all(np.abs(dA.cpu().numpy() - rA) <= REL * bA)
    assert np.all(np.abs(dB.cpu().numpy() - rB) <= REL * bB)


@pytest.mark.parametrize("d,per_row", [(1, 1), (32, 3), (33, 8), (64, 9), (100, 16), (129, 17), (256, 40), (257, 6)])
@pytest.mark.parametrize("tuning", [{}, {"pack_b": 2}])
def test_widths_and_long_columns(d, per_row, tuning):
    # columns of 512, 513, 1024 and 1700 entries beside short and empty ones
    n = 1700
    rng = np.random.default_rng(d)
    rows = [set(rng.choice(n, 3, replace=False)) - {11, 12, 13, 14, 15} for _ in range(n)]
    for c, m in ((11, 512), (12, 513), (13, 1024), (14, n)):
        for r in rng.choice(n, m, replace=False):
            rows[r].add(c)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    rowptr[1:] = np.cumsum([len(r) for r in rows])
    A = CSR(n, n, rowptr, np.concatenate([np.sort(np.array(list(r), dtype=np.int32)) for r in rows]),
            synth.uniform(int(rowptr[-1]), 8))
    B = synth.tall_skinny(n, d, per_row / d, 9)
    lens = np.where(rng.random(n) < 0.1, 0, B.row_lengths())
    B = CSR(n, d, np.concatenate([[0], np.cumsum(lens)]).astype(np.int64), B.col[np.repeat(lens > 0, B.row_lengths())])
    B.val = synth.normal(B.nnz, 10)
    _check(A, B, tuning)


@pytest.mark.parametrize("n,k", [(1, 1), (2, 2), (1024, 8), (1025, 8), (2730, 3), (8704, 1), (8705, 1), (17408, 1), (4096, 4), (33000, 1), (70000, 2)])
def test_sizes_of_the_sort(n, k):
    A, B = synth.er_product(n=n, k=k, d=48, density=0.08, seed=11)
    _check(A, B, {})
