"""Light rows as the row-group kernels deal them out: rows shared by a warp's
slots, rows in a slot each, with row lengths at the lines between them, tile
remainders in d, and few rows or (threshold raised) rows far above the usual
line; forward and both gradients against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from _cmp import REL, compare_full
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR, Plan

ENTRIES = [0, 1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 513, 1023, 1025]


def _inputs(n, d, per_row, copies, seed):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 6, n)
    at = rng.permutation(n)[:copies * len(ENTRIES)]
    lens[at] = np.tile([min(x, n) for x in ENTRIES], copies)[:at.size]
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rowptr[1:])
    A = CSR(n, n, rowptr, np.concatenate([np.sort(rng.choice(n, m, replace=False)) for m in lens]).astype(np.int32))
    A.val = synth.uniform(A.nnz, seed + 1)
    B = synth.tall_skinny(n, d, per_row / d, seed + 2)
    B.val = synth.normal(B.nnz, seed + 3)
    return A, B


@pytest.mark.parametrize("n,d,per_row,copies", [(1100, 256, 4.0, 1), (1100, 33, 2.5, 3), (2000, 128, 8.0, 20),
                                                (2000, 250, 1.0, 5), (40, 64, 16.0, 1), (9000, 512, 3.3, 100)])
@pytest.mark.parametrize("tuning", [None, {"cta_min_flops": 1 << 20}, {"warps_per_cta": 1}, {"row_lanes": 4},
                                    {"row_lanes": 16}])
def test_units(n, d, per_row, copies, tuning):
    if d > 256 and tuning and "row_lanes" in tuning:
        pytest.skip("row groups over one tile: d <= 256")
    A, B = _inputs(n, d, per_row, copies, n + d)
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    plan = Plan(Ad, Bd, tuning=tuning)
    C = plan.forward(Ad, Bd)
    Cp, Ci, _, _ = compare_full(C, A, B)
    dC = synth.grad_output(C.nnz, 5)
    dA, dB = plan.backward(Ad, Bd, C, torch.as_tensor(dC, device="cuda"))
    plan.check()
    rA, bA, rB, bB = oracle.backward(A, B, Cp, Ci, dC.astype(np.float64))
    assert np.all(np.abs(dA.cpu().numpy() - rA) <= REL * bA)
    assert np.all(np.abs(dB.cpu().numpy() - rB) <= REL * bB)
