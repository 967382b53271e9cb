"""Light rows of a product of so many rows that every warp has many units: only
rows of 2048 products and more are shared by a warp's slots then (numeric and
backward from some 780,000 light rows on, the symbolic pass from twice as many, on
152 SMs).  Forward and gradients against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from _cmp import REL, compare_full
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR, Plan


@pytest.mark.parametrize("d,per_row", [(64, 10.0), (100, 12.0)])
def test_many_units(d, per_row):
    n = 1_750_000
    rng = np.random.default_rng(d)
    lens = np.ones(n, dtype=np.int64)  # one entry, so that almost every row is light
    at = rng.permutation(n)
    # products about per_row times these: 100 .. 511, 512 .. 2047, 2048 .. 4095, and block rows
    want = [12, 40, 51, 52, 60, 120, 200, 204, 205, 206, 300, 400, 409, 410, 500, 1100]
    lens[at[:40 * len(want)]] = np.tile(want, 40)
    lens[at[-50_000:]] = 0
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rowptr[1:])
    rows = np.repeat(np.arange(n), lens)
    key = np.unique(rows * n + rng.integers(0, n, rows.size))
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=rowptr[1:])
    A = CSR(n, n, rowptr, (key % n).astype(np.int32))
    A.val = synth.uniform(A.nnz, 1)
    B = synth.tall_skinny(n, d, per_row / d, 2)
    B.val = synth.normal(B.nnz, 3)
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    plan = Plan(Ad, Bd)
    assert plan.tuning["cta_min_flops"] == 4096
    C = plan.forward(Ad, Bd)
    Cp, Ci, _, _ = compare_full(C, A, B)
    dC = synth.grad_output(C.nnz, 4)
    dA, dB = plan.backward(Ad, Bd, C, torch.as_tensor(dC, device="cuda"))
    plan.check()
    rA, bA, rB, bB = oracle.backward(A, B, Cp, Ci, dC.astype(np.float64))
    assert np.all(np.abs(dA.cpu().numpy() - rA) <= REL * bA)
    assert np.all(np.abs(dB.cpu().numpy() - rB) <= REL * bB)
