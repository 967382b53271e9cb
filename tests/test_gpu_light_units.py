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

from paper_2408_11988_gb300 import OR_SELECT2ND, DeviceCSR, Plan

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


@pytest.mark.parametrize("n,d,per_row,copies", [(1100, 513, 6.0, 3), (1100, 1024, 3.0, 1), (1300, 700, 12.0, 2),
                                                (1500, 2050, 7.0, 1)])
@pytest.mark.parametrize("tuning", [None, {"cta_min_flops": 1 << 20}, {"warps_per_cta": 1}, {"bwd_group": 1},
                                    {"pack_b": 2}])
def test_rows_of_a_whole_warp(n, d, per_row, copies, tuning):
    test_units(n, d, per_row, copies, tuning)


def _line(n, d, per_row, **plan):
    nnz = int(n * per_row + 1)
    rowptr = np.minimum(np.arange(n + 1, dtype=np.int64) * -(-nnz // n), nnz)
    lens = np.diff(rowptr)
    B = CSR(n, d, rowptr, (np.arange(nnz) - np.repeat(rowptr[:-1], lens)).astype(np.int32))
    B.val = np.ones(nnz, np.float32)
    A = CSR(n, n, np.zeros(n + 1, np.int64), np.zeros(0, np.int32))
    A.val = np.zeros(0, np.float32)
    return Plan(DeviceCSR.from_host(A), DeviceCSR.from_host(B), **plan).tuning["cta_min_flops"]


@pytest.mark.parametrize("n,want", [((1 << 17) - 1, 1024), (1 << 17, 4096)])
@pytest.mark.parametrize("d,plan", [(600, {"semiring": OR_SELECT2ND}), (600, {"tuning": {"col_tile": 256}}), (1025, {})])
def test_line_without_the_wide_kernel(n, want, d, plan):
    assert _line(n, d, 4.6, **plan) == want


@pytest.mark.parametrize("n,d,per_row,want", [(3000, 64, 4.0, 1024), (3000, 512, 4.6, 2048), (3000, 513, 4.6, 1024),
                                              (3000, 513, 4.4, 1024), (3000, 513, 9.0, 4096),
                                              (1 << 20, 513, 4.6, 4096), ((1 << 20) - 1, 513, 4.6, 1024),
                                              (1 << 20, 512, 4.6, 2048)])
def test_line_of_the_heavy_rows(n, d, per_row, want):
    assert _line(n, d, per_row) == want
