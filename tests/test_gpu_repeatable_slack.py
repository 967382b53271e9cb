"""Repeatable dB of an A whose arrays hold more entries than its rows (room
before the first row and behind the last): the entries of no row take no part in
C, dA and dB, and dB repeats bit for bit.  (The groups a column is summed in count
its stored entries, those of no row among them, so its bits may differ from the
trimmed matrix's.)"""
import numpy as np
import pytest
import torch

import oracle
import synth
from _cmp import REL, compare_full

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR, Plan


@pytest.mark.parametrize("n", [64, 2048, 2049, 5000])
@pytest.mark.parametrize("d", [40, 300])
@pytest.mark.parametrize("lead,slack", [(0, 1), (0, 700), (33, 5), (600, 1300)])
def test_entries_of_no_row(n, d, lead, slack):
    scale = max(1, (n - 1).bit_length())
    A = synth.rmat(scale, 6, 7)
    rp = np.minimum(A.rowptr[:n + 1], A.rowptr[n])
    col = (A.col[:rp[n]] % n).astype(np.int32)
    # distinct columns in every row after the fold
    key = np.unique(np.repeat(np.arange(n), np.diff(rp)) * n + col)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=rp[1:])
    A = synth.CSR(n, n, rp, (key % n).astype(np.int32))
    A.val = synth.uniform(A.nnz, 8)
    B = synth.tall_skinny(n, d, 6 / d, 9)
    B.val = synth.normal(B.nnz, 10)
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    rng = np.random.default_rng(11)
    junk = rng.integers(0, 2 * n, lead + slack).astype(np.int32)  # columns past the last among them
    col = np.concatenate([junk[:lead], A.col, junk[lead:]])
    val = np.concatenate([np.full(lead, np.nan, np.float32), A.val, np.full(slack, np.nan, np.float32)])
    Aw = DeviceCSR(n, n, torch.as_tensor(A.rowptr + lead).cuda(), torch.as_tensor(col).cuda(), torch.as_tensor(val).cuda())
    got = []
    for M in (Ad, Aw, Aw):
        plan = Plan(M, Bd, tuning={"dB_mode": 2})
        C = plan.forward(M, Bd)
        plan.workspace().fill_(0x11)  # rows that read what nobody wrote would show
        C = plan.forward(M, Bd)
        dC = torch.as_tensor(synth.grad_output(C.nnz, 12), device="cuda")
        dA, dB = plan.backward(M, Bd, C, dC)
        plan.check()
        got.append((C, dA, dB))
    Cp, Ci, _, _ = compare_full(got[1][0], A, B)
    rA, bA, rB, bB = oracle.backward(A, B, Cp, Ci, dC.cpu().numpy().astype(np.float64))
    assert np.all(np.abs(got[1][1].cpu().numpy()[lead:lead + A.nnz] - rA) <= REL * bA)
    dB = got[1][2].cpu().numpy()
    assert np.all(np.abs(dB - rB) <= REL * bB)
    np.testing.assert_array_equal(dB.view(np.int32), got[2][2].cpu().numpy().view(np.int32))
