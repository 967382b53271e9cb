"""Backward kernels at the lines between four and five blocks per SM (groups of 8,
16 and 32 lanes, by the width of the dense row of dC), packed B and B's own
arrays, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from _cmp import REL

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR, Plan


@pytest.mark.parametrize("pack_b", [1, 2])
@pytest.mark.parametrize("group", [4, 8, 16, 32])
@pytest.mark.parametrize("d", [100, 1024, 1344, 1345, 2000, 5000])
def test_groups_and_widths(d, group, pack_b):
    A, B = synth.rmat_embedding(scale=11, edge_factor=12, d=d, density=12 / d, seed=d, b_values="uniform")
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    # d <= 512 with packed B: one warp per row, so that this kernel takes the light rows
    tuning = {"bwd_group": group, "pack_b": pack_b, "row_lanes": 32 if d <= 512 else 0}
    plan = Plan(Ad, Bd, tuning=tuning)
    C = plan.forward(Ad, Bd)
    dC = synth.grad_output(C.nnz, 3)
    dA, dB = plan.backward(Ad, Bd, C, torch.as_tensor(dC, device="cuda"))
    plan.check()
    Cp, Ci = C.rowptr.cpu().numpy(), C.col.cpu().numpy()
    rA, bA, rB, bB = oracle.backward(A, B, Cp, Ci, dC.astype(np.float64))
    assert np.all(np.abs(dA.cpu().numpy() - rA) <= REL * bA)
    assert np.all(np.abs(dB.cpu().numpy() - rB) <= REL * bB)
