"""Batches of one large graph among many small ones, the large one first, in the
middle or last, at sizes that give units of 8, 16 and 32 rows; forward and
gradients against the oracle, both semirings."""
import numpy as np
import pytest
import torch

import oracle
import synth
from _cmp import REL, compare_full
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import OR_SELECT2ND, PLUS_TIMES, DeviceCSR
from paper_2408_11988_gb300.batched import BatchedProduct


def _instance(n, d, per_row, seed):
    rng = np.random.default_rng(seed)
    lens = np.minimum(rng.integers(0, 6, n), n)
    if n > 5000:
        lens[rng.permutation(n)[:8]] = (62, 63, 64, 65, 200, 700, 1500, 3000)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rowptr[1:])
    col = rng.integers(0, n, int(rowptr[-1]))
    rows = np.repeat(np.arange(n), lens)
    key = np.unique(rows * n + col)  # distinct columns in every row
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=rowptr[1:])
    A = CSR(n, n, rowptr, (key % n).astype(np.int32))
    A.val = synth.uniform(A.nnz, seed + 1)
    B = synth.tall_skinny(n, d, per_row / d, seed + 2)
    B.val = synth.normal(B.nnz, seed + 3)
    return A, B


@pytest.mark.parametrize("semiring", [PLUS_TIMES, OR_SELECT2ND])
@pytest.mark.parametrize("at", [0, 150, 300])
@pytest.mark.parametrize("n", [80_000, 170_001, 330_000])
def test_large_among_small(n, at, semiring):
    rng = np.random.default_rng(n + at)
    shapes = [(int(rng.integers(1, 70)), int(rng.choice([32, 40, 64])), 1.5) for _ in range(300)]
    shapes.insert(at, (n, 100, 2.5))
    host = [_instance(m, d, p, 7 * i) for i, (m, d, p) in enumerate(shapes)]
    batch = BatchedProduct([DeviceCSR.from_host(A) for A, _ in host], [DeviceCSR.from_host(B) for _, B in host], semiring)
    for _ in range(2):
        Cs = batch.forward()
    batch.check()
    out = [compare_full(C, A, B, semiring) for C, (A, B) in zip(Cs, host)]
    if semiring != PLUS_TIMES:
        return
    dCs = [synth.grad_output(int(o[0][-1]), 20 + i) for i, o in enumerate(out)]
    batch.bind_grads([torch.as_tensor(x, device="cuda") if x.size else torch.zeros(1, device="cuda") for x in dCs])
    dAs, dBs = batch.backward()
    batch.check()
    for (A, B), (Cp, Ci, _, _), dC, dA, dB in zip(host, out, dCs, dAs, dBs):
        rA, bA, rB, bB = oracle.backward(A, B, Cp, Ci, dC.astype(np.float64))
        assert np.all(np.abs(dA.cpu().numpy()[:A.nnz] - rA) <= REL * bA)
        assert np.all(np.abs(dB.cpu().numpy()[:B.nnz] - rB) <= REL * bB)
