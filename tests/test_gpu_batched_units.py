"""Batched products at the lines of their units and groups: instances of a few
rows, of parts of a chunk, of one scan tile exactly and one row more, rows of A
at the length from which a row is shared by a warp's slots, heavy rows, widths
below and above 256 columns, both semirings; forward and gradients."""
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
    lens = rng.integers(0, 6, n)
    want = [min(x, n) for x in (62, 63, 64, 65, 200, 700, 1500)][:n]
    lens[rng.permutation(n)[:len(want)]] = want
    rowptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rowptr[1:])
    A = CSR(n, n, rowptr, np.concatenate([np.sort(rng.choice(n, m, replace=False)) for m in lens]).astype(np.int32))
    A.val = synth.uniform(A.nnz, seed + 1)
    B = synth.tall_skinny(n, d, per_row / d, seed + 2)
    B.val = synth.normal(B.nnz, seed + 3)
    return A, B


SHAPES = [(1, 32, 2), (5, 33, 1), (33, 64, 9), (800, 250, 3.3), (4096, 96, 2.5), (4097, 128, 1.2), (9000, 32, 0.4)]


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("semiring", [PLUS_TIMES, OR_SELECT2ND])
@pytest.mark.parametrize("heavy", [0, 1 << 20])
def test_units(wide, semiring, heavy):
    host = [_instance(n, 4 * d if wide else d, p, 10 * i) for i, (n, d, p) in enumerate(SHAPES)]
    As, Bs = ([DeviceCSR.from_host(h[k]) for h in host] for k in (0, 1))
    batch = BatchedProduct(As, Bs, semiring, tuning={"cta_min_flops": heavy} if heavy else None)
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
