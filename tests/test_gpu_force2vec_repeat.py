"""A Force2Vec step repeats bit for bit, and rows on both sides of the lines
between a warp's row, a block's and several parts agree with the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR
from paper_2408_11988_gb300.force2vec import Force2Vec


def _graph(n, lens, seed):
    rng = np.random.default_rng(seed)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    return CSR(n, n, rp, np.concatenate([np.sort(rng.choice(n, m, replace=False)) for m in lens]).astype(np.int32))


@pytest.mark.parametrize("d,k", [(1, 1), (64, 8), (128, 26), (100, 50), (520, 70), (4096, 30)])
def test_step_repeats_and_matches(d, k):
    n, s, b, r0 = 3000, 4, 80, 11
    rng = np.random.default_rng(d)
    lens = rng.integers(0, 60, n)
    # terms = entries + 4: 31 .. 33, 63 .. 65, 255 .. 257, 511 .. 513, 1023 .. 1025, hubs
    edge = [t + e for t in (32, 64, 256, 512, 1024) for e in (-1, 0, 1)] + [2052, 2600, n + s]
    lens[r0:r0 + len(edge)] = np.array(edge) - s
    A = _graph(n, lens, d + 1)
    Z = synth.sparse_embedding(n, d, k, 150 + d, scale=0.3)
    neg = synth.negatives(b, s, n, 151)
    Ad = DeviceCSR.from_host(A, with_values=False)
    got = []
    for _ in range(8):
        Zd = DeviceCSR.from_host(Z)
        f = Force2Vec(Ad, Zd, k, negatives=s, lr=0.2, batch=b)
        U = f.step(r0, torch.as_tensor(neg), want_u=True)
        got.append([t.cpu().numpy().view(np.int32) for t in (U, Zd.col, Zd.val)])
    for g in got[1:]:
        for x, y in zip(got[0], g):
            np.testing.assert_array_equal(x, y)
    Ug = got[0][0].view(np.float32).astype(np.float64)
    Uo, Ub, _, _ = oracle.f2v_step(A, Z, r0, b, neg, s, 0.2, k)
    assert np.all(np.abs(Ug - Uo) <= 1e-5 * Ub)
    ncol, nval = oracle.f2v_topk(Ug, k)
    np.testing.assert_array_equal(got[0][1].reshape(n, k)[r0:r0 + b], ncol)
    np.testing.assert_array_equal(got[0][2].view(np.float32).reshape(n, k)[r0:r0 + b].astype(np.float64), nval)
