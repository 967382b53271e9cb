"""A Force2Vec step that reports a failed device check leaves Z as it was."""
import numpy as np
import pytest
import torch

import synth
from synth import CSR

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import DeviceCSR, TSError
from paper_2408_11988_gb300.force2vec import Force2Vec


@pytest.mark.parametrize("d,k", [(64, 8), (128, 40), (700, 70)])
@pytest.mark.parametrize("what", ["rowptr", "A", "neg", "Z"])
def test_failed_step_leaves_the_embedding(what, d, k):
    n, s, b, r0 = 700, 4, 60, 13
    A = synth.rmat(10, 8, 140, symmetrize=True)
    A = CSR(n, n, np.minimum(A.rowptr[:n + 1], A.rowptr[n]), A.col[:A.rowptr[n]] % n)
    rp, ci = A.rowptr.copy(), A.col.copy()
    neg = synth.negatives(b, s, n, 141)
    Z = synth.sparse_embedding(n, d, k, 142, scale=0.3)
    zc = Z.col.copy()
    if what == "rowptr":  # every other row holds all of A: more terms than A has entries
        rp[0::2], rp[1::2] = 0, rp[-1]
    elif what == "A":
        ci[rp[r0]:rp[r0 + b]] = 1 << 20
    elif what == "neg":
        neg[7] = -3
    else:
        zc[(r0 + 1) * k] = 1 << 20
    Ad = DeviceCSR.from_host(CSR(n, n, rp, ci), with_values=False)
    Zd = DeviceCSR.from_host(CSR(n, d, Z.rowptr, zc, Z.val))
    f = Force2Vec(Ad, Zd, k, negatives=s, lr=0.2, batch=b)
    f._ws.fill_(0x5A)
    with pytest.raises(TSError):
        f.step(r0, torch.as_tensor(neg))
    np.testing.assert_array_equal(Zd.col.cpu().numpy(), zc)
    np.testing.assert_array_equal(Zd.val.cpu().numpy(), Z.val)
