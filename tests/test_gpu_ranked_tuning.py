"""Products of more than 4096 columns run the accumulator their tuning names,
whether it came with the plan or by set_tuning, and the autotuner tries both."""
import pytest

import synth
from _cmp import compare_full

pytestmark = pytest.mark.gpu

from paper_2408_11988_gb300 import ACC_HASH, DeviceCSR, Plan
from paper_2408_11988_gb300 import _native as N

RANKED = {"accum": ACC_HASH, "hash_slots": N.HASH_RANKED}


def _run(plan, A, B):
    """The product, and the kernels its numeric pass launched (two when ranked: very long rows, the others)."""
    rowptr, nnz = plan.symbolic(A, B)
    C = plan.alloc_c(rowptr, nnz)
    before = N.lib().ts_kernel_launches()
    plan.numeric(A, B, C)
    launches = N.lib().ts_kernel_launches() - before
    plan.check()
    return C, launches


@pytest.mark.parametrize("d", [4097, 9000])
def test_kernel_follows_the_tuning(d):
    A, B = synth.rmat_embedding(scale=10, edge_factor=12, d=d, density=6 / d, seed=5, b_values="uniform")
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    auto = Plan(Ad, Bd)
    for tuning, launches in ((None, 2), ({"accum": ACC_HASH}, 1), ({"hash_slots": 512}, 1), (RANKED, 2),
                             (auto.tuning, 2)):
        C, seen = _run(Plan(Ad, Bd, tuning=tuning), Ad, Bd)
        assert seen == launches, tuning
        compare_full(C, A, B)
    plan = Plan(Ad, Bd)
    for tuning, launches in (({"accum": ACC_HASH, "hash_slots": 256}, 1), ({}, 2), ({"accum": ACC_HASH}, 1),
                             (auto.tuning, 2)):
        plan.set_tuning(tuning)
        C, seen = _run(plan, Ad, Bd)
        assert seen == launches, tuning
        compare_full(C, A, B)


def test_autotune_reports_what_it_chose():
    A, B = synth.rmat_embedding(scale=11, edge_factor=12, d=6000, density=8 / 6000, seed=6, b_values="uniform")
    Ad, Bd = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    plan = Plan(Ad, Bd)
    C = plan.forward(Ad, Bd)
    chosen = plan.autotune(Ad, Bd, C, reps=1)
    compare_full(C, A, B)
    assert chosen == plan.tuning
    again = Plan(Ad, Bd, tuning=chosen)
    assert again.tuning == chosen
    C, seen = _run(again, Ad, Bd)
    compare_full(C, A, B)
    assert _run(plan, Ad, Bd)[1] == seen
