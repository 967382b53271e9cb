"""The tuning of products of more than 4096 columns names the accumulator it
runs: ranked columns or the hash table (plan creation only, no launch)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def N():
    from paper_2408_11988_gb300.build import build
    from paper_2408_11988_gb300 import _native as N
    build()
    N.lib()
    return N


class Handle:
    def __init__(self, N, d, force=None, semiring=0, n=1000):
        self.N, self.h = N, ctypes.c_void_p()
        A, B = N.CsrDesc(n, n, 8 * n, 8, 8, 8), N.CsrDesc(n, d, 10 * n, 8, 8, 8)
        f = N.Tuning.from_dict(force)
        self.status = N.lib().ts_plan_create(ctypes.byref(A), ctypes.byref(B), semiring, ctypes.byref(f),
                                             ctypes.byref(self.h))

    def __del__(self):
        if self.h.value:
            self.N.lib().ts_plan_destroy(self.h)

    def tuning(self):
        t = self.N.Tuning()
        assert self.N.lib().ts_plan_get_tuning(self.h, ctypes.byref(t)) == self.N.TS_OK
        return t.as_dict()

    def set(self, tuning):
        t = self.N.Tuning.from_dict(tuning)
        return self.N.lib().ts_plan_set_tuning(self.h, ctypes.byref(t))

    def kind(self):
        t = self.tuning()
        return t["accum"], t["hash_slots"]


@pytest.mark.parametrize("semiring", [0, 1])
@pytest.mark.parametrize("d", [4097, 8192, 32768])
def test_ranked_plan_reports_a_tuning_that_makes_it_again(N, d, semiring):
    auto = Handle(N, d, semiring=semiring)
    assert auto.kind() == (N.ACC_HASH, N.HASH_RANKED)
    assert Handle(N, d, auto.tuning(), semiring).tuning() == auto.tuning()
    # a table asked for by its kind or its size, and taken back
    for ask, slots in (({"accum": N.ACC_HASH}, 1024), ({"accum": N.ACC_HASH, "hash_slots": 512}, 512),
                       ({"hash_slots": 256}, 256)):
        asked = Handle(N, d, ask, semiring)
        assert asked.kind() == (N.ACC_HASH, slots)
        assert Handle(N, d, asked.tuning(), semiring).kind() == (N.ACC_HASH, slots)
        p = Handle(N, d, semiring=semiring)
        assert p.set(ask) == N.TS_OK and p.kind() == (N.ACC_HASH, slots)
        assert p.set({}) == N.TS_OK and p.kind() == (N.ACC_HASH, N.HASH_RANKED)
        assert asked.set(auto.tuning()) == N.TS_OK and asked.kind() == (N.ACC_HASH, N.HASH_RANKED)


def test_where_ranking_does_not_fit(N):
    assert Handle(N, 32769).kind() == (N.ACC_HASH, 1024)
    assert Handle(N, 32769, {"accum": N.ACC_HASH, "hash_slots": N.HASH_RANKED}).kind() == (N.ACC_HASH, 1024)
    assert Handle(N, 4096).kind() == (N.ACC_DENSE, 1024)
    assert Handle(N, 300, {"accum": N.ACC_HASH, "hash_slots": N.HASH_RANKED}).kind() == (N.ACC_HASH, 1024)
    for bad in (-2, 1, 63, 100, 16384):
        assert Handle(N, 8192, {"accum": N.ACC_HASH, "hash_slots": bad}).status == N.TS_ERR_INVALID_ARG
        assert Handle(N, 8192, {"hash_slots": bad}).status == N.TS_ERR_INVALID_ARG
