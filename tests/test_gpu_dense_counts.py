"""Counters and selections of cohorts with rows too dense to list, against the oracle: few
rounds (most tumors share a cover round) and many, fewer column words than a warp has lanes
and more, and more tumors in a row than a warp lists at a time."""
import numpy as np
import pytest

import oracle
from test_oracle_pins import _random_cohort

pytestmark = pytest.mark.gpu

# G, Nt, Nn, h, tumor density, normal density
CASES = [
    (64, 500, 40, 2, 0.5, 0.1),
    (65, 2048, 16, 2, 0.9, 0.1),     # 1,843 tumors a row
    (40, 1990, 3, 2, 0.99, 0.5),     # about 1,970: the list is filled a second time
    (30, 1552, 0, 2, 1.0, 0.0),      # all tumors in every row, one round
    (70, 300, 30, 3, 0.4, 0.2),
    (2100, 90, 20, 2, 0.4, 0.2),     # two chunks of column words
    (1025, 200, 300, 2, 0.15, 0.1),
    (24, 150, 20, 5, 0.5, 0.2),
    (33, 700, 10, 3, 0.12, 0.3),     # many rounds
]


@pytest.fixture(scope="module")
def mh():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_16721_gb300 import mh as m
    return m


@pytest.mark.parametrize("build", ["", "large"])
@pytest.mark.parametrize("case", CASES, ids=str)
def test_dense_cohorts_match_the_oracle(mh, case, build, monkeypatch):
    monkeypatch.setenv("MH_PERSISTENT_BUILD", build)
    G, Nt, Nn, h, dt, dn = case
    bm, _, _ = _random_cohort(np.random.default_rng(G + Nt), G, Nt, Nn, dt, dn)
    ref = oracle.pdfs(bm, G, Nt, Nn, h)
    with mh.mh_create(bm, G, Nt, Nn) as H:
        for rounds in (0, 1, 3):
            got = mh.mh_solve_ex(H, h, max_rounds=rounds)
            n = rounds or len(ref.visited)
            assert got.records() == ref.records()[:n]
            assert np.array_equal(got.visited, ref.visited[:n]) and np.array_equal(got.pruned, ref.pruned[:n])
