"""The exhaustive enumeration where its expansions hand out 32 children of a record and where
they hand out whole records: few and many depth-1 parents, deeper parents fewer and more than
the warps of a launch (2,432 of 16-warp blocks), in both modes, against the oracle."""
import numpy as np
import pytest

import oracle
from test_oracle_pins import _random_cohort

pytestmark = pytest.mark.gpu

# G, Nt, Nn, h; depth-2 parents: C(G - h + 2, 2)
CASES = [(71, 40, 20, 4), (72, 40, 20, 4), (73, 40, 20, 4),  # 2,346, 2,415 and 2,485
         (33, 130, 10, 5), (20, 70, 64, 6), (400, 30, 10, 3)]


@pytest.fixture(scope="module")
def mh():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_16721_gb300 import mh as m
    return m


@pytest.mark.parametrize("case", CASES, ids=str)
def test_enumeration_matches_the_oracle(mh, case):
    G, Nt, Nn, h = case
    bm, _, _ = _random_cohort(np.random.default_rng(G), G, Nt, Nn, 0.15, 0.1)
    ref = oracle.pdfs(bm, G, Nt, Nn, h, prune=False, max_rounds=2)
    with mh.mh_create(bm, G, Nt, Nn) as H:
        for mode in (mh.MH_MODE_PERSISTENT, mh.MH_MODE_LAUNCHES):
            got = mh.mh_solve_ex(H, h, prune=mh.MH_PRUNE_OFF, max_rounds=2, mode=mode)
            assert got.records() == ref.records()
            assert np.array_equal(got.visited, ref.visited) and np.array_equal(got.pruned, ref.pruned)
