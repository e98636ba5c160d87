"""A cohort keeps to one way of solving over all launches of a batch, whatever build of
the kernel each launch is: nine hits and 1,800 tumors (three tuple words per tumor, the most
scratch the picks of a score level take) solved beside cohorts that finish earlier, so
that it begins in one build and ends in another, equal to its solve alone and to the
oracle."""
import numpy as np
import pytest

import oracle
from test_oracle_pins import _random_cohort

pytestmark = pytest.mark.gpu

# G, Nt, Nn, h, tumor density, normal density
COHORTS = [(13, 1800, 10, 9, 0.7, 0.3), (13, 2048, 40, 9, 0.6, 0.2), (40, 90, 30, 3, 0.1, 0.1), (60, 12, 5, 2, 0.3, 0.1)]


@pytest.fixture(scope="module")
def mh():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_16721_gb300 import mh as m
    return m


@pytest.mark.parametrize("build", ["", "large"])
@pytest.mark.parametrize("choice", ["1", "101.5", "210.75", "1000", "2002"])
def test_nine_hits_in_every_build(mh, monkeypatch, choice, build):
    monkeypatch.setenv("MH_BATCH_CHOICE", choice)
    monkeypatch.setenv("MH_PERSISTENT_BUILD", build)
    rng = np.random.default_rng(9)
    bms = [_random_cohort(rng, G, Nt, Nn, dt, dn)[0] for G, Nt, Nn, _, dt, dn in COHORTS]
    handles = [mh.mh_create(bm, G, Nt, Nn) for bm, (G, Nt, Nn, *_) in zip(bms, COHORTS)]
    try:
        got = mh.mh_solve_batch(handles, [c[3] for c in COHORTS])
        for bm, H, g, (G, Nt, Nn, h, _, _) in zip(bms, handles, got, COHORTS):
            for want in (oracle.pdfs(bm, G, Nt, Nn, h), mh.mh_solve(H, h)):
                assert g.records() == want.records()
                assert np.array_equal(g.visited, want.visited) and np.array_equal(g.pruned, want.pruned)
    finally:
        for H in handles:
            H.close()
