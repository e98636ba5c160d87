"""Levels with a great many combinations of one score: groups of tumors that share all of a
set of genes, every one of them in the same normals, give every h-subset of the set the same
score, and groups that overlap leave records a part of whose tumors a pick has taken.  The
picks are made from a list, or one by one where the list would be long or has no room
(buffers of one record, a budget that they may not pass), alone, in batches that stop a
solve between two picks, served, and without allocation: whole numbers, equal to the oracle."""
import numpy as np
import pytest

import oracle
from test_oracle_pins import pack

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mh():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_16721_gb300 import mh as m
    return m


def _groups(P, m, k, step, normals, seed):
    """P groups of k tumors sharing m genes, a group begins `step` tumors after the last; one
    gene of each tumor's own, in no normal and first in the rows, so that its best
    combination on its own is found at once."""
    rng = np.random.default_rng(seed)
    Nt = (P - 1) * step + k
    t = np.zeros((P * m, Nt), dtype=np.uint8)
    for p in range(P):
        t[p * m:(p + 1) * m, p * step:p * step + k] = 1
    t = np.concatenate([np.eye(Nt, dtype=np.uint8), t[rng.permutation(P * m)]])
    n = np.ones((len(t), normals), dtype=np.uint8)
    n[:Nt] = 0
    return pack(t, n), len(t), Nt, normals


# groups, genes, tumors each, offset, normals, h, alpha
CASES = [
    (6, 30, 14, 14, 1, 3, (1, 10)),     # listed records, FP = 1 everywhere
    (8, 30, 14, 7, 1, 3, (1, 10)),      # half of a group's tumors are the next one's too
    (5, 24, 30, 30, 1, 3, (1, 10)),     # rows too dense to list
    (5, 24, 30, 11, 1, 3, (1, 10)),     # and overlapping
    (9, 110, 5, 3, 1, 2, (5, 1)),
    (4, 120, 22, 9, 2, 2, (3, 1)),
    (5, 17, 16, 5, 1, 4, (1, 10)),
    (3, 13, 19, 8, 1, 6, (1, 5)),
    (40, 3, 2, 1, 65, 2, (70, 1)),      # few members, many picks
]


def _same(got, want):
    assert got.records() == want.records()
    assert np.array_equal(got.visited, want.visited) and np.array_equal(got.pruned, want.pruned)


# (no growth: a budget that the frontiers of the cases up to three hits just keep to, 2.1 MB)
@pytest.mark.parametrize("case,room", [(c, r) for c in CASES for r in ("default", "one record", "no growth")
                                       if r != "no growth" or c[5] <= 3], ids=str)
def test_equal_scores_match_the_oracle(mh, case, room, monkeypatch):
    *g, h, alpha = case
    bm, G, Nt, Nn = _groups(*g, seed=sum(g))
    if room != "default":
        monkeypatch.setenv("MH_FRONTIER_MIN_RECORDS", "1")
    if room == "no growth":
        monkeypatch.setenv("MH_FRONTIER_BUDGET_MB", "3")
    ref = oracle.pdfs(bm, G, Nt, Nn, h, alpha)
    with mh.mh_create(bm, G, Nt, Nn) as H:
        for rounds in (0, 2, 0):
            got = mh.mh_solve_ex(H, h, alpha, max_rounds=rounds)
            assert got.records() == ref.records()[:rounds or None]
            assert np.array_equal(got.visited, ref.visited[:rounds or None])
            assert np.array_equal(got.pruned, ref.pruned[:rounds or None])


def test_all_ones_within_the_budget(mh, monkeypatch):
    """40 genes in all of 64 tumors: 91,390 combinations of one score, 14.6 MB with room to
    spare; the buffers of a handle stay within a budget of 4 MB."""
    monkeypatch.setenv("MH_FRONTIER_MIN_RECORDS", "64")
    monkeypatch.setenv("MH_FRONTIER_BUDGET_MB", "4")
    G, Nt, h = 40, 64, 4
    bm = pack(np.ones((G, Nt), dtype=np.uint8), np.ones((G, 0), dtype=np.uint8))
    with mh.mh_create(bm, G, Nt, 0) as H:
        before = mh.mh_handle_info(H)[3]
        _same(mh.mh_solve(H, h), oracle.pdfs(bm, G, Nt, 0, h))
        assert mh.mh_handle_info(H)[3] - before <= 5 << 20  # and under 1 MB of workspace


@pytest.mark.parametrize("choice", ["1", "101.5", "210.75", "1000"])
def test_batches_of_equal_scores(mh, choice, monkeypatch):
    monkeypatch.setenv("MH_BATCH_CHOICE", choice)
    monkeypatch.setenv("MH_FRONTIER_MIN_RECORDS", "1")
    cases = [(_groups(*c[:5], seed=i), c[5]) for i, c in enumerate(CASES)]
    handles = [mh.mh_create(*c) for c, _ in cases]
    try:
        got = mh.mh_solve_batch(handles, [h for _, h in cases])
        for ((bm, G, Nt, Nn), h), r in zip(cases, got):
            _same(r, oracle.pdfs(bm, G, Nt, Nn, h))
    finally:
        for H in handles:
            H.close()


def test_served_equal_scores(mh):
    cases = [(_groups(*c[:5], seed=i), c[5]) for i, c in enumerate(CASES)]
    with mh.Server(slots=4) as S:
        tickets = [S.submit(*c, h) for c, h in cases for _ in range(2)]
        got = [S.wait(t, 60000) for t in tickets]
    for i, ((bm, G, Nt, Nn), h) in enumerate(cases):
        ref = oracle.pdfs(bm, G, Nt, Nn, h)
        _same(got[2 * i], ref)
        _same(got[2 * i + 1], ref)


@pytest.mark.parametrize("case", [c for c in CASES if c[5] <= 4], ids=str)
def test_noalloc_equal_scores(mh, case):
    import torch

    *g, h, alpha = case
    bm, G, Nt, Nn = _groups(*g, seed=sum(g))
    ref = oracle.pdfs(bm, G, Nt, Nn, h, alpha)
    d = torch.from_numpy(bm.view(np.int64)).to("cuda")
    out = [torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in (Nt * h, Nt, Nt)]
    k, rounds = mh.mh_solve_noalloc(d.data_ptr(), G, Nt, Nn, h, alpha, torch.cuda.current_stream().cuda_stream,
                                    *(x.data_ptr() for x in out), Nt)
    gn, tp, fp = (x.cpu().numpy() for x in out)
    assert [(tuple(gn[i * h:(i + 1) * h].tolist()), int(tp[i]), int(fp[i])) for i in range(k)] == ref.records()
    assert rounds == len(ref.visited)
