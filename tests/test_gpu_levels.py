"""Edges of the solve by score levels and of the expansions beside it, against the
CPU oracle (whole numbers: equal).

Cases: weights from 0 (a level is one TP count) to far above the normals' term, two
to nine hits, sample counts at word boundaries and at the largest, thousands of equal
scores (bands beyond the pool of picks), buffers of one record (grown on the way,
bands that do not fit), rows too dense to list; the exhaustive enumeration by 32
children of a record, the score bound, and the allocation-free solve inside and
beyond its lists."""
import numpy as np
import pytest

import oracle
from test_oracle_pins import _random_cohort

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mh():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_16721_gb300 import mh as m
    return m


# G, Nt, Nn, h, tumor density, normal density, alpha, smallest buffers, prune
CASES = [
    (2, 1, 0, 2, 1.0, 0.0, (1, 10), None, "paper"),
    (40, 63, 1, 2, 0.1, 0.3, (0, 1), None, "paper"),
    (60, 64, 64, 3, 0.08, 0.1, (7, 2), None, "paper"),
    (60, 65, 65, 3, 0.08, 0.1, (1000, 1), None, "paper"),
    (30, 129, 40, 4, 0.2, 0.2, (1, 10), None, "paper"),
    (22, 90, 33, 6, 0.35, 0.3, (1, 10), None, "paper"),
    (13, 60, 10, 9, 0.7, 0.3, (1, 3), None, "paper"),
    (500, 300, 20, 2, 0.015, 0.0, (1, 10), None, "paper"),   # thousands of equal scores
    (120, 200, 0, 3, 0.03, 0.0, (1, 10), None, "paper"),
    (100, 120, 30, 3, 0.05, 0.1, (1, 10), 1, "paper"),       # every buffer grows
    (300, 90, 20, 2, 0.04, 0.0, (0, 1), 1, "paper"),
    (90, 2047, 65, 2, 0.3, 0.2, (1, 10), None, "paper"),     # dense: no listed samples
    (40, 2048, 2048, 3, 0.1, 0.05, (1, 10), None, "paper"),
    (120, 2048, 16, 2, 0.004, 0.1, (3, 1), None, "paper"),
    (33, 70, 70, 3, 0.1, 0.1, (1, 10), None, "off"),         # a word of children and one more
    (64, 40, 20, 4, 0.2, 0.2, (1, 10), None, "off"),         # and its depth-2 records
    (97, 500, 300, 2, 0.3, 0.3, (1, 10), 1, "off"),
    (120, 257, 31, 3, 0.06, 0.05, (1, 2), None, "bound"),    # listed parents
    (60, 300, 20, 3, 0.4, 0.1, (2, 1), None, "bound"),       # dense ones
    (22, 200, 64, 5, 0.3, 0.2, (1, 10), 1, "bound"),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"G{c[0]}-Nt{c[1]}-h{c[3]}-{c[8]}" + ("-grown" if c[7] else ""))
def test_edges_match_the_oracle(mh, case, monkeypatch):
    G, Nt, Nn, h, dt, dn, alpha, least, prune = case
    if least:
        monkeypatch.setenv("MH_FRONTIER_MIN_RECORDS", str(least))
        monkeypatch.setenv("MH_FRONTIER_PRESIZE", "0")
    bm, _, _ = _random_cohort(np.random.default_rng(G * 7919 + Nt), G, Nt, Nn, dt, dn)
    opt = {"paper": mh.MH_PRUNE_PAPER, "off": mh.MH_PRUNE_OFF, "bound": mh.MH_PRUNE_BOUND}[prune]
    ref = oracle.pdfs(bm, G, Nt, Nn, h, alpha, prune=prune != "off")
    with mh.mh_create(bm, G, Nt, Nn) as H:
        for rounds in (0, 3, 0):  # the whole solve, its first rounds, the whole again in the same workspace
            for mode in (mh.MH_MODE_PERSISTENT, mh.MH_MODE_LAUNCHES):
                got = mh.mh_solve_ex(H, h, alpha, prune=opt, max_rounds=rounds, mode=mode)
                n = min(rounds, len(ref.visited)) if rounds else len(ref.visited)
                assert got.records() == ref.records()[:rounds or None] and len(got.visited) == n
                if prune == "bound":
                    assert (got.visited <= ref.visited[:n]).all() and (got.cut <= got.visited - got.pruned).all()
                else:
                    assert np.array_equal(got.visited, ref.visited[:n]) and np.array_equal(got.pruned, ref.pruned[:n])
                    assert not got.cut.any()


@pytest.mark.parametrize("G,Nt,Nn,h,dt", [(1, 1, 0, 1, 1.0), (33, 64, 1, 2, 0.2), (300, 65, 0, 3, 0.05), (8192, 1024, 64, 1, 0.01),
                                          (4096, 257, 30, 2, 0.9), (4600, 257, 30, 2, 0.9)])  # 0.95 and 1.06 million mutations
def test_noalloc_matches_the_solve(mh, G, Nt, Nn, h, dt):
    import torch

    bm, _, _ = _random_cohort(np.random.default_rng(G + Nt), G, Nt, Nn, dt, 0.1)
    with mh.mh_create(bm, G, Nt, Nn) as H:
        ref = mh.mh_solve(H, h)
    d = torch.from_numpy(bm.view(np.int64)).to("cuda")
    out = [torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in (Nt * h, Nt, Nt)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    k, rounds = mh.mh_solve_noalloc(d.data_ptr(), G, Nt, Nn, h, (1, 10), stream.cuda_stream, *(x.data_ptr() for x in out), Nt)
    g, tp, fp = (x.cpu().numpy() for x in out)
    assert [(tuple(g[i * h:(i + 1) * h].tolist()), int(tp[i]), int(fp[i])) for i in range(k)] == ref.records()
    assert rounds == ref.rounds and (tp[k:] == -1).all()
