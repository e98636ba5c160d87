"""What a call that fails at its end leaves behind, the failures made on the host: a batch
that cannot make one of its results leaves no copy in flight into the handles' buffers
(each handle on a stream of its own), which later handles get again; the allocation-free
solve returns the error of its persistent kernel."""
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
    yield m
    m.mh_set_fault(None)


def _cohorts(n, seed=3):
    rng = np.random.default_rng(seed)
    return [(_random_cohort(rng, 60, 120 + 40 * i, 30, 0.1, 0.05)[0], 60, 120 + 40 * i, 30) for i in range(n)]


@pytest.mark.parametrize("at", [1, 2, 4])
def test_batch_without_memory_for_a_result(mh, monkeypatch, at):
    import torch

    monkeypatch.setenv("MH_AUTOTUNE", "0")
    cohorts = _cohorts(4)
    refs = [oracle.pdfs(bm, G, Nt, Nn, 3) for bm, G, Nt, Nn in cohorts]
    for _ in range(2):  # the second handles get the first ones' buffers
        streams = [torch.cuda.Stream() for _ in cohorts]
        handles = [mh.mh_create(*c) for c in cohorts]
        for H, s in zip(handles, streams):
            mh.mh_set_stream(H, s.cuda_stream)
        mh.mh_set_fault(f"result_fail={at}")
        with pytest.raises(mh.MHError) as e:
            mh.mh_solve_batch(handles, [3] * 4)
        assert e.value.code == mh.MH_ENOMEM
        assert all(s.query() for s in streams)  # nothing is left in flight
        mh.mh_set_fault(None)
        for H, r in zip(handles[:2], refs):
            assert mh.mh_solve(H, 3).records() == r.records()
        for got, r in zip(mh.mh_solve_batch(handles, [3] * 4), refs):
            assert got.records() == r.records() and np.array_equal(got.visited, r.visited)
        for H in handles:
            H.close()


def test_noalloc_reports_a_timeout(mh):
    """A bounded wait that ran out is an error here too, not a silent second solve."""
    import torch

    (bm, G, Nt, Nn), h = _cohorts(1)[0], 3
    ref = oracle.pdfs(bm, G, Nt, Nn, h)
    d = torch.from_numpy(bm.view(np.int64)).to("cuda")

    def solve():
        out = [torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in (Nt * h, Nt, Nt)]
        k, _ = mh.mh_solve_noalloc(d.data_ptr(), G, Nt, Nn, h, (1, 10), torch.cuda.current_stream().cuda_stream,
                                   *(x.data_ptr() for x in out), Nt)
        g, tp, fp = (x.cpu().numpy() for x in out)
        return [(tuple(g[i * h:(i + 1) * h].tolist()), int(tp[i]), int(fp[i])) for i in range(k)]

    mh.mh_set_fault("timeout_after=1")
    with pytest.raises(mh.MHError) as e:
        solve()
    assert e.value.code == mh.MH_ETIMEOUT
    assert solve() == ref.records()
