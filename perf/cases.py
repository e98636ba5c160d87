"""What the framework is timed on: whole calls of its public entry points.

A user brings the mutation bitmaps of a cohort (genes x tumor and normal samples)
and gets the ordered multi-hit combinations of the greedy weighted set cover, with
their counts and the search's per-round counters.  Every case is such a call: a
solve on a resident cohort (two to five hits, the smallest to the largest cohorts),
its pruning options, a training / test evaluation from host rows, a batch of
cohorts, a burst of served requests and the allocation-free solve.  All results are
whole numbers (gene indices, counts, 64-bit counters).

Cohorts are drawn on the GPU from the seed: per-gene mutation rates of one of three
laws (log-normal; a power tail under twenty frequent genes; a power tail with a
log-normal burden per sample), normals at 0.3 of the tumors' rates, and a few
combinations of h genes planted in a share of the tumors; genes in random order.
"""
import math

import numpy as np
import torch

from paper_2603_16721_gb300 import mh

ALPHA = (1, 10)  # the usual weight 0.1, as a rational


def listed():
    return [
        # a panel of a few hundred genes: the smallest solve, all latency
        {"name": "panel_h3", "what": "solve", "law": "top", "G": 600, "Nt": 130, "Nn": 70, "h": 3},
        # two hits on a thousand genes
        {"name": "pairs_h2", "what": "solve", "law": "lognormal", "G": 1000, "Nt": 200, "Nn": 100, "h": 2},
        # three hits on a middle-sized cohort: the ordinary solve
        {"name": "triples_h3", "what": "solve", "law": "top", "G": 5000, "Nt": 500, "Nn": 300, "h": 3},
        # four hits over a whole exome
        {"name": "exome_h4", "what": "solve", "law": "burden", "G": 19000, "Nt": 800, "Nn": 400, "h": 4},
        # as many samples as a pan-cancer cohort brings (the widest rows)
        {"name": "wide_h3", "what": "solve", "law": "burden", "G": 19000, "Nt": 1999, "Nn": 1001, "h": 3},
        # five hits, sizes off every word boundary
        {"name": "ragged_h5", "what": "solve", "law": "burden", "G": 2111, "Nt": 333, "Nn": 129, "h": 5},
        # the score-bound pruning option
        {"name": "bound_h3", "what": "bound", "law": "top", "G": 5000, "Nt": 500, "Nn": 300, "h": 3},
        # pruning switched off: the exhaustive enumeration
        {"name": "exhaustive_h3", "what": "exhaustive", "law": "lognormal", "G": 300, "Nt": 150, "Nn": 75, "h": 3},
        # from host rows: a handle for the training and one for the test split, learn, evaluate both
        {"name": "train_test_h3", "what": "train_test", "law": "top", "G": 5000, "Nt": 500, "Nn": 300, "h": 3},
        # eight uneven cohorts in one call
        {"name": "batch_8", "what": "batch", "law": "top", "n": 8, "sizes": 100, "G": 19000, "Nt": 1000, "Nn": 500, "h": 3},
        # a burst of served requests with mixed hit counts
        {"name": "served_8", "what": "served", "law": "burden", "n": 8, "sizes": 0, "G": 19000, "Nt": 800, "Nn": 400, "h": 3},
        # the solve for callers that may not allocate, rows and results on the device
        {"name": "noalloc_h3", "what": "noalloc", "law": "top", "G": 2000, "Nt": 300, "Nn": 200, "h": 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["solve", "solve", "solve", "solve", "bound", "exhaustive", "train_test", "batch", "served", "noalloc"])
    h = {"solve": rng.choice([2, 3, 3, 4, 5]), "exhaustive": rng.choice([2, 3]), "noalloc": rng.choice([2, 3])}.get(what, 3)
    law = {2: "lognormal", 3: rng.choice(["top", "burden"]), 4: "burden", 5: "burden"}[h]
    if what == "batch":  # shapes between a tenth and the whole of these, drawn per cohort
        return {"what": what, "law": "top", "n": rng.randint(3, 8), "sizes": rng.randint(0, 9999), "G": _log(rng, 2000, 12000),
                "Nt": _log(rng, 100, 800), "Nn": _log(rng, 50, 400), "h": 3}
    if what == "served":
        return {"what": what, "law": "burden", "n": rng.randint(3, 8), "sizes": 0, "G": _log(rng, 2000, 19000),
                "Nt": _log(rng, 100, 800), "Nn": _log(rng, 50, 400), "h": 3}
    if what == "exhaustive":
        g, nt = (_log(rng, 200, 900), 200) if h == 2 else (_log(rng, 60, 260), 140)
    elif what == "noalloc":
        g, nt = (_log(rng, 300, 8000), 500) if h == 2 else (_log(rng, 300, 2000), 300)
        law = "lognormal" if h == 2 else "top"
    else:
        g, nt = {2: (_log(rng, 200, 3000), 600), 3: (_log(rng, 300, 9000), 900), 4: (_log(rng, 1000, 16000), 700),
                 5: (_log(rng, 500, 2000), 320)}[h]
    return {"what": what, "law": law, "G": g, "Nt": _log(rng, 60, nt), "Nn": _log(rng, 30, nt // 2), "h": h}


def _device():
    return torch.device("cuda")


def _power(n, mean, cap):
    """Rates min(cap, c r^-0.65) for r = 1..n with the given mean."""
    r = torch.arange(1, n + 1, dtype=torch.float64) ** -0.65
    lo, hi = 0.0, 1e6
    for _ in range(80):
        c = (lo + hi) / 2
        if float(torch.clamp(c * r, max=cap).mean()) < mean:
            lo = c
        else:
            hi = c
    return torch.clamp(c * r, max=cap)


def _words(bits):
    """Bits [G, n] as 64-bit words, least significant bit first, zero padding (int64)."""
    g, n = bits.shape
    w = (n + 63) // 64
    full = torch.zeros(g, w * 64, dtype=torch.int64, device=bits.device)
    full[:, :n] = bits
    return (full.view(g, w, 64) << torch.arange(64, device=bits.device)).sum(2)


def _cohort(law, G, Nt, Nn, h, seed):
    """Mutation bits (tumor [G, Nt], normal [G, Nn]) on the GPU."""
    dev = _device()
    cpu = torch.Generator().manual_seed(seed)
    gen = torch.Generator(device=dev).manual_seed(seed)
    burden = torch.ones(Nt + Nn, dtype=torch.float64)
    if law == "lognormal":
        p = torch.clamp(torch.exp(math.log(0.01) + torch.randn(G, generator=cpu, dtype=torch.float64)), 0.001, 0.30)
        plants, lo, hi = 2, 0.20, 0.20
    elif law == "top":
        top = 0.10 + 0.30 * torch.rand(min(20, G), generator=cpu, dtype=torch.float64)
        p = torch.cat([top, _power(G - 20, 0.008, 0.10)]) if G > 20 else top
        plants, lo, hi = 3, 0.10, 0.15
    else:
        p = _power(G, 0.003, 0.30)
        burden = torch.exp(0.7 * torch.randn(Nt + Nn, generator=cpu, dtype=torch.float64) - 0.245)
        plants, lo, hi = 4, 0.05, 0.10
    p = p[torch.randperm(G, generator=cpu)]
    scale = burden * torch.cat([torch.ones(Nt), torch.full((Nn,), 0.3)]).double()
    prob = torch.clamp(p[:, None].to(dev) * scale[None, :].to(dev), max=0.95).float()
    bits = torch.rand(prob.shape, generator=gen, device=dev) < prob
    for _ in range(plants):
        share = lo + (hi - lo) * float(torch.rand(1, generator=cpu))
        who = torch.randperm(Nt, generator=cpu)[: max(1, int(round(share * Nt)))].to(dev)
        for g in torch.randperm(G, generator=cpu)[:h].tolist():
            bits[g, who] = True
    return bits[:, :Nt], bits[:, Nt:]


def _rows(tumor, normal):
    return torch.cat([_words(tumor), _words(normal)], dim=1).contiguous()


def _host(rows):
    return np.ascontiguousarray(rows.cpu().numpy()).view(np.uint64)


def _members(case):
    """Sizes and hit counts of the cohorts of a batch or a burst of requests."""
    out = []
    r = np.random.RandomState(case["sizes"])
    for i in range(case["n"]):
        if case["what"] == "batch":
            f = r.uniform(0.1, 1.0, 3)
            out.append((max(300, int(case["G"] * f[0])), max(60, int(case["Nt"] * f[1])), max(30, int(case["Nn"] * f[2])),
                        4 if i >= (3 * case["n"]) // 4 else 3))
        else:
            out.append((case["G"], case["Nt"], case["Nn"], (3, 2, 3, 4)[i % 4]))
    return out


def prepare(case, seed):
    what, law, G, Nt, Nn, h = (case[k] for k in ("what", "law", "G", "Nt", "Nn", "h"))
    if what in ("batch", "served"):
        many = []
        for i, (g, nt, nn, hh) in enumerate(_members(case)):
            many.append((_host(_rows(*_cohort(law, g, nt, nn, hh, seed * 1009 + i))), g, nt, nn, hh))
        if what == "served":
            return {"what": what, "server": mh.Server(slots=case["n"]), "requests": many}
        stream = torch.cuda.Stream()
        handles = [mh.mh_create(rows, g, nt, nn) for rows, g, nt, nn, _ in many]
        for x in handles:
            mh.mh_set_stream(x, stream.cuda_stream)
        hits = [m[4] for m in many]
        mh.mh_solve_batch(handles, hits)  # the schedule is chosen on a batch's first solve
        return {"what": what, "handles": handles, "hits": hits, "stream": stream, "tumors": [m[2] for m in many]}
    tumor, normal = _cohort(law, G, Nt, Nn, h, seed)
    if what == "train_test":
        kt, kn = max(1, (3 * Nt) // 4), (3 * Nn) // 4  # samples are exchangeable: the first three quarters train
        parts = [(tumor[:, :kt], normal[:, :kn]), (tumor[:, kt:], normal[:, kn:])]
        return {"what": what, "h": h, "G": G,
                "splits": [(_host(_rows(t.contiguous(), n.contiguous())), t.shape[1], n.shape[1]) for t, n in parts]}
    rows = _rows(tumor, normal)
    if what == "noalloc":
        dev = _device()
        out = [torch.zeros(n, dtype=torch.int32, device=dev) for n in (Nt * h, Nt, Nt)]
        return {"what": what, "rows": rows, "size": (G, Nt, Nn, h), "out": out}
    return {"what": what, "h": h, "Nt": Nt, "handle": mh.mh_create(_host(rows), G, Nt, Nn)}


def _padded(a, rows):
    out = np.full((rows,) + a.shape[1:], -1, dtype=a.dtype)
    out[: len(a)] = a
    return out


def _whole(r, nt):
    """A result, its rows (selections, rounds) followed by -1 up to the most a cohort of nt tumors can have."""
    out = {"genes": _padded(r.genes, nt), "tp": _padded(r.tp, nt), "fp": _padded(r.fp, nt)}
    return dict(out, visited=_padded(r.visited.view(np.int64), nt + 1), pruned=_padded(r.pruned.view(np.int64), nt + 1))


def run(state):
    what = state["what"]
    if what == "solve":
        return _whole(mh.mh_solve(state["handle"], state["h"], ALPHA), state["Nt"])
    if what == "bound":  # which prefixes are cut depends on when candidates are found: the selections do not
        r = mh.mh_solve_ex(state["handle"], state["h"], ALPHA, prune=mh.MH_PRUNE_BOUND)
        return {k: v for k, v in _whole(r, state["Nt"]).items() if k in ("genes", "tp", "fp")}
    if what == "exhaustive":
        return _whole(mh.mh_solve_ex(state["handle"], state["h"], ALPHA, prune=mh.MH_PRUNE_OFF), state["Nt"])
    if what == "train_test":
        (train, nt, nn), (test, mt, mn) = state["splits"]
        with mh.mh_create(train, state["G"], nt, nn) as a, mh.mh_create(test, state["G"], mt, mn) as b:
            r = mh.mh_solve(a, state["h"], ALPHA)
            out = _whole(r, nt)
            for name, x in (("train", a), ("test", b)):
                v = mh.mh_evaluate(x, r.genes)
                out[name] = {k: v[k].view(np.int64) if isinstance(v[k], np.ndarray) else v[k] for k in v}
        return out
    if what == "batch":
        return [_whole(r, nt) for r, nt in zip(mh.mh_solve_batch(state["handles"], state["hits"]), state["tumors"])]
    if what == "served":
        server = state["server"]
        tickets = [server.submit(rows, g, nt, nn, hh, ALPHA) for rows, g, nt, nn, hh in state["requests"]]
        return [_whole(server.wait(t), q[2]) for t, q in zip(tickets, state["requests"])]
    g, nt, nn, h = state["size"]
    genes, tp, fp = state["out"]
    k, rounds = mh.mh_solve_noalloc(state["rows"].data_ptr(), g, nt, nn, h, ALPHA, torch.cuda.current_stream().cuda_stream,
                                    genes.data_ptr(), tp.data_ptr(), fp.data_ptr(), nt)
    return {"genes": genes.view(nt, h), "tp": tp, "fp": fp, "k": k, "rounds": rounds}


def work(case):
    """Bytes: the packed rows read once and the results written once (a selection per
    four tumors is usual).  The path is integer work on bits: it has no floating-point
    operations to count."""
    members = _members(case) if "n" in case else [(case["G"], case["Nt"], case["Nn"], case["h"])]
    total = 0
    for g, nt, nn, h in members:
        total += 8 * g * ((nt + 63) // 64 + (nn + 63) // 64)
        total += (nt // 4 + 1) * (4 * (h + 2) + 16 * h)
    return {"bytes": total, "flops": 0}


def exact(case, seed):
    """The two-hit solve by its definition: every pair of every round, counted in 64 bits."""
    if case["what"] != "solve" or case["h"] != 2 or case["G"] > 1500:
        return None
    tumor, normal = _cohort(case["law"], case["G"], case["Nt"], case["Nn"], 2, seed)
    G, Nn = case["G"], case["Nn"]
    order = torch.sort(tumor.sum(1), stable=True).indices  # search order: fewest tumors first, ties by row
    T, N = tumor[order].double(), normal[order].double()
    lo, hi = torch.minimum(order[:, None], order[None, :]), torch.maximum(order[:, None], order[None, :])
    pair = lo * G + hi  # ascending original rows, in lexicographic order
    upper = torch.ones(G, G, dtype=torch.bool, device=T.device).triu(1)
    fp = (N @ N.T).long()
    places = torch.arange(G, device=T.device)
    genes, tps, fps, visited, pruned = [], [], [], [], []
    while T.shape[1] and bool((T.sum() > 0)):
        tp = (T @ T.T).long()
        alive = T[: G - 1].sum(1) > 0
        leaves = int((G - 1 - places[: G - 1])[alive].sum())
        full = int(((tp > 0) & upper).sum())
        visited.append([G - 1, leaves])
        pruned.append([G - 1 - int(alive.sum()), leaves - full])
        if not full:
            break
        score = torch.where((tp > 0) & upper, ALPHA[0] * tp + ALPHA[1] * (Nn - fp), torch.full_like(tp, -1))
        best = int(score.max())
        key = torch.where(score == best, pair, torch.full_like(pair, G * G))
        k = int(key.argmin())
        i, j = k // G, k % G
        genes.append([int(lo[i, j]), int(hi[i, j])])
        tps.append(int(tp[i, j]))
        fps.append(int(fp[i, j]))
        T = T[:, ~((T[i] > 0) & (T[j] > 0))]
    if T.shape[1] and not bool(T.sum() > 0):  # tumors without a mutated gene: a last round finds nothing
        visited.append([G - 1, 0])
        pruned.append([G - 1, 0])
    a = lambda v, t, s, rows: _padded(np.array(v, dtype=t).reshape(s), rows)  # noqa: E731
    nt = case["Nt"]
    return {"genes": a(genes, np.int32, (-1, 2), nt), "tp": a(tps, np.int32, -1, nt), "fp": a(fps, np.int32, -1, nt),
            "visited": a(visited, np.int64, (-1, 2), nt + 1), "pruned": a(pruned, np.int64, (-1, 2), nt + 1)}
