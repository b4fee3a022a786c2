"""The resident round loop (the default for rows of up to 8 words) against the
oracle and the round-by-round schedules, where its parts have edges: words per
row, frontier rows around 32 and 256 out-arcs (pushed by a lane, or in pieces
by a warp), a full frontier stage, one-row counts windows, rows full before
and during a round, and packed batches whose graphs sweep and push."""
import functools

import numpy as np
import pytest

import oracle
import paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _hubs(degrees, directed):
    """Nodes of the given out-degrees, chained; leaves shared between them."""
    k, n = len(degrees), len(degrees) + max(degrees)
    src = np.concatenate([np.full(d, i) for i, d in enumerate(degrees)] + [np.arange(k - 1)])
    dst = np.concatenate([k + np.arange(d) for d in degrees] + [np.arange(1, k)])
    return I.from_arcs(n, src, dst, symmetrise=not directed)


@functools.lru_cache(maxsize=None)
def _graph(kind):
    if kind == "hubs":
        return _hubs([1, 31, 32, 33, 255, 256, 257, 511, 512, 513, 2000], False)
    if kind == "hubs_directed":
        return _hubs([600, 33, 32, 1, 256, 257, 700, 5], True)
    if kind == "grid":
        return I.grid(37, 41, 0.05, 401)
    if kind == "er":
        return I.er(3001, 7, 402)
    return I.rmat(11, 12, 403, directed=True)


@pytest.mark.parametrize("kind", ["hubs", "hubs_directed", "grid", "er", "rmat"])
@pytest.mark.parametrize("s", [1, 64, 65, 128, 129, 257, 512])
def test_resident_matches_oracle_and_round_by_round(kind, s):
    g = _graph(kind)
    seeds = I.seeds(g.n, min(s, g.n), 404)
    want = oracle.run(g, seeds)
    per_pass = np.zeros(want["rounds"] + 2, np.uint64)
    for k in range(0, seeds.size, 64):
        b = oracle.run(g, seeds[k:k + 64])["m_active"]
        per_pass[:b.size] += b
    with pg.Graph.from_inputs(g) as G:
        totals = {}
        for kw in (dict(sparse_push=1), dict(), dict(direction=pg.PG_DIR_DENSE),
                   dict(direction=pg.PG_DIR_SPARSE), dict(window_rows=1),
                   dict(window_rows=3, test_changed=1, dense_threshold=0.3)):
            o = pg.options(**kw)
            r = pg.propagate_p(G, seeds, opts=o)
            st = G.last_stats()
            assert r.rounds == want["rounds"], kw
            assert np.array_equal(r.counts, want["counts"]), kw
            assert np.array_equal(r.m_active, want["m_active"]), kw
            for f in ("active_rows", "changed_rows", "seed_edge_traversals", "m_active_total"):
                assert totals.setdefault(f, st[f]) == st[f], (kw, f)
            if not kw.get("sparse_push") and not kw.get("window_rows"):
                assert st["launches"] == 1, kw
            r = pg.propagate_s(G, seeds, opts=o)
            assert r.rounds == want["rounds"], kw
            assert np.array_equal(r.counts, want["counts"]), kw
            assert np.array_equal(r.m_active, per_pass[:r.m_active.size]), kw


@pytest.mark.parametrize("window_rows", [0, 1, 4])
@pytest.mark.parametrize("threshold", [0.0, 0.02, 1.0])
def test_resident_packed_batch(window_rows, threshold):
    kinds = ("er", "grid", "rmat", "hubs", "hubs_directed", "grid")
    b = pg.Batch()
    want = []
    for i, (kind, s) in enumerate(zip(kinds, (200, 130, 256, 129, 190, 255))):
        g = _graph(kind)
        seeds = I.seeds(g.n, s, 405 + i)
        b.add_inputs(g, seeds)
        want.append(oracle.run(g, seeds))
    kw = dict(window_rows=window_rows)
    if threshold:
        kw["dense_threshold"] = threshold
    for streams in (4, 1):
        b.set_streams(streams)
        b.run(opts=pg.options(**kw))
        for i, w in enumerate(want):
            r = b.result(i)
            assert r.rounds == w["rounds"], i
            assert np.array_equal(r.counts, w["counts"]), i
            assert np.array_equal(r.m_active, w["m_active"]), i


def test_delta_buffers_carried_between_calls():
    """Calls leave their delta buffers zero for the next one; widths, schedules
    and calls that stop short (counts capacity) in any order do not mix."""
    g = _graph("er")
    with pg.Graph.from_inputs(g) as G:
        seeds = {s: I.seeds(g.n, s, 410 + s) for s in (512, 64, 1500, 300)}
        want = {s: oracle.run(g, x) for s, x in seeds.items()}
        for kw in (dict(), dict(sparse_push=1), dict(window_rows=1), dict(timing=1)):
            for s in (64, 512, 1500, 300, 64, 1500):
                for fn in (pg.propagate_p, pg.propagate_s):
                    r = fn(G, seeds[s], opts=pg.options(**kw))
                    assert r.rounds == want[s]["rounds"], (s, kw)
                    assert np.array_equal(r.counts, want[s]["counts"]), (s, kw)
                with pytest.raises(pg.PropagateError):
                    pg.propagate_p(G, seeds[s], max_rounds=2, opts=pg.options(**kw))
