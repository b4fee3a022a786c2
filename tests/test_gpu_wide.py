"""Rows of 16 and more words of one graph: the pull writes signatures, deltas,
their parts and the saturated rows, the post kernel counts in bit-sliced form.
Against the oracle where those have edges: words per row around the parts and
the column blocks, rows cut into pieces, rows that fill up in different rounds,
seeds that never leave their node."""
import functools

import numpy as np
import pytest

import oracle
import paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@functools.lru_cache(maxsize=None)
def _graph(kind):
    if kind == "er":
        return I.er(4500, 6, 501)
    if kind == "rmat":  # isolated nodes, hubs in pieces
        return I.rmat(13, 24, 502, directed=True)
    n = 4400  # a star of 2,100 leaves on a path, in pieces; the rest a cycle
    src = np.concatenate([np.zeros(2100), np.arange(2100, 2160), np.arange(2200, n)])
    dst = np.concatenate([np.arange(1, 2101), np.arange(2101, 2161),
                          np.append(np.arange(2201, n), 2200)])
    return I.from_arcs(n, src.astype(np.int32), dst.astype(np.int32), symmetrise=True)


@functools.lru_cache(maxsize=None)
def _want(kind, s):
    g = _graph(kind)
    seeds = I.seeds(g.n, s, 503)
    want = oracle.run(g, seeds)
    per_pass = np.zeros(want["rounds"] + 2, np.uint64)
    for k in range(0, s, 64):
        b = oracle.run(g, seeds[k:k + 64])["m_active"]
        per_pass[:b.size] += b
    return seeds, want, per_pass


@pytest.mark.parametrize("kind", ["er", "rmat", "star"])
@pytest.mark.parametrize("s", [961, 1024, 1090, 2100, 4160])
def test_wide_rows(kind, s):
    g = _graph(kind)
    seeds, want, per_pass = _want(kind, s)
    with pg.Graph.from_inputs(g) as G:
        for kw in (dict(), dict(direction=pg.PG_DIR_DENSE, test_changed=2),
                   dict(direction=pg.PG_DIR_SPARSE), dict(window_rows=1, use_graphs=0)):
            o = pg.options(**kw)
            r = pg.propagate_p(G, seeds, opts=o)
            assert r.rounds == want["rounds"], kw
            assert np.array_equal(r.counts, want["counts"]), kw
            assert np.array_equal(r.m_active, want["m_active"]), kw
            r = pg.propagate_s(G, seeds, opts=o)
            assert r.rounds == want["rounds"], kw
            assert np.array_equal(r.counts, want["counts"]), kw
            assert np.array_equal(r.m_active, per_pass[:r.m_active.size]), kw
