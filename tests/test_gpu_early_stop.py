"""Dense rounds stop a row once it can gain nothing more: counts and m_active
against the oracle where seeds stop growing at different rounds, rows fill up
part of the way through their arcs, and rows are cut into pieces."""
import functools

import numpy as np
import pytest

import oracle
import paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _union(parts):
    """Disjoint union of undirected graphs."""
    rp, col, n = [np.zeros(1, np.int64)], [], 0
    for g in parts:
        rp.append(g.row_ptr[1:] + rp[-1][-1])
        col.append(g.col.astype(np.int64) + n)
        n += g.n
    return I.Graph(n=n, row_ptr=np.concatenate(rp), col=np.concatenate(col).astype(np.int32),
                   directed=False)


@functools.lru_cache(maxsize=None)
def _graph(kind):
    """Graphs of more than 2^22 arcs (smaller ones are swept whole)."""
    if kind == "rmat":  # many seeds isolated, hubs in pieces
        return I.rmat(15, 100, 301, directed=False)
    if kind == "rmat_directed":
        return I.rmat(16, 128, 302, directed=True)
    # balls that end at rounds 0, 1, 2, ~6 and 60; rows full after one arc
    return _union([I.complete(2100), I.er(900, 9, 303), I.star(700), I.path(61),
                   I.from_arcs(5, [0], [1], symmetrise=True)])


@pytest.mark.parametrize("kind", ["rmat", "rmat_directed", "depths"])
@pytest.mark.parametrize("s", [1, 65, 200, 257, 300, 512])
def test_dense_rounds_stop_early(kind, s):
    g = _graph(kind)
    assert g.m >= 1 << 22
    seeds = I.seeds(g.n, s, 304)
    want = oracle.run(g, seeds)
    blocks = [oracle.run(g, seeds[k:k + 64])["m_active"] for k in range(0, s, 64)]
    per_pass = np.zeros(want["rounds"] + 2, np.uint64)
    for b in blocks:
        per_pass[:b.size] += b
    with pg.Graph.from_inputs(g) as G:
        for kw in (dict(direction=pg.PG_DIR_DENSE), dict(),
                   dict(direction=pg.PG_DIR_DENSE, window_rows=2, test_changed=1),
                   dict(direction=pg.PG_DIR_DENSE, words_per_thread=1),
                   dict(direction=pg.PG_DIR_DENSE, test_changed=2, use_graphs=0)):
            r = pg.propagate_p(G, seeds, opts=pg.options(**kw))
            assert r.rounds == want["rounds"], kw
            assert np.array_equal(r.counts, want["counts"]), kw
            assert np.array_equal(r.m_active, want["m_active"]), kw
            r = pg.propagate_s(G, seeds, opts=pg.options(**kw))
            assert r.rounds == want["rounds"], kw
            assert np.array_equal(r.counts, want["counts"]), kw
            assert np.array_equal(r.m_active, per_pass[:r.m_active.size]), kw
