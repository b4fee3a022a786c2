"""arcs_scanned and rows_gathered of calls whose dense rounds read every arc."""
import numpy as np
import pytest

import oracle
import paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _graph():
    """A graph of more than 2^22 arcs whose balls meet after three rounds, and
    two paths of 40 nodes."""
    er = I.er(20_000, 230, 701)
    ends = er.n + np.array([0, 40])
    path = np.concatenate([e + np.arange(39) for e in ends])
    v = np.repeat(np.arange(er.n), np.diff(er.row_ptr))
    src = np.concatenate([er.col, path, path + 1])
    dst = np.concatenate([v, path + 1, path])
    return I.from_arcs(er.n + 80, src, dst), ends


def test_lane_pairs_count_what_either_lane_reads():
    """Rows of eight words, a lane per half. The paths' seeds are in the second
    half (by degree, and by index for PROPAGATE-S) and grow to the last round, so
    every row lacks a growing bit there, and all its arcs are read, in each of the
    T + 1 rounds; the first half is done after three."""
    g, ends = _graph()
    assert g.m >= 1 << 22
    seeds = np.concatenate([I.seeds(20_000, 510, 702), ends]).astype(np.int32)
    want = oracle.run(g, seeds)
    assert want["rounds"] == 39
    with pg.Graph.from_csr(g.row_ptr, g.col, directed=False) as G:
        for fn in (pg.propagate_p, pg.propagate_s):
            r = fn(G, seeds, opts=pg.options(direction=pg.PG_DIR_DENSE, test_changed=2))
            assert np.array_equal(r.counts, want["counts"])
            st = G.last_stats()
            assert st["launches"] == 1
            assert st["arcs_scanned"] == 40 * g.m, fn
            assert st["rows_gathered"] == 40 * g.m, fn
