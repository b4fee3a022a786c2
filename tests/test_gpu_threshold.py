"""dense_threshold: the rounds that are full sweeps, from the oracle's distances."""
import numpy as np
import pytest

import oracle
import paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_every_threshold_can_be_asked_for():
    """A round is swept when the out-arcs of the rows that changed in the round
    before are more than the threshold's part of all: at the caller's threshold,
    0.05 too, in the resident loop and round by round; at the library's own where
    the caller names none."""
    g = I.er(50_000, 8, 901)
    seeds = I.seeds(g.n, 1, 902)
    want = oracle.run(g, seeds)
    _, _, dist = oracle.seed_histograms(g, seeds, with_distances=True)
    deg = np.diff(g.row_ptr)
    assert deg.max() <= 64  # the library's threshold is 0.2 then
    sums = [int(deg[(dist == t).any(axis=1)].sum()) for t in range(want["rounds"] + 1)]
    assert any(0.05 < x / g.m < 0.2 for x in sums)
    with pg.Graph.from_inputs(g) as G:
        for thr in (0.0, 0.01, 0.05, 0.2, 0.5):
            for push, default in ((0, 0.2), (2, 0.05)):
                r = pg.propagate_p(G, seeds, opts=pg.options(dense_threshold=thr, sparse_push=push))
                assert np.array_equal(r.counts, want["counts"])
                part = np.float32(thr or default)
                assert G.last_stats()["dense_rounds"] == sum(x > float(part) * g.m for x in sums), \
                    (thr, push)
        pg.propagate_p(G, seeds)
        own = G.last_stats()["dense_rounds"]
        pg.propagate_p(G, seeds, opts=pg.options(dense_threshold=0.2))
        assert G.last_stats()["dense_rounds"] == own
