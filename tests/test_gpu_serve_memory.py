"""A server slot is charged at least what it holds after the run, whatever kinds
of rows the runs before it left buffers for."""
import numpy as np
import pytest

import oracle
import paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("kw", [{}, {"sparse_push": 1}, {"wide_rows": 2}])
def test_charges_cover_what_a_slot_holds(directed, kw):
    g = I.rmat(15, 8, 951, directed=directed)
    sizes = (64, 600, 64, 1500, 130, 512, 2500, 300)  # rows of words, wide rows, in turn
    seeds = {s: I.seeds(g.n, s, 952) for s in sizes}
    want = {s: oracle.run(g, x) for s, x in seeds.items()}
    with pg.Server(slots=1, opts=pg.options(**kw)) as srv:
        gid = srv.add_inputs(g)
        for s in sizes:
            res, info = srv.result(srv.submit(gid, seeds[s]))
            assert res.rounds == want[s]["rounds"] and np.array_equal(res.counts, want[s]["counts"])
            st = srv.stats()
            assert info["footprint"] >= st["inflight_bytes"], s
            assert st["peak_bytes"] >= st["resident_bytes"] + st["inflight_bytes"]


def test_charges_cover_a_union():
    """Requests on several graphs that queue behind a long one run as a union, on
    a slot that has run wide rows."""
    long_g = I.grid(500, 500, 0.05, 953)
    graphs = [I.rmat(13, 8, 954 + k, directed=bool(k & 1)) for k in range(4)]
    seeds = [I.seeds(g.n, 100, 960) for g in graphs]
    with pg.Server(slots=1) as srv:
        lg = srv.add_inputs(long_g)
        gids = [srv.add_inputs(g) for g in graphs]
        srv.result(srv.submit(gids[0], I.seeds(graphs[0].n, 900, 961)))
        first = srv.submit(lg, I.seeds(long_g.n, 64, 962))
        rids = [srv.submit(i, x) for i, x in zip(gids, seeds)]
        srv.result(first)
        for g, x, rid in zip(graphs, seeds, rids):
            res, info = srv.result(rid)
            want = oracle.run(g, x)
            assert res.rounds == want["rounds"] and np.array_equal(res.counts, want["counts"])
        assert info["merged"] == 4
        st = srv.stats()
        assert info["footprint"] >= st["inflight_bytes"]
        assert st["peak_bytes"] >= st["resident_bytes"] + st["inflight_bytes"]
