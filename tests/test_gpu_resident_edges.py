"""The resident round loop at the sizes where its parts change: frontier rows of
exactly as many out-arcs as one group of lanes pushes (32) or a piece holds (128),
one less and one more; warps whose stage of changed rows runs full in the middle
of a pushed and of a swept round."""
import functools

import numpy as np
import pytest

import oracle
import paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DEGREES = (1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 384, 385, 2000)


@functools.lru_cache(maxsize=None)
def _hubs(directed):
    """A chain of nodes with exactly these out-degrees, its arcs among them; the
    leaves are shared."""
    k = len(DEGREES)
    chain = np.arange(k - 1)
    on_chain = np.full(k, 2) if not directed else np.full(k, 1)
    on_chain[-1] -= 1
    if not directed:
        on_chain[0] -= 1
    leaves = np.array(DEGREES) - on_chain
    src = np.concatenate([np.full(d, i) for i, d in enumerate(leaves)] + [chain])
    dst = np.concatenate([k + np.arange(d) for d in leaves] + [chain + 1])
    g = I.from_arcs(k + max(DEGREES), src, dst, symmetrise=not directed)
    if not directed:
        out = np.diff(g.row_ptr)[:k]
    else:
        out = np.bincount(g.col, minlength=g.n)[:k]
    assert tuple(out) == DEGREES
    return g


def _check(G, g, seeds, kw):
    want = oracle.run(g, seeds)
    per_pass = np.zeros(want["rounds"] + 2, np.uint64)
    for k in range(0, seeds.size, 64):
        b = oracle.run(g, seeds[k:k + 64])["m_active"]
        per_pass[:b.size] += b
    for fn, act in ((pg.propagate_p, want["m_active"]), (pg.propagate_s, per_pass)):
        r = fn(G, seeds, opts=pg.options(**kw))
        assert G.last_stats()["launches"] == 1
        assert r.rounds == want["rounds"], kw
        assert np.array_equal(r.counts, want["counts"]), kw
        assert np.array_equal(r.m_active, act[:r.m_active.size]), kw


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("s", [17, 64, 130, 300, 512])
def test_rows_of_a_group_and_of_a_piece(directed, s):
    g = _hubs(directed)
    # the hubs first: several rows of every length are in one frontier
    seeds = np.concatenate([np.arange(len(DEGREES)),
                            np.arange(len(DEGREES), g.n)[::3]])[:s].astype(np.int32)
    assert seeds.size == s
    with pg.Graph.from_inputs(g) as G:
        for kw in (dict(direction=pg.PG_DIR_SPARSE), dict(), dict(direction=pg.PG_DIR_DENSE)):
            _check(G, g, seeds, kw)


@pytest.mark.parametrize("s", [1, 65])
@pytest.mark.parametrize("direction", [pg.PG_DIR_SPARSE, pg.PG_DIR_DENSE])
def test_a_full_stage(s, direction):
    """A star of 1.2 million leaves: its centre's arcs are 9,375 pieces of 128, at
    least three for some warp of any launch of up to 256 blocks of 16 warps, and a
    stage holds two; its leaves are 37,500 chunks of 32 rows, at least nine for
    some warp, and a stage holds eight."""
    n = 1_200_001
    assert (n - 1) / 128 > 2 * 256 * 16 and n / 32 > 8 * 256 * 16
    g = I.star(n)
    assert np.diff(g.row_ptr).max() == n - 1
    centre = int(np.diff(g.row_ptr).argmax())
    seeds = np.concatenate([[centre], I.seeds(n, 2 * s, 971)])
    seeds = np.unique(seeds[seeds != centre])[:s - 1]
    seeds = np.concatenate([[centre], seeds]).astype(np.int32)
    assert seeds.size == s
    with pg.Graph.from_inputs(g) as G:
        _check(G, g, seeds, dict(direction=direction))
