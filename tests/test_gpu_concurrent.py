"""Calls on different graphs from different host threads, and other work on the
device, beside a resident round loop; a loop that ends its launch and goes on."""
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

import oracle
import paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _check(res, want):
    assert res.rounds == want["rounds"]
    assert np.array_equal(res.counts, want["counts"])
    assert np.array_equal(res.m_active, want["m_active"])


def test_a_long_call_lets_others_through():
    """A path of 150,000 nodes takes 150,000 rounds. Calls on another graph (one
    launch; kernels round by round; wide rows) and a kernel of torch, each on a
    stream of its own, take far less than that call does: they run beside it."""
    import torch
    n = 150_000
    g = I.er(50_000, 8, 801)
    seeds = {s: I.seeds(g.n, s, 802) for s in (64, 600)}
    want = {s: oracle.run(g, x) for s, x in seeds.items()}
    x = torch.zeros(1 << 20, device="cuda")
    with pg.Graph.from_inputs(I.path(n)) as L, pg.Graph.from_inputs(g) as G:
        def others():
            for s, kw in ((64, {}), (64, dict(sparse_push=2)), (600, {})):
                _check(pg.propagate_p(G, seeds[s], opts=pg.options(**kw)), want[s])
                yield
            x.add_(1)
            torch.cuda.current_stream().synchronize()
            yield

        def long_call(out):
            with torch.cuda.stream(torch.cuda.Stream()):
                t = time.perf_counter()
                out.append(pg.propagate_p(L, np.zeros(1, np.int32)))
                out.append(time.perf_counter() - t)

        took = []
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in others():  # what a first call sets up
                pass
            out = []
            long_call(out)
            out.clear()
            th = threading.Thread(target=long_call, args=(out,))
            th.start()
            time.sleep(0.1)
            for _ in range(3):
                t = time.perf_counter()
                for _ in others():
                    took.append(time.perf_counter() - t)
                    t = time.perf_counter()
            th.join()
    res, length = out
    assert res.rounds == n - 1 and (res.counts == 1).all()
    assert max(took) < length / 4, (took, length)


def test_two_threads_on_two_graphs():
    """Calls of several kinds from two threads at once: every result as alone."""
    import torch
    graphs = [I.grid(200, 210, 0.05, 803), I.rmat(15, 100, 804, directed=False)]
    work = []
    for g in graphs:
        seeds = [I.seeds(g.n, s, 805) for s in (64, 300)]
        work.append([(x, oracle.run(g, x)) for x in seeds])
    errors = []

    def thread(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()), pg.Graph.from_inputs(graphs[k]) as G:
                for i in range(12):
                    for x, want in work[k]:
                        _check(pg.propagate_p(G, x), want)
                        r = pg.propagate_s(G, x)
                        assert r.rounds == want["rounds"]
                        assert np.array_equal(r.counts, want["counts"])
        except BaseException as e:  # noqa: B902 - the main thread raises it
            errors.append(e)

    th = [threading.Thread(target=thread, args=(k,)) for k in range(2)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    if errors:
        raise errors[0]


def test_a_batch_beside_calls():
    """A packed batch whose part of the SMs changes as another thread's calls come
    and go: its counts windows end at rounds of their own, each graph's m_active
    among them."""
    import torch
    graphs = [I.grid(260, 250, 0.05, 806), I.grid(300, 120, 0.05, 807), I.er(20_000, 6, 808)]
    seeds = [I.seeds(g.n, 100, 809) for g in graphs]
    want = [oracle.run(g, x) for g, x in zip(graphs, seeds)]
    other = I.er(50_000, 8, 810)
    x = I.seeds(other.n, 64, 811)
    want_other = oracle.run(other, x)
    stop, errors = threading.Event(), []

    def calls():
        try:
            with torch.cuda.stream(torch.cuda.Stream()), pg.Graph.from_inputs(other) as G:
                while not stop.is_set():
                    for _ in range(3):
                        _check(pg.propagate_p(G, x), want_other)
                    time.sleep(0.003)
        except BaseException as e:  # noqa: B902 - the main thread raises it
            errors.append(e)

    th = threading.Thread(target=calls)
    th.start()
    split = False  # the loop ended its launch and went on
    try:
        with pg.Batch() as b:
            for g, sd in zip(graphs, seeds):
                b.add_inputs(g, sd)
            for k in range(100):
                b.set_streams(4 if k == 1 else 1)
                b.run()
                for i, w in enumerate(want):
                    _check(b.result(i), w)
                split = split or b.stats()["launches"] > b.stats()["groups"]
                if split and k >= 3:
                    break
    finally:
        stop.set()
        th.join()
    if errors:
        raise errors[0]
    assert split


def test_a_loop_that_ends_after_every_round():
    """Launches of one round each (and so a counts window of one row): pushed and
    swept rounds, passes as words, copies as a packed batch, rows on lane pairs
    with the seeds placed by degree. Counts and m_active as the oracle's."""
    code = """
import ctypes, numpy as np, oracle, paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I, _abi
L = _abi.lib()
L.pg_debug_slice.argtypes = [ctypes.c_void_p, ctypes.c_int64]
L.pg_debug_slice.restype = None
for g in (I.grid(37, 41, 0.05, 401), I.er(3001, 7, 402), I.rmat(11, 12, 403, directed=True),
          I.rmat(15, 100, 301, directed=False)):
    G = pg.Graph.from_inputs(g)
    L.pg_debug_slice(G._h, 1)
    for s in (1, 64, 130, 300, 512):
        seeds = I.seeds(g.n, s, 404)
        want = oracle.run(g, seeds)
        for kw in ({}, dict(direction=pg.PG_DIR_DENSE), dict(direction=pg.PG_DIR_SPARSE)):
            r = pg.propagate_p(G, seeds, opts=pg.options(**kw))
            assert G.last_stats()["launches"] == want["rounds"] + 1 or s > 64, G.last_stats()
            assert r.rounds == want["rounds"] and np.array_equal(r.counts, want["counts"]), (s, kw)
            assert np.array_equal(r.m_active, want["m_active"]), (s, kw)
            for planes in (64, 32):
                r = pg.propagate_s(G, seeds, opts=pg.options(planes_per_pass=planes, **kw))
                act = np.zeros(want["rounds"] + 2, np.uint64)
                for k in range(0, s, planes):
                    a = oracle.run(g, seeds[k:k + planes])["m_active"]
                    act[:a.size] += a
                assert r.rounds == want["rounds"] and np.array_equal(r.counts, want["counts"]), (s, kw)
                assert np.array_equal(r.m_active, act[:r.m_active.size]), (s, kw, planes)
print("slices ok")
"""
    out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True,
                         env=dict(os.environ, PG_LIBRARY_VARIANT="debug-bounds"), timeout=1200)
    assert out.returncode == 0, out.stderr[-3000:]
    assert "slices ok" in out.stdout
