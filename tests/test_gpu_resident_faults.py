"""The resident round loop where a launch does not run as asked: a wait of its
barrier that runs out."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _child(code, **env):
    out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, **env),
                         capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stderr[-3000:]
    return out.stdout


@pytest.mark.gpu
def test_barrier_wait_that_runs_out():
    """Every block gives up after the limit (a millisecond, for a block that
    never comes), the call returns PG_ETIMEOUT, and the next one on the graph,
    on another stream, is whole. One graph and a packed batch, whose blocks wait
    for a release."""
    assert "timeouts ok" in _child("""
import ctypes, numpy as np, torch, oracle, paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I, _abi
L = _abi.lib()
L.pg_debug_short_barrier.argtypes = [ctypes.c_void_p, ctypes.c_uint64]
L.pg_debug_short_barrier.restype = None
g = I.er(30011, 7, 601)
seeds = {s: I.seeds(g.n, s, 602) for s in (64, 300)}
want = {s: oracle.run(g, x) for s, x in seeds.items()}
G = pg.Graph.from_inputs(g)
streams = [torch.cuda.Stream() for _ in range(2)]
for k, (fn, s, kw) in enumerate([(pg.propagate_p, 64, {}), (pg.propagate_p, 300, {}),
                                 (pg.propagate_s, 300, {}),
                                 (pg.propagate_s, 300, {"planes_per_pass": 32})]):
    for again in range(2):  # after calls of other kinds, and after one of its own
        L.pg_debug_short_barrier(G._h, 1_000_000)
        with torch.cuda.stream(streams[k % 2]):
            try:
                fn(G, seeds[s], opts=pg.options(**kw))
                raise SystemExit("the wait did not run out")
            except pg.PropagateError as e:
                assert e.status == _abi.PG_ETIMEOUT, e
        with torch.cuda.stream(streams[1 - k % 2]):
            r = fn(G, seeds[s], opts=pg.options(**kw))
        assert G.last_stats()["launches"] == 1 or kw
        assert r.rounds == want[s]["rounds"] and np.array_equal(r.counts, want[s]["counts"])
print("timeouts ok")
""", PG_LIBRARY_VARIANT="debug-bounds")
