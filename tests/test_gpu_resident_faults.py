"""The resident round loop where a launch does not run as asked: a wait of its
barrier that runs out, a cooperative launch that the device refuses."""
import os
import shutil
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


# A stand-in for the runtime's cooperative launch that refuses grids of more
# blocks than a limit (one for the first launch, one for the others), as the
# runtime does for a stream that owns fewer SMs than the device has.
FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
typedef struct { unsigned x, y, z; } D3;
typedef int (*Fn)(const void *, D3, D3, void **, size_t, void *);
int coop_limit_first = 1 << 30, coop_limit = 1 << 30, coop_launched, coop_refused;
int cudaLaunchCooperativeKernel(const void *f, D3 g, D3 b, void **a, size_t m, void *s) {
  if ((int)g.x > (coop_launched ? coop_limit : coop_limit_first)) {
    ++coop_refused;
    return 720; /* cudaErrorCooperativeLaunchTooLarge */
  }
  ++coop_launched;
  return ((Fn)dlsym(RTLD_NEXT, "cudaLaunchCooperativeKernel"))(f, g, b, a, m, s);
}
"""


@pytest.mark.gpu
def test_refused_cooperative_launch(tmp_path):
    """A refused loop runs on fewer SMs, on the first launch as after a counts
    window, and round by round where none fits; the results are the same."""
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no host C compiler")
    src, so = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    subprocess.run([cc, "-shared", "-fPIC", "-o", str(so), str(src), "-ldl"], check=True)
    assert "refusals ok" in _child(f"""
import ctypes, numpy as np, torch, oracle, paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs as I
fake = ctypes.CDLL({str(so)!r})
first, rest, launched, refused = (ctypes.c_int.in_dll(fake, x) for x in
                                  ("coop_limit_first", "coop_limit", "coop_launched", "coop_refused"))
graphs = [I.er(30011, 7, 603), I.rmat(12, 12, 604, directed=True)]
seeds = [I.seeds(g.n, 300, 605) for g in graphs]
want = [oracle.run(g, x) for g, x in zip(graphs, seeds)]
G = pg.Graph.from_inputs(graphs[0])
for a, b, loops in ((1000, 1000, True), (40, 40, True), (1, 1, True), (1000, 20, True), (0, 0, False)):
    def start():
        first.value, rest.value, launched.value, refused.value = a, b, 0, 0
    def check(r, k=0):
        assert r.rounds == want[k]["rounds"] and np.array_equal(r.counts, want[k]["counts"])
        assert (launched.value > 0) == loops and (refused.value > 0) == (a < 1000 or b < 1000)
    for fn, kw in ((pg.propagate_p, {{}}), (pg.propagate_s, {{}}),
                   (pg.propagate_s, {{"planes_per_pass": 32}})):
        start()
        check(fn(G, seeds[0], opts=pg.options(window_rows=2, **kw)))
    start()
    with pg.Batch() as B:
        for g, x in zip(graphs, seeds):
            B.add_inputs(g, x)
        B.set_streams(1)
        B.run(opts=pg.options(window_rows=2))
        for k in range(2):
            check(B.result(k), k)
            assert np.array_equal(B.result(k).m_active, want[k]["m_active"])
print("refusals ok")
""", LD_PRELOAD=str(so))
