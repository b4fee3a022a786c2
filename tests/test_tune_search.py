"""The tuner's search, with given times for its runs: it times the options that
the schedule reads, and no others."""
import ctypes

import pytest

from paper_2301_06499_gb300 import _abi, build


@pytest.fixture(scope="module")
def search():
    f = ctypes.CDLL(build.build(variant="debug-bounds")).pg_debug_tune
    cb = ctypes.CFUNCTYPE(ctypes.c_double, ctypes.POINTER(_abi.Options))
    f.argtypes = [ctypes.c_int32, ctypes.c_int32, ctypes.c_int32, cb,
                  ctypes.POINTER(_abi.Options), ctypes.POINTER(_abi.TuneReport)]

    def call(s, s_mode, ms, **kw):
        o = _abi.Options(**{"use_graphs": 1, "planes_per_pass": 64, **kw})
        tried, rep = [], _abi.TuneReport()

        def run(p):
            tried.append({k: getattr(p.contents, k) for k, _ in p.contents._fields_})
            return ms(tried[-1])
        assert f(s, s_mode, 1000, cb(run), ctypes.byref(o), ctypes.byref(rep)) == _abi.PG_OK
        return {k: getattr(o, k) for k, _ in o._fields_}, tried[::3], rep
    return call


@pytest.mark.parametrize("s,s_mode", [(64, 0), (256, 0), (512, 0), (64, 1), (300, 1)])
def test_lanes_are_tried_where_they_are_read(search, s, s_mode):
    lanes = lambda tried: sorted({t["group_lanes"] for t in tried})  # noqa: E731
    _, tried, _ = search(s, s_mode, lambda o: 1.0)
    assert lanes(tried) == [0]  # the resident loop
    assert {round(t["dense_threshold"], 3) for t in tried} == {0, 0.01, 0.02, 0.05, 0.1, 0.2, 0.5}
    every = [0, 1, 2, 4, 8, 16, 32]
    # round by round: asked for, or found to be faster
    for kw in (dict(sparse_push=2), dict(use_graphs=0), dict(timing=1), dict(tma_gather=2)):
        assert lanes(search(s, s_mode, lambda o: 1.0, **kw)[1]) == every, kw
    got, tried, rep = search(s, s_mode, lambda o: 0.5 if o["sparse_push"] == 1 else 1.0)
    assert got["sparse_push"] == 1 and lanes(tried) == every
    assert 0.05 not in [round(t["dense_threshold"], 3) for t in tried]  # what 0 is there
    if s > 64 and not s_mode:
        got, tried, rep = search(s, s_mode, lambda o: 0.5 if o["words_per_thread"] == 1 else 1.0)
        assert got["words_per_thread"] == 1 and lanes(tried) == every


@pytest.mark.parametrize("s", [600, 5568])
def test_wide_rows_have_no_lanes(search, s):
    _, tried, _ = search(s, 0, lambda o: 1.0)
    assert {t["group_lanes"] for t in tried} == {0}
