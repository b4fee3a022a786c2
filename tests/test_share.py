"""Parts of the SMs that propagations side by side get: equal up to what each can
use, together never more than there are."""
import ctypes
import itertools

import pytest

from paper_2301_06499_gb300 import build


@pytest.fixture(scope="module")
def parts():
    f = ctypes.CDLL(build.build(variant="debug-bounds")).pg_debug_share_parts
    f.restype = None

    def call(cap, need, total=152):
        n = len(cap)
        out = (ctypes.c_int * n)()
        f(n, (ctypes.c_int * n)(*cap), (ctypes.c_int * n)(*need), total, out)
        return list(out)
    return call


@pytest.mark.parametrize("cap,need,want", [
    ([152], [8], [152]),  # alone: all it may use
    ([40], [40], [40]),
    ([152, 152], [152, 152], [76, 76]),
    ([152, 152], [152, 8], [144, 8]),  # a small one beside a large one
    ([152, 152, 152], [152, 152, 152], [50, 51, 51]),
    ([38, 38, 38, 38], [38, 38, 38, 38], [38, 38, 38, 38]),  # limits that fit stay
    ([152, 38, 38], [152, 38, 38], [76, 38, 38]),
    ([1000], [8], [152]),
])
def test_parts(parts, cap, need, want):
    assert sorted(parts(cap, need)) == sorted(want)
    assert parts(cap, need)[0] == want[0]


def test_parts_fit_and_are_even(parts):
    for n in (2, 3, 5, 64, 151, 152, 153, 200):
        for pattern in itertools.product((1, 8, 60, 152), repeat=2):
            need = [pattern[i % 2] for i in range(n)]
            cap = [152 if i % 3 else 100 for i in range(n)]
            use = [min(c, x) for c, x in zip(cap, need)]
            got = parts(cap, need)
            assert all(1 <= g <= u for g, u in zip(got, use))
            assert sum(got) <= max(152, n)
            short = [g for g, u in zip(got, use) if g < u]
            if short:  # nothing is left over, and no one has much more than who lacks
                assert sum(got) >= 152 or n > 152
                assert max(got) <= min(short) + 1
