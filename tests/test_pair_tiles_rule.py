"""The widths of pair tiles (host only): what the pair kernel's halves, copies
and epilogue rest on, over shapes of every size."""

import ctypes
import random

import pytest


@pytest.fixture(scope="module")
def rule():
    from paper_1608_05265_gb300 import build
    f = ctypes.CDLL(build.build()).gbgemm_internal_pair_tiles
    i64 = ctypes.c_int64
    f.argtypes = [i64, i64, i64, i64, ctypes.c_int, ctypes.c_int, ctypes.POINTER(i64)]

    def tiles(*args):
        out = (i64 * 3)()
        f(*args, out)
        return tuple(out)

    return tiles


@pytest.mark.parametrize("seed", range(4))
def test_widths_and_halves(rule, seed):
    r = random.Random(seed)
    size = lambda hi: min(hi, int(2 ** r.uniform(0, 15)) + r.randrange(3))
    for _ in range(2000):
        m, n, batch, pairs = max(129, size(40000)), size(40000), size(64), r.choice([1, 7, 70, 76])
        bn, tiles, tail = rule(m, n, batch, size(2048), r.randrange(2), pairs)
        assert 64 <= bn <= 256 and bn % 32 == 0
        assert tiles == (m + 255) // 256 * ((n + bn - 1) // bn) * batch
        assert 0 <= tail <= tiles
        if tail < tiles:  # the last ones in halves: whole rounds before, halves that the MMA takes
            assert tail % pairs == 0 and bn % 64 == 0
        width = bn // 2 if tail < tiles else bn
        assert n + 2 * bn < 2 ** 31 and width % 32 == 0
