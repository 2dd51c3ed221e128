"""Which launches of the compaction let CTAs go on with other units: a host decision, asked for the sizes that the GPU tests rely
on and on both sides of its two lines."""
import ctypes

import pytest

from paper_2603_00907_b200 import binding, build
from tests import test_gpu_compact_shares as shares, test_gpu_short_waits as waits

SINK, TILE = 32, 64


@pytest.fixture(scope="module")
def decide():
    build.build()
    fn = binding.lib().kvs_detail_compact_shares

    def ask(hkv, tiles):
        per_unit = ctypes.c_int32()
        helped = fn((ctypes.c_int32 * len(tiles))(*tiles), len(tiles), hkv, ctypes.byref(per_unit))
        return helped, per_unit.value

    return ask


def _tiles(lens):
    return [max(0, (n - SINK + TILE - 1) // TILE) for n in lens]


@pytest.mark.parametrize("hkv,lens,want", [(h, n, 1) for h, n, _ in shares.HELPED + waits.HELPING] +
                         [(h, n, 0) for h, n, _ in shares.NOT_HELPED + waits.APART])
def test_the_sizes_of_the_gpu_tests(decide, hkv, lens, want):
    assert decide(hkv, _tiles(lens))[0] == want


def test_the_lines(decide):
    # 160 units on 296 CTAs, 1.85 of the average on the busiest: from 40 tiles on, and then up to two CTAs a unit
    assert decide(8, [39] * 20) == (0, 1) and decide(8, [40] * 20) == (1, 2)
    # 232 and 240 units: 1.28 and 1.23 of the average
    assert decide(8, [100] * 29) == (1, 2) and decide(8, [100] * 30) == (0, 1)
    # empty units count for nothing
    assert decide(8, [0] * 30 + [39] * 20)[0] == 0 and decide(8, [0] * 30 + [40] * 20)[0] == 1
