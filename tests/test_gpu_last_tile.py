"""GPU parity tests of the scatter passes' last tile, which is ranked slot by slot in a
loop: tiles of one item, around a warp's slots and all but full, as whole arrays above the
MSD-first order's sizes and as segments, against the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1008_2849_gb300 import inputs
from tests.gpu_util import oracle_sort, to_dev, to_host

pytestmark = pytest.mark.gpu

PAIR_TILE, KEY_TILE = 384 * 13, 384 * 18
LAST = [1, 31, 32, 33, 415, 416, 417, 577, 3000]


@pytest.fixture(scope="module")
def rs():
    from paper_1008_2849_gb300 import build, rs as _rs
    build.build_library()
    _rs.lib()
    return _rs


@pytest.mark.parametrize("last", LAST + [-1])
@pytest.mark.parametrize("dist", ["uniform", "and4", "equal"])
def test_whole_arrays(rs, last, dist):
    n = 400 * PAIR_TILE + last
    k, v = inputs.keys(dist, n, 60 + len(dist)), inputs.index_values(n)
    ko, vo = oracle_sort(k, v)
    kd, vd = to_dev(k, 1), to_dev(v, 3)
    rs.sort_pairs(kd, vd)
    assert np.array_equal(to_host(kd), ko) and np.array_equal(to_host(vd), vo)
    n = 290 * KEY_TILE + last
    kd = to_dev(k[:n], 2)
    rs.sort_keys(kd)
    assert np.array_equal(to_host(kd), np.sort(k[:n]))
    kd = to_dev(k[:n])
    rs.sort_typed(kd, None, "i32")
    assert np.array_equal(to_host(kd), np.sort(k[:n].view(np.int32)).view(np.uint32))


@pytest.mark.parametrize("dist", ["uniform", "and4"])
@pytest.mark.parametrize("pairs", [True, False])
def test_segments(rs, dist, pairs):
    sizes = np.array([2 * PAIR_TILE + r for r in LAST], dtype=np.uint64)
    off = inputs.offsets_from_sizes(sizes)
    n = int(off[-1])
    k, v = inputs.keys(dist, n, 71) & np.uint32(0xFFFFFF), inputs.index_values(n)
    ko, vo = oracle.sort_pairs_segmented(k, v, off)
    kd, vd, od = to_dev(k, 1), to_dev(v, 1), to_dev(off)
    if pairs:
        rs.sort_pairs_segmented(kd, vd, od)
        assert np.array_equal(to_host(vd), vo)
    else:
        rs.sort_keys_segmented(kd, od)
    assert np.array_equal(to_host(kd), ko)
