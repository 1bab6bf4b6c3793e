"""GPU parity tests of the large segments' two orders (one pass by the top digit and
its buckets on chip, or all passes), mixed in one call, against the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1008_2849_gb300 import inputs
from tests.gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu

SIZES = [4097, 5120, 5121, 9_999, 0, 40_961, 1, 65_537, 300_007, 700, 1_100_000, 1_300_003, 8_000]


@pytest.fixture(scope="module")
def rs():
    from paper_1008_2849_gb300 import build, rs as _rs
    build.build_library()
    _rs.lib()
    return _rs


def _segment(kind, m, seed):
    if kind == "two buckets":  # the top digit takes two values
        return inputs.keys("uniform", m, seed) & np.uint32(0x01FFFFFF)
    if kind == "one bucket large":  # one bucket of more than 3584 keys, the rest spread
        k = inputs.keys("uniform", m, seed)
        k[:4700] &= np.uint32(0x00FFFFFF)
        return k
    return inputs.keys(kind, m, seed)


@pytest.mark.parametrize("key_type", ["u32", "i32", "f32"])
@pytest.mark.parametrize("pairs", [True, False])
def test_orders_mixed(rs, key_type, pairs):
    kinds = ["uniform", "and4", "low16", "equal", "sorted", "two buckets", "one bucket large"]
    sizes = np.array(SIZES * 2, dtype=np.uint64)
    off = inputs.offsets_from_sizes(sizes) + np.uint32(3)
    n = int(off[-1]) + 5
    k = inputs.keys("uniform", n, 17)
    for i, (a, m) in enumerate(zip(off[:-1].astype(np.int64), sizes.astype(np.int64))):
        k[a:a + m] = _segment(kinds[i % len(kinds)], int(m), 500 + i)
    v = inputs.index_values(n)
    ko, vo = oracle.sort_kv_segmented(k, v, off, key_type)
    full = rs.alloc_workspace(n, pairs, sizes.size)
    # A workspace without the MSD-first order's parts is taken too: all passes.
    for ws in (full, full[:-256]):
        kd, vd, od = to_dev(k, 1), to_dev(v, 2), to_dev(off)
        rs.sort_segmented_typed_ex(kd, vd if pairs else None, od, key_type, ws)
        rs.check_stream()
        assert np.array_equal(to_host(kd), ko)
        if pairs:
            assert np.array_equal(to_host(vd), vo)


@pytest.mark.parametrize("segments", [1, 1023, 1024, 1025, 5000])
def test_segment_counts(rs, segments):
    """Segment tables at the edges of the planner's CTAs, replayed from a graph."""
    k, v, off = inputs.segmented_batch(segments, 4, 16, seed=segments, scale_to=1 << 22)
    kd, vd, od = to_dev(k), to_dev(v), to_dev(off)
    ko, vo = oracle.sort_pairs_segmented(k, v, off)
    g = rs.Graph(kd, vd, od)
    for _ in range(2):
        kd.copy_(to_dev(k))
        vd.copy_(to_dev(v))
        g.launch()
        rs.check_stream()
        assert np.array_equal(to_host(kd), ko) and np.array_equal(to_host(vd), vo)
    g.close()
