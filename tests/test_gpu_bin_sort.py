"""GPU parity tests of the one-CTA bin sort: arrays at the edges of its CTA
sizes and bin counts, keys that spread over the bins, crowd into few (the digit
passes), differ in few bits or not at all, against the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1008_2849_gb300 import inputs
from tests.gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 3, 31, 32, 33, 127, 128, 129, 511, 512, 513, 1023, 1024, 1025, 2047, 2049, 4095,
         4096, 4097, 5000, 8191, 8192]


@pytest.fixture(scope="module")
def rs():
    from paper_1008_2849_gb300 import build, rs as _rs
    build.build_library()
    _rs.lib()
    return _rs


def _keys(dist, n, seed):
    if dist == "crowded":  # half the keys in one bin, the rest spread
        k = inputs.keys("uniform", n, seed)
        half = inputs.splitmix32(seed, n, 5) & np.uint32(1)
        return np.where(half == 1, k, (k & np.uint32(0xFFF)) | np.uint32(0x40000000)).astype(np.uint32)
    if dist == "narrow":  # seven bits differ, below common ones
        return (inputs.keys("uniform", n, seed) & np.uint32(0x7F00)) | np.uint32(0xABCD0011)
    if dist == "ends":  # the smallest and largest words
        return np.where(inputs.keys("uniform", n, seed) >> np.uint32(31), np.uint32(0xFFFFFFFF),
                        np.uint32(0)).astype(np.uint32)
    return inputs.keys(dist, n, seed)


DISTS = ["uniform", "and2", "and4", "equal", "sorted", "reverse", "low16", "crowded", "narrow",
         "ends"]


@pytest.mark.parametrize("dist", DISTS)
@pytest.mark.parametrize("pairs", [True, False])
def test_segments_of_every_cta_size(rs, dist, pairs):
    sizes = np.array(SIZES * 3, dtype=np.uint64)
    off = inputs.offsets_from_sizes(sizes)
    n = int(off[-1])
    k = np.concatenate([_keys(dist, int(m), 700 + i) for i, m in enumerate(sizes)])
    v = inputs.index_values(n)
    saved = {c: {kn: rs.tune_get_class(c, kn) for kn in ("small_max", "warp_max")}
             for c in range(rs.NUM_SIZE_CLASSES)}
    try:
        for warp_max in (0, 512):
            rs.tune_set("small_max", 8192)
            rs.tune_set("warp_max", warp_max)
            kd, vd, od = to_dev(k, 1), to_dev(v, 3), to_dev(off)
            if pairs:
                rs.sort_pairs_segmented(kd, vd, od)
            else:
                rs.sort_keys_segmented(kd, od)
            ko, vo = oracle.sort_pairs_segmented(k, v, off)
            assert np.array_equal(to_host(kd), ko)
            if pairs:
                assert np.array_equal(to_host(vd), vo)
    finally:
        for c, kn in saved.items():
            for name, val in kn.items():
                rs.tune_set_class(c, name, val)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("key_type", ["u32", "i32", "f32"])
def test_single_arrays(rs, n, key_type):
    for dist in ("uniform", "crowded", "ends"):
        k = _keys(dist, n, 900 + n)
        v = inputs.index_values(n)
        kd, vd = to_dev(k), to_dev(v)
        rs.sort_typed(kd, vd, key_type)
        ko, vo = oracle.sort_typed(k, v, key_type)
        assert np.array_equal(to_host(kd), ko) and np.array_equal(to_host(vd), vo)
        kd = to_dev(k)
        rs.sort_typed(kd, None, key_type)
        assert np.array_equal(to_host(kd), ko)
