"""GPU parity tests of the on-chip sorts where keys repeat: bins longer than the windows'
first rounds, bins that hold one key each, words that differ in their index only, and
arrays of one key, against the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1008_2849_gb300 import inputs
from tests.gpu_util import oracle_sort, to_dev, to_host

pytestmark = pytest.mark.gpu

SIZES = [2, 3, 9, 33, 64, 100, 255, 256, 512, 513, 1000, 1024, 1025, 2048, 3000, 4095, 4096, 5000,
         9000, 40_000]


@pytest.fixture(scope="module")
def rs():
    from paper_1008_2849_gb300 import build, rs as _rs
    build.build_library()
    _rs.lib()
    return _rs


def _segment(m, times, near, bits, seed):
    """m keys, each some `times` times; near: every other of them one more in its lowest
    bits, which a word with an index in its place does not hold."""
    rng = np.random.default_rng(seed)
    words = rng.integers(0, 1 << bits, max(1, m // times), dtype=np.uint64)
    k = words[rng.integers(0, words.size, m)]
    if near:
        k ^= rng.integers(0, 2, m, dtype=np.uint64)
    return k.astype(np.uint32 if bits == 32 else np.uint64)


@pytest.mark.parametrize("times", [2, 4, 9, 16, 40, 70, 200, 5000])
@pytest.mark.parametrize("near", [False, True])
@pytest.mark.parametrize("key_type,value_bits", [("u32", 0), ("u32", 32), ("u64", 0), ("f64", 32),
                                                 ("i32", 64)])
def test_segments(rs, times, near, key_type, value_bits):
    import torch
    bits = 64 if key_type[1:] == "64" else 32
    sizes = np.array(SIZES + SIZES[:16], dtype=np.uint64)
    off = inputs.offsets_from_sizes(sizes)
    n = int(off[-1])
    k = np.concatenate([_segment(int(m), times, near, bits, 31 * times + i)
                        for i, m in enumerate(sizes)])
    v = None
    if value_bits:
        v = np.arange(n, dtype=np.uint64 if value_bits == 64 else np.uint32)
    kd = torch.from_numpy(k.view(np.int64 if bits == 64 else np.int32)).cuda()
    vd = None
    if v is not None:
        vd = torch.from_numpy(v.view(np.int64 if value_bits == 64 else np.int32)).cuda()
    ws = torch.empty(rs.workspace_bytes_kv_segmented(n, key_type, value_bits, sizes.size) + 256,
                     dtype=torch.uint8, device="cuda")
    pad = -ws.data_ptr() % 256
    rs.sort_kv_segmented_ex(kd, vd, to_dev(off), key_type, ws[pad:])
    rs.check_stream()
    ko, vo = k.copy(), None if v is None else v.copy()
    for a, b in zip(off[:-1].astype(int), off[1:].astype(int)):
        sk, sv = oracle.sort_kv(k[a:b], None if v is None else v[a:b], key_type)
        ko[a:b] = sk
        if v is not None:
            vo[a:b] = sv
    assert np.array_equal(kd.cpu().numpy().view(k.dtype), ko)
    if v is not None:
        assert np.array_equal(vd.cpu().numpy().view(v.dtype), vo)


@pytest.mark.parametrize("n", [20_000, 1_000_003, 1_500_001, (1 << 25) + 3])
@pytest.mark.parametrize("times", [4, 16, 100])
def test_whole_arrays(rs, n, times):
    k = _segment(n, times, times == 16, 32, n + times)
    v = inputs.index_values(n)
    ko, vo = oracle_sort(k, v)
    kd, vd = to_dev(k, 1), to_dev(v, 2)
    rs.sort_pairs(kd, vd)
    assert np.array_equal(to_host(kd), ko) and np.array_equal(to_host(vd), vo)
    kd = to_dev(k)
    rs.sort_keys(kd)
    assert np.array_equal(to_host(kd), ko)
