"""GPU parity tests of the on-chip sort of small arrays and segments of wide items
(64-bit keys, or 32-bit keys with 64-bit values) at the edges of its CTA sizes, with
keys that spread, crowd, tie in all but their lowest bits or are few, against the
CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1008_2849_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 3, 32, 33, 511, 512, 513, 1023, 1024, 1025, 2049, 4095, 4096, 4097]
WIDE = [("u64", 0), ("i64", 32), ("f64", 64), ("f64", 0), ("u64", 32), ("f32", 64), ("u32", 64)]


@pytest.fixture(scope="module")
def rs():
    from paper_1008_2849_gb300 import build, rs as _rs
    build.build_library()
    _rs.lib()
    return _rs


def _keys(dist, key_type, n, seed):
    lo, hi = (inputs.splitmix32(seed, n, i).astype(np.uint64) for i in (0, 1))
    ones = np.uint64(0xFFFFFFFF)
    if dist == "few":
        lo, hi = lo & np.uint64(3), hi & np.uint64(1)
    elif dist == "crowded":  # half the keys in one bin, the rest spread
        lo, hi = np.where(lo & np.uint64(1), lo >> np.uint64(20), lo), np.where(
            lo & np.uint64(1), np.uint64(0x40000000), hi)
    elif dist == "low bits":  # one of five keys, and the five lowest bits
        hi = hi % np.uint64(5) * np.uint64(0x33333333)
        lo = lo & np.uint64(31) | hi & np.uint64(0xFFFFFF00)
    elif dist == "ends":
        lo = hi = np.where(lo & np.uint64(1), ones, np.uint64(0))
    if key_type.endswith("32"):
        return (hi if dist in ("crowded", "few") else lo).astype(np.uint32)
    return hi << np.uint64(32) | lo


def _values(bits, n):
    idx = np.arange(n, dtype=np.uint64)
    return None if bits == 0 else idx.astype(np.uint32) if bits == 32 else idx << np.uint64(31) | idx


def _dev(a):
    import torch
    return None if a is None else torch.from_numpy(
        a.view(np.int64 if a.dtype == np.uint64 else np.int32)).cuda()


@pytest.mark.parametrize("dist", ["uniform", "few", "crowded", "low bits", "ends"])
@pytest.mark.parametrize("key_type,bits", WIDE)
def test_wide_small(rs, key_type, bits, dist):
    sizes = np.array(SIZES * 2 + [0, 9000], dtype=np.uint64)
    off = inputs.offsets_from_sizes(sizes) + np.uint32(1)
    n = int(off[-1]) + 2
    k = np.concatenate([_keys(dist, key_type, int(m), 40 + i) for i, m in enumerate([1, *sizes, 2])])
    v = _values(bits, n)
    ko, vo = oracle.sort_kv_segmented(k, v, off, key_type)
    kd, vd = _dev(k), _dev(v)
    rs.sort_kv_segmented(kd, vd, _dev(off), key_type)
    assert np.array_equal(kd.cpu().numpy().view(k.dtype), ko)
    assert bits == 0 or np.array_equal(vd.cpu().numpy().view(v.dtype), vo)
    for m in SIZES:
        ko, vo = oracle.sort_kv(k[:m], None if v is None else v[:m], key_type)
        kd, vd = _dev(k[:m]), None if v is None else _dev(v[:m])
        rs.sort_kv(kd, vd, key_type)
        assert np.array_equal(kd.cpu().numpy().view(k.dtype), ko)
        assert bits == 0 or np.array_equal(vd.cpu().numpy().view(v.dtype), vo)
