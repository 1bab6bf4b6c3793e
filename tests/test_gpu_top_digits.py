"""GPU parity tests of the top-digits order of whole arrays (two scatter passes
by the highest digits, then chunks sorted on chip), against the CPU oracle: at
the ends of its size ranges, for keys that the plan takes and refuses, and with
chunks too long for the chip."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1008_2849_gb300 import inputs
from tests.gpu_util import oracle_sort, to_dev, to_host

pytestmark = pytest.mark.gpu

FIRST = 1 << 25  # the smallest array it is tried for


@pytest.fixture(scope="module")
def rs():
    from paper_1008_2849_gb300 import build, rs as _rs
    build.build_library()
    _rs.lib()
    return _rs


def _keys(kind, n, seed):
    k = inputs.keys("uniform", n, seed)
    if kind == "same digits":  # each digit even, the top two always equal
        return (k & np.uint32(0x00FFFFFF)) | ((k << np.uint32(8)) & np.uint32(0xFF000000))
    if kind == "long chunks":  # two prefixes with 2400 keys more than their share
        k[5:4805:2] = (k[5:4805:2] & np.uint32(0xFFFF)) | np.uint32(0x12340000)
        k[-4801::2] = (k[-4801::2] & np.uint32(0xFF)) | np.uint32(0xFFFFFF00)
        return k
    if kind == "few low bits":  # chunks whose keys crowd into few bins
        return k & np.uint32(0xFFFF000F)
    if kind in ("uniform", "no low digits"):
        return k if kind == "uniform" else k & np.uint32(0xFFFF0000)
    return inputs.keys(kind, n, seed)


@pytest.mark.parametrize("kind,taken", [
    ("uniform", True), ("sorted", True), ("reverse", True), ("few low bits", True),
    ("long chunks", True), ("same digits", False), ("no low digits", False), ("and2", False),
    ("distinct256", False), ("equal", False), ("low16", False)])
def test_order_and_result(rs, kind, taken):
    n = FIRST
    k = _keys(kind, n, 40 + n % 13)
    v = inputs.index_values(n)
    ko, vo = oracle_sort(k, v)
    for pairs in (True, False):
        ws = rs.alloc_workspace(n, pairs)
        kd, vd = to_dev(k, 1), to_dev(v, 3)
        if pairs:
            rs.sort_pairs_ex(kd, vd, ws)
        else:
            rs.sort_keys_ex(kd, ws)
        rs.check_stream()
        assert np.array_equal(to_host(kd), ko), (kind, pairs)
        if pairs:
            assert np.array_equal(to_host(vd), vo), kind
        # Control block, word 25: the chunks of this order (0: another order).
        assert (int(ws[100:104].cpu().numpy().view(np.uint32)[0]) > 0) == taken, kind


@pytest.mark.parametrize("key_type", ["i32", "f32"])
def test_typed_keys(rs, key_type):
    n = FIRST + 5
    k = _keys("long chunks", n, 61)
    v = inputs.index_values(n)
    kd, vd = to_dev(k), to_dev(v)
    rs.sort_typed(kd, vd, key_type)
    ko, vo = oracle.sort_typed(k, v, key_type)
    assert np.array_equal(to_host(kd), ko) and np.array_equal(to_host(vd), vo)


@pytest.mark.parametrize("n", [FIRST + 8192, (1 << 26) + 3, (1 << 28) + 65536])
def test_chunk_sizes(rs, n):
    """The first arrays with other chunks (the last with the larger CTA), replayed
    from a graph."""
    k = inputs.keys("uniform", n, 71)
    v = inputs.index_values(n)
    ko, vo = oracle_sort(k, v)
    kd, vd = to_dev(k), to_dev(v)
    k0, v0 = kd.clone(), vd.clone()
    g = rs.Graph(kd, vd)
    for _ in range(2):
        kd.copy_(k0)
        vd.copy_(v0)
        g.launch()
        rs.check_stream()
        assert np.array_equal(to_host(kd), ko) and np.array_equal(to_host(vd), vo)
    g.close()
    kd.copy_(k0)
    rs.sort_keys(kd)
    assert np.array_equal(to_host(kd), ko)


def _wide_keys(kind, n, seed, bits):
    k = inputs.splitmix32(seed, n, 0).astype(np.uint64)
    if bits == 32:
        return k.astype(np.uint32)
    k = (k << np.uint64(32)) | inputs.splitmix32(seed, n, 1).astype(np.uint64)
    if kind == "long chunks":  # one prefix with 1500 keys more, their low words nearly equal
        k[7:3007:2] = (k[7:3007:2] & np.uint64(0x3)) | np.uint64(0x1234000000000000)
    elif kind == "equal low":  # chunks of few distinct keys
        k &= np.uint64(0xFFFFFF0000000000)
    return k


@pytest.mark.parametrize("n", [(1 << 14) - 1, 1 << 14, 100_003, (1 << 20) + 5, 3_000_001])
@pytest.mark.parametrize("key_type,value_bits", [("u64", 0), ("u64", 32), ("i64", 64), ("f64", 32),
                                                 ("f64", 64)])
def test_wide_keys(rs, n, key_type, value_bits):
    for kind in ("uniform", "long chunks", "equal low"):
        if kind != "uniform" and n < (1 << 20):
            continue
        k = _wide_keys(kind, n, 80 + n % 17, 64)
        v = None
        if value_bits:
            v = np.arange(n, dtype=np.uint64 if value_bits == 64 else np.uint32)
        import torch
        signed = np.int64 if value_bits == 64 else np.int32
        kd = torch.from_numpy(k.view(np.int64)).cuda()
        vd = None if v is None else torch.from_numpy(v.view(signed)).cuda()
        rs.sort_kv(kd, vd, key_type)
        ko, vo = oracle.sort_kv(k, v, key_type)
        assert np.array_equal(kd.cpu().numpy().view(np.uint64), ko), kind
        if v is not None:
            assert np.array_equal(vd.cpu().numpy().view(v.dtype), vo), kind


def test_32_bit_keys_with_64_bit_values(rs):
    import torch
    n = FIRST + 3
    k = inputs.keys("uniform", n, 91)
    v = np.arange(n, dtype=np.uint64) << np.uint64(20)
    kd, vd = to_dev(k), torch.from_numpy(v.view(np.int64)).cuda()
    rs.sort_kv(kd, vd, "i32")
    place = np.argsort(k.view(np.int32), kind="stable")
    assert np.array_equal(to_host(kd), k[place])
    assert np.array_equal(vd.cpu().numpy().view(np.uint64), v[place])


def _uneven_keys(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "normal":
        return rng.standard_normal(n).view(np.uint64)
    if kind == "low40":   # the top digits never differ
        return rng.integers(0, 1 << 40, n, dtype=np.uint64)
    if kind == "and2":
        return rng.integers(0, 1 << 63, n, dtype=np.uint64) & rng.integers(0, 1 << 63, n, dtype=np.uint64)
    if kind == "hidden crowd":  # some 6000 keys of one prefix, too few to be sampled
        k = rng.standard_normal(n).view(np.uint64)
        k[11:12_011:2] = (k[11:12_011:2] & np.uint64(0xFFFF)) | np.uint64(0x3FF1234500000000)
        return k
    return np.sort(rng.standard_normal(n)).view(np.uint64)[::-1].copy()  # "reverse"


@pytest.mark.parametrize("n", [1 << 14, 65_537, (1 << 20) + 5, 4_500_003])
@pytest.mark.parametrize("key_type,value_bits", [("u64", 0), ("i64", 32), ("f64", 64)])
def test_uneven_wide_keys(rs, n, key_type, value_bits):
    """Keys that take more than two passes by their highest digits, and chunks by
    position: 64-bit keys that crowd, with digits that never differ, and with a
    crowd that the plan cannot see."""
    import torch
    for kind in ("normal", "low40", "and2", "hidden crowd", "reverse"):
        k = _uneven_keys(kind, n, 7 + n % 11)
        v = None
        if value_bits:
            v = np.arange(n, dtype=np.uint64 if value_bits == 64 else np.uint32)
        kd = torch.from_numpy(k.view(np.int64)).cuda()
        vd = None
        if v is not None:
            vd = torch.from_numpy(v.view(np.int64 if value_bits == 64 else np.int32)).cuda()
        rs.sort_kv(kd, vd, key_type)
        ko, vo = oracle.sort_kv(k, v, key_type)
        assert np.array_equal(kd.cpu().numpy().view(np.uint64), ko), kind
        if v is not None:
            assert np.array_equal(vd.cpu().numpy().view(v.dtype), vo), kind
