"""GPU tests of which order the plan chooses, read from the control block at the start of
the workspace, beside the results against the CPU oracle: keys that repeat or share few
prefixes take the passes by all digits, as does an array with one hot key; wide items and
large segments take the orders that their other tests mean to reach."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1008_2849_gb300 import inputs
from tests.gpu_util import oracle_sort, to_dev, to_host

pytestmark = pytest.mark.gpu

# Words of the control block (rs_device.cuh).
CHUNKS, MSD_TILES, LSD_TILES, STEP, SRC = 25, 26, 27, 29, 30


@pytest.fixture(scope="module")
def rs():
    from paper_1008_2849_gb300 import build, rs as _rs
    build.build_library()
    _rs.lib()
    return _rs


def _ctrl(ws):
    return ws[:128].cpu().numpy().view(np.uint32)


def _workspace(nbytes):
    import torch
    raw = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    pad = -raw.data_ptr() % 256
    return raw[pad:pad + nbytes]


def _words(rng, n, bits):
    return rng.integers(0, 1 << bits, n, dtype=np.uint64).astype(
        np.uint32 if bits == 32 else np.uint64)


def _keys(kind, n, bits, seed):
    rng = np.random.default_rng(seed)
    name, _, count = kind.partition(" ")
    if name == "distinct":
        return _words(rng, int(count), bits)[rng.integers(0, int(count), n)]
    if name == "prefixes":  # of the upper half of the bits
        high = _words(rng, int(count), bits)[rng.integers(0, int(count), n)]
        half = bits // 2
        return (high >> half << half) | (_words(rng, n, bits) >> half)
    k = _words(rng, n, bits)
    if name == "and4":  # words that differ in few bits
        for _ in range(3):
            k &= _words(rng, n, bits)
    if name == "hot":  # `count` in 1000 items have one key
        k[rng.random(n) < float(count) / 1000] = k[0]
    if name == "slope":  # denser towards the greatest key, by 1 - c to 1 + c of the mean
        c = float(count) / 100
        x = (np.sqrt((1 - c) ** 2 + 4 * c * rng.random(n)) - (1 - c)) / (2 * c)
        high = np.minimum(x, 1 - 2.0 ** -53) * 2.0 ** 32
        k = high.astype(np.uint32) if bits == 32 else (high.astype(np.uint64) << 32) | (k >> 32)
    return k


def _sort32(rs, k):
    v = inputs.index_values(k.size)
    ws = rs.alloc_workspace(k.size, True)
    kd, vd = to_dev(k), to_dev(v)
    rs.sort_pairs_ex(kd, vd, ws)
    rs.check_stream()
    ko, vo = oracle_sort(k, v)
    assert np.array_equal(to_host(kd), ko) and np.array_equal(to_host(vd), vo)
    return _ctrl(ws)


def _sort64(rs, k, key_type="u64"):
    import torch
    ws = _workspace(rs.workspace_bytes_kv(k.size, key_type, 32))
    v = np.arange(k.size, dtype=np.uint32)
    kd, vd = torch.from_numpy(k.view(np.int64)).cuda(), to_dev(v)
    rs.sort_kv_ex(kd, vd, key_type, ws)
    rs.check_stream()
    ko, vo = oracle.sort_kv(k, v, key_type)
    assert np.array_equal(kd.cpu().numpy().view(np.uint64), ko)
    assert np.array_equal(to_host(vd), vo)
    return _ctrl(ws)


@pytest.mark.parametrize("n", [1 << 25, 1 << 26])
@pytest.mark.parametrize("kind", ["distinct 5000", "distinct 16000", "distinct 40000",
                                  "distinct 1000000", "prefixes 3000", "prefixes 30000", "hot 4"])
def test_32_bit_keys_that_crowd_are_refused(rs, n, kind):
    assert _sort32(rs, _keys(kind, n, 32, n % 97 + len(kind)))[CHUNKS] == 0


@pytest.mark.parametrize("kind", ["distinct 12000000", "uniform"])
def test_32_bit_keys_that_spread_are_taken(rs, kind):
    assert _sort32(rs, _keys(kind, 1 << 25, 32, 3))[CHUNKS] > 0


@pytest.mark.parametrize("n,kind", [(1 << 22, "distinct 5000"), (1 << 24, "distinct 16000"),
                                    (1 << 24, "distinct 40000"), (1 << 24, "prefixes 1500"),
                                    (1 << 22, "hot 6")])
def test_64_bit_keys_that_crowd_are_refused(rs, n, kind):
    assert _sort64(rs, _keys(kind, n, 64, 11))[CHUNKS] == 0


@pytest.mark.parametrize("bits,n", [(64, 1 << 22), (64, 5_000_011), (32, 1 << 25)])
def test_keys_that_differ_in_few_bits(rs, bits, n):
    """The plan's table of sampled keys has to spread such keys too: 64-bit ones took
    linear probes of some hundred slots each, 0.4 ms of the plan's one CTA."""
    import torch
    k = _keys("and4", n, bits, 21)
    (_sort64 if bits == 64 else _sort32)(rs, k)
    ws = _workspace(rs.workspace_bytes_kv(n, "u%d" % bits, 32))
    src = torch.from_numpy(k.view(np.int64 if bits == 64 else np.int32)).cuda()
    kd, vd = src.clone(), torch.arange(n, dtype=torch.int32, device="cuda")
    rs.profile_enable(True)
    try:
        for _ in range(4):
            kd.copy_(src)
            rs.sort_kv_ex(kd, vd, "u%d" % bits, ws)
        torch.cuda.synchronize()
        launches, ms = rs.profile_read()["plan"]
    finally:
        rs.profile_enable(False)
    assert launches == 4 and ms / launches < 0.1


@pytest.mark.parametrize("n", [1 << 14, 100_003, (1 << 20) + 5, 4_500_003])
def test_orders_of_64_bit_keys(rs, n):
    c = _sort64(rs, _keys("uniform", n, 64, 5))
    assert c[CHUNKS] > 0 and c[STEP] == 0 and c[SRC] == 0     # two passes, by prefix
    k = np.random.default_rng(n).standard_normal(n).view(np.uint64)
    c = _sort64(rs, k, "f64")                                  # by position
    passes = int((c[1:9] > 0).sum())
    assert c[CHUNKS] > 0 and c[STEP] > 0 and c[SRC] == passes % 2 and 2 <= passes <= 4


@pytest.mark.parametrize("full", [True, False])
def test_orders_of_segments(rs, full):
    """Uniform segments take one pass and runs, one of equal digits the four passes; all do
    in a workspace without the parts for the former."""
    import torch
    sizes = np.array([20_000, 50_000, 300_000, 5000], dtype=np.uint64)
    off = inputs.offsets_from_sizes(sizes)
    n = int(off[-1])
    k = inputs.keys("uniform", n, 9)
    k[int(off[1]):int(off[2])] &= np.uint32(0xFFFF)  # digits 3 and 2 are the same
    v = inputs.index_values(n)
    nbytes = rs.workspace_bytes(n, True, sizes.size)
    if not full:  # the size before the parts of the routes: a geometry and a run list less
        tiles = -(-n // 4096) + min(sizes.size, n // 4097 + 1)
        runs = (n // 512 + 2 * min(sizes.size, n // 4097 + 1) + 2) * 8
        nbytes -= -(-tiles * 16 // 256) * 256 + -(-runs // 256) * 256
    ws = _workspace(nbytes)
    kd, vd = to_dev(k), to_dev(v)
    rs.sort_pairs_segmented_ex(kd, vd, to_dev(off), ws)
    rs.check_stream()
    ko, vo = oracle.sort_pairs_segmented(k, v, off)
    assert np.array_equal(to_host(kd), ko) and np.array_equal(to_host(vd), vo)
    c = _ctrl(ws)
    assert (c[MSD_TILES] > 0) == full and (c[LSD_TILES] > 0) == full
    torch.cuda.empty_cache()


@pytest.mark.parametrize("kind", ["distinct 256", "and4"])
@pytest.mark.parametrize("pairs", [True, False])
def test_orders_of_crowded_segments(rs, kind, pairs):
    """Pairs of segments whose middle digits crowd take the four passes; segments whose
    other digits are the same in all their keys are not crowded."""
    sizes = np.array([20_000, 4097, 60_000, 9000], dtype=np.uint64)
    off = inputs.offsets_from_sizes(sizes)
    n = int(off[-1])
    k = _keys(kind, n, 32, 3)
    if kind == "and4":  # but in the top digit, so that no bucket of it is too large
        k = (k & np.uint32(0x00FFFFFF)) | (_words(np.random.default_rng(4), n, 32)
                                           & np.uint32(0xFF000000))
    same = slice(int(off[0]), int(off[1]))
    k[same] = _keys("uniform", 20_000, 32, 6) & np.uint32(0xFF0000FF)
    v = inputs.index_values(n)
    ws = _workspace(rs.workspace_bytes(n, pairs, sizes.size))
    kd, vd = to_dev(k), to_dev(v)
    if pairs:
        rs.sort_pairs_segmented_ex(kd, vd, to_dev(off), ws)
    else:
        rs.sort_keys_segmented_ex(kd, to_dev(off), ws)
    rs.check_stream()
    ko, vo = oracle.sort_pairs_segmented(k, v, off)
    assert np.array_equal(to_host(kd), ko)
    if pairs:
        assert np.array_equal(to_host(vd), vo)
    c = _ctrl(ws)
    assert c[MSD_TILES] > 0 and (c[LSD_TILES] > 0) == pairs


@pytest.mark.parametrize("slope, taken", [(0.05, True), (0.35, False), (0.7, False)])
def test_density_of_32_bit_keys(rs, slope, taken):
    """2^25 keys whose chunks grow too long for a CTA where they are denser take the
    passes."""
    n = 1 << 25
    k = _keys("slope %g" % (100 * slope), n, 32, 12)
    ws = _workspace(rs.workspace_bytes(n, False))
    kd = to_dev(k)
    rs.sort_keys_ex(kd, ws)
    rs.check_stream()
    assert np.array_equal(to_host(kd), np.sort(k))
    assert (_ctrl(ws)[CHUNKS] > 0) == taken


@pytest.mark.parametrize("n, slope, by_prefix", [(1 << 18, 0.35, True), (1 << 22, 0.6, True),
                                                 ((1 << 23) + 5, 0.9, False)])
def test_density_of_64_bit_keys(rs, n, slope, by_prefix):
    """Where a CTA takes far more than an even chunk, denser chunks fit too; else the keys
    go by position."""
    c = _sort64(rs, _keys("slope %g" % (100 * slope), n, 64, 13))
    assert c[CHUNKS] > 0 and (c[STEP] == 0) == by_prefix
