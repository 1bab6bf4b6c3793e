"""The measured work: sorts as programs call them through ``paper_1008_2849_gb300.rs``
and ``serve``.

The sorts work in place, so a program that keeps its input sorts a copy: every
pass copies the input into the working buffers and sorts those, with a
workspace (or a captured graph) kept from call to call.

A case is one of three kinds:

* ``whole``      one array: ``n`` items, ``key`` type, ``value_bits``, ``dist``;
* ``segmented``  many arrays of one buffer sorted in one call: ``segments``
  arrays with sizes floor(2^U), U uniform on [``lo``, ``hi``], rescaled to about
  ``total`` items in all when that is not 0; ``graph`` replays a captured call;
* ``serve``      a request stream through the serving loop: ``requests``
  requests of 10^3 to 10^``hi10`` items, sizes drawn from ``stream``.

Keys are drawn from ``dist``: uniform words, the AND of 2 to 4 words (low
entropy), 256 distinct words, one word, sorted, reverse, words below 2^16
(32-bit) or 2^40 (64-bit), and for floating-point keys standard normal
variates.  Values are the item's index in its array, as for an argsort.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1008_2849_gb300 import rs, serve

KEY_BYTES = {"u32": 4, "i32": 4, "f32": 4, "u64": 8, "i64": 8, "f64": 8}
MAX_BYTES = 2 * 8 * (1 << 28)  # the largest listed case's


def _whole(name, n, key="u32", value_bits=32, dist="uniform"):
    return {"name": name, "kind": "whole", "n": n, "key": key, "value_bits": value_bits,
            "dist": dist}


def _segmented(name, segments, lo, hi, total=0, key="u32", value_bits=32, graph=False):
    return {"name": name, "kind": "segmented", "segments": segments, "lo": lo, "hi": hi,
            "total": total, "key": key, "value_bits": value_bits, "dist": "uniform",
            "graph": graph}


def listed():
    return [
        # The smallest serving request: one launch, pure latency.
        _whole("keys 1000", 1000, value_bits=0),
        # A table column of an odd size, carried with row numbers.
        _whole("pairs 50021", 50021),
        # The latency benchmark: 2^20 uniform keys.
        _whole("keys 2^20", 1 << 20, value_bits=0),
        # A large serving request: low-entropy keys, a size that is no power of two.
        _whole("keys and2 10M", 10_000_019, value_bits=0, dist="and2"),
        # The throughput benchmark: 2^28 pairs.
        _whole("pairs 2^28", 1 << 28),
        # The distribution sweep's low-entropy keys at its size.
        _whole("pairs and3 2^27", 1 << 27, dist="and3"),
        # Argsort of measured values: normal floats.
        _whole("f32 argsort 16M", 16_777_259, key="f32", dist="normal"),
        # Hash or composite keys with row numbers (a join or a group-by).
        _whole("u64 pairs 2^26", 1 << 26, key="u64"),
        # Argsort of doubles with 64-bit row numbers.
        _whole("f64 v64 3M", 3_000_001, key="f64", value_bits=64, dist="normal"),
        # 4096 uneven arrays in one captured call, 2^28 pairs in all.
        _segmented("batch 4096 arrays", 4096, 8.0, 22.0, total=1 << 28, graph=True),
        # Many short arrays (neighbour lists, rows of a sparse matrix).
        _segmented("short arrays 2^15", 1 << 15, 1.0, 12.0),
        # The serving loop: 40 requests of 10^3 to 10^7 items, all waiting.
        {"name": "serve 40 requests", "kind": "serve", "requests": 40, "hi10": 7.0, "stream": 11},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | rng.randint(0, 1)

    kind = rng.choices(("whole", "segmented", "serve"), (12, 4, 1))[0]
    if kind == "serve":
        return {"kind": "serve", "requests": rng.randint(8, 40), "hi10": rng.uniform(5.0, 7.0),
                "stream": rng.randint(1, 1 << 20)}
    key = rng.choices(("u32", "i32", "f32", "u64", "i64", "f64"), (10, 1, 3, 3, 1, 2))[0]
    value_bits = rng.choice((0, 32, 32)) if key == "u32" else rng.choice((0, 32, 64))
    item = KEY_BYTES[key] + value_bits // 8
    if kind == "whole":
        n = log_int(1000, MAX_BYTES // 4 // item)
        if key in ("f32", "f64"):
            dist = rng.choice(("normal", "normal", "uniform"))
        elif KEY_BYTES[key] == 8:
            dist = rng.choice(("uniform", "uniform", "and2", "low40"))
        else:
            dist = rng.choice(("uniform", "uniform", "uniform", "uniform", "and2", "and2", "and3",
                               "and4", "distinct256", "equal", "sorted", "reverse", "low16"))
        return {"kind": kind, "n": n, "key": key, "value_bits": value_bits, "dist": dist}
    lo = rng.uniform(1.0, 10.0)
    hi = rng.uniform(lo + 1.0, 22.0)
    total = log_int(1 << 18, MAX_BYTES // 4 // item)
    mean = (2.0 ** hi - 2.0 ** lo) / ((hi - lo) * math.log(2.0))
    segments = max(2, min(1 << 16, int(total / mean)))
    return {"kind": kind, "segments": segments, "lo": lo, "hi": hi, "total": total, "key": key,
            "value_bits": value_bits, "dist": "uniform",
            "graph": key == "u32" and value_bits < 64 and rng.random() < 0.5}


def _words(n, bits, gen):
    if bits == 64:
        return torch.randint(-(1 << 63), (1 << 63) - 1, (n,), dtype=torch.int64, device="cuda",
                             generator=gen)
    return torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int32, device="cuda",
                         generator=gen)


def _keys(case, n, gen):
    """n keys' bit patterns (int32 or int64) of the case's distribution."""
    bits = 8 * KEY_BYTES[case["key"]]
    dist = case["dist"]
    word = torch.int64 if bits == 64 else torch.int32
    if dist == "normal":
        return torch.randn(n, dtype=torch.float64 if bits == 64 else torch.float32, device="cuda",
                           generator=gen).view(word)
    if dist == "equal":
        return _words(1, bits, gen).repeat(n)
    if dist == "distinct256":
        pick = torch.randint(0, 256, (n,), device="cuda", generator=gen)
        return _words(256, bits, gen)[pick]
    k = _words(n, bits, gen)
    if dist in ("and2", "and3", "and4"):
        for _ in range(int(dist[3]) - 1):
            k &= _words(n, bits, gen)
    elif dist in ("sorted", "reverse"):
        k = _unsigned_order(k).sort(descending=dist == "reverse").values.to(word)
        k ^= -(1 << (bits - 1))
    elif dist == "low16":
        k &= 0xFFFF
    elif dist == "low40":
        k &= (1 << 40) - 1
    return k


def _segment_sizes(case, seed):
    """The same sizes for every seed (drawn once), in an order of the seed's own."""
    u = np.random.default_rng(10).random(case["segments"])
    sizes = np.floor(np.exp2(case["lo"] + (case["hi"] - case["lo"]) * u))
    if case["total"]:
        sizes = np.maximum(np.floor(sizes * (case["total"] / sizes.sum())), 1)
    return np.random.default_rng(seed).permutation(sizes.astype(np.int64))


def _inputs(case, seed):
    """(keys, values or None, segment offsets or None) on the device."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    off = None
    if case["kind"] == "segmented":
        sizes = torch.from_numpy(_segment_sizes(case, seed)).cuda()
        off = torch.zeros(sizes.numel() + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(sizes, 0, out=off[1:])
        n = int(off[-1])
    else:
        n = case["n"]
    keys = _keys(case, n, gen)
    vals = None
    if case["value_bits"]:
        vals = torch.arange(n, dtype=torch.int64 if case["value_bits"] == 64 else torch.int32,
                            device="cuda")
        if off is not None:
            vals -= torch.repeat_interleave(off[:-1], sizes).to(vals.dtype)
    return keys, vals, None if off is None else off.to(torch.int32)


def _requests(case, seed):
    reqs = serve.make_requests(case["requests"], case["stream"], 3.0, case["hi10"])
    for r in reqs:
        r.key_seed = seed * 1000003 + r.id
    return reqs


def prepare(case, seed):
    if case["kind"] == "serve":
        return {"case": case, "executor": serve.GpuExecutor(pool_n=1 << 24),
                "requests": _requests(case, seed)}
    src_k, src_v, off = _inputs(case, seed)
    key, n = case["key"], src_k.numel()
    state = {"case": case, "src_k": src_k, "src_v": src_v, "off": off,
             "keys": torch.empty_like(src_k),
             "vals": None if src_v is None else torch.empty_like(src_v)}
    narrow = KEY_BYTES[key] == 4 and case["value_bits"] <= 32
    segments = 0 if off is None else case["segments"]
    if case.get("graph"):
        state["graph"] = rs.Graph(state["keys"], state["vals"], off)
    elif narrow:
        state["ws"] = rs.alloc_workspace(n, src_v is not None, segments)
    else:
        nbytes = (rs.workspace_bytes_kv_segmented(n, key, case["value_bits"], segments)
                  if segments else rs.workspace_bytes_kv(n, key, case["value_bits"]))
        raw = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
        pad = -raw.data_ptr() % 256
        state["ws"] = raw[pad:pad + nbytes]
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        server = serve.SortServer(state["executor"], keep_results=True)
        done = server.run(state["requests"], realtime=False)["done"]
        return [(d.keys, d.vals) for d in done]
    keys, vals, off = state["keys"], state["vals"], state["off"]
    keys.copy_(state["src_k"])
    if vals is not None:
        vals.copy_(state["src_v"])
    key = case["key"]
    if "graph" in state:
        state["graph"].launch()
    elif off is not None:
        if key == "u32" and case["value_bits"] == 32:
            rs.sort_pairs_segmented_ex(keys, vals, off, state["ws"])
        elif key == "u32" and vals is None:
            rs.sort_keys_segmented_ex(keys, off, state["ws"])
        else:
            rs.sort_kv_segmented_ex(keys, vals, off, key, state["ws"])
    elif key == "u32" and case["value_bits"] == 32:
        rs.sort_pairs_ex(keys, vals, state["ws"])
    elif key == "u32" and vals is None:
        rs.sort_keys_ex(keys, state["ws"])
    elif KEY_BYTES[key] == 4 and case["value_bits"] <= 32:
        rs.sort_typed_ex(keys, vals, key, state["ws"])
    else:
        rs.sort_kv_ex(keys, vals, key, state["ws"])
    return [keys] if vals is None else [keys, vals]


def work(case):
    """Every item read once and written once; a sort of integers has no
    floating-point work."""
    if case["kind"] == "serve":
        return {"bytes": sum(2 * r.n * (8 if r.with_values else 4) for r in _requests(case, 0)),
                "flops": 0}
    n = case["n"] if case["kind"] == "whole" else int(_segment_sizes(case, 0).sum())
    return {"bytes": 2 * n * (KEY_BYTES[case["key"]] + case["value_bits"] // 8), "flops": 0}


def _unsigned_order(k):
    """The words' unsigned order as a signed order."""
    return k ^ -(1 << (8 * k.element_size() - 1))


def exact(case, seed):
    """The stable sort by torch: keys mapped onto integers of the same order
    (unsigned order, two's complement, or IEEE totalOrder)."""
    if case["kind"] == "serve":
        return None
    keys, vals, off = _inputs(case, seed)
    if case["key"][0] == "u":
        order = _unsigned_order(keys)
    elif case["key"][0] == "i":
        order = keys
    else:  # a negative float's larger magnitude comes first
        order = torch.where(keys < 0, keys ^ ((1 << (8 * keys.element_size() - 1)) - 1), keys)
    place = torch.sort(order, stable=True).indices
    del order
    if off is not None:
        seg = torch.repeat_interleave(torch.arange(case["segments"], dtype=torch.int32,
                                                   device="cuda"), off[1:] - off[:-1])
        place = place[torch.sort(seg[place], stable=True).indices]
    return [keys[place]] if vals is None else [keys[place], vals[place]]
