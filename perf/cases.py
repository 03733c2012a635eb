"""Sorts that a program using this library makes, as it makes them.

Each case is one call of ``BucketSorter``: a keys-only sort, a key-value
sort, a batch of independent arrays, or a sort of host buffers.  The listed
cases take their sizes and key distributions from the benchmark's workloads
(one array of 2^20 and of 2^24 to 2^28 keys on several distributions, 2^27
pairs with heavily repeated keys, thousands of arrays of 2^7 to 2^20 keys in
one call, host buffers copied both ways) and add the small and the ragged
calls around them; ``draw`` spreads over the same ranges.  (The request loop
of ``SortServer`` sorts its jobs by the batch path, which the two batch cases
take at those jobs' sizes.)

A case's fields: ``kind`` (keys, pairs, batch, host), ``key`` (u32, f32, u64),
``val`` (value bytes of a pair, 0 without values), ``n`` (keys; arrays of a
batch), ``dist`` (the keys' distribution) and, for batches, the smallest and
largest array as powers of two and the seed of the array sizes.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1002_4464_gb300 import BucketSorter

KEY_BYTES = {"u32": 4, "f32": 4, "u64": 8}


def _case(name, kind, key, n, dist="uniform", val=0, lo=0, hi=0, sizes_seed=0):
    return {"name": name, "kind": kind, "key": key, "val": val, "n": n, "dist": dist,
            "lo": lo, "hi": hi, "sizes_seed": sizes_seed}


def listed():
    return [
        # the smallest call: a few thousand keys, one CTA, all latency
        _case("keys_u32_2k", "keys", "u32", 2000),
        # the paper's small single array: launches and latency of every step
        _case("keys_u32_1m", "keys", "u32", 1 << 20),
        # an ordinary array of measurements, ragged, bell-shaped float keys
        _case("keys_f32_16m_odd", "keys", "f32", (1 << 24) + 12345, "gaussian"),
        # identifiers drawn from a few popular values (repeated keys)
        _case("keys_u32_4m_zipf", "keys", "u32", (1 << 22) + 77, "zipf"),
        # partly ordered data: chunks of narrow ranges
        _case("keys_u32_64m_staggered", "keys", "u32", 1 << 26, "staggered"),
        # the headline workload
        _case("keys_u32_256m", "keys", "u32", 1 << 28),
        # hashes and timestamps: 64-bit keys
        _case("keys_u64_16m_odd", "keys", "u64", (1 << 24) + 3),
        # a stable sort of records by a popular attribute, value = row number
        _case("pairs_u32_128m_zipf", "pairs", "u32", 1 << 27, "zipf", val=4),
        # records with 64-bit keys and 64-bit payloads, ragged
        _case("pairs_u64_4m_odd", "pairs", "u64", (1 << 22) + 1001, val=8),
        # thousands of independent arrays of all sizes in one call
        _case("batch_u32_4000", "batch", "u32", 4000, lo=7, hi=20, sizes_seed=4),
        # the same with 64-bit keys
        _case("batch_u64_800", "batch", "u64", 800, lo=10, hi=20, sizes_seed=8),
        # keys that live in pinned host memory, sorted and copied back
        _case("host_u32_32m", "host", "u32", (1 << 25) + 5),
    ]


def draw(rng: random.Random):
    """One more case: any kind, key type and distribution, sizes spread over
    their logarithm."""
    def log_size(lo, hi):
        return int(2.0 ** rng.uniform(lo, hi))

    kind = rng.choice(["keys", "keys", "keys", "pairs", "pairs", "batch", "host"])
    if kind == "keys":
        key = rng.choice(["u32", "u32", "f32", "u64"])
        dist = rng.choice(["uniform", "uniform", "gaussian", "staggered", "sorted", "zipf"])
        c = _case(None, kind, key, log_size(10, 26 if key == "u64" else 28), dist)
    elif kind == "pairs":
        key = rng.choice(["u32", "u32", "f32", "u64"])
        dist = rng.choice(["uniform", "zipf", "few"])
        c = _case(None, kind, key, log_size(10, 24 if key == "u64" else 26.5), dist,
                  val=rng.choice([4, 8]))
    elif kind == "batch":
        key = rng.choice(["u32", "f32", "u64"])
        hi = rng.choice([14, 17, 20])
        most = 4000 if key != "u64" else 1200
        c = _case(None, kind, key, log_size(4, math.log2(most)),
                  rng.choice(["uniform", "uniform", "zipf"]), lo=7, hi=hi,
                  sizes_seed=rng.randrange(1 << 30))
    else:
        c = _case(None, kind, rng.choice(["u32", "f32", "u64"]), log_size(12, 25))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _offsets(case):
    """Host offsets of a batch's arrays: sizes log-uniform in [2^lo, 2^hi]."""
    rng = np.random.default_rng(case["sizes_seed"])
    sizes = np.floor(2.0 ** rng.uniform(case["lo"], case["hi"], case["n"])).astype(np.int64)
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)


def _total(case):
    return int(_offsets(case)[-1]) if case["kind"] == "batch" else case["n"]


def _bits32(n, dist, gen):
    """n 32-bit keys as bit patterns in int32, on the GPU."""
    dev = gen.device
    lo, hi = -(1 << 31), 1 << 31
    if dist in ("uniform", "sorted"):
        v = torch.randint(lo, hi, (n,), dtype=torch.int32, device=dev, generator=gen)
        if dist == "sorted":  # ascending as unsigned words
            v = torch.sort(v).values ^ (-(1 << 31))
        return v
    if dist == "gaussian":  # mean of four uniform draws
        acc = torch.zeros(n, dtype=torch.int64, device=dev)
        for _ in range(4):
            acc += torch.randint(0, 1 << 32, (n,), dtype=torch.int64, device=dev, generator=gen)
        acc >>= 2
        return (acc - (1 << 31)).to(torch.int32) ^ (-(1 << 31))
    if dist == "zipf":  # 1024 values, P(k) ~ k^-1.1
        cdf = torch.cumsum(torch.arange(1, 1025, dtype=torch.float64, device=dev) ** -1.1, 0)
        cdf /= cdf[-1].clone()
        values = torch.randint(lo, hi, (1024,), dtype=torch.int32, device=dev, generator=gen)
        x = torch.rand(n, dtype=torch.float64, device=dev, generator=gen)
        return values[torch.searchsorted(cdf, x).clamp_(max=1023)]
    if dist == "few":  # 16 values
        v = torch.randint(0, 16, (n,), dtype=torch.int32, device=dev, generator=gen)
        return v << 28
    if dist == "staggered":  # chunk c of 128 holds the range (2c + 1) mod 128
        c = torch.arange(n, dtype=torch.int64, device=dev)
        c.div_(max(1, n // 128), rounding_mode="floor").clamp_(max=127)
        v = torch.randint(0, 1 << 25, (n,), dtype=torch.int32, device=dev, generator=gen)
        return (((2 * c + 1) % 128) << 25).to(torch.int32) | v
    raise ValueError(dist)


def _keys(case, n, gen):
    dist, key = case["dist"], case["key"]
    if key == "u32":
        return _bits32(n, dist, gen)
    if key == "f32":  # the 32-bit draws mapped in order to [-1, 1)
        u = _bits32(n, dist, gen)
        return ((u ^ (-(1 << 31))) >> 8).to(torch.float32) * 2.0 ** -23
    hi = _bits32(n, dist, gen).to(torch.int64) << 32
    if dist in ("zipf", "few"):  # repeated keys repeat whole
        return hi | (~(hi >> 32) & 0xFFFFFFFF)
    return hi | torch.randint(0, 1 << 32, (n,), dtype=torch.int64, device=gen.device,
                              generator=gen)


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n = _total(case)
    keys = _keys(case, n, gen)
    vals = None
    if case["kind"] == "pairs":  # the row numbers
        vals = torch.arange(n, dtype=torch.int32 if case["val"] == 4 else torch.int64,
                            device="cuda")
    return keys, vals


def prepare(case, seed):
    """Buffers and the handle that a program keeps for its sorts."""
    keys, vals = _inputs(case, seed)
    state = {"case": case, "sorter": BucketSorter()}
    if case["kind"] == "host":
        state["keys"] = keys.cpu().pin_memory()
        state["out"] = torch.empty_like(state["keys"], pin_memory=True)
        return state
    state["keys"], state["out"] = keys, torch.empty_like(keys)
    if vals is not None:
        state["vals"], state["out_vals"] = vals, torch.empty_like(vals)
    if case["kind"] == "batch":
        state["offsets"] = _offsets(case)
    return state


def run(state):
    """One sort through the public wrapper; the result is in the caller's
    output buffers once the stream's work is done."""
    case, sorter = state["case"], state["sorter"]
    kind, key = case["kind"], case["key"]
    if kind == "keys":
        return sorter.sort_keys(state["keys"], state["out"], key)
    if kind == "pairs":
        return sorter.sort_pairs(state["keys"], state["vals"], state["out"], state["out_vals"],
                                 key)
    if kind == "batch":
        return sorter.sort_batch(state["keys"], state["offsets"], state["out"], key)
    return sorter.sort_keys_host(state["keys"], state["out"], key)


def work(case):
    """Every key (and value) read once and written once; a sort has no
    floating-point work (its comparisons and digit steps are not counted)."""
    return {"bytes": 2 * _total(case) * (KEY_BYTES[case["key"]] + case["val"]), "flops": 0}


# ------------------------------------------------------------------ results

def _order_code(keys, key):
    """int64 codes whose signed order is the library's key order."""
    if key == "u32":
        return keys.to(torch.int64) & 0xFFFFFFFF
    if key == "f32":  # negative: all bits inverted, else the sign bit set
        b = keys.view(torch.int32).to(torch.int64) & 0xFFFFFFFF
        return torch.where(b >= 1 << 31, 0xFFFFFFFF - b, b + (1 << 31))
    return keys ^ (-(1 << 63))


def exact(case, seed):
    """The same sorts by torch, on 64-bit codes of the keys."""
    keys, vals = _inputs(case, seed)
    key = case["key"]
    if case["kind"] == "batch":
        off = [int(x) for x in _offsets(case)]
        out = torch.empty_like(keys)
        for a, b in zip(off, off[1:]):
            part = keys[a:b]
            out[a:b] = part[torch.sort(_order_code(part, key)).indices]
        return out
    code = _order_code(keys, key)
    order = torch.sort(code, stable=case["kind"] == "pairs").indices
    del code
    out = keys[order]
    if case["kind"] == "pairs":
        return out, vals[order]
    return out.cpu() if case["kind"] == "host" else out
