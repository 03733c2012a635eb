"""GPU parity of the CTAs that sort by bins (one counting pass over linear
bins of the unit's key range, then neighbour exchanges), against the oracle's
textbook sort, bit for bit: fills at the warp and unit edges, and the key
distributions that take each route through the sort: even keys, repeated
keys (bins that hold one value, and bins that mix a repeated value with
another), keys that crowd into few bins, ranges below the bin count, and
float keys with infinities, NaNs and subnormals."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, run on the GPU machine
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1002_4464_gb300 as pkg  # noqa: E402


def _keys(kind, n, bits, seed):
    """n unsigned keys of 32 or 64 bits."""
    u = synth.draws64(seed, n)
    if bits == 32:
        u = u >> np.uint64(32)
    top = np.uint64((1 << bits) - 1)
    if kind == "even":
        k = u
    elif kind == "narrow":  # 5000 consecutive values
        k = top - np.uint64(7000) + u % np.uint64(5000)
    elif kind == "few":
        k = u & np.uint64(0xF << (bits - 4))
    elif kind == "zipf":  # 1024 values, P(k) ~ k^-1.1
        rank = synth.keys_zipf(n, seed)
        vals = synth.draws64(seed + 1, 1024) >> np.uint64(64 - bits)
        _, inv = np.unique(rank, return_inverse=True)
        k = vals[inv]
    elif kind == "pairs":  # popular values one apart: every popular bin is mixed
        k = (u % np.uint64(8) << np.uint64(bits - 3)) + (u >> np.uint64(9)) % np.uint64(2)
    elif kind == "outlier":  # all keys in the first bin but one
        k = u % np.uint64(100000)
        k[n // 2] = top
    elif kind == "log":  # crowded towards zero
        x = (u >> np.uint64(bits - 24)).astype(np.float64) / 2.0 ** 24
        k = np.floor(2.0 ** (x * (bits - 1))).astype(np.uint64)
    elif kind == "clusters":  # even, with a cluster of a few hundred keys
        k = u.copy()
        k[: n // 50] = np.uint64(1 << (bits - 2)) + u[: n // 50] % np.uint64(50000)
    elif kind == "sorted":
        k = np.sort(u)
    else:
        raise ValueError(kind)
    return k.astype(np.uint32 if bits == 32 else np.uint64)


KINDS = ["even", "narrow", "few", "zipf", "pairs", "outlier", "log", "clusters", "sorted"]


def _check(keys, key_type, **kw):
    sorter = pkg.BucketSorter(**kw)
    d = torch.from_numpy(keys.view(np.int32 if keys.itemsize == 4 else np.int64)).cuda()
    if key_type == "f32":
        d = d.view(torch.float32)
    out = sorter.sort_keys(d, key_type=key_type)
    sorter.sync()
    got = out.cpu().numpy().view(np.uint32 if keys.itemsize == 4 else np.uint64)
    want = oracle.textbook_sort(keys.view(np.float32) if key_type == "f32" else keys, key_type)
    assert np.array_equal(got, want.view(got.dtype))
    sorter.close()


@pytest.mark.parametrize("n", [33, 511, 2048, 2049, 4096, 8191, 8192, 16383, 16384, 16385, 30719,
                               30721, 32767, 32768, 65536, 150001])
@pytest.mark.parametrize("kind", KINDS)
def test_units_u32(kind, n):
    _check(_keys(kind, n, 32, synth.seed_for(7, 1, n)), "u32")


@pytest.mark.parametrize("n", [300007, 1 << 20])
@pytest.mark.parametrize("kind", KINDS)
def test_sampled_u32(kind, n):
    _check(_keys(kind, n, 32, synth.seed_for(7, 2, n)), "u32")


@pytest.mark.parametrize("n", [2000, 5000, 16384, 32768, 70001, 400003])
@pytest.mark.parametrize("kind", ["even", "special", "wide", "zipf", "bits"])
def test_units_f32(kind, n):
    """Codes of floats: values in [-1, 1), with infinities and NaNs, over the
    whole exponent range, repeated, and arbitrary bit patterns."""
    u = synth.keys_u32("uniform", n, synth.seed_for(7, 3, n))
    if kind == "bits":
        f = u.view(np.float32).copy()
    elif kind == "zipf":
        f = synth.u32_to_f32(synth.keys_zipf(n, synth.seed_for(7, 4, n)))
    else:
        f = synth.u32_to_f32(u).copy()
    if kind == "wide":
        f = np.ldexp(f, (u >> np.uint32(8)).astype(np.int64) % 250 - 125).astype(np.float32)
    if kind == "special":
        f[::97] = np.float32(np.inf)
        f[1::89] = np.float32(-np.inf)
        f[2::83] = np.float32(np.nan)
        f[3::79] = np.float32(-0.0)
        f[4::73] = np.float32(1e-45)
    _check(f.view(np.uint32), "f32")


@pytest.mark.parametrize("n", [33, 2048, 2049, 8191, 8192, 16383, 16384, 16385, 40001, 300007])
@pytest.mark.parametrize("kind", KINDS)
def test_units_u64(kind, n):
    _check(_keys(kind, n, 64, synth.seed_for(7, 5, n)), "u64")


@pytest.mark.parametrize("n", [33, 2047, 2048, 4097, 8192, 16383, 16384, 40001, 300007])
@pytest.mark.parametrize("kind", KINDS + ["equal"])
def test_units_pairs(kind, n):
    """Key-value pairs, value = input index: equal keys keep their order."""
    keys = (np.full(n, 0xFFFFFFFF, np.uint32) if kind == "equal"
            else _keys(kind, n, 32, synth.seed_for(7, 6, n)))
    sorter = pkg.BucketSorter()
    d_k = torch.from_numpy(keys.view(np.int32)).cuda()
    d_v = torch.arange(n, dtype=torch.int32, device="cuda")
    ok, ov = sorter.sort_pairs(d_k, d_v)
    sorter.sync()
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(ok.cpu().numpy().view(np.uint32), keys[order])
    assert np.array_equal(ov.cpu().numpy(), order.astype(np.int32))
    sorter.close()


@pytest.mark.parametrize("key_type", ["u32", "u64"])
@pytest.mark.parametrize("kind", KINDS)
def test_batch_units(kind, key_type):
    """Batch segments of every unit shape (sizes at the shapes' edges)."""
    bits = 32 if key_type == "u32" else 64
    sizes = [2, 33, 2047, 2048, 2049, 4096, 8192, 8193, 16384, 16385, 32767, 32768, 50000, 140001]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    keys = _keys(kind, int(off[-1]), bits, synth.seed_for(7, 7))
    sorter = pkg.BucketSorter()
    d = torch.from_numpy(keys.view(np.int32 if bits == 32 else np.int64)).cuda()
    out = sorter.sort_batch(d, off, key_type=key_type)
    sorter.sync()
    got = out.cpu().numpy().view(keys.dtype)
    for a, b in zip(off[:-1].astype(int), off[1:].astype(int)):
        assert np.array_equal(got[a:b], np.sort(keys[a:b]))
    sorter.close()


@pytest.mark.parametrize("kind", ["even", "zipf", "sorted"])
def test_batch_joined_segments(kind):
    """Segments above the sampled size: up to 2^21 keys in one sequence of
    launches, or one plain sort each in a workspace that only holds those."""
    sizes = [524288, 524289, 3, 1 << 20, (1 << 20) + 1, 900001, 1 << 21, (1 << 21) + 1, 40000]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    keys = _keys(kind, int(off[-1]), 32, synth.seed_for(7, 8))
    d = torch.from_numpy(keys.view(np.int32)).cuda()
    want = np.concatenate([np.sort(keys[a:b]) for a, b in
                           zip(off[:-1].astype(int), off[1:].astype(int))])
    free = pkg.BucketSorter()
    need = free.plan_batch(off).workspace_bytes
    small = 48 << 20
    assert small < need
    tight = pkg.BucketSorter(workspace_bytes=small)
    assert tight.plan_batch(off).workspace_bytes <= small
    for sorter in (free, tight):
        info = sorter.plan_batch(off)
        assert (info.sampled_segs, info.large_segs) == (1, 6)
        out = sorter.sort_batch(d, off)
        sorter.sync()
        assert np.array_equal(out.cpu().numpy().view(np.uint32), want)
        sorter.close()


@pytest.mark.parametrize("kind", ["even", "zipf", "few"])
def test_batch_joined_direct_segments(kind):
    """Enough 64-bit segments above one CTA's unit take the sampled route (two
    to eight sublists each); with the limit given they stay with clusters."""
    unit, most = 16384, 131072
    sizes = [unit, 5]
    k = 0
    while sum(sizes) < (1 << 22) + 2 * unit:
        sizes.append(unit + 1 + (k * 7919) % (most - unit))
        k += 1
    sizes += [unit + 1, 2 * unit, most]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    keys = _keys(kind, int(off[-1]), 64, synth.seed_for(7, 9))
    d = torch.from_numpy(keys.view(np.int64)).cuda()
    outs = []
    for limit in (0, most):
        sorter = pkg.BucketSorter(batch_direct_max=limit)
        assert sorter.plan_batch(off, "u64").direct_segs == len(sizes)
        out = sorter.sort_batch(d, off, key_type="u64")
        sorter.sync()
        outs.append(out.cpu().numpy().view(keys.dtype))
        sorter.close()
    for a, b in zip(off[:-1].astype(int), off[1:].astype(int)):
        assert np.array_equal(outs[0][a:b], np.sort(keys[a:b]))
    assert np.array_equal(outs[0], outs[1])
