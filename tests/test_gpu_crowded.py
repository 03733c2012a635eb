"""Units whose keys do not spread over their key range: the sorts by bins must
not lose to the sorts that they replaced on them, and must stay exact.

The times are compared inside one process, as ratios between sorts of the same
size on different keys, with room for noise: each limit lies well above what
the sound code measures and well below what the fault measured."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, run on the GPU machine
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1002_4464_gb300 as pkg  # noqa: E402


def _time(fn, reps=25):
    """Lower-quartile time of one call in us (device events)."""
    for _ in range(5):
        fn()
    torch.cuda.synchronize()
    ts = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        ts.append(1000.0 * a.elapsed_time(b))
    return sorted(ts)[reps // 4]


def _draws(n, seed):
    return synth.draws64(synth.seed_for(9, seed), n)


# ------------------------------------------------ padding of the last unit
def test_padding_does_not_crowd_the_last_unit():
    """A ragged sort of small keys (below 10^6): the padding codes are far
    above every key; taken for keys they crowd the last unit's real ones into
    a few bins, and their samples in Step 4 the others (1.48 times the time of
    keys over the whole range; 1.00 with the padding left out)."""
    n = 400001
    u = _draws(n, 1)
    wide = torch.from_numpy((u >> np.uint64(32)).astype(np.uint32).view(np.int32)).cuda()
    small = torch.from_numpy((u % np.uint64(1000000)).astype(np.uint32).view(np.int32)).cuda()
    out = torch.empty_like(wide)
    sorter = pkg.BucketSorter()
    t_wide = min(_time(lambda: sorter.sort_keys(wide, out)) for _ in range(2))
    t_small = min(_time(lambda: sorter.sort_keys(small, out)) for _ in range(2))
    sorter.close()
    assert t_small < 1.25 * t_wide, (t_small, t_wide)


@pytest.mark.parametrize("n", [300007, 400001, (1 << 20) + 3])
@pytest.mark.parametrize("key_type", ["u32", "f32", "u64"])
def test_real_keys_equal_to_the_padding(n, key_type):
    """Real keys with the padding's code, and few keys besides: the last units
    hold real maxima, padding, or padding alone."""
    u = _draws(n, 2)
    if key_type == "u64":
        k = np.where(u % np.uint64(3) == 0, u, np.uint64(0xFFFFFFFFFFFFFFFF))
        d = torch.from_numpy(k.view(np.int64)).cuda()
    else:
        top = np.uint32(0xFFFFFFFF if key_type == "u32" else 0x7FFFFFFF)
        k = np.where(u % np.uint64(3) == 0, (u >> np.uint64(32)).astype(np.uint32), top)
        d = torch.from_numpy(k.view(np.int32)).cuda()
        if key_type == "f32":
            d, k = d.view(torch.float32), k.view(np.float32)
    sorter = pkg.BucketSorter()
    got = sorter.sort_keys(d, key_type=key_type)
    sorter.sync()
    sorter.close()
    want = oracle.textbook_sort(k, key_type)
    word = np.uint64 if key_type == "u64" else np.uint32
    assert np.array_equal(got.cpu().numpy().view(word), want.view(word))


@pytest.mark.parametrize("low_memory", [False, True])
def test_pairs_equal_to_the_padding(low_memory):
    n = 300007
    k = np.where(_draws(n, 3) % np.uint64(3) == 0, np.uint32(5), np.uint32(0xFFFFFFFF))
    sorter = pkg.BucketSorter(low_memory=low_memory)
    ok, ov = sorter.sort_pairs(torch.from_numpy(k.view(np.int32)).cuda(),
                               torch.arange(n, dtype=torch.int32, device="cuda"))
    sorter.sync()
    sorter.close()
    order = np.argsort(k, kind="stable")
    assert np.array_equal(ok.cpu().numpy().view(np.uint32), k[order])
    assert np.array_equal(ov.cpu().numpy(), order.astype(np.int32))
