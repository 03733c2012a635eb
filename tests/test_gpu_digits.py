"""The digit sort of crowded 32768-key units, against the oracle's textbook
sort: units whose keys fill two narrow groups at the ends of a span (half of
the unit in one bin each, eight values or more to a group, so that neither
the bins, nor a cut of them, nor those of the logarithm part them), with the
span on both sides of the pass boundaries of 6-bit digits, at the ends and in
the middle of the key space; floats by their codes."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, run on the GPU machine
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1002_4464_gb300 as pkg  # noqa: E402

SPANS = [(1 << 18) - 1, 1 << 18, (1 << 18) + 1, (1 << 20) + 7, (1 << 24) - 1, 1 << 24,
         (1 << 24) + 1, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, 0xFFFFFFFF]


def _two_groups(n, lo, span, seed):
    """n keys of [lo, lo + span], both ends present, half in its lowest and
    half in its highest 1/40000."""
    u = synth.draws64(synth.seed_for(13, seed), n)
    width = np.uint64(max(6, span // 40000))
    near = (u >> np.uint64(8)) % width
    k = np.where(u & np.uint64(1) == 0, near, np.uint64(span) - near)
    k[n // 3], k[(2 * n) // 3] = 0, span
    return (k + np.uint64(lo)).astype(np.uint32)


def _sort(keys, key_type):
    d = torch.from_numpy(keys.view(np.int32)).cuda()
    if key_type == "f32":
        d = d.view(torch.float32)
    sorter = pkg.BucketSorter()
    out = sorter.sort_keys(d, key_type=key_type)
    sorter.sync()
    sorter.close()
    return out.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("n", [16385, 20000, 32767, 32768])
@pytest.mark.parametrize("span", SPANS)
def test_two_groups_u32(n, span):
    for lo in {0, 0xFFFFFFFF - span, 0x12345678 % (0xFFFFFFFF - span + 1)}:
        keys = _two_groups(n, lo, span, span % 991 + n)
        assert np.array_equal(_sort(keys, "u32"), oracle.textbook_sort(keys, "u32"))


@pytest.mark.parametrize("n", [16385, 32767, 32768])
@pytest.mark.parametrize("span", [1 << 18, 1 << 24, (1 << 30) + 1, 0xFFFFFFFF])
def test_two_groups_f32(n, span):
    """Codes of the two groups: around zero, and to both infinities and NaN."""
    for lo in {0, 0xFFFFFFFF - span, (0x80000000 - span // 2) % (0xFFFFFFFF - span + 1)}:
        code = _two_groups(n, lo, span, span % 983 + n)
        bits = np.where(code & np.uint32(0x80000000), code ^ np.uint32(0x80000000), ~code)
        f = bits.astype(np.uint32).view(np.float32)
        want = oracle.textbook_sort(f, "f32").view(np.uint32)
        assert np.array_equal(_sort(bits.astype(np.uint32), "f32"), want)


@pytest.mark.parametrize("span", [1 << 18, (1 << 24) + 1, 0xFFFFFFFF])
def test_two_groups_in_a_batch(span):
    sizes = [32768, 16385, 30000, 32767, 9000]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    keys = np.concatenate([_two_groups(n, 0xFFFFFFFF - span, span, n) for n in sizes])
    sorter = pkg.BucketSorter()
    out = sorter.sort_batch(torch.from_numpy(keys.view(np.int32)).cuda(), off)
    sorter.sync()
    sorter.close()
    got = out.cpu().numpy().view(np.uint32)
    for a, b in zip(off[:-1].astype(int), off[1:].astype(int)):
        assert np.array_equal(got[a:b], np.sort(keys[a:b]))
