"""Which segments of a batch join the sampled ones, and the workspace that
this takes: host plans only, no GPU."""
import numpy as np
import pytest

import paper_1002_4464_gb300 as pkg

U32, U64 = pkg.BSORT_U32, pkg.BSORT_U64
JOIN_LIMIT = 4 << 30  # joined segments' tiles and relocated keys


def _plan(sizes, kt=U32, **cfg):
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    h = pkg.bsort_create(pkg.bsort_config(device=0, **cfg))
    try:
        return pkg.bsort_plan_batch(h, kt, off)
    finally:
        pkg.bsort_destroy(h)


def _plain(n, kt=U32, **cfg):
    h = pkg.bsort_create(pkg.bsort_config(device=0, **cfg))
    try:
        return pkg.bsort_plan(h, kt, 0, n)
    finally:
        pkg.bsort_destroy(h)


@pytest.mark.parametrize("sizes,kt", [([(1 << 20) - 8] * 4000, U32), ([1 << 17] * 16000, U64),
                                      ([1500000] * 2000, U32)])
def test_joined_workspace_is_bounded(sizes, kt):
    """Batches of 12 to 17 GB whose joined segments would take twice that at
    once: they are sorted in parts of at most 4 GiB (records, runs and
    descriptors come to less than an eighth of that)."""
    p = _plan(sizes, kt)
    assert p.workspace_bytes <= JOIN_LIMIT * 9 // 8
    assert p.num_segs == len(sizes) and p.n == sum(sizes)
    per_part = JOIN_LIMIT // (2 * sizes[0] * (8 if kt == U64 else 4))
    assert 7 * (len(sizes) // per_part) <= p.num_kernels <= 7 * (len(sizes) // per_part + 3)


def test_parts_count_every_segment_once():
    sizes = ([2000000] * 200 + [7, 0, 1, 5000, 300000]) * 3 + [1 << 22]
    p, small = _plan(sizes), _plan([5000, 300000] * 3 + [7] * 3)
    assert (p.direct_segs, p.sampled_segs) == (small.direct_segs, small.sampled_segs)
    assert p.large_segs == 601 and p.n == sum(sizes)
    assert (p.sublists, p.buckets) == (small.sublists, small.buckets)


@pytest.mark.parametrize("n", [524289, 900001, 1 << 20, 1 << 21])
def test_low_memory_and_lone_segments_are_plain_sorts(n):
    low = dict(flags=pkg.BSORT_FLAG_LOW_MEMORY)
    assert _plan([n], **low).workspace_bytes == _plain(n, **low).workspace_bytes
    assert _plan([n] * 20, **low).workspace_bytes == _plain(n, **low).workspace_bytes
    one = _plan([n])  # (another's sequence of launches costs more than it saves)
    assert one.num_kernels == _plain(n).num_kernels and one.large_segs == 1
    assert _plan([n, n]).num_kernels == 7
    assert _plan([n, 300000]).num_kernels == 7
    assert _plan([n, 5000]).num_kernels == one.num_kernels + 1


def test_low_memory_u64_stays_with_clusters():
    sizes = [100000] * 200
    assert _plan(sizes, U64).num_kernels == 7
    assert _plan(sizes, U64, flags=pkg.BSORT_FLAG_LOW_MEMORY).num_kernels == 1


@pytest.mark.parametrize("n,joins", [(16385, False), (32768, False), (65536, False),
                                     (65537, True), (131072, True)])
def test_u64_direct_segments_that_join(n, joins):
    """2^24 keys in all: clusters of 2 and 4 CTAs are faster by themselves."""
    p = _plan([n] * ((1 << 24) // n + 1), U64)
    assert p.num_kernels == (7 if joins else 1)
    few = _plan([n] * ((1 << 21) // n), U64)
    assert few.num_kernels == 1
    beside = _plan([n] * ((1 << 24) // n + 1) + [500000], U64)  # a sampled segment
    assert beside.num_kernels == (7 if n > 32768 else 8)
