"""Batches whose joined segments' workspace cannot be had, or comes in parts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, run on the GPU machine
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1002_4464_gb300 as pkg  # noqa: E402
import synth  # noqa: E402

SIZES = [600001, 1 << 20, 300000, 5000, 1500001, 1, 700000] * 4


def _batch(seed, bits=32, sizes=SIZES):
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.uint64)
    k = synth.draws64(synth.seed_for(10, seed), int(off[-1]))
    if bits == 32:
        k = (k >> np.uint64(32)).astype(np.uint32)
    want = np.concatenate([np.sort(k[a:b]) for a, b in
                           zip(off[:-1].astype(int), off[1:].astype(int))])
    return off, torch.from_numpy(k.view(np.int32 if bits == 32 else np.int64)).cuda(), want


def _same(out, want):
    torch.cuda.synchronize()
    return np.array_equal(out.cpu().numpy().view(want.dtype), want)


@pytest.mark.parametrize("bits,sizes", [(32, SIZES), (64, [100000] * 60 + [20000, 3])])
def test_out_of_memory_sorts_without_joining(bits, sizes):
    """A handle that grows its workspace, on a device whose free memory holds
    the plan without joined segments only."""
    key_type = "u32" if bits == 32 else "u64"
    kt = pkg.BSORT_U32 if bits == 32 else pkg.BSORT_U64
    off, d, want = _batch(1, bits, sizes)
    out = torch.empty_like(d)
    h = pkg.bsort_create(pkg.bsort_config(device=0))
    need = pkg.bsort_plan_batch(h, kt, off).workspace_bytes
    warm = pkg.BucketSorter()  # the library's kernels are loaded
    warm.sort_batch(d, off, out, key_type)
    warm.sync()
    warm.close()
    del warm
    out.zero_()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    left = need * 2 // 3
    stream = torch.cuda.current_stream().cuda_stream
    hog = torch.empty(free - left, dtype=torch.uint8, device="cuda")
    try:  # (nothing else may want device memory here)
        pkg.bsort_sort_batch(h, kt, d.data_ptr(), out.data_ptr(), off, stream)
        pkg.bsort_sync(h, stream)
        assert torch.cuda.mem_get_info()[0] > 0
    finally:
        del hog
        torch.cuda.empty_cache()
    assert _same(out, want)
    # as much is not asked for again
    out.zero_()
    pkg.bsort_sort_batch(h, kt, d.data_ptr(), out.data_ptr(), off, stream)
    pkg.bsort_sync(h, stream)
    assert _same(out, want)
    pkg.bsort_destroy(h)


def test_wrapper_out_of_memory(monkeypatch):
    """The same through the wrapper, whose workspace is a torch tensor: its
    allocation fails above a limit."""
    off, d, want = _batch(2)
    sorter = pkg.BucketSorter()
    need = sorter.plan_batch(off).workspace_bytes
    limit = need // 2
    real = torch.empty

    def empty(*a, **kw):
        if kw.get("dtype") == torch.uint8 and a[0] > limit:
            raise torch.cuda.OutOfMemoryError("no room")
        return real(*a, **kw)

    out = torch.empty_like(d)
    monkeypatch.setattr(torch, "empty", empty)
    sorter.sort_batch(d, off, out)
    sorter.sync()
    assert sorter.ws.numel() <= limit
    assert _same(out, want)
    kept = sorter.ws.data_ptr()
    out.zero_()
    sorter.sort_batch(d, off, out)  # (as much is not asked for again)
    assert sorter.ws.data_ptr() == kept
    assert _same(out, want)
    sorter.close()


def test_wrapper_plans_do_not_depend_on_earlier_calls():
    """A small batch first: the workspace it leaves must not decide how the
    next one is sorted."""
    off, d, want = _batch(3)
    small_off, small, small_want = _batch(4, sizes=[5000, 600])
    sorter = pkg.BucketSorter()
    need = sorter.plan_batch(off).workspace_bytes
    out_s, out = torch.empty_like(small), torch.empty_like(d)
    sorter.sort_batch(small, small_off, out_s)
    assert sorter.plan_batch(off).workspace_bytes == need
    sorter.sort_batch(d, off, out)
    assert sorter.ws.numel() >= need
    assert _same(out_s, small_want) and _same(out, want)
    sorter.close()


def test_capture_with_a_small_workspace():
    """Under the caller's capture the workspace cannot grow: the plan that fits
    what is there is taken."""
    off, d, want = _batch(5)
    out = torch.empty_like(d)
    h = pkg.bsort_create(pkg.bsort_config(device=0))
    one = np.array([0, 1500001], np.uint64)  # grows the workspace to one plain sort's
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        pkg.bsort_sort_batch(h, pkg.BSORT_U32, d.data_ptr(), out.data_ptr(), one, s.cuda_stream)
        pkg.bsort_sync(h, s.cuda_stream)
        lone = np.concatenate([[0], np.cumsum([5000] * 3000)]).astype(np.uint64)
        pkg.bsort_sort_batch(h, pkg.BSORT_U32, d.data_ptr(), out.data_ptr(), lone, s.cuda_stream)
        pkg.bsort_sync(h, s.cuda_stream)  # (grows the staging of descriptors)
    two = np.array([0, 600001, 1200002], np.uint64)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s, capture_error_mode="relaxed"):
        pkg.bsort_sort_batch(h, pkg.BSORT_U32, d.data_ptr(), out.data_ptr(), two, s.cuda_stream)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    k = d.cpu().numpy().view(np.uint32)
    got = out.cpu().numpy().view(np.uint32)
    assert np.array_equal(got[:600001], np.sort(k[:600001]))
    assert np.array_equal(got[600001:1200002], np.sort(k[600001:1200002]))
    pkg.bsort_destroy(h)


def test_parts_of_a_large_batch():
    """300 segments of 2^21 keys: 5 GB of joined segments, two parts."""
    rows, n = 300, 1 << 21
    off = (np.arange(rows + 1, dtype=np.uint64) * np.uint64(n))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)
    d = torch.randint(-(1 << 31), 1 << 31, (rows, n), dtype=torch.int32, device="cuda",
                      generator=gen)
    sorter = pkg.BucketSorter()
    assert sorter.plan_batch(off).num_kernels == 14
    out = sorter.sort_batch(d.view(-1), off).view(rows, n)
    sorter.sync()
    sorter.close()
    flip = torch.tensor(-(1 << 31), dtype=torch.int32, device="cuda")
    for a in range(0, rows, 50):
        want = torch.sort(d[a:a + 50] ^ flip, dim=1).values ^ flip
        assert torch.equal(out[a:a + 50], want)
