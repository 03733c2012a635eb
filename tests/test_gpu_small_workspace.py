"""Sorts in a workspace too small for the tabled plan: a plan with fewer
records and runs takes its place, as the sizes that held these sorts before
the plans were tabled still must."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, run on the GPU machine
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1002_4464_gb300 as pkg  # noqa: E402

KT = {"u32": pkg.BSORT_U32, "u64": pkg.BSORT_U64}
# key type, value bytes, n, the bytes that once held the sort
CASES = [("u32", 0, 1 << 23, 72056576), ("u32", 0, 1 << 24, 153832448),
         ("u32", 4, (1 << 23) - 1, 144038400), ("u32", 8, 1 << 26, 1822533120),
         ("u64", 8, (1 << 23) - 1, 446028288)]


def _data(key_type, n):
    k = synth.draws64(synth.seed_for(12, n % 1000), n)
    if key_type == "u32":
        k = (k >> np.uint64(44)).astype(np.uint32)  # (repeated keys)
    return k, torch.from_numpy(k.view(np.int32 if key_type == "u32" else np.int64)).cuda()


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("key_type,vb,n,held", CASES)
def test_fixed_workspace(key_type, vb, n, held, in_place):
    k, d = _data(key_type, n)
    sorter = pkg.BucketSorter(workspace_bytes=held)
    free = pkg.BucketSorter()
    assert free.plan(n, key_type, vb).workspace_bytes > held
    assert sorter.plan(n, key_type, vb).workspace_bytes <= held
    free.close()
    out = d if in_place else torch.empty_like(d)
    if vb:
        v = torch.arange(n, dtype=torch.int32 if vb == 4 else torch.int64, device="cuda")
        ov = v if in_place else torch.empty_like(v)
        sorter.sort_pairs(d, v, out, ov, key_type)
    else:
        sorter.sort_keys(d, out, key_type)
    sorter.sync()
    assert sorter.ws.numel() == held
    sorter.close()
    if vb:
        order = np.argsort(k, kind="stable")
        assert np.array_equal(ov.cpu().numpy(), order.astype(ov.cpu().numpy().dtype))
        k = k[order]
    else:
        k = np.sort(k)
    assert np.array_equal(out.cpu().numpy().view(k.dtype), k)


def test_fixed_workspace_host_buffers():
    n = 1 << 23
    k, _ = _data("u32", n)
    h_in = torch.from_numpy(k.view(np.int32)).pin_memory()
    out = torch.empty_like(h_in, pin_memory=True)
    ws = torch.empty(72056576 + 4 * n + 256, dtype=torch.uint8, device="cuda")
    h = pkg.bsort_create(pkg.bsort_config(device=0, workspace=ws.data_ptr(),
                                          workspace_bytes=ws.numel()))
    stream = torch.cuda.current_stream().cuda_stream
    pkg.bsort_sort_keys_host(h, pkg.BSORT_U32, h_in.data_ptr(), out.data_ptr(), n, stream)
    pkg.bsort_sync(h, stream)
    pkg.bsort_destroy(h)
    assert np.array_equal(out.numpy().view(np.uint32), np.sort(k))


def test_out_of_memory_takes_the_smallest_plan():
    n, least = 1 << 23, 72056576
    k, d = _data("u32", n)
    out = torch.empty_like(d)
    for held in (0, least):  # (the kernels of both plans are loaded)
        warm = pkg.BucketSorter(workspace_bytes=held)
        warm.sort_keys(d, out)
        warm.sync()
        need = warm.plan(n).workspace_bytes
        assert need > least + (12 << 20) or held
        warm.close()
    del warm
    out.zero_()
    h = pkg.bsort_create(pkg.bsort_config(device=0))
    stream = torch.cuda.current_stream().cuda_stream
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - (least + (8 << 20)), dtype=torch.uint8, device="cuda")
    try:  # (nothing else may want device memory here)
        for _ in range(2):
            pkg.bsort_sort_keys(h, pkg.BSORT_U32, d.data_ptr(), out.data_ptr(), n, stream)
        pkg.bsort_sync(h, stream)
    finally:
        del hog
        torch.cuda.empty_cache()
    pkg.bsort_destroy(h)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), np.sort(k))
