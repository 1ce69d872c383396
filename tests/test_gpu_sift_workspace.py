"""sff_match_views_sift in a workspace that is enough for sff_match_views alone:
same fields, and no device memory allocated on the way (the library's calls work in
the caller's buffers)."""
import ctypes

import pytest

import scenegen

pytestmark = pytest.mark.gpu

USED_MEM_HIGH = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH


@pytest.mark.parametrize("w,h,S", [(64, 40, 4), (131, 57, 4), (45, 33, 2), (33, 20, 1)])
def test_small_workspace_allocates_nothing(w, h, S):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1710_10096_gb300 as sff
    sff.build()
    p = sff.default_params(num_scales=S)
    dev = [torch.as_tensor(im).cuda() for im in scenegen.make_quad("planes", w, h, 5).images()]
    full = torch.empty(sff.workspace_bytes(w, h, p), dtype=torch.uint8, device="cuda")
    pyr = [torch.empty(sff.pyramid_bytes(w, h, p), dtype=torch.uint8, device="cuda") for _ in range(4)]
    for im, q in zip(dev, pyr):
        sff.features(im, q, full, p)
    phis = [torch.empty((S, h, w, 4), dtype=torch.float32, device="cuda") for _ in range(4)]
    sff.sift_features(dev, phis, torch.empty(sff.sift_workspace_bytes(w, h), dtype=torch.uint8, device="cuda"), p)

    # the smallest workspace that sff_match_views takes
    lo, hi = 0, full.numel() // 256 * 256
    out = [(torch.empty((h, w, 4), dtype=torch.int16, device="cuda"), torch.empty((h, w), dtype=torch.int32, device="cuda"))
           for _ in range(2)]
    while lo < hi:
        mid = (lo + hi) // 2 // 256 * 256
        try:
            sff.match_views(*pyr, w, h, 0, 7, *out[0], full[:mid], p)
            hi = mid
        except sff.SffError:
            lo = mid + 256
    small = torch.empty(lo, dtype=torch.uint8, device="cuda")
    sff.match_views_sift(*pyr, *phis, w, h, 0, 7, *out[0], full, p)
    torch.cuda.synchronize()

    cu = ctypes.CDLL("libcuda.so.1")
    pool, high = ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), ctypes.c_int(torch.cuda.current_device())) == 0
    assert cu.cuMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    sff.match_views_sift(*pyr, *phis, w, h, 0, 7, *out[1], small, p)
    torch.cuda.synchronize()
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(high)) == 0
    assert high.value == 0
    for a, b in zip(*out):
        assert torch.equal(a, b)
