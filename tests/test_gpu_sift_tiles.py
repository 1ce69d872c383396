"""SIFT-PCA features at the edges of the descriptor tiles (32 x 16 pixels of
one residue class mod the stride): sizes one below, at and one above a whole
number of tiles at strides 1 and 8, and images smaller than a stride's tile.
Bit-exact against the oracle, which follows the same operation order."""
import os

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h", [(8, 8), (9, 15), (31, 16), (32, 17), (33, 33), (257, 129), (255, 127), (300, 50)])
def test_phi_at_tile_edges(w, h):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    images = scenegen.random_images(w, h, seed=w + 1000 * h, n=4)
    images[1][:] = 77  # no gradient: all-zero descriptors
    images[2][:, : w // 2] = images[2][:1, :1]  # flat beside noise
    p = sff.default_params(num_scales=4)
    dev = [torch.as_tensor(np.ascontiguousarray(im)).cuda() for im in images]
    phis = [torch.full((4, h, w, 4), float("nan"), dtype=torch.float32, device="cuda") for _ in range(4)]
    ws = torch.empty(sff.sift_workspace_bytes(w, h), dtype=torch.uint8, device="cuda")
    sff.sift_features(dev, phis, ws, p)
    torch.cuda.synchronize()
    want, _, _ = oracle.sift_phi(images, num_scales=4)
    for got, o in zip(phis, want):
        assert np.array_equal(got.cpu().numpy(), o)


@pytest.mark.parametrize("w,h", [(1416, 904), (500, 37)])
def test_axes_of_many_descriptors(w, h):
    """The covariance's sums over more descriptors than one 32-bit partial
    sum takes (1416 x 904), and over a count that is no multiple of a step."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    images = scenegen.random_images(w, h, seed=w, n=4)
    images[3] //= 8
    p = sff.default_params(num_scales=1)
    dev = [torch.as_tensor(np.ascontiguousarray(im)).cuda() for im in images]
    phis = [torch.empty((1, h, w, 4), dtype=torch.float32, device="cuda") for _ in range(4)]
    ws = torch.empty(sff.sift_workspace_bytes(w, h), dtype=torch.uint8, device="cuda")
    sff.sift_features(dev, phis, ws, p)
    assert sff.device_status() == sff.OK
    want, _, _ = oracle.sift_phi(images, num_scales=1)
    for got, o in zip(phis, want):
        assert np.array_equal(got.cpu().numpy(), o)


def test_scratch_of_one_scale_gives_the_same_phi():
    """The order of the scales does not depend on the results: scratch for one
    scale's descriptors (what larger images get) and for all of them, on a side
    stream and inside a captured graph."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1710_10096_gb300 as sff
    sff.build()
    w, h = 161, 83
    p = sff.default_params()
    dev = [torch.as_tensor(im).cuda() for im in scenegen.make_quad("planes", w, h, 5).images()]
    full = sff.sift_workspace_bytes(w, h)
    small = full - 3 * 4 * w * h * 128
    outs = []
    for nbytes in (full, small + 4096):
        phis = [torch.full((4, h, w, 4), float("nan"), device="cuda") for _ in range(4)]
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            sff.sift_features(dev, phis, ws, p, stream=s)
            s.synchronize()
            outs.append([t.clone() for t in phis])
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                sff.sift_features(dev, phis, ws, p, stream=torch.cuda.current_stream())
            for t in phis:
                t.zero_()
            g.replay()
        s.synchronize()
        outs.append([t.clone() for t in phis])
    for o in outs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(outs[0], o))
    with pytest.raises(sff.SffError):
        sff.sift_features(dev, phis, torch.empty(small - 4096, dtype=torch.uint8, device="cuda"), p)


@pytest.mark.parametrize("w,h,S,knn_t,knn_e", [(8, 8, 4, 8, 8), (9, 11, 1, 3, 1), (67, 35, 4, 4, 2), (130, 33, 3, 8, 3),
                                               (16, 40, 2, 1, 8)])
def test_sift_fields_at_tile_edges(w, h, S, knn_t, knn_e):
    """The matching with the SIFT cost where tiles, windows and candidate lists
    are partial (images smaller than a window's reach, one to eight
    combinations and more), on features with exact zeros among the distances
    (flat areas shared by the views) and with values outside the fast root's
    range: the fields and the costs' bit patterns equal the oracle's."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    rng = np.random.default_rng(w * h + S)
    images = scenegen.random_images(w, h, seed=w + h, n=4)
    for im in images:
        im[: h // 2, : w // 2] = 90
    p = sff.default_params(num_scales=S, iterations=5, knn_temporal=knn_t, knn_epipolar=knn_e)
    op = oracle.default_params(**p.as_dict())
    dev = [torch.as_tensor(im).cuda() for im in images]
    ws = torch.empty(sff.workspace_bytes(w, h, p), dtype=torch.uint8, device="cuda")
    pyr = [torch.empty(sff.pyramid_bytes(w, h, p), dtype=torch.uint8, device="cuda") for _ in range(4)]
    for im, py in zip(dev, pyr):
        sff.features(im, py, ws, p)
    phis = [(rng.standard_normal((S, h, w, 4)) * 40).astype(np.float32) for _ in range(4)]
    for f in phis:
        f[..., 3] = 0
        f[:, : h // 2, : w // 2] = 1.5                      # exact zero distances
        f[:, h // 2:, : w // 4, :3] *= np.float32(1e-18)     # squares below 2^-96
        f[0, -1, -1, 0] = np.float32(3e17)                   # a square above 2^100
    dphi = [torch.as_tensor(f).cuda() for f in phis]
    for mirror, order in ((0, (0, 2, 1, 3)), (1, (3, 1, 2, 0))):
        field = torch.empty((h, w, 4), dtype=torch.int16, device="cuda")
        cost = torch.empty((h, w), dtype=torch.int32, device="cuda")
        sff.match_views_sift(*[pyr[k] for k in order], *[dphi[k] for k in order], w, h, mirror, 77, field, cost, ws, p)
        torch.cuda.synchronize()
        feats = [oracle.features(im, op)[0] for im in images]
        wf, wc = oracle.match_views_sift(*[feats[k] for k in order], *[phis[k] for k in order], w, h, mirror, 77, op)
        assert np.array_equal(cost.cpu().numpy(), wc)
        assert np.array_equal(field.cpu().numpy(), wf)


@pytest.mark.parametrize("w,h", [(64, 40), (37, 23)])
def test_workspace_of_two_fields_gives_the_same_field(w, h):
    """A workspace without room for the repacked phi: the scratch of the WHT
    matching calls, 39 to 64 bytes per pixel at four scales, is enough for both."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1710_10096_gb300 as sff
    sff.build()
    p = sff.default_params(num_scales=4)
    dev = [torch.as_tensor(np.ascontiguousarray(im)).cuda() for im in scenegen.random_images(w, h, seed=5, n=4)]
    full = torch.empty(sff.workspace_bytes(w, h, p), dtype=torch.uint8, device="cuda")
    pyr = [torch.empty(sff.pyramid_bytes(w, h, p), dtype=torch.uint8, device="cuda") for _ in range(4)]
    for im, q in zip(dev, pyr):
        sff.features(im, q, full, p)
    phis = [torch.empty((4, h, w, 4), dtype=torch.float32, device="cuda") for _ in range(4)]
    sff.sift_features(dev, phis, torch.empty(sff.sift_workspace_bytes(w, h), dtype=torch.uint8, device="cuda"), p)

    def field(call, ws):
        f = torch.empty((h, w, 4), dtype=torch.int16, device="cuda")
        c = torch.empty((h, w), dtype=torch.int32, device="cuda")
        call(f, c, ws)
        torch.cuda.synchronize()
        return f, c

    def sift(f, c, ws):
        sff.match_views_sift(*pyr, *phis, w, h, 0, 7, f, c, ws, p)

    def wht(f, c, ws):
        sff.match_views(*pyr, w, h, 0, 7, f, c, ws, p)

    # the smallest workspace that sff_match_views takes
    lo, hi = 0, full.numel()
    while lo < hi:
        mid = (lo + hi) // 2 // 256 * 256
        try:
            field(wht, full[:mid])
            hi = mid
        except sff.SffError:
            lo = mid + 256
    assert lo < full.numel()
    for a, b in zip(field(sift, full), field(sift, full[:lo].clone())):
        assert torch.equal(a, b)
    with pytest.raises(sff.SffError):
        field(sift, full[: lo - 256])
