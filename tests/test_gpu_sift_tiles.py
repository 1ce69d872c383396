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
