"""The exact nearest-neighbour initialisation around its tiles (128 queries,
256 candidates): grids of one less, exactly and one more than whole tiles, fewer
candidates than neighbours asked for, and images whose distances tie everywhere
(constant) or in large groups (stripes), which overflow the candidate buffers.
No iterations: the fields are the initialisation, equal to the oracle's."""
import os

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["random", "flat", "stripes"])
@pytest.mark.parametrize("w,h,S", [(8, 8, 4), (16, 8, 1), (17, 15, 1), (16, 16, 1), (19, 27, 1), (61, 9, 2), (100, 77, 2)])
def test_knn_tile_edges(w, h, S, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    images = scenegen.random_images(w, h, seed=w + 5 * h, n=4)
    if kind == "flat":
        images = [np.full_like(im, 10 * k) for k, im in enumerate(images)]
    elif kind == "stripes":
        images = [np.ascontiguousarray(np.broadcast_to(im[:1] // 64 * 64, im.shape)) for im in images]
    p = sff.default_params(num_scales=S, iterations=0, knn_temporal=8)
    op = oracle.default_params(**p.as_dict())
    ws = torch.empty(sff.workspace_bytes(w, h, p), dtype=torch.uint8, device="cuda")
    pyr = [torch.empty(sff.pyramid_bytes(w, h, p), dtype=torch.uint8, device="cuda") for _ in range(4)]
    for im, py in zip(images, pyr):
        sff.features(torch.as_tensor(im).cuda(), py, ws, p)
    feats = [oracle.features(im, op)[0] for im in images]
    for mirror, o in ((0, (0, 2, 1, 3)), (1, (3, 1, 2, 0))):
        field = torch.empty((h, w, 4), dtype=torch.int16, device="cuda")
        cost = torch.empty((h, w), dtype=torch.int32, device="cuda")
        sff.match_views(*[pyr[k] for k in o], w, h, mirror, 5, field, cost, ws, p)
        assert sff.device_status() == sff.OK
        wf, wc = oracle.match_views(*[feats[k] for k in o], mirror, 5, op)
        assert np.array_equal(cost.cpu().numpy(), wc)
        assert np.array_equal(field.cpu().numpy(), wf)
