"""The sequential sweeps where the number of rows changes the work split: at
and past 128 and 256 rows (lanes per row), past 512 rows (blocks of rows go round
the warps, the last warp's rows reaching the first through memory) with rows
longer than the ring between two warps.  Fields and costs equal the oracle's
scan order."""
import os

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h", [(33, 128), (33, 129), (72, 256), (40, 257), (200, 1100), (9, 530)])
def test_sequential_rows(w, h):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    images = scenegen.random_images(w, h, seed=w + 3 * h, n=4)
    for k in (1, 2, 3):  # related views, so that vectors travel along the rows
        images[k] = np.roll(images[0], (k, -2 * k), (0, 1)) // 2 + images[k] // 2
    p = sff.default_params(num_scales=4, iterations=4)
    op = oracle.default_params(**p.as_dict())
    op.order_mode = oracle.SEQUENTIAL_SCAN
    ws = torch.empty(sff.workspace_bytes(w, h, p), dtype=torch.uint8, device="cuda")
    pyr = [torch.empty(sff.pyramid_bytes(w, h, p), dtype=torch.uint8, device="cuda") for _ in range(4)]
    for im, py in zip(images, pyr):
        sff.features(torch.as_tensor(im).cuda(), py, ws, p)
    feats = [oracle.features(im, op)[0] for im in images]
    for mirror, o in ((0, (0, 2, 1, 3)), (1, (3, 1, 2, 0))):
        field = torch.empty((h, w, 4), dtype=torch.int16, device="cuda")
        cost = torch.empty((h, w), dtype=torch.int32, device="cuda")
        sff.match_views_sequential(*[pyr[k] for k in o], w, h, mirror, 5, field, cost, ws, p)
        assert sff.device_status() == sff.OK
        wf, wc = oracle.match_views(*[feats[k] for k in o], mirror, 5, op)
        assert np.array_equal(cost.cpu().numpy(), wc)
        assert np.array_equal(field.cpu().numpy(), wf)
