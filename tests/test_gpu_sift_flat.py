"""Matching with the SIFT cost where flat areas are shared by the views (saturated
sky, bars, a constant image): exact zeros among the distances send a candidate
through the general form.  Fields and costs' bit patterns equal the oracle's."""
import os

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h", [(61, 47), (120, 64)])
@pytest.mark.parametrize("what", ["sky", "bars", "constant", "speckle"])
def test_fields_on_flat_areas(w, h, what):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    images = [im.copy() for im in scenegen.make_quad("planes", w, h, 7).images()]
    for k, im in enumerate(images):
        if what == "sky":
            im[: h * 3 // 10] = 255
        elif what == "bars":
            im[: h // 8] = 0
            im[-(h // 8):] = 0
        elif what == "constant":
            im[:] = 128
        else:
            im[np.random.default_rng(k).random((h, w)) < 0.5] = 255
    p = sff.default_params(iterations=6)
    op = oracle.default_params(**p.as_dict())
    dev = [torch.as_tensor(im).cuda() for im in images]
    ws = torch.empty(sff.workspace_bytes(w, h, p), dtype=torch.uint8, device="cuda")
    pyr = [torch.empty(sff.pyramid_bytes(w, h, p), dtype=torch.uint8, device="cuda") for _ in range(4)]
    for im, py in zip(dev, pyr):
        sff.features(im, py, ws, p)
    phis = [torch.empty((4, h, w, 4), dtype=torch.float32, device="cuda") for _ in range(4)]
    sff.sift_features(dev, phis, torch.empty(sff.sift_workspace_bytes(w, h), dtype=torch.uint8, device="cuda"), p)
    field = torch.empty((h, w, 4), dtype=torch.int16, device="cuda")
    cost = torch.empty((h, w), dtype=torch.int32, device="cuda")
    feats = [oracle.features(im, op)[0] for im in images]
    ophi, _, _ = oracle.sift_phi(images, num_scales=4)
    for mirror, order in ((0, (0, 2, 1, 3)), (1, (3, 1, 2, 0))):
        sff.match_views_sift(*[pyr[k] for k in order], *[phis[k] for k in order], w, h, mirror, 5, field, cost, ws, p)
        torch.cuda.synchronize()
        wf, wc = oracle.match_views_sift(*[feats[k] for k in order], *[ophi[k] for k in order], w, h, mirror, 5, op)
        assert np.array_equal(cost.cpu().numpy(), wc)
        assert np.array_equal(field.cpu().numpy(), wf)
