"""The disparity map where the path kernel's splits are partial: every
disparity range with lines that do not fill a warp (heights and widths around
multiples of the lines per warp), lines shorter and longer than the costs kept
in flight, and segments of the cost kernel cut by the image edge.  Equal to the
oracle's."""
import os

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [32, 64, 128, 256])
@pytest.mark.parametrize("w,h", [(8, 9), (15, 33), (63, 8), (64, 17), (65, 31), (129, 12)])
def test_sgm_partial_splits(w, h, D):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    L, R = scenegen.random_images(w, h, seed=D + w * h, n=2)
    R[:, : w // 3] = L[:, : w // 3]  # a part that matches at 0, ties elsewhere
    p1, p2 = (0, 193) if w % 2 else (12, 90)
    p = sff.default_sgm_params(max_disp=D, p1=p1, p2=p2)
    disp = torch.full((h, w), -7, dtype=torch.int16, device="cuda")
    ws = torch.empty(sff.sgm_workspace_bytes(w, h, p), dtype=torch.uint8, device="cuda")
    sff.sgm(torch.as_tensor(L).cuda(), torch.as_tensor(R).cuda(), disp, ws, p)
    torch.cuda.synchronize()
    assert np.array_equal(disp.cpu().numpy(), oracle.sgm(L, R, oracle.sgm_params(max_disp=D, p1=p1, p2=p2)))
