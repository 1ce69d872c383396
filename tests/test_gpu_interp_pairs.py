"""Interpolation of odd and tiny numbers of seeds: a warp fits two seeds side by
side, so an odd count leaves one alone, and a pair may differ in the size of its
neighbourhoods (fewer seeds than k, a seed without motion neighbours nearby).
Within the bound of test_gpu_interp (1e-3 px + 1e-5 relative, element by
element: both sides sum the same doubles in different orders)."""
import os

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 2, 3, 5, 64, 129])
@pytest.mark.parametrize("kg,km", [(160, 80), (17, 33)])
def test_seed_pairs(count, kg, km):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    w, h = 123, 77
    gt, occ, f, b = scenegen.ground_truth("planes", w, h, 3)
    s = scenegen.sparse_seeds(gt, np.zeros_like(occ), seed=count, keep=1.0, noise=0.3)
    s = s[np.sort(np.random.default_rng(count).permutation(len(s))[:count])]
    s["d1"][1::3] = 0  # geometry only
    cap = sff.seed_capacity(w, h)
    buf = np.zeros(cap, sff.SEED_DTYPE)
    buf[:count] = s.view(sff.SEED_DTYPE)
    ip = sff.default_interp_params(w, h, f, b, k_geo=kg, k_motion=km)
    field = torch.empty((h, w, 4), dtype=torch.float32, device="cuda")
    ws = torch.empty(sff.interp_workspace_bytes(w, h, cap), dtype=torch.uint8, device="cuda")
    sff.interpolate(torch.as_tensor(buf.view(np.uint8).copy()).cuda(),
                    torch.tensor([count], dtype=torch.int32, device="cuda"), cap, w, h, ip, field, ws)
    torch.cuda.synchronize()
    assert sff.interp_status(ws, w, h, cap) == 0
    want = oracle.interpolate(s, w, h, oracle.interp_params(w, h, f, b, k_geo=kg, k_motion=km))
    assert np.allclose(field.cpu().numpy(), want, rtol=1e-5, atol=1e-3)
