"""Interpolation on both sides of each line of its split (one or two seeds per
warp, by the number of seeds, the 152 x 20 warps resident at the default
neighbourhoods and the number of blocks), odd numbers among them, against the
oracle at sampled pixels within the bound of test_gpu_interp."""
import os

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

R = 152 * 20


@pytest.mark.parametrize("w,h,count", [
    (265, 200, R - 1), (265, 200, R), (265, 200, R + 1), (265, 200, R + 2),  # 89 x 67 blocks
    (421, 253, 5992), (421, 253, 5993),                                      # half of 141 x 85 blocks
    (421, 253, 2 * R), (421, 253, 2 * R + 1), (421, 253, 10 * R // 3), (421, 253, 10 * R // 3 + 1),
    (421, 253, 10 * R // 3 + 2),
])
def test_counts_at_the_splits(w, h, count):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    gt, occ, f, b = scenegen.ground_truth("planes", w, h, 3)
    s = scenegen.sparse_seeds(gt, np.zeros_like(occ), seed=4, keep=1.0, noise=0.3)
    assert len(s) >= count
    s = s[np.sort(np.random.default_rng(count).permutation(len(s))[:count])]
    s["d1"][1::3] = 0  # geometry only
    cap = sff.seed_capacity(w, h)
    buf = np.zeros(cap, sff.SEED_DTYPE)
    buf[:count] = s.view(sff.SEED_DTYPE)
    field = torch.empty((h, w, 4), dtype=torch.float32, device="cuda")
    ws = torch.empty(sff.interp_workspace_bytes(w, h, cap), dtype=torch.uint8, device="cuda")
    sff.interpolate(torch.as_tensor(buf.view(np.uint8).copy()).cuda(),
                    torch.tensor([count], dtype=torch.int32, device="cuda"), cap, w, h,
                    sff.default_interp_params(w, h, f, b), field, ws)
    torch.cuda.synchronize()
    assert sff.interp_status(ws, w, h, cap) == 0
    rng = np.random.default_rng(6)
    pix = np.stack([rng.integers(0, w, 3000), rng.integers(0, h, 3000)], 1).astype(np.int32)
    pix = np.concatenate([pix, [[s["x"][k], s["y"][k]] for k in (0, 1, count - 2, count - 1)]]).astype(np.int32)
    p = oracle.interp_params(w, h, f, b)
    sd = np.ascontiguousarray(s, oracle.SEED_DTYPE)
    zero = (np.zeros((len(sd), 3)), np.zeros((len(sd), 15)), np.zeros(len(sd), np.int32))
    _, closest = oracle.interpolate_pixels(sd, p, pix, models=zero)
    want, _ = oracle.interpolate_pixels(sd, p, pix, models=oracle.seed_models(sd, p, which=closest))
    assert {0, 1, count - 2, count - 1} <= set(closest.tolist())
    np.testing.assert_allclose(field.cpu().numpy()[pix[:, 1], pix[:, 0]], want, rtol=1e-5, atol=1e-3)


@pytest.mark.parametrize("kg,km", [(200, 100), (240, 120), (250, 125), (400, 300), (1024, 1024), (7, 1024)])
@pytest.mark.parametrize("count", [1, 33, 4001])
def test_neighbourhoods_at_the_split(kg, km, count):
    # two seeds per warp up to 220 / 110 neighbours, one each above
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    w, h = 265, 200
    gt, occ, f, b = scenegen.ground_truth("planes", w, h, 3)
    s = scenegen.sparse_seeds(gt, np.zeros_like(occ), seed=5, keep=1.0, noise=0.3)
    s = s[np.sort(np.random.default_rng(kg + count).permutation(len(s))[:count])]
    s["d1"][1::3] = 0  # geometry only
    raw = torch.as_tensor(np.frombuffer(np.ascontiguousarray(s).tobytes(), np.uint8).copy()).cuda()
    field = torch.empty((h, w, 4), dtype=torch.float32, device="cuda")
    ws = torch.empty(sff.interp_workspace_bytes(w, h, count), dtype=torch.uint8, device="cuda")
    sff.interpolate(raw, torch.tensor([count], dtype=torch.int32, device="cuda"), count, w, h,
                    sff.default_interp_params(w, h, f, b, k_geo=kg, k_motion=km), field, ws)
    torch.cuda.synchronize()
    assert sff.interp_status(ws, w, h, count) == 0
    want = oracle.interpolate(s, w, h, oracle.interp_params(w, h, f, b, k_geo=kg, k_motion=km))
    np.testing.assert_allclose(field.cpu().numpy(), want, rtol=1e-5, atol=1e-3)
