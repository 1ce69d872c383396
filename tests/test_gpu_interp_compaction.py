"""Interpolation where a set reaches its k-th member inside the ring of blocks
that overflows the candidate slots: a lone seed in a hole of a dense lattice,
and a seed inside a patch of geometry-only seeds (what the disparity fill emits)
surrounded by motion seeds.  The compaction then has to bound the k-th distances
by the seeds of that ring too.  Against the oracle, which holds every seed,
within the bound of test_gpu_interp (1e-3 px + 1e-5 relative: both sides sum the
same doubles in different orders)."""
import os

import numpy as np
import pytest

import scenegen

pytestmark = pytest.mark.gpu

FLAT = dict(alpha=0.1)  # weights that let far neighbours count beside the seed itself


def _lattice(blocks, half, jitter):
    """One seed per block of a blocks x blocks grid, and per seed the Chebyshev
    distance of its block from the middle one."""
    by, bx = np.mgrid[0:blocks, 0:blocks]
    rng = np.random.default_rng(blocks + half)
    o = rng.integers(0, 3, (2,) + bx.shape) if jitter else np.ones((2,) + bx.shape, int)
    s = np.zeros(bx.size, scenegen.SEED_RECORD)
    s["x"], s["y"] = (3 * bx + o[0]).ravel(), (3 * by + o[1]).ravel()
    s["d0"] = 20 + s["x"] // 40 + (s["x"] + 2 * s["y"]) % 3
    s["d1"] = s["d0"] + 2 + s["y"] // 100
    s["u"], s["v"] = 3 + s["y"] // 60, -2
    return s, np.maximum(np.abs(bx - blocks // 2), np.abs(by - blocks // 2)).ravel()


def _check(s, w, h, **over):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_1710_10096_gb300 as sff
    sff.build()
    oracle.build()
    oracle.set_threads(os.cpu_count() or 1)
    raw = torch.as_tensor(np.frombuffer(np.ascontiguousarray(s).tobytes(), np.uint8).copy()).cuda()
    count = torch.tensor([len(s)], dtype=torch.int32, device="cuda")
    field = torch.full((h, w, 4), float("nan"), dtype=torch.float32, device="cuda")
    ws = torch.empty(sff.interp_workspace_bytes(w, h, len(s)), dtype=torch.uint8, device="cuda")
    sff.interpolate(raw, count, len(s), w, h, sff.default_interp_params(w, h, 400.0, 0.5, **over), field, ws)
    torch.cuda.synchronize()
    assert sff.interp_status(ws, w, h, len(s)) == 0
    rng = np.random.default_rng(w)
    pix = np.concatenate([w // 2 + rng.integers(-40, 41, (200, 2)), rng.integers(0, min(w, h), (100, 2)),
                          [[w // 2, h // 2]]]).astype(np.int32)
    p = oracle.interp_params(w, h, 400.0, 0.5, **over)
    sd = np.ascontiguousarray(s, oracle.SEED_DTYPE)
    zero = (np.zeros((len(sd), 3)), np.zeros((len(sd), 15)), np.zeros(len(sd), np.int32))
    _, closest = oracle.interpolate_pixels(sd, p, pix, models=zero)
    want, _ = oracle.interpolate_pixels(sd, p, pix, models=oracle.seed_models(sd, p, which=closest))
    np.testing.assert_allclose(field.cpu().numpy()[pix[:, 1], pix[:, 0]], want, rtol=1e-5, atol=1e-3)


@pytest.mark.parametrize("half,over", [
    (80, FLAT),                             # 480 px: the k-th member in an earlier ring than the overflow
    (105, FLAT), (130, FLAT), (155, FLAT),  # 630, 780 and 930 px: in the same ring
    (40, dict(k_geo=8, k_motion=8, **FLAT)),  # 240 px, few neighbours, few slots
])
@pytest.mark.parametrize("jitter", [False, True])
def test_lone_seed_in_a_hole(half, over, jitter):
    blocks = 2 * half + 31
    s, ring = _lattice(blocks, half, jitter)
    s = s[(ring >= half) | (ring == 0)]
    _check(s, 3 * blocks, 3 * blocks, **over)


@pytest.mark.parametrize("half,keep", [(75, 1), (80, 1), (80, 4), (100, 1), (100, 4), (125, 1), (125, 7)])
def test_geometry_only_patch_among_motion_seeds(half, keep):
    # inside, one seed in `keep` of a dense lattice, none with motion
    blocks = 2 * half + 31
    s, ring = _lattice(blocks, half, True)
    inside = ring < half
    s["u"][inside] = s["v"][inside] = s["d1"][inside] = 0
    s["kind"][inside] = 1
    s = s[~inside | (np.arange(len(s)) % keep == 0)]
    _check(s, 3 * blocks, 3 * blocks)


@pytest.mark.parametrize("half", [110, 160])
def test_only_the_geometry_set_fills_in_the_overflowing_ring(half):
    # around the hole one seed in 16 moves, so the motion set fills many rings later
    blocks = 2 * half + 61
    s, ring = _lattice(blocks, half, True)
    s = s[(ring >= half) | (ring == 0)]
    still = np.random.default_rng(half).random(len(s)) > 1 / 16
    s["u"][still] = s["v"][still] = s["d1"][still] = 0
    s["kind"][still] = 1
    _check(s, 3 * blocks, 3 * blocks, **FLAT)
