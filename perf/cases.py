"""The work a user has this library do, as cases that can be timed.

A case names one of the public paths (KINDS) with its image size, its scene
and its parameters.  The images are rendered here from layered textured
surfaces with known disparities and motions, in the ranges of the
configurations in the repository (disparities up to a tenth of the width,
flows up to an eighth, about a tenth of the pixels occluded, sensor noise), so
the matcher meets smooth fields, motion boundaries, occlusions and pixels
without a correspondence as it does on rendered or recorded quads.

exact() states the computed numbers in 64 bits in plain torch.  The matching
stage, the filter, the seeds and the disparity map are whole numbers (the
SIFT costs too: bit patterns of a fixed operation order), so their cases have
no such value.
"""
import math

import numpy as np
import torch

import paper_1710_10096_gb300 as sff

DEV = "cuda"
FOCAL_PER_WIDTH, BASELINE = 0.58, 0.54  # 721 px at 1242, as the driving scenes


def _case(name, kind, width, height, **more):
    c = {"kind": kind, "width": width, "height": height, "scales": 4, "iterations": 12, "quant_shift": 4,
         "knn_temporal": 4, "knn_epipolar": 2, "max_disp": 128, "quads": 1, "keep": 0.75, "layers": 16}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest configured quad (planes scene): launches and latency count
        _case("quad_256x80", "quad", 256, 80, layers=6),
        # one driving quad, images already on the device: the flagship call
        _case("quad_1242x375", "quad", 1242, 375, layers=24),
        # a movie-shaped quad from host arrays to host seeds: the call a first program makes
        _case("host_1024x436", "host", 1024, 436),
        # full-HD-like and ragged: no side is a multiple of a tile
        _case("quad_1917x1083", "quad", 1917, 1083, layers=24),
        # 32 quads of uneven sizes as one CUDA graph: an offline or multi-camera job
        _case("batch_32", "batch", 1242, 375, quads=32),
        # the dense method: features, fields, filter, SGM fill, seeds and interpolation, call by call
        _case("method_1242x375", "method", 1242, 375, layers=24),
        # the paper's own cost: SIFT-PCA features of four images at every scale
        _case("sift_features_1242x375", "sift_features", 1242, 375),
        # both fields of a quad with that cost, features resident
        _case("sift_match_1242x375", "sift_match", 1242, 375),
        # the disparity map of a driving pair
        _case("sgm_1242x375_d128", "sgm", 1242, 375),
        # a small ragged pair with the shorter disparity range: few lines in flight
        _case("sgm_515x161_d64", "sgm", 515, 161, max_disp=64),
        # dense interpolation of a driving quad's seeds
        _case("interp_1242x375", "interp", 1242, 375, layers=24),
        # the paper's sequential propagation order on the small configured quad
        _case("sequential_256x80", "sequential", 256, 80, layers=6),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["quad", "quad", "quad", "host", "batch", "method", "sift_features", "sift_match", "sgm", "sgm",
                       "interp", "interp", "sequential"])
    most = {"quad": 1917, "host": 1280, "batch": 1242, "method": 1242, "sift_features": 1242, "sift_match": 1242,
            "sgm": 1600, "interp": 1400, "sequential": 256}[kind]
    least = {"batch": 640, "sequential": 96}.get(kind, 160)
    w = _log_uniform(rng, least, most)
    h = max(48, min(1083, int(round(w * rng.uniform(0.28, 0.56)))))
    if kind == "sequential":
        h = min(h, 80)
    if kind in ("sift_features", "sift_match", "method", "batch"):
        h = min(h, 436)
    c = _case(None, kind, w, h, layers=rng.randint(4, 24), quant_shift=rng.choice([4, 4, 3, 5]),
              iterations=rng.choice([12, 12, 8, 6]), knn_temporal=rng.choice([4, 4, 3, 8]),
              knn_epipolar=rng.choice([2, 2, 1, 4]), max_disp=rng.choice([32, 64, 128, 128, 256]),
              keep=round(rng.uniform(0.2, 0.95), 3))
    if w <= 320 and rng.random() < 0.5:
        c["scales"] = 3
    if kind == "batch":
        c["quads"] = rng.choice([2, 5, 8, 13, 24])
    return c


# ---------------------------------------------------------------- the scenes

def _affine_inverse(a):
    """Inverse of the 2x3 affine map a (nested lists of Python numbers)."""
    (m00, m01, m02), (m10, m11, m12) = a
    det = m00 * m11 - m01 * m10
    i00, i01, i10, i11 = m11 / det, -m01 / det, -m10 / det, m00 / det
    return [[i00, i01, -(i00 * m02 + i01 * m12)], [i10, i11, -(i10 * m02 + i11 * m12)]]


def _scene(w, h, layers, seed):
    """(images [4][H, W, 3] uint8 on the device in the order L0, R0, L1, R1,
    vectors [H, W, 4] float64 of L0, visible [H, W] bool).

    Surface k has an affine disparity d0, flow (u, v) and d1 over L0's
    coordinates; its points appear at (x, y), (x - d0, y), (x + u, y + v) and
    (x + u - d1, y + v).  Every view is rendered by the inverse maps, the
    nearest surface that covers the pixel winning."""
    rs = np.random.RandomState((seed * 2654435761 + 12345) % (1 << 32))
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(rs.randint(1 << 30)))
    dmax, umax, vmax = 0.1 * w, 0.125 * w, 0.06 * h
    surf = []  # (rectangle in L0 coordinates, affine d0, u, v, d1 as (constant, per x, per y))
    far = 0.01 * w + 0.5
    ego = rs.uniform(0.02, 0.05)  # forward motion: flow away from the centre, growing with nearness
    # background wall, ground plane, then boxes from far to near
    rects = [((-w, -h, 2 * w, 2 * h), (far, 0.0, 0.0)),
             ((-w, 0.45 * h, 2 * w, 2 * h), (far - 0.45 * h * 0.7 * dmax / (0.55 * h), 0.0, 0.7 * dmax / (0.55 * h)))]
    near = np.sort(rs.uniform(0.03, 0.95, max(0, layers - 2)) ** 2) * dmax + far
    for d in near:
        bw, bh = rs.uniform(0.06, 0.22) * w, rs.uniform(0.15, 0.45) * h
        x0, y0 = rs.uniform(-0.05, 0.95) * w, rs.uniform(0.05, 0.75) * h
        rects.append(((x0, y0, x0 + bw, y0 + bh), (d, 0.0, 0.0)))
    for k, (r, d) in enumerate(rects):
        slant = rs.uniform(-0.02, 0.02) if k > 1 else 0.0
        cx, cy = 0.5 * (r[0] + r[2]), 0.5 * (r[1] + r[3])
        d = (d[0] - slant * cx, d[1] + slant, d[2])
        dc = d[0] + d[1] * cx + d[2] * cy if k != 1 else 0.35 * dmax
        grow = ego * min(1.0, dc / dmax) + 0.01
        tu, tv = (rs.uniform(-1, 1) * umax * dc / dmax, rs.uniform(-1, 1) * vmax * dc / dmax) if k > 1 else (0.0, 0.0)
        if k > 1 and rs.rand() < 0.2:  # an independently moving object
            tu, tv = rs.uniform(-1, 1) * umax, rs.uniform(-1, 1) * vmax
        u = (tu - grow * 0.5 * w, grow, 0.0)
        v = (tv - grow * 0.4 * h, 0.0, grow)
        s = 1.0 + grow * rs.uniform(0.3, 1.0)
        surf.append((r, d, u, v, tuple(s * t for t in d)))
    lat = torch.rand((3, 256, 256), generator=gen, device=DEV)
    off = rs.randint(0, 256, (len(surf), 2))
    offt = torch.as_tensor(off, device=DEV)
    tint = torch.as_tensor(rs.uniform(0.5, 1.0, (len(surf), 3)), device=DEV, dtype=torch.float32)
    yy, xx = torch.meshgrid(torch.arange(h, device=DEV, dtype=torch.float32),
                            torch.arange(w, device=DEV, dtype=torch.float32), indexing="ij")

    def maps(d, u, v, e):
        return ([[1.0, 0.0, 0.0], [0.0, 1.0, 0.0]],
                [[1.0 - d[1], -d[2], -d[0]], [0.0, 1.0, 0.0]],
                [[1.0 + u[1], u[2], u[0]], [v[1], 1.0 + v[2], v[0]]],
                [[1.0 + u[1] - e[1], u[2] - e[2], u[0] - e[0]], [v[1], 1.0 + v[2], v[0]]])

    images, owner = [], []
    for view in range(4):
        ids = torch.zeros((h, w), dtype=torch.long, device=DEV)
        X, Y = xx.clone(), yy.clone()
        for k, (r, d, u, v, e) in enumerate(surf):
            i = _affine_inverse(maps(d, u, v, e)[view])
            px = i[0][0] * xx + i[0][1] * yy + i[0][2]
            py = i[1][0] * xx + i[1][1] * yy + i[1][2]
            inside = (px >= r[0]) & (px < r[2]) & (py >= r[1]) & (py < r[3])
            ids = torch.where(inside, k, ids)
            X, Y = torch.where(inside, px, X), torch.where(inside, py, Y)
        tex = torch.zeros((3, h, w), device=DEV)
        for cell, amp in ((2.7, 0.4), (9.0, 0.35), (31.0, 0.25)):
            gx = X / cell + offt[ids, 0]
            gy = Y / cell + offt[ids, 1]
            ix, iy = torch.floor(gx), torch.floor(gy)
            fx, fy = gx - ix, gy - iy
            ix, iy = ix.long() & 255, iy.long() & 255
            jx, jy = (ix + 1) & 255, (iy + 1) & 255
            tex += amp * ((lat[:, iy, ix] * (1 - fx) + lat[:, iy, jx] * fx) * (1 - fy)
                          + (lat[:, jy, ix] * (1 - fx) + lat[:, jy, jx] * fx) * fy)
        img = tex.permute(1, 2, 0) * tint[ids] * 250.0 + 2.0 * torch.randn((h, w, 3), generator=gen, device=DEV)
        images.append(torch.clamp(torch.round(img), 0, 255).to(torch.uint8).contiguous())
        owner.append(ids)
    coef = torch.as_tensor(np.array([[s[2], s[3], s[1], s[4]] for s in surf]), device=DEV)  # [k, 4, 3]
    c = coef[owner[0]]
    vec = c[..., 0] + c[..., 1] * xx[..., None].double() + c[..., 2] * yy[..., None].double()
    visible = torch.ones((h, w), dtype=torch.bool, device=DEV)
    u, v, d0, d1 = vec.unbind(-1)
    for view, (tx, ty) in ((1, (xx - d0, yy + 0.0 * v)), (2, (xx + u, yy + v)), (3, (xx + u - d1, yy + v))):
        ix, iy = torch.round(tx).long(), torch.round(ty).long()
        ok = (ix >= 0) & (ix < w) & (iy >= 0) & (iy < h)
        visible &= ok & (owner[view][iy.clamp(0, h - 1), ix.clamp(0, w - 1)] == owner[0])
    return images, vec, visible


def _sparse_seeds(w, h, layers, keep, seed):
    """A device byte buffer of seeds as the matcher writes them (block raster
    order, at most one per 3x3 block), and their number: visible pixels with
    their rounded vectors plus noise, a few wrong ones, and in a part of the
    remaining blocks disparity-only seeds."""
    _, vec, visible = _scene(w, h, layers, seed)
    vec, visible = vec.cpu().numpy(), visible.cpu().numpy()
    rs = np.random.RandomState((seed + 977) % (1 << 32))
    by, bx = np.mgrid[0:(h + 2) // 3, 0:(w + 2) // 3]
    x = np.minimum(w - 1, 3 * bx + rs.randint(0, 3, bx.shape)).ravel()
    y = np.minimum(h - 1, 3 * by + rs.randint(0, 3, by.shape)).ravel()
    vis = visible[y, x]
    full = vis & (rs.rand(x.size) < keep)
    only = ~full & (rs.rand(x.size) < 0.5 * keep)
    take = full | only
    x, y, only = x[take], y[take], only[take]
    val = vec[y, x] + 0.4 * rs.randn(x.size, 4)
    wrong = rs.rand(x.size) < 0.02
    val[wrong] += rs.uniform(-0.05, 0.05, (int(wrong.sum()), 4)) * w
    val = np.rint(val)
    val[:, 2:] = np.maximum(val[:, 2:], 0)
    val[only, 0] = val[only, 1] = val[only, 3] = 0
    out = np.zeros(sff.seed_capacity(w, h), sff.SEED_DTYPE)
    n = x.size
    for name, col in (("x", x), ("y", y), ("u", val[:, 0]), ("v", val[:, 1]), ("d0", val[:, 2]), ("d1", val[:, 3]),
                      ("cost", rs.randint(0, 1 << 18, n)), ("cerr", rs.randint(0, 4, n)), ("kind", only)):
        out[name][:n] = col
    return torch.as_tensor(out.view(np.uint8).copy()).to(DEV), n


# ------------------------------------------------------------ prepare and run

def _params(case):
    return sff.default_params(num_scales=case["scales"], iterations=case["iterations"],
                              quant_shift=case["quant_shift"], knn_temporal=case["knn_temporal"],
                              knn_epipolar=case["knn_epipolar"])


def _empty(shape, dtype):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _bytes(n):
    return torch.zeros(n, dtype=torch.uint8, device=DEV)


def _quad_outputs(b):
    return [b.seeds, b.count, b.fwd, b.fwd_cost, b.inv, b.inv_cost, b.keep, b.cerr]


def _batch_sizes(case):
    """Uneven sizes in the proportions of the configured batch (1242x375,
    1024x436, 640x192 and 512x160 in turn, scaled with the case's width)."""
    f = case["width"] / 1242.0
    sizes = [(1242, 375), (1024, 436), (640, 192), (512, 160)]
    return [(int(round(f * sizes[k % 4][0])), int(round(f * sizes[k % 4][1]))) for k in range(case["quads"])]


def prepare(case, seed):
    kind, w, h = case["kind"], case["width"], case["height"]
    p = _params(case)
    st = {"kind": kind, "w": w, "h": h, "p": p, "seed": 1000 + seed}
    if kind == "interp":
        st["seeds"], n = _sparse_seeds(w, h, case["layers"], case["keep"], seed)
        st["capacity"] = sff.seed_capacity(w, h)
        st["count"] = torch.tensor([n], dtype=torch.int32, device=DEV)
        _prepare_interp(st)
        return st
    if kind == "batch":
        sizes = _batch_sizes(case)
        m = sff.BatchMatcher(sizes, p, DEV)
        for k, (qw, qh) in enumerate(sizes):
            m.load(k, *_scene(qw, qh, case["layers"], 64 * seed + k)[0])
            m.quads[k].seeds.zero_()
        st["m"] = m
        st["graph"] = m.capture([st["seed"] + k for k in range(len(sizes))])
        return st
    images = _scene(w, h, case["layers"], seed)[0]
    st["images"] = images
    if kind in ("quad", "host", "method"):
        st["m"] = sff.QuadMatcher(w, h, p, DEV, mode="calls" if kind == "method" else "batch")
        st["m"].seeds.zero_()
        if kind == "host":
            st["images"] = [im.cpu().numpy() for im in images]
            st["taken"] = np.zeros(20 * st["m"].capacity, np.uint8)
    if kind in ("sgm", "method"):
        st["sp"] = sff.default_sgm_params(max_disp=case["max_disp"])
        st["disp"] = _empty((h, w), torch.int16)
        st["sgm_ws"] = _empty(sff.sgm_workspace_bytes(w, h, st["sp"]), torch.uint8)
    if kind == "method":
        st["capacity"] = st["m"].capacity
        st["seeds"], st["count"] = _bytes(20 * st["capacity"]), torch.zeros(1, dtype=torch.int32, device=DEV)
        st["ws"] = _empty(sff.workspace_bytes(w, h, p), torch.uint8)
        _prepare_interp(st)
    if kind in ("sift_features", "sift_match"):
        st["phi"] = [_empty((p.num_scales, h, w, 4), torch.float32) for _ in range(4)]
        st["sift_ws"] = _empty(sff.sift_workspace_bytes(w, h), torch.uint8)
    if kind in ("sift_match", "sequential"):
        st["ws"] = _empty(sff.workspace_bytes(w, h, p), torch.uint8)
        st["pyr"] = [_empty(sff.pyramid_bytes(w, h, p), torch.uint8) for _ in range(4)]
        for im, pyr in zip(images, st["pyr"]):
            sff.features(im, pyr, st["ws"], p)
        st["fields"] = [_empty((h, w, 4), torch.int16) for _ in range(2)]
        st["costs"] = [_empty((h, w), torch.int32) for _ in range(2)]
        if kind == "sift_match":
            sff.sift_features(images, st["phi"], st["sift_ws"], p)
            del st["sift_ws"]
    return st


def _prepare_interp(st):
    w, h = st["w"], st["h"]
    st["ip"] = sff.default_interp_params(w, h, FOCAL_PER_WIDTH * w, BASELINE)
    st["field"] = _empty((h, w, 4), torch.float32)
    st["interp_ws"] = _empty(sff.interp_workspace_bytes(w, h, st["capacity"]), torch.uint8)


def run(st):
    kind, w, h, p = st["kind"], st["w"], st["h"], st["p"]
    if kind == "quad":
        st["m"].run(*st["images"], seed=st["seed"])
        return _quad_outputs(st["m"].buf)
    if kind == "host":
        seeds = st["m"].run_host(*st["images"], seed=st["seed"])
        st["taken"][:20 * len(seeds)] = seeds.view(np.uint8)  # their number depends on the images
        return [len(seeds), st["taken"]]
    if kind == "batch":
        st["graph"].replay()
        return [t for q in st["m"].quads for t in (q.seeds, q.count)]
    if kind == "sgm":
        sff.sgm(st["images"][0], st["images"][1], st["disp"], st["sgm_ws"], st["sp"])
        return st["disp"]
    if kind == "interp":
        sff.interpolate(st["seeds"], st["count"], st["capacity"], w, h, st["ip"], st["field"], st["interp_ws"])
        return st["field"]
    if kind == "sift_features":
        sff.sift_features(st["images"], st["phi"], st["sift_ws"], p)
        return st["phi"]
    if kind == "method":
        m = st["m"]
        m.run(*st["images"], seed=st["seed"])
        sff.sgm(st["images"][0], st["images"][1], st["disp"], st["sgm_ws"], st["sp"])
        sff.emit_seeds_geo(m.fwd, m.fwd_cost, m.keep, m.cerr, st["disp"], st["seeds"], st["capacity"], st["count"],
                           st["ws"], p)
        sff.interpolate(st["seeds"], st["count"], st["capacity"], w, h, st["ip"], st["field"], st["interp_ws"])
        return _quad_outputs(m.buf) + [st["disp"], st["seeds"], st["count"], st["field"]]
    L0, R0, L1, R1 = st["pyr"]
    (f, g), (c, d) = st["fields"], st["costs"]
    if kind == "sift_match":
        a, b, e, k = st["phi"]
        sff.match_views_sift(L0, L1, R0, R1, a, e, b, k, w, h, 0, st["seed"], f, c, st["ws"], p)
        sff.match_views_sift(R1, R0, L1, L0, k, b, e, a, w, h, 1, st["seed"], g, d, st["ws"], p)
    else:
        sff.match_views_sequential(L0, L1, R0, R1, w, h, 0, st["seed"], f, c, st["ws"], p)
        sff.match_views_sequential(R1, R0, L1, L0, w, h, 1, st["seed"], g, d, st["ws"], p)
    return [f, c, g, d]


# ----------------------------------------------------------------------- work

def _match_flops(w, h, case, per_candidate):
    """K-NN of the coarsest grid and three candidates (two predecessors, one
    random) per grid pixel and iteration, of both fields."""
    n = 1 << (case["scales"] - 1)
    gq = -(-w // n) * -(-h // n)
    grid = sum(-(-w // (1 << s)) * -(-h // (1 << s)) for s in range(case["scales"]))
    return 2 * (2 * 48 * gq * gq + grid * case["iterations"] * 3 * per_candidate)


def _stage_work(w, h, case):
    np_ = w * h
    # images in; fields, costs, masks and (at most) the seeds out
    by = 12 * np_ + 2 * (8 + 4) * np_ + 2 * np_ + 20 * np_ / 9
    fl = 4 * case["scales"] * 250 * np_ + _match_flops(w, h, case, 3 * 96)
    return by, fl


def work(case):
    kind, w, h = case["kind"], case["width"], case["height"]
    np_, S, D = w * h, case["scales"], case["max_disp"]
    sgm = (8 * np_, np_ * D * (2 + 8 * 6))
    interp = (20 * np_ / 9 * case["keep"] + 16 * np_, np_ / 9 * case["keep"] * (20 * 160 + 53 * 80) + 60 * np_)
    if kind in ("quad", "host"):
        by, fl = _stage_work(w, h, case)
        if kind == "host":
            by = 12 * np_ + 20 * np_ / 9
    elif kind == "batch":
        by, fl = (sum(t) for t in zip(*(_stage_work(qw, qh, case) for qw, qh in _batch_sizes(case))))
    elif kind == "sgm":
        by, fl = sgm
    elif kind == "interp":
        by, fl = interp
    elif kind == "sift_features":
        # images in, phi out; 16 cells of 9 samples, two norms and divisions,
        # quantisation and projection per descriptor; the covariance
        by = 12 * np_ + 4 * S * 16 * np_
        fl = 4 * S * np_ * (144 + 128 * 6 + 768) + 4 * np_ * 128 * 128
    elif kind == "method":
        by, fl = (a + b + c for a, b, c in zip(_stage_work(w, h, case), sgm, interp))
    else:
        per = 147 * 9 if kind == "sift_match" else 3 * 96
        by = 4 * S * (52 + (16 if kind == "sift_match" else 0)) * np_ + 2 * 12 * np_
        fl = _match_flops(w, h, case, per)
    return {"bytes": float(by), "flops": float(fl)}


# ------------------------------------------------------- the values in 64 bits

def exact(case, seed):
    if case["kind"] == "interp":
        return _exact_interp(case, seed)
    if case["kind"] == "sift_features":
        return _exact_sift(case, seed)
    return None  # whole numbers (the method's dense field depends on all of them)


def _nearest(x, y, sx, sy, k):
    """(squared distance, index) of the k nearest of (sx, sy) to every (x, y), ties to the lower index."""
    d = (x[:, None] - sx[None]) ** 2 + (y[:, None] - sy[None]) ** 2
    key = (d << 20) | torch.arange(sx.numel(), device=DEV)[None]
    v = torch.topk(key, min(k, sx.numel()), dim=1, largest=False, sorted=True)[0] if k > 1 else key.amin(1, True)
    return v >> 20, v & ((1 << 20) - 1)


def _solve(M, b):
    """M x = b for symmetric positive definite batches; b [n, dim, columns]."""
    L = torch.linalg.cholesky(M)
    return torch.cholesky_solve(b, L)


def _exact_interp(case, seed):
    w, h = case["width"], case["height"]
    raw, n = _sparse_seeds(w, h, case["layers"], case["keep"], seed)
    s = raw.cpu().numpy().view(sff.SEED_DTYPE)[:n]
    k_geo, k_motion, alpha, unit = 160, 80, 2.2, 20.0
    f, cx, cy = FOCAL_PER_WIDTH * w, (w - 1) / 2, (h - 1) / 2
    sx, sy = (torch.as_tensor(s[c].astype(np.int64), device=DEV) for c in ("x", "y"))
    u, v, d0, d1 = (torch.as_tensor(s[c].astype(np.float64), device=DEV) for c in ("u", "v", "d0", "d1"))

    def lift(x, y, d):
        z = f * BASELINE / d
        return torch.stack([(x - cx) * z / f, (y - cy) * z / f, z], -1)

    def ridge(M):
        lam = 1e-9 * M.diagonal(dim1=1, dim2=2).sum(1) / M.shape[1] + 1e-300
        r = torch.zeros(M.shape[0], M.shape[1], M.shape[1], dtype=torch.float64, device=DEV)
        k = M.shape[1] - 1
        r[:, range(k), range(k)] = lam[:, None]
        return r

    fx, fy = sx.double(), sy.double()
    moving = torch.nonzero((d0 >= 1) & (d1 >= 1)).ravel()
    X0 = lift(fx[moving], fy[moving], d0[moving])
    X1 = lift((fx + u)[moving], (fy + v)[moving], d1[moving])
    plane = torch.empty((n, 3), dtype=torch.float64, device=DEV)
    A = torch.zeros((n, 4, 3), dtype=torch.float64, device=DEV)
    cen = torch.zeros((n, 3), dtype=torch.float64, device=DEV)
    for a in range(0, n, 2048):
        b = min(n, a + 2048)
        d2, idx = _nearest(sx[a:b], sy[a:b], sx, sy, k_geo)
        wt = torch.exp(-alpha * torch.sqrt(d2.double()) / unit)
        r = torch.stack([fx[idx] - fx[a:b, None], fy[idx] - fy[a:b, None], torch.ones_like(wt)], -1)
        M = torch.einsum("nk,nka,nkb->nab", wt, r, r)
        rhs = torch.einsum("nk,nka,nk->na", wt, r, d0[idx])
        plane[a:b] = _solve(M + ridge(M), rhs[..., None])[..., 0]
        if moving.numel():
            d2, idx = _nearest(sx[a:b], sy[a:b], sx[moving], sy[moving], k_motion)
            wt = torch.exp(-alpha * torch.sqrt(d2.double()) / unit)
            P, Q = X0[idx], X1[idx]
            cen[a:b] = (wt[..., None] * P).sum(1) / wt.sum(1, keepdim=True)
            r = torch.cat([P - cen[a:b, None], torch.ones_like(wt)[..., None]], -1)
            M = torch.einsum("nk,nka,nkb->nab", wt, r, r)
            R = ridge(M)
            A[a:b] = _solve(M + R, torch.einsum("nk,nka,nkj->naj", wt, r, Q) + R[:, :, :3])
    out = torch.zeros((w * h, 4), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 27) // max(1, n))
    for a in range(0, w * h, step) if n else ():
        i = torch.arange(a, min(w * h, a + step), device=DEV)
        x, y = i % w, i // w
        k = _nearest(x, y, sx, sy, 1)[1][:, 0]
        x, y = x.double(), y.double()
        d = (plane[k] * torch.stack([x - fx[k], y - fy[k], torch.ones_like(x)], -1)).sum(1)
        out[i, 2] = out[i, 3] = d
        if moving.numel():
            r = torch.cat([lift(x, y, d.clamp(min=1.0)) - cen[k], torch.ones_like(x)[:, None]], -1)
            p = torch.einsum("na,naj->nj", r, A[k])
            ok = p[:, 2] > 0
            j, p = i[ok], p[ok]
            out[j, 0] = f * p[:, 0] / p[:, 2] + cx - x[ok]
            out[j, 1] = f * p[:, 1] / p[:, 2] + cy - y[ok]
            out[j, 3] = f * BASELINE / p[:, 2]
    return out.view(h, w, 4)


def _exact_sift(case, seed):
    w, h, S = case["width"], case["height"], case["scales"]
    images = _scene(w, h, case["layers"], seed)[0]
    ys, xs = torch.arange(h, device=DEV), torch.arange(w, device=DEV)
    rx, ry = (1, 1, 0, -1, -1, -1, 0, 1, 1), (0, 1, 1, 1, 0, -1, -1, -1, 0)

    def descriptors(img, n):
        img = img.long()
        if n > 1:  # n x n box mean with clamped positions, rounded half up
            t = sum(img[(ys + j).clamp(0, h - 1)] for j in range(-n // 2, n // 2))
            t = sum(t[:, (xs + i).clamp(0, w - 1)] for i in range(-n // 2, n // 2))
            img = (t + n * n // 2) // (n * n)
        g = (img[..., 0] + 2 * img[..., 1] + img[..., 2] + 2) >> 2
        dx = g[:, (xs + n).clamp(max=w - 1)] - g[:, (xs - n).clamp(min=0)]
        dy = g[(ys + n).clamp(max=h - 1)] - g[(ys - n).clamp(min=0)]
        mag = torch.sqrt((dx * dx + dy * dy).double())
        part = torch.stack([torch.where((rx[k] * dy - ry[k] * dx >= 0) & (rx[k + 1] * dy - ry[k + 1] * dx < 0), mag, 0.0)
                            for k in range(8)], -1)
        cells = []
        for cy in range(4):
            rows = sum(part[(ys + (3 * cy + j - 6) * n).clamp(0, h - 1)] for j in range(3))
            for cx in range(4):
                cells.append(sum(rows[:, (xs + (3 * cx + i - 6) * n).clamp(0, w - 1)] for i in range(3)))
        d = torch.cat(cells, -1)
        nr = d.norm(dim=-1, keepdim=True)
        d = torch.where(nr > 0, d / nr, d).clamp(max=0.2)
        nr = d.norm(dim=-1, keepdim=True)
        d = torch.where(nr > 0, d / nr, torch.zeros_like(d))
        return torch.floor(d * 512 + 0.5).clamp(max=255)

    out = [torch.zeros((S, h, w, 4), dtype=torch.float64, device=DEV) for _ in range(4)]
    axes = mean = None
    for s in range(S):
        desc = [descriptors(im, 1 << s) for im in images]
        if s == 0:
            q = torch.cat([d.view(-1, 128) for d in desc])
            m, C = q.mean(0), q.T @ q / q.shape[0]
            C = (C - m[:, None] * m[None]).cpu().numpy()
            ax = []
            for _ in range(3):
                v = np.ones(128)
                for _ in range(200):
                    v = C @ v
                    for e in ax:
                        v = v - (e @ v) * e
                    v = v / np.linalg.norm(v) if np.linalg.norm(v) > 0 else 0 * v
                ax.append(v * (-1.0 if v[np.argmax(np.abs(v))] < 0 else 1.0))
            axes, mean = torch.as_tensor(np.stack(ax), device=DEV), m
        for o, d in zip(out, desc):
            o[s, ..., :3] = (d - mean) @ axes.T
    return out
