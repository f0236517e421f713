"""Cases of the layer-editing path, for measuring it through the package's public entry points.

A case names one kind of call a program makes on a model, with its sizes:

  strokes   sphere strokes on a label layer, one lcl_select_sphere call
  values    sphere strokes on a numeric layer, one lcl_numeric_sphere call
  lassos    screen lassos on a label layer, one lcl_select_lasso call each
  tool      the paper's editing tool (window with an inscribed circle), texture padding included
  batch     queued strokes and lassos of several models, one lcl_batch_edit call
  atlas     the UV atlas of a mesh, one lcl_atlas_build call
  depth     the depth map of a camera, one lcl_depth_render call
  query     the overlay of two label layers and the result's per-label area
  analysis  the difference of two numeric layers, a selection by value from it and its zonal statistics

Models are vessels (surfaces of revolution with a seeded relief) with a cylindrical unwrap, which
covers the whole texture, or cut into square charts with gutters between them, as the atlases of
scanned models are.  Everything follows from the case and the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2501_14807_gb300 import lcl

GRID_MAX = (1 << 21) - 1
DIAG = 4.2      # about the bounding box diagonal of a vessel (radius up to 1.3, height 2)
SURFACE = 14.0  # about its surface area
U8, U16 = 1, 2
VALUE_BYTES = {"u8": 1, "i8": 1, "u16": 2, "i16": 2, "f16": 2, "u32": 4, "i32": 4, "f32": 4}


def listed():
    return [
        # one click of a brush on a small model: the call itself, its launches and little else
        dict(name="stroke-1024-u8", kind="strokes", w=1024, h=1024, tile=32, mesh="cylinder", tris=20000, bytes=U8,
             n=1, r_lo=0.02, r_hi=0.02, pad=0),
        # many small strokes on a layer of a chart atlas with many labels
        dict(name="strokes-4096-u16", kind="strokes", w=4096, h=4096, tile=32, mesh="charts", tris=1000000, bytes=U16,
             n=625, r_lo=0.001, r_hi=0.05, pad=0),
        # strokes of every radius on a layer of the largest texture
        dict(name="strokes-16384-u8", kind="strokes", w=16384, h=16384, tile=32, mesh="cylinder", tris=8000000,
             bytes=U8, n=250, r_lo=0.01, r_hi=0.30, pad=0),
        # value strokes on an integer layer whose sides fit neither tiles nor words
        dict(name="values-5004x3310-i16", kind="values", w=5004, h=3310, tile=16, mesh="charts", tris=400000,
             type="i16", n=40, r_lo=0.01, r_hi=0.10, pad=0),
        # lassos drawn on a chart atlas with many labels
        dict(name="lassos-4096-u16", kind="lassos", w=4096, h=4096, tile=32, mesh="charts", tris=1000000, bytes=U16,
             n=12, screen_w=2048, screen_h=2048, pad=0),
        # lassos drawn on the largest texture
        dict(name="lassos-16384-u8", kind="lassos", w=16384, h=16384, tile=32, mesh="cylinder", tris=8000000, bytes=U8,
             n=5, screen_w=2048, screen_h=2048, pad=0),
        # one application of the paper's tool with padding, the operation the paper times
        dict(name="tool-8192-u8", kind="tool", w=8192, h=8192, tile=32, mesh="charts", tris=313600, bytes=U8,
             radius_px=70, screen_w=1920, screen_h=1080, pad=2),
        # one epoch of a server: the queued edits of its models
        dict(name="batch-24", kind="batch", models=24, tri_lo=5000, tri_hi=500000, spheres=48, lassos=16, screen=1024),
        # a model arrives: its atlas
        dict(name="atlas-16384", kind="atlas", w=16384, h=16384, tile=32, mesh="cylinder", tris=8000000),
        # the camera moved: its depth map
        dict(name="depth-2048-8m", kind="depth", w=4096, h=4096, tile=32, mesh="cylinder", tris=8000000, screen_w=2048,
             screen_h=2048),
        # how much surface two layers share, by label
        dict(name="query-16384-u8", kind="query", w=16384, h=16384, tile=32, mesh="cylinder", tris=8000000, bytes=U8,
             labels=256, op="xor"),
        # change of a float property between two surveys, where it is large and what it is per zone
        dict(name="analysis-8192-f32", kind="analysis", w=8192, h=8192, tile=32, mesh="charts", tris=2000000,
             type="f32", bytes=U8, zones=40),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _texture(rng, hi=16384):
    """Sides of a texture of about hi^2 texels at most, square ones and odd ones (widths are multiples of 4)."""
    if rng.random() < 0.4:
        side = 2 ** rng.randint(9, int(math.log2(hi)))
        return side, side, rng.choice([16, 32, 32, 64])
    side = _log(rng, 512, hi / 1.3)
    aspect = rng.uniform(0.6, 1.3)
    w, h = min(hi, int(side * aspect)), min(hi, int(side / aspect))
    return w // 4 * 4, h, rng.choice([16, 32, 32, 64])


def _model(rng, hi=16384):
    w, h, tile = _texture(rng, hi)
    most = max(5000.0, min(8e6, 0.03 * w * h))
    return dict(w=w, h=h, tile=tile, mesh=rng.choice(["cylinder", "charts"]), tris=int(_log(rng, most / 20, most)))


def draw(rng):
    kind = rng.choice(["strokes", "strokes", "values", "lassos", "lassos", "tool", "batch", "atlas", "depth", "query",
                       "analysis"])
    if kind == "strokes":
        m = _model(rng)
        most = max(1.0, min(1000.0, 250 * 16384.0 ** 2 / (m["w"] * m["h"])))
        pad = rng.choice([0, 0, 0, 1, 2]) if m["w"] * m["h"] <= 4096 ** 2 else 0
        n = int(_log(rng, 1, 16 if pad else most))
        r_lo = _log(rng, 0.001, 0.05)
        return dict(kind=kind, **m, bytes=rng.choice([U8, U16]), n=n, r_lo=r_lo, r_hi=min(0.3, r_lo * _log(rng, 1, 30)),
                    pad=pad)
    if kind == "values":
        m = _model(rng, 8192)
        r_lo = _log(rng, 0.005, 0.05)
        return dict(kind=kind, **m, type=rng.choice(["u8", "i16", "f16", "f32", "f32"]), n=int(_log(rng, 1, 64)),
                    r_lo=r_lo, r_hi=min(0.2, r_lo * _log(rng, 1, 10)), pad=0)
    if kind in ("lassos", "tool"):
        m = _model(rng)
        screen = dict(screen_w=rng.choice([800, 1280, 1920, 2048]), screen_h=rng.choice([600, 1080, 2048]))
        if kind == "lassos":
            pad = rng.choice([0, 0, 0, 2]) if m["w"] * m["h"] <= 4096 ** 2 else 0
            return dict(kind=kind, **m, bytes=rng.choice([U8, U16]), n=int(_log(rng, 1, 4 if pad else 12)), **screen,
                        pad=pad)
        return dict(kind=kind, **m, bytes=rng.choice([U8, U16]), radius_px=int(_log(rng, 10, 200)), **screen,
                    pad=rng.choice([0, 1, 2, 2, 4]))
    if kind == "batch":
        lo = _log(rng, 5e3, 1e5)
        return dict(kind=kind, models=int(_log(rng, 1, 24)), tri_lo=int(lo), tri_hi=int(min(5e5, lo * _log(rng, 1, 50))),
                    spheres=rng.randint(1, 48), lassos=rng.randint(0, 16), screen=rng.choice([512, 1024]))
    if kind == "atlas":
        return dict(kind=kind, **_model(rng))
    if kind == "depth":
        return dict(kind=kind, **_model(rng, 4096) | dict(tris=int(_log(rng, 2e4, 8e6))),
                    screen_w=rng.choice([800, 1920, 2048]), screen_h=rng.choice([600, 1080, 2048]))
    if kind == "query":
        width = rng.choice([U8, U16])
        return dict(kind=kind, **_model(rng), bytes=width, labels=rng.choice([16, 256] if width == U8 else [256, 1024]),
                    op=rng.choice(["and", "or", "xor", "mask"]))
    return dict(kind=kind, **_model(rng, 8192), type=rng.choice(["i16", "f16", "f32", "f32"]),
                bytes=rng.choice([U8, U16]), zones=rng.choice([1, 12, 40, 200]))


# ---- models ---------------------------------------------------------------------------------------------

def _relief(seed):
    """Phases and frequencies of a vessel's relief: whole numbers of waves around it, so that its seam closes."""
    rng = np.random.default_rng([7, seed])
    return [(int(rng.integers(3, 9) * 4 ** k), float(rng.uniform(4, 9) * 4 ** k), float(rng.uniform(0, 6.28)),
             float(rng.uniform(0, 6.28)), 0.012 / 3 ** k) for k in range(3)]


def _surface(theta, h, relief, sin, cos, stack):
    r = 1.0 + 0.3 * sin(3.0 * math.pi * h)
    for a, b, p, q, amp in relief:
        r = r + amp * sin(a * theta + p) * sin(b * math.pi * h + q)
    return stack([r * cos(theta), r * sin(theta), 2.0 * h], -1)


def _vessel(case, seed, tris=None, w=None, h=None):
    """The case's vessel on the GPU, as lcl.Mesh.  Charts are blocks of 16 x 16 quads on a regular grid with
    gutters of four texels."""
    tris, w, h = tris or case["tris"], w or case["w"], h or case["h"]
    dev = "cuda"
    n_h = max(16, int(math.sqrt(tris / 4)))
    n_t = max(32, tris // (2 * n_h))
    if case.get("mesh") == "charts":
        n_h, n_t = max(16, n_h // 16 * 16), max(16, n_t // 16 * 16)
    theta = torch.arange(n_t, device=dev, dtype=torch.float64) * (2.0 * math.pi / n_t)
    hh = torch.arange(n_h + 1, device=dev, dtype=torch.float64) / n_h
    pos = _surface(theta[None, :].expand(n_h + 1, n_t), hh[:, None].expand(n_h + 1, n_t), _relief(seed), torch.sin,
                   torch.cos, torch.stack).reshape(-1, 3).to(torch.float32).contiguous()
    j, i = torch.meshgrid(torch.arange(n_h, device=dev), torch.arange(n_t, device=dev), indexing="ij")
    i, j = i.reshape(-1), j.reshape(-1)
    right = (i + 1) % n_t
    p = [j * n_t + i, j * n_t + right, (j + 1) * n_t + right, (j + 1) * n_t + i]
    if case.get("mesh") == "charts":
        c = 16
        ci, cj, li, lj = i // c, j // c, i % c, j % c
        nx, ny = n_t // c, n_h // c
        base = (cj * nx + ci) * (c + 1) * (c + 1)
        u = [base + lj * (c + 1) + li, base + lj * (c + 1) + li + 1, base + (lj + 1) * (c + 1) + li + 1,
             base + (lj + 1) * (c + 1) + li]
        step = torch.arange(c + 1, device=dev, dtype=torch.float64) / c
        gx, gy = min(2.0, 0.1 * w / nx), min(2.0, 0.1 * h / ny)
        cx, cy = w / nx, h / ny  # a chart's cell in texels
        uu = (torch.arange(nx, device=dev, dtype=torch.float64)[:, None] * cx + gx + step[None, :] * (cx - 2 * gx)) / w
        vv = (torch.arange(ny, device=dev, dtype=torch.float64)[:, None] * cy + gy + step[None, :] * (cy - 2 * gy)) / h
        shape = (ny, nx, c + 1, c + 1)
        uv = torch.stack([uu[None, :, None, :].expand(shape), vv[:, None, :, None].expand(shape)], -1)
    else:
        s = n_t + 1
        u = [j * s + i, j * s + i + 1, (j + 1) * s + i + 1, (j + 1) * s + i]
        uu = torch.arange(n_t + 1, device=dev, dtype=torch.float64) / n_t
        uv = torch.stack([uu[None, :].expand(n_h + 1, s), hh[:, None].expand(n_h + 1, s)], -1)
    uv = uv.reshape(-1, 2).to(torch.float32).contiguous()

    def triangles(q):
        return torch.stack([torch.stack([q[0], q[1], q[2]], 1), torch.stack([q[0], q[2], q[3]], 1)],
                           1).reshape(-1, 3).to(torch.int32).contiguous()

    return lcl.Mesh(pos, uv, triangles(p), triangles(u))


def _atlas(mesh, w, h, tile):
    return lcl.lcl_atlas_build(mesh, lcl.Atlas(w, h, tile, mesh.n_tri))


def _on_surface(rng, n, seed):
    return _surface(rng.uniform(0, 2 * math.pi, n), rng.uniform(0, 1, n), _relief(seed), np.sin, np.cos, np.stack)


def _spheres(atlas, rng, seed, n, r_lo, r_hi, label_hi, pad=0, erase=0.0):
    """Stroke records with centres on the surface; radii are fractions of the diagonal, log-uniform."""
    r = np.exp(rng.uniform(math.log(r_lo), math.log(max(r_hi, r_lo)), n)) * DIAG
    recs = lcl.lcl_quantize_spheres(atlas, _on_surface(rng, n, seed), r, rng.integers(1, label_hi + 1, n))
    recs["flags"] = lcl.pad_flags(pad, pad) | np.where(rng.random(n) < erase, lcl.LCL_ERASE, 0)
    return recs


def _camera(atlas, rng, width, height):
    """A camera on an orbit around the vessel, and its view-projection matrix."""
    az, el = rng.uniform(0, 2 * math.pi), math.radians(rng.uniform(-30, 60))
    dist, reach = 2.5 * DIAG / 2, 1.1 * DIAG / 2
    eye = np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)]) * dist
    f = -eye / np.linalg.norm(eye)
    s = np.cross(f, [0.0, 0.0, 1.0])
    s /= np.linalg.norm(s)
    view = np.eye(4)
    view[0, :3], view[1, :3], view[2, :3] = s, np.cross(s, f), -f
    view[:3, 3] = -view[:3, :3] @ (eye + np.array([0.0, 0.0, 1.0]))  # it looks at the middle of the height
    near, far, c = dist - reach, dist + reach, 1.0 / math.tan(math.radians(20))
    proj = np.zeros((4, 4))
    proj[0, 0], proj[1, 1], proj[2, 2] = c * height / width, c, far / (near - far)
    proj[2, 3], proj[3, 2] = near * far / (near - far), -1.0
    vp = proj @ view
    return lcl.lcl_camera_from_vp(atlas, vp, width, height), vp


def _view(mesh, atlas, rng, width, height):
    cam, vp = _camera(atlas, rng, width, height)
    depth = torch.empty((height, width), dtype=torch.float32, device="cuda")
    lcl.lcl_depth_render(mesh, atlas, cam, depth)
    return cam, vp, depth


def _screen_point(vp, rng, seed, width, height):
    """A surface point's place on the screen."""
    for _ in range(50):
        q = vp @ np.append(_on_surface(rng, 1, seed)[0], 1.0)
        x, y = (q[0] / q[3] * 0.5 + 0.5) * width, (q[1] / q[3] * 0.5 + 0.5) * height
        if 0 <= x < width and 0 <= y < height:
            break
    return float(x), float(y)


def _star(rng, centre, width, height):
    """A hand-drawn outline: 8 to 64 vertices around the centre at 5 to 40% of the screen."""
    n = int(rng.integers(8, 65))
    ang = 2 * math.pi * np.arange(n) / n + rng.uniform(-0.95, 0.95, n) * math.pi / n
    rad = rng.uniform(0.3, 1.0, n) * rng.uniform(0.05, 0.40) * min(width, height)
    return np.stack([centre[0] + rad * np.cos(ang), centre[1] + rad * np.sin(ang)], 1).astype(np.float32)


def _layer(h, w, size):
    return torch.zeros((h, w), dtype=torch.uint8 if size == U8 else torch.int16, device="cuda")


def _edited(atlas, rng, seed, size, n, label_hi):
    """A label layer as some editing leaves it."""
    layer = _layer(atlas.height, atlas.width, size)
    lcl.lcl_select_sphere(atlas, layer, _spheres(atlas, rng, seed, n, 0.02, 0.2, label_hi))
    return layer


def _values(atlas, rng, gen, ntype):
    """A numeric layer: a smooth property with measuring noise, known on nine tenths of the texture."""
    w, h = atlas.width, atlas.height
    layer = lcl.NumericLayer(w, h, ntype)
    x = torch.arange(w, device="cuda", dtype=torch.float32) * float(rng.uniform(4, 12) / w)
    y = torch.arange(h, device="cuda", dtype=torch.float32) * float(rng.uniform(4, 12) / h)
    v = torch.randn((h, w), device="cuda", generator=gen).mul_(0.1)
    v.add_(torch.sin(x)[None, :]).add_(torch.cos(y)[:, None]).add_(3.0)
    layer.data.copy_(v if ntype in ("f16", "f32") else v.mul_(8.0 if VALUE_BYTES[ntype] == 1 else 1000.0))
    words = layer.mask.numel()
    known = torch.rand(words // 16 + 1, device="cuda", generator=gen) < 0.9
    layer.mask.copy_(torch.where(known, -1, 0).repeat_interleave(16)[:words])
    return layer


# ---- prepare and run ------------------------------------------------------------------------------------

def prepare(case, seed):
    rng = np.random.default_rng([11, seed])
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, seed, rng)
    w, h, tile = case["w"], case["h"], case["tile"]
    mesh = _vessel(case, seed)
    if kind == "atlas":
        ws = torch.empty(lcl.lcl_atlas_workspace_bytes(mesh, w, h), dtype=torch.uint8, device="cuda")
        return dict(kind=kind, mesh=mesh, atlas=lcl.Atlas(w, h, tile, mesh.n_tri), ws=ws)
    atlas = _atlas(mesh, w, h, tile)
    s = dict(kind=kind, atlas=atlas)
    if kind in ("strokes", "values"):
        if kind == "strokes":
            s["layer"], label_hi = _layer(h, w, case["bytes"]), 255 if case["bytes"] == U8 else 1000
        else:
            s["layer"], label_hi = lcl.NumericLayer(w, h, case["type"]), 100
        s["strokes"] = _spheres(atlas, rng, seed, case["n"], case["r_lo"], case["r_hi"], label_hi, case["pad"],
                                0.1 if kind == "values" else 0.0)
        if kind == "values" and case["type"] in ("f16", "f32"):  # a value travels as its bits
            v = s["strokes"]["label"].astype(np.float16 if case["type"] == "f16" else np.float32)
            s["strokes"]["label"] = v.view(np.uint16 if case["type"] == "f16" else np.uint32)
        s["hits"] = torch.zeros(case["n"], dtype=torch.int64, device="cuda")
        s["ws"] = torch.empty(lcl.lcl_select_workspace_bytes(atlas, case["n"]), dtype=torch.uint8, device="cuda")
        return s
    if kind in ("lassos", "tool"):
        views = [_view(mesh, atlas, rng, case["screen_w"], case["screen_h"]) for _ in range(1 if kind == "tool" else 2)]
        s["layer"] = _layer(h, w, case["bytes"])
        s["ws"] = torch.empty(lcl.lcl_select_workspace_bytes(atlas, 1), dtype=torch.uint8, device="cuda")
        n = case.get("n", 1)
        s["hits"] = torch.zeros(n, dtype=torch.int64, device="cuda")
        s["edits"] = []
        for k in range(n):
            cam, vp, depth = views[k % len(views)]
            at = _screen_point(vp, rng, seed, case["screen_w"], case["screen_h"])
            label = int(rng.integers(1, 256))
            if kind == "tool":
                shape = lcl.make_tool(at, (2 * case["radius_px"], 2 * case["radius_px"]),
                                      flags=lcl.pad_flags(case["pad"], case["pad"]))
            else:
                shape = _star(rng, at, case["screen_w"], case["screen_h"])
            s["edits"].append((cam, depth, shape, label, s["hits"][k:k + 1]))
        s["flags"] = lcl.pad_flags(case["pad"], case["pad"])  # a lasso's; a tool carries its own
        return s
    if kind == "depth":
        s["mesh"] = mesh
        s["cam"], _ = _camera(atlas, rng, case["screen_w"], case["screen_h"])
        s["depth"] = torch.empty((case["screen_h"], case["screen_w"]), dtype=torch.float32, device="cuda")
        s["ws"] = torch.empty(lcl.lcl_depth_workspace_bytes(mesh, case["screen_w"], case["screen_h"]),
                              dtype=torch.uint8, device="cuda")
        return s
    if kind == "query":
        hi = min(case["labels"], 255 if case["bytes"] == U8 else 1000)
        s["a"], s["b"] = (_edited(atlas, rng, seed, case["bytes"], 60, hi) for _ in range(2))
        s["out"] = torch.empty_like(s["a"])
        s["op"], s["labels"] = case["op"], case["labels"]
        s["count"], s["area"] = (torch.empty(case["labels"], dtype=torch.int64, device="cuda") for _ in range(2))
        return s
    s["a"], s["b"] = (_values(atlas, rng, gen, case["type"]) for _ in range(2))
    s["out"] = lcl.NumericLayer(w, h, case["type"])
    one_zone = case["zones"] == 1
    s["zones"] = None if one_zone else _edited(atlas, rng, seed, case["bytes"], 2 * case["zones"], case["zones"] - 1)
    s["n_zones"] = case["zones"]
    s["marked"] = _layer(h, w, case["bytes"])
    s["threshold"] = {"f32": int(np.float32(0.5).view(np.uint32)), "f16": int(np.float16(0.5).view(np.uint16))}.get(
        case["type"], 500)
    s["hits"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    s["stats"] = torch.empty(48 * case["zones"], dtype=torch.uint8, device="cuda")
    return s


def _prepare_batch(case, seed, rng):
    models, queues = [], []
    # sizes spread over the range, the large ones among the small ones; the same for every seed
    order = np.random.default_rng(5).permutation(case["models"])
    for k in range(case["models"]):
        tris = int(case["tri_lo"] * (case["tri_hi"] / case["tri_lo"]) ** ((order[k] + 0.5) / case["models"]))
        side = int(2 ** np.clip(round(math.log2(math.sqrt(8.0 * tris))), 9, 11))
        sub = 1000 * seed + k
        mesh = _vessel(dict(mesh=("cylinder", "charts")[k % 2]), sub, tris, side, side)
        atlas = _atlas(mesh, side, side, 32)
        views = [_view(mesh, atlas, rng, case["screen"], case["screen"]) for _ in range(2)]
        queue = [("sphere", r) for r in _spheres(atlas, rng, sub, case["spheres"], 0.005, 0.10, 255)]
        for j in range(case["lassos"]):
            cam, vp, depth = views[j % 2]
            at = _screen_point(vp, rng, sub, case["screen"], case["screen"])
            queue.append(("lasso", (cam, depth, _star(rng, at, case["screen"], case["screen"]),
                                    int(rng.integers(1, 256)), lcl.DEFAULT_BIAS)))
        queues.append([queue[i] for i in rng.permutation(len(queue))])
        models.append((atlas, _layer(side, side, U8)))
    return dict(kind="batch", batch=lcl.Batch(models, queues), layers=[layer for _, layer in models])


def run(s):
    kind = s["kind"]
    if kind == "strokes":
        lcl.lcl_select_sphere(s["atlas"], s["layer"], s["strokes"], s["hits"], s["ws"])
        return {"layer": s["layer"], "hits": s["hits"]}
    if kind == "values":
        lcl.lcl_numeric_sphere(s["atlas"], s["layer"], s["strokes"], s["hits"], s["ws"])
        return {"data": s["layer"].data, "mask": s["layer"].mask, "hits": s["hits"]}
    if kind == "lassos":
        for cam, depth, poly, label, hits in s["edits"]:
            lcl.lcl_select_lasso(s["atlas"], s["layer"], cam, depth, poly, label, hits_out=hits, workspace=s["ws"],
                                 flags=s["flags"])
        return {"layer": s["layer"], "hits": s["hits"]}
    if kind == "tool":
        for cam, depth, tool, label, hits in s["edits"]:
            lcl.lcl_select_tool(s["atlas"], s["layer"], cam, depth, tool, label, hits_out=hits, workspace=s["ws"])
        return {"layer": s["layer"], "hits": s["hits"]}
    if kind == "batch":
        lcl.lcl_batch_edit(s["batch"])
        return {"layers": s["layers"]}
    if kind == "atlas":
        a = lcl.lcl_atlas_build(s["mesh"], s["atlas"], s["ws"])
        return {"planes": [a.plane(p) for p in ("pos_x", "pos_y", "pos_z", "tri")], "cover": a.cover(),
                "tiles": a.tile_box(), "supers": a.super_box(), "area_w": a.area_w(), "bbox_min": a.bbox_min,
                "scale": a.scale}
    if kind == "depth":
        return {"depth": lcl.lcl_depth_render(s["mesh"], s["atlas"], s["cam"], s["depth"], s["ws"])}
    if kind == "query":
        lcl.lcl_overlay(s["atlas"], s["a"], s["b"], s["out"], s["op"])
        lcl.lcl_label_area(s["atlas"], s["out"], s["labels"], s["count"], s["area"])
        return {"out": s["out"], "count": s["count"], "area": s["area"]}
    lcl.lcl_numeric_arith(s["atlas"], s["a"], s["b"], s["out"], "sub")
    lcl.lcl_numeric_select(s["atlas"], s["out"], "gt", s["threshold"], s["marked"], 7, s["hits"])
    lcl.lcl_numeric_stats(s["atlas"], s["out"], s["zones"], s["n_zones"], s["stats"])
    ints, floats = s["stats"].view(torch.int64).view(-1, 6), s["stats"].view(torch.float64).view(-1, 6)
    return {"data": s["out"].data, "mask": s["out"].mask, "marked": s["marked"], "hits": s["hits"],
            "counts": ints[:, :2], "sums": floats[:, 2:]}


# ---- what a pass cannot do without ----------------------------------------------------------------------

def _covered(case):
    return case["w"] * case["h"] * (0.8 if case["mesh"] == "charts" else 1.0)


def _stroke_share(f):
    """About the share of the surface within a radius of f diagonals of a surface point."""
    return min(0.95, math.pi * (f * DIAG) ** 2 / SURFACE)


def _union(n, r_lo, r_hi):
    """About the share of the surface that n strokes with log-uniform radii reach together."""
    steps = 64
    miss = [math.log(1.0 - _stroke_share(r_lo * (r_hi / r_lo) ** ((k + 0.5) / steps))) for k in range(steps)]
    return 1.0 - math.exp(n * sum(miss) / steps)


LASSO_SHARE = 0.02  # about the share of the surface that one lasso of the drawn sizes selects


def work(case):
    kind = case["kind"]
    if kind in ("strokes", "values"):
        texels = _covered(case) * _union(case["n"], case["r_lo"], case["r_hi"])
        size = case["bytes"] if kind == "strokes" else VALUE_BYTES[case["type"]] + 0.125
        return {"bytes": texels * (12 + size) + 32 * case["n"], "flops": 8 * texels}
    if kind in ("lassos", "tool"):
        pixels = case["screen_w"] * case["screen_h"]
        if kind == "lassos":
            share, seen = 1.0 - (1.0 - LASSO_SHARE) ** case["n"], 0.06 * pixels * case["n"]
        else:
            seen = math.pi * case["radius_px"] ** 2
            share = min(0.4, seen / (0.3 * case["screen_h"] ** 2) * 0.4)  # the vessel fills part of the height
        texels = _covered(case) * share
        return {"bytes": texels * (12 + case["bytes"]) + 4 * seen, "flops": 40 * texels}
    if kind == "batch":
        tris = math.sqrt(case["tri_lo"] * case["tri_hi"])
        texels = case["models"] * min(2048.0 ** 2, 8 * tris) * 0.9
        share = 1.0 - (1.0 - _union(case["spheres"], 0.005, 0.10)) * (1.0 - LASSO_SHARE) ** case["lassos"]
        return {"bytes": texels * share * 13 + case["models"] * 4 * case["screen"] ** 2 * 0.3,
                "flops": 40 * texels * share}
    corners = case["tris"] / 2
    if kind == "atlas":
        return {"bytes": 12 * corners + 8 * corners + 24 * case["tris"] + case["w"] * case["h"] * 16.125 +
                8 * case["tris"], "flops": 40 * _covered(case)}
    if kind == "depth":
        pixels = case["screen_w"] * case["screen_h"]
        return {"bytes": 12 * corners + 12 * case["tris"] + 4 * pixels, "flops": 40 * corners + 20 * pixels}
    texels = case["w"] * case["h"]
    if kind == "query":
        return {"bytes": texels * (3 * case["bytes"] + 0.125 + 4) + 8 * case["tris"] + 16 * case["labels"],
                "flops": 2 * texels}
    v = VALUE_BYTES[case["type"]]
    zones = 0 if case["zones"] == 1 else case["bytes"]
    return {"bytes": texels * (3 * v + 0.5 + 4 + zones + 0.1 * case["bytes"]) + 8 * case["tris"] + 48 * case["zones"],
            "flops": 4 * texels}


# ---- the computed numbers in 64 bits --------------------------------------------------------------------

def _exact_depth(s):
    """The depth map from its definition: grid positions projected in binary32, snapped to 1/256 pixel, and per
    covered pixel centre the smallest depth interpolated in 64 bits."""
    m, c = s["mesh"], s["cam"]
    mat = torch.tensor(list(c.m), dtype=torch.float32).tolist()
    lo = torch.tensor(s["atlas"].bbox_min.astype(np.float64), device="cuda")
    q = torch.floor((m.pos.double() - lo) * s["atlas"].scale + 0.5).clamp(0, GRID_MAX).float()

    def row(k):
        return ((q[:, 0] * mat[k] + q[:, 1] * mat[k + 1]) + q[:, 2] * mat[k + 2]) + mat[k + 3]

    cw = row(12)
    z = row(8) / cw
    x = torch.round((row(0) / cw * 0.5 + 0.5) * float(c.width) * 256.0).long()
    y = torch.round((row(4) / cw * 0.5 + 0.5) * float(c.height) * 256.0).long()
    kept = (cw > 0) & (z >= 0) & (z <= 1) & (x.abs() <= 1 << 28) & (y.abs() <= 1 << 28)
    depth = torch.full((c.height * c.width,), math.inf, dtype=torch.float64, device="cuda")
    for tri in m.tri_pos.long().split(1 << 20):
        tri = tri[kept[tri].all(1)]
        X, Y, Z = x[tri], y[tri], z[tri].double()
        A = (X[:, 1] - X[:, 0]) * (Y[:, 2] - Y[:, 0]) - (Y[:, 1] - Y[:, 0]) * (X[:, 2] - X[:, 0])
        order = torch.where((A < 0)[:, None], torch.tensor([0, 2, 1], device="cuda"), torch.tensor([0, 1, 2], device="cuda"))
        X, Y, Z, A = X.gather(1, order), Y.gather(1, order), Z.gather(1, order), A.abs()
        i0, i1 = ((X.amin(1) + 127) // 256).clamp(min=0), ((X.amax(1) - 128) // 256).clamp(max=c.width - 1)
        j0, j1 = ((Y.amin(1) + 127) // 256).clamp(min=0), ((Y.amax(1) - 128) // 256).clamp(max=c.height - 1)
        n = torch.where((A > 0) & (i1 >= i0) & (j1 >= j0), (i1 - i0 + 1) * (j1 - j0 + 1), 0)
        t = torch.repeat_interleave(torch.arange(len(n), device="cuda"), n)
        k = torch.arange(len(t), device="cuda") - (torch.cumsum(n, 0) - n)[t]
        wide = (i1 - i0 + 1)[t]
        i, j = i0[t] + k % wide, j0[t] + k // wide
        px, py = 256 * i + 128, 256 * j + 128
        inside, total = None, 0.0
        for e in range(3):  # the edge opposite corner e
            ax, ay, bx, by = X[t, (e + 1) % 3], Y[t, (e + 1) % 3], X[t, (e + 2) % 3], Y[t, (e + 2) % 3]
            weight = (bx - ax) * (py - ay) - (by - ay) * (px - ax)
            owned = (by < ay) | ((by == ay) & (bx < ax))
            ok = (weight > 0) | ((weight == 0) & owned)
            inside = ok if inside is None else inside & ok
            total = total + weight.double() * Z[t, e]
        depth.scatter_reduce_(0, (j * c.width + i)[inside], (total / A[t].double())[inside], "amin")
    return depth.view(c.height, c.width)


def _bits(words, n):
    w = words[:(n + 31) // 32]
    return ((w[:, None] >> torch.arange(32, device=w.device, dtype=torch.int32)) & 1).bool().reshape(-1)[:n]


def _exact_analysis(case, s):
    n = case["w"] * case["h"]
    cover = _bits(s["atlas"].cover(), n)
    valid = _bits(s["a"].mask, n) & _bits(s["b"].mask, n) & cover
    d = torch.where(valid, s["a"].data.reshape(-1).double() - s["b"].data.reshape(-1).double(), 0.0)
    if case["type"] == "i16":
        d = (d + 32768) % 65536 - 32768
    data = d.view(case["h"], case["w"])
    # the statistics are of the stored layer, so of the differences rounded to its type
    v = d if case["type"] == "i16" else d.to(s["a"].data.dtype).double()
    zone = torch.zeros(n, dtype=torch.int64, device="cuda") if s["zones"] is None else s["zones"].reshape(-1).long()
    at = valid & (zone < s["n_zones"])
    zone, v, tri = zone[at], v[at], s["atlas"].plane("tri").reshape(-1)[at].long()
    area = s["atlas"].area_w()[tri].double()
    new = lambda fill: torch.full((s["n_zones"],), fill, dtype=torch.float64, device="cuda")  # noqa: E731
    sums = torch.stack([new(math.inf).scatter_reduce(0, zone, v, "amin"),
                        new(-math.inf).scatter_reduce(0, zone, v, "amax"),
                        new(0.0).index_add(0, zone, v), new(0.0).index_add(0, zone, v * area)], 1)
    return {"data": data if case["type"] != "i16" else None, "mask": None, "marked": None, "hits": None, "counts": None,
            "sums": sums}


def exact(case, seed):
    if case["kind"] not in ("depth", "analysis", "atlas"):
        return None  # labels, values that are copied, and counts
    s = prepare(case, seed)
    if case["kind"] == "depth":
        return {"depth": _exact_depth(s)}
    if case["kind"] == "analysis":
        return _exact_analysis(case, s)
    lo, hi = s["mesh"].pos.double().amin(0), s["mesh"].pos.double().amax(0)
    return {"planes": [None] * 4, "cover": None, "tiles": None, "supers": None, "area_w": None, "bbox_min": lo,
            "scale": GRID_MAX / float((hi - lo).max())}
