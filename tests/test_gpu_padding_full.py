"""Padded edits on tiles without uncovered texels (csrc/select.cu), which take the route of edits without padding,
beside tiles with them: textures covered whole, covered but for their last rows, and charts, tiles of every side,
sides that end inside a tile, against the oracle; and a padded stroke on a covered texture costs about what it
costs without padding."""
import os
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, sphere_recs, to_dev, to_np
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu

SHAPES = [(64, 40, 8), (300, 170, 16), (256, 256, 32), (204, 130, 32), (384, 256, 128), (160, 150, 64)]
PADS = [(1, 1), (8, 8), (8, 1), (1, 8), (3, 0)]


def covered(rows=1.0):
    mesh = synth.vessel_cylindrical(96, 48, noise_amp=0.03, seed=5)
    uv = mesh.uv.copy()
    uv[:, 1] *= np.float32(rows)
    return synth.Mesh(mesh.pos, uv, mesh.tri_pos, mesh.tri_uv)


@pytest.fixture(scope="module", params=[(s, r) for s in SHAPES for r in (1.0, 0.8)],
                ids=lambda p: "%dx%d-t%d-%g" % (*p[0], p[1]))
def model(request):
    (W, H, T), rows = request.param
    mesh = covered(rows)
    o = oracle.Atlas(mesh, W, H, tile=T)
    assert (o.tri != 0xFFFFFFFF).all() == (rows == 1.0)
    return o, gpu_atlas(mesh, W, H, T), mesh


@pytest.mark.parametrize("pad", PADS, ids=lambda p: "r%d-t%d" % p)
@pytest.mark.parametrize("numeric", [False, True])
def test_spheres(model, pad, numeric):
    o, (_, a), mesh = model
    recs = sphere_recs(o, synth.sphere_strokes(mesh, 6, 17, 0.01, 0.9, 1, 255))
    recs["flags"] = oracle.pad_flags(*pad)
    recs["flags"][2] = 0
    exp = np.zeros(o.tri.shape, np.uint8)
    exp_hits, _ = oracle.select_sphere_2d(o, exp, recs)
    hits = torch.full((6,), -1, dtype=torch.int64, device="cuda")
    if numeric:
        layer = lcl.NumericLayer(o.tri.shape[1], o.tri.shape[0], "u8")
        lcl.lcl_numeric_sphere(a, layer, recs, hits_out=hits)
        got = to_np(layer.data, np.uint8)
        n = got.size
        known = np.unpackbits(layer.mask.cpu().numpy().view(np.uint8), bitorder="little")[:n].reshape(got.shape)
        assert np.array_equal(known.astype(bool), exp > 0)
    else:
        layer = to_dev(np.zeros(o.tri.shape, np.uint8))
        lcl.lcl_select_sphere(a, layer, recs, hits_out=hits)
        got = to_np(layer, np.uint8)
    assert np.array_equal(got, exp) and np.array_equal(to_np(hits, np.uint64), exp_hits)


@pytest.mark.parametrize("pad", PADS, ids=lambda p: "r%d-t%d" % p)
def test_lasso_and_tool(model, pad):
    o, (m, a), mesh = model
    cam = synth.orbit_camera(mesh, 240, 180, np.random.default_rng(5))
    M = oracle.camera_mq(cam.vp, o.mn, o.S)
    dm = oracle.depth(mesh, o.mn, o.S, M, 240, 180)
    d = to_dev(dm)
    flags = oracle.pad_flags(*pad)
    for radius in (60.0, 400.0):  # across the model, and around it: tiles inside the polygon
        poly = synth.star_lasso((120.0, 90.0), 12, radius, np.random.default_rng(6))
        exp = np.zeros(o.tri.shape, np.uint8)
        exp_hits, _, amb = oracle.select_lasso_2d(o, exp, M, dm, poly, 7, flags=flags)
        layer = to_dev(np.zeros(o.tri.shape, np.uint8))
        h = torch.full((1,), -1, dtype=torch.int64, device="cuda")
        lcl.lcl_select_lasso(a, layer, lcl.camera(M, 240, 180), d, poly, 7, flags=flags, hits_out=h)
        assert exp_hits and not ((to_np(layer, np.uint8) != exp) & (amb == 0)).any()
        assert abs(int(h) - exp_hits) <= int((amb != 0).sum())
    exp = np.zeros(o.tri.shape, np.uint8)
    _, _, amb = oracle.select_tool_2d(o, exp, M, dm, (120.0, 90.0), (120.0, 90.0), label=9, flags=flags)
    layer = to_dev(np.zeros(o.tri.shape, np.uint8))
    tool = lcl.make_tool((120.0, 90.0), (120.0, 90.0), flags=flags)
    lcl.lcl_select_tool(a, layer, lcl.camera(M, 240, 180), d, tool, 9)
    assert not ((to_np(layer, np.uint8) != exp) & (amb == 0)).any() and exp.any()


@pytest.mark.skipif(os.environ.get("LCL_DEBUG_BOUNDS") == "1", reason="times of the bounds-checking build")
def test_padding_costs_little_on_a_covered_texture():
    W = H = 4096
    mesh = covered()
    _, a = gpu_atlas(mesh, W, H, 32)
    o = oracle.Atlas(mesh, 64, 64, tile=32)  # the grid only
    recs = sphere_recs(o, synth.sphere_strokes(mesh, 3, 17, 0.4, 0.8, 1, 255))
    layer = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
    ws = torch.empty(lcl.lcl_select_workspace_bytes(a, 3), dtype=torch.uint8, device="cuda")

    def time_of(f):
        best = float("inf")
        for _ in range(5):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(20):
                f()
            t1.record()
            t1.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best

    def each():
        for k in range(3):
            lcl.lcl_select_sphere(a, layer, recs[k:k + 1], workspace=ws)

    plain = time_of(each)
    recs = recs.copy()
    recs["flags"] = lcl.pad_flags(8, 8)
    assert time_of(lambda: lcl.lcl_select_sphere(a, layer, recs, workspace=ws)) < 1.5 * plain
