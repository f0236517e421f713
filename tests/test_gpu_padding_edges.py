"""Texture padding from row bits (csrc/select.cu) at its edges, against the oracle: every tile side (blocks of
8, 16 and 32 texels, several blocks per tile), textures that end inside a block, kernels and outlines up to 8,
each larger than the other, strokes with and without padding in one call."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, sphere_recs, to_dev, to_np
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu

SHAPES = [(64, 40, 8), (300, 170, 16), (256, 256, 32), (204, 130, 32), (384, 256, 128), (160, 150, 64)]
PADS = [(1, 1), (2, 2), (8, 8), (8, 1), (1, 8), (3, 0)]


@pytest.fixture(scope="module", params=SHAPES, ids=lambda s: "%dx%d-t%d" % s)
def model(request):
    W, H, T = request.param
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    return oracle.Atlas(mesh, W, H, tile=T), gpu_atlas(mesh, W, H, T), mesh


@pytest.mark.parametrize("pad", PADS, ids=lambda p: "r%d-t%d" % p)
@pytest.mark.parametrize("dt", [np.uint8, np.uint16])
def test_spheres(model, dt, pad):
    o, (_, a), mesh = model
    recs = sphere_recs(o, synth.sphere_strokes(mesh, 6, 17, 0.01, 0.4, 1, 255))
    recs["flags"] = oracle.pad_flags(*pad)
    recs["flags"][2] = 0
    exp = np.random.default_rng(1).integers(0, 9, size=o.tri.shape).astype(dt)
    layer = to_dev(exp)
    exp_hits, _ = oracle.select_sphere_2d(o, exp, recs)
    hits = torch.full((6,), -1, dtype=torch.int64, device="cuda")
    lcl.lcl_select_sphere(a, layer, recs, hits_out=hits)
    assert np.array_equal(to_np(layer, dt), exp)
    assert np.array_equal(to_np(hits, np.uint64), exp_hits)


@pytest.mark.parametrize("pad", PADS, ids=lambda p: "r%d-t%d" % p)
def test_lasso_and_tool(model, pad):
    o, (m, a), mesh = model
    cam = synth.orbit_camera(mesh, 240, 180, np.random.default_rng(5))
    M = oracle.camera_mq(cam.vp, o.mn, o.S)
    dm = oracle.depth(mesh, o.mn, o.S, M, 240, 180)
    d = torch.empty((180, 240), dtype=torch.float32, device="cuda")
    lcl.lcl_depth_render(m, a, lcl.camera(M, 240, 180), d)
    poly = synth.star_lasso((120.0, 90.0), 12, 70.0, np.random.default_rng(6))
    flags = oracle.pad_flags(*pad)
    exp = np.zeros(o.tri.shape, np.uint8)
    _, _, amb = oracle.select_lasso_2d(o, exp, M, dm, poly, 7, flags=flags)
    layer = to_dev(np.zeros(o.tri.shape, np.uint8))
    lcl.lcl_select_lasso(a, layer, lcl.camera(M, 240, 180), d, poly, 7, flags=flags)
    assert not ((to_np(layer, np.uint8) != exp) & (amb == 0)).any() and exp.any()
    # the tool over the whole view with the same padding as an inscribed circle
    exp = np.zeros(o.tri.shape, np.uint8)
    _, _, amb = oracle.select_tool_2d(o, exp, M, dm, (120.0, 90.0), (120.0, 90.0), label=9, flags=flags)
    layer = to_dev(np.zeros(o.tri.shape, np.uint8))
    tool = lcl.make_tool((120.0, 90.0), (120.0, 90.0), flags=flags)
    lcl.lcl_select_tool(a, layer, lcl.camera(M, 240, 180), d, tool, 9)
    assert not ((to_np(layer, np.uint8) != exp) & (amb == 0)).any() and exp.any()
