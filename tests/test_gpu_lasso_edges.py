"""The lasso's apply (csrc/select.cu) at its edges: tiles of every side, so that an item of a CTA is part of a
tile, one tile or several small ones with a remainder; tiles inside the polygon and across it; and operands on
both sides of the fast division's window.  Scaling a camera matrix by a power of two scales every clip
coordinate exactly, so the selection is the same to the bit while the window is left."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, to_dev, to_np
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu

SHAPES = [(64, 40, 8), (300, 170, 16), (204, 130, 32), (160, 150, 64), (384, 256, 128)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "%dx%d-t%d" % s)
@pytest.mark.parametrize("radius", [25.0, 160.0])
def test_lasso_items_and_division_window(shape, radius):
    W, H, T = shape
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    o, (m, a) = oracle.Atlas(mesh, W, H, tile=T), gpu_atlas(mesh, W, H, T)
    cam = synth.orbit_camera(mesh, 240, 180, np.random.default_rng(5))
    M = oracle.camera_mq(cam.vp, o.mn, o.S)
    dm = oracle.depth(mesh, o.mn, o.S, M, 240, 180)
    d = torch.empty((180, 240), dtype=torch.float32, device="cuda")
    lcl.lcl_depth_render(m, a, lcl.camera(M, 240, 180), d)
    poly = synth.star_lasso((120.0, 90.0), 12, radius, np.random.default_rng(6))
    exp = np.zeros(o.tri.shape, np.uint16)
    hits, amb = oracle.select_lasso(o, exp, M, dm, poly, 7)
    got = {}
    for k in (0, -45, 45):
        layer = to_dev(np.zeros(o.tri.shape, np.uint16))
        h = torch.full((1,), -1, dtype=torch.int64, device="cuda")
        lcl.lcl_select_lasso(a, layer, lcl.camera(np.ldexp(M, k).astype(np.float32), 240, 180), d, poly, 7, hits_out=h)
        got[k] = to_np(layer, np.uint16)
        assert int(h) == int((got[k] == 7).sum())
    assert hits and not ((got[0] != exp) & (amb == 0)).any()
    assert np.array_equal(got[-45], got[0]) and np.array_equal(got[45], got[0])
