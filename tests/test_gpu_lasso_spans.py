"""Lasso polygons whose vertices are any finite floats (csrc/select_common.cuh, lasso_band_range): a frame around the
view at +-B, and one whose left or upper edge cuts through it, select the same texels for every B up to the
largest float, where the polygon's height no longer fits in a float; in single calls and batched."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, to_dev, to_np
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu

MAX = float(np.finfo(np.float32).max)


def frame(B, left, top):
    x0, y1 = -B if left is None else left, B if top is None else top
    return np.array([[x0, -B], [B, -B], [B, y1], [x0, y1]], np.float32)


@pytest.mark.parametrize("left,top", [(None, None), (100.2, None), (None, 90.3)])
@pytest.mark.parametrize("batched", [False, True])
def test_polygons_around_the_view(left, top, batched):
    W, H, T = 300, 170, 16
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    o, (m, a) = oracle.Atlas(mesh, W, H, tile=T), gpu_atlas(mesh, W, H, T)
    cam = synth.orbit_camera(mesh, 240, 180, np.random.default_rng(5))
    M = oracle.camera_mq(cam.vp, o.mn, o.S)
    dm = oracle.depth(mesh, o.mn, o.S, M, 240, 180)
    d = to_dev(dm)
    got = {}
    for B in (1e4, 1e20, 1e38, 2e38, MAX):
        poly = frame(B, left, top)
        layer = to_dev(np.zeros(o.tri.shape, np.uint8))
        if batched:
            lcl.lcl_batch_edit(lcl.Batch([(a, layer)], [[("lasso", (lcl.camera(M, 240, 180), d, poly, 7, lcl.DEFAULT_BIAS))]]))
        else:
            lcl.lcl_select_lasso(a, layer, lcl.camera(M, 240, 180), d, poly, 7)
        got[B] = to_np(layer, np.uint8)
    exp = np.zeros(o.tri.shape, np.uint8)
    _, amb = oracle.select_lasso(o, exp, M, dm, frame(1e4, left, top), 7)
    assert exp.any() and not ((got[1e4] != exp) & (amb == 0)).any()
    for B, layer in got.items():
        assert np.array_equal(layer, got[1e4]), B
