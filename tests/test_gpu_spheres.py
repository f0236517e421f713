"""Unpadded sphere strokes (csrc/spheres.cu) at the edges of its launch shapes, against the oracle: stroke
counts around the two launch sizes, tiles of every side, textures whose blocks are bands of one tile, single
tiles and several tiles, widths that are and are not whole 32-texel words.  All results are integers: exact."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, sphere_recs, to_dev, to_np
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu

SHAPES = [(64, 40, 8), (300, 170, 16), (256, 256, 32), (1000, 600, 32), (384, 256, 128), (512, 512, 64)]
COUNTS = [1, 32, 33, 512, 515]


@pytest.fixture(scope="module", params=SHAPES, ids=lambda s: "%dx%d-t%d" % s)
def model(request):
    W, H, T = request.param
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    return oracle.Atlas(mesh, W, H, tile=T), gpu_atlas(mesh, W, H, T), mesh


def strokes(o, mesh, n):
    recs = sphere_recs(o, synth.sphere_strokes(mesh, n, 91 + n, 0.005, 0.5, 1, 255))
    recs["r2"][n // 2] = 1 << 62  # one that contains everything, with older and newer ones around it
    return recs


@pytest.mark.parametrize("n", COUNTS)
@pytest.mark.parametrize("dt", [np.uint8, np.uint16])
def test_label_layer(model, dt, n):
    o, (_, a), mesh = model
    recs = strokes(o, mesh, n)
    exp = np.random.default_rng(n).integers(0, 9, size=o.tri.shape).astype(dt)
    layer, uncounted = to_dev(exp), to_dev(exp)
    exp_hits = oracle.select_sphere(o, exp, recs)
    hits = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    lcl.lcl_select_sphere(a, layer, recs, hits_out=hits)
    lcl.lcl_select_sphere(a, uncounted, recs)
    assert np.array_equal(to_np(layer, dt), exp)
    assert np.array_equal(to_np(uncounted, dt), exp)
    assert np.array_equal(to_np(hits, np.uint64), exp_hits)


@pytest.mark.parametrize("n", [1, 33])
@pytest.mark.parametrize("ntype", ["u8", "i16", "f32"])
def test_numeric_layer(model, ntype, n):
    o, (_, a), mesh = model
    H, W = o.tri.shape
    recs = strokes(o, mesh, n)
    if n > 1:
        recs["flags"][::3] = oracle.ERASE
    rng = np.random.default_rng(n)
    data = rng.integers(0, 100, size=(H, W)).astype(oracle.NUM_NP[ntype])
    mask = rng.integers(0, 2, size=(H, W)).astype(np.uint8)
    layer = lcl.NumericLayer(W, H, ntype)
    layer.data.copy_(torch.from_numpy(data))
    words = np.zeros(layer.mask.numel() * 4, np.uint8)
    packed = np.packbits(mask.reshape(-1), bitorder="little")
    words[:packed.size] = packed
    layer.mask.copy_(torch.from_numpy(words.view(np.int32)))
    hits = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    lcl.lcl_numeric_sphere(a, layer, recs, hits_out=hits)
    exp_hits, _ = oracle.num_select_sphere(o, data, mask, recs)
    assert np.array_equal(layer.data.cpu().numpy().view(np.uint8), data.view(np.uint8))
    assert np.array_equal(layer.mask_bits(), mask.astype(bool))
    assert np.array_equal(to_np(hits, np.uint64), exp_hits)
