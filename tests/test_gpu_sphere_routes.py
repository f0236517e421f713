"""Sphere calls on both sides of the rule that sends few strokes on a large texture through candidate lists
(by_lists in csrc/select.cu): a texture of 160,000 tiles (tile 8), calls of 1, 2, 4, 5, 32, 33 (small and with
one large radius), 96 and 97 strokes, on label and value layers, against one call per stroke on a tile of 32,
which the rule never sends there."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, sphere_recs
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu

W, H = 3200, 3200


@pytest.fixture(scope="module")
def atlases():
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    o = oracle.Atlas(mesh, 64, 64, tile=32)  # the grid only
    return mesh, o, gpu_atlas(mesh, W, H, 8)[1], gpu_atlas(mesh, W, H, 32)[1]


@pytest.mark.parametrize("n,large", [(1, False), (2, False), (2, True), (4, False), (5, True), (32, True), (33, False),
                                     (33, True), (96, False), (97, False)])
@pytest.mark.parametrize("numeric", [False, True])
def test_routes_agree(atlases, n, large, numeric):
    mesh, o, fine, coarse = atlases
    recs = sphere_recs(o, synth.sphere_strokes(mesh, n, 17, 0.01, 0.04, 1, 255))
    if large:
        recs["r2"][n // 2] = 1 << 38
    assert (recs["r2"] <= 1 << 36).sum() == n - (1 if large else 0)
    layers, hits = [], []
    for a in (fine, coarse):
        layer = lcl.NumericLayer(W, H, "u8") if numeric else torch.zeros((H, W), dtype=torch.uint8, device="cuda")
        edit = lcl.lcl_numeric_sphere if numeric else lcl.lcl_select_sphere
        h = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        if a is fine:
            edit(a, layer, recs, hits_out=h)
        else:
            for k in range(n):
                edit(a, layer, recs[k:k + 1], hits_out=h[k:k + 1])
        layers.append(layer)
        hits.append(h)
    if numeric:
        assert torch.equal(layers[0].mask, layers[1].mask)
        layers = [v.data for v in layers]
    assert torch.equal(layers[0], layers[1]) and torch.equal(hits[0], hits[1]) and int(hits[0].sum()) > 0
