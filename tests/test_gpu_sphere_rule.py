"""Sphere calls on both sides of the rule that sends some through candidate lists (by_lists in csrc/select.cu), by texture
size, tile side, number of strokes and radius, on label and value layers, against the definition on the
atlas's planes: textures just above the sizes from which the rule changes, with tiles of every side."""
import os

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, sphere_recs
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mesh():
    return synth.vessel_charts(80, 40, 20, 10, 512, seed=6)


def definition(a, recs, layer, erase_value=None):
    px, py, pz = (a.plane(k).long() for k in ("pos_x", "pos_y", "pos_z"))
    covered = px != -2 ** 31
    hits = []
    for r in recs:
        at = covered & ((px - int(r["cx"])) ** 2 + (py - int(r["cy"])) ** 2 + (pz - int(r["cz"])) ** 2 <= int(r["r2"]))
        layer[at] = int(r["label"])
        hits.append(int(at.sum()))
    return hits


@pytest.mark.parametrize("side", [2048, 3552, 7104])
@pytest.mark.parametrize("T", [8, 16, 32, 64, 128])
def test_every_route_is_the_definition(mesh, side, T):
    o = oracle.Atlas(mesh, 64, 64, tile=32)  # the grid only
    _, a = gpu_atlas(mesh, side, side, T)
    for n, wide in ((1, False), (1, True), (2, False), (5, True), (9, False), (16, False), (17, True), (33, False)):
        recs = sphere_recs(o, synth.sphere_strokes(mesh, n, 17 + n, 0.01, 0.04, 1, 255))
        if wide:
            recs["r2"][n // 2] = 1 << 38
        assert (recs["r2"] > 1 << 36).any() == wide
        exp = torch.zeros((side, side), dtype=torch.uint8, device="cuda")
        want = definition(a, recs, exp)
        layer, value = torch.zeros_like(exp), lcl.NumericLayer(side, side, "u8")
        h = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        lcl.lcl_select_sphere(a, layer, recs, hits_out=h)
        assert torch.equal(layer, exp) and h.tolist() == want and sum(want) > 0, (n, wide)
        h.fill_(-1)
        lcl.lcl_numeric_sphere(a, value, recs, hits_out=h)
        assert torch.equal(value.data, exp) and h.tolist() == want, (n, wide, "value")
        known = np.unpackbits(value.mask.cpu().numpy().view(np.uint8), bitorder="little")[:side * side]
        assert np.array_equal(known.reshape(side, side).astype(bool), (exp > 0).cpu().numpy())


@pytest.mark.skipif(os.environ.get("LCL_DEBUG_BOUNDS") == "1", reason="times of the bounds-checking build")
def test_one_wide_stroke_costs_the_same_with_larger_tiles(mesh):
    o = oracle.Atlas(mesh, 64, 64, tile=32)  # the grid only
    recs = sphere_recs(o, synth.sphere_strokes(mesh, 1, 17, 0.2, 0.2, 1, 255))

    def time_of(T):
        side = 16384
        _, a = gpu_atlas(mesh, side, side, T)
        layer = torch.zeros((side, side), dtype=torch.uint8, device="cuda")
        ws = torch.empty(lcl.lcl_select_workspace_bytes(a, 1), dtype=torch.uint8, device="cuda")
        best = float("inf")
        for _ in range(6):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(20):
                lcl.lcl_select_sphere(a, layer, recs, workspace=ws)
            t1.record()
            t1.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best

    assert time_of(64) < 1.8 * time_of(32)  # three times by blocks, as a rule that counted tiles had it
