"""Atlases whose triangles share texels of the texture (csrc/atlas.cu): of the triangles that cover a texel the one of
the smallest id has it, whatever their order, and a mesh with a shared texel costs no second build."""
import os
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import assert_atlas_equal, gpu_atlas, to_np
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu


def overlapping(kind, n_theta=64, n_h=40):
    m = synth.vessel_cylindrical(n_theta, n_h, noise_amp=0.03, seed=5)
    uv, tp, tu = m.uv.copy(), m.tri_pos, m.tri_uv
    if kind == "mirror":    # the right half over the left
        uv[:, 0] = np.where(uv[:, 0] <= 0.5, 2 * uv[:, 0], 2 - 2 * uv[:, 0])
    elif kind == "one":     # a triangle again, as the last one
        tp, tu = np.concatenate([tp, tp[:1]]), np.concatenate([tu, tu[:1]])
    elif kind == "first":   # every tenth again, before the others
        tp, tu = np.concatenate([tp[::10], tp]), np.concatenate([tu[::10], tu])
    return synth.Mesh(m.pos, uv, np.ascontiguousarray(tp), np.ascontiguousarray(tu))


@pytest.mark.parametrize("kind", ["mirror", "one", "first"])
@pytest.mark.parametrize("W,H,T", [(160, 96, 32), (300, 170, 16), (1024, 512, 64)])
def test_smallest_id_wins(kind, W, H, T):
    mesh = overlapping(kind)
    o = oracle.Atlas(mesh, W, H, tile=T)
    _, a = gpu_atlas(mesh, W, H, T)
    assert_atlas_equal(a, o)
    assert np.array_equal(to_np(a.area_w(), np.uint64), o.area_w)
    assert np.array_equal(to_np(a.tile_box(), np.int32), o.tile_aabb())
    assert np.array_equal(to_np(a.cover(), np.uint32), o.cover_bits())


@pytest.mark.skipif(os.environ.get("LCL_DEBUG_BOUNDS") == "1", reason="times of the bounds-checking build")
def test_a_shared_texel_costs_no_second_build():
    def time_of(kind):
        mesh = lcl.Mesh.from_host(overlapping(kind, 400, 150), "cuda")
        a = lcl.Atlas(2048, 2048, 32, mesh.n_tri, "cuda")
        ws = torch.empty(lcl.lcl_atlas_workspace_bytes(mesh, 2048, 2048), dtype=torch.uint8, device="cuda")
        best = float("inf")
        for _ in range(6):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(5):
                lcl.lcl_atlas_build(mesh, a, ws)
            t1.record()
            t1.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best

    time_of("none")
    assert time_of("one") < 1.3 * time_of("none")  # 1.6 with a second raster and resolve
