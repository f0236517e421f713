"""The atlas build and the depth map where their binary32 and fixed-point shortcuts end, bit for bit against
the oracle: vertices on and next to rounding boundaries of the grid, models far from the origin, tiny and
huge ones (the binary64 quantisation), texture coordinates on snapping ties, triangles that overlap in the
texture, slivers, one triangle over the whole texture, and steep and nearly flat position planes."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import DEV, assert_atlas_equal, gpu_atlas, to_np
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu


def soup(pos, uv):
    n = np.arange(len(pos), dtype=np.uint32).reshape(-1, 3)
    return synth.Mesh(np.asarray(pos, np.float32), np.asarray(uv, np.float32), n, n.copy())


def check(mesh, W, H, T):
    o = oracle.Atlas(mesh, W, H, tile=T)
    m, a = gpu_atlas(mesh, W, H, T)
    assert_atlas_equal(a, o)
    assert np.array_equal(to_np(a.area_w(), np.uint64), o.area_w)
    assert np.array_equal(to_np(a.tile_box(), np.int32), o.tile_aabb())
    assert np.array_equal(to_np(a.cover(), np.uint32), o.cover_bits())
    return o, m, a


@pytest.mark.parametrize("scale,shift", [(1.0, 0.0), (1.0, 1e4), (3e-30, 0.0), (2e25, 0.0), (1e-3, 7.0)])
def test_quantisation(scale, shift):
    mesh = synth.vessel_cylindrical(64, 40, noise_amp=0.03, seed=5)
    pos = (mesh.pos.astype(np.float64) * scale + shift).astype(np.float32)
    mesh = synth.Mesh(pos, mesh.uv, mesh.tri_pos, mesh.tri_uv)
    o, m, a = check(mesh, 160, 96, 32)
    cam = synth.orbit_camera(mesh, 150, 110, np.random.default_rng(4))
    M = oracle.camera_mq(cam.vp, o.mn, o.S)
    if np.isfinite(M).all():
        d = torch.empty((110, 150), dtype=torch.float32, device=DEV)
        lcl.lcl_depth_render(m, a, lcl.camera(M, 150, 110), d)
        assert np.array_equal(to_np(d, np.uint32), oracle.depth(mesh, o.mn, o.S, M, 150, 110).view(np.uint32))


def test_grid_rounding_boundaries():
    # extent 2^21 - 1: the scale is 1 and positions k + 1/2 and their neighbours lie on its boundaries
    rng = np.random.default_rng(1)
    k = rng.integers(0, 1 << 21, size=(300, 3)).astype(np.float64)
    pos = (k + 0.5).astype(np.float32)
    pos[1::3] = np.nextafter(pos[1::3], np.float32(np.inf))
    pos[2::3] = np.nextafter(pos[2::3], np.float32(-np.inf))
    pos = np.clip(pos, 0, (1 << 21) - 1).astype(np.float32)
    pos[0], pos[1] = 0, (1 << 21) - 1
    check(soup(pos, rng.random((300, 2))), 128, 128, 16)


def test_snapping_ties():
    # u * 256 * W on halves (ties to even) and one ulp to either side
    rng = np.random.default_rng(2)
    W, H = 96, 64
    n = 240
    uv = np.stack([(rng.integers(-100, 256 * W, n) + 0.5) / (256 * W), (rng.integers(0, 256 * H, n) + 0.5) / (256 * H)], 1)
    uv = uv.astype(np.float32)
    uv[1::3] = np.nextafter(uv[1::3], np.float32(np.inf))
    uv[2::3] = np.nextafter(uv[2::3], np.float32(-np.inf))
    check(soup(rng.random((n, 3)), np.clip(uv, -1, 2)), W, H, 8)


@pytest.mark.parametrize("n,W,H,T", [(3, 128, 96, 32), (60, 256, 256, 64), (900, 300, 170, 16)])
def test_overlaps_and_slivers(n, W, H, T):
    rng = np.random.default_rng(n)
    uv = rng.random((n, 2)).astype(np.float32) * 1.5 - 0.25
    uv[2::9] = uv[1::9] + np.float32(1e-3)  # needles: their planes are too steep to use
    pos = rng.random((n, 3)) * [1.0, 1e-4, 1.0]
    check(soup(pos, uv), W, H, T)


def test_single_triangle_over_the_texture():
    uv = np.array([[-0.5, -0.5], [2.0, -0.5], [-0.5, 2.0]], np.float32)
    check(soup([[0, 0, 0], [1, 0.3, 0], [0, 0.2, 1e-3]], uv), 512, 256, 32)


def test_degenerate_next_to_a_full_cover():
    # two copies of one square (every texel covered twice: the smallest id wins) and triangles without area
    uv = np.array([[0, 0], [1, 0], [1, 1], [0, 0], [1, 1], [0, 1]] * 2 + [[0.5, 0.5]] * 3, np.float32)
    pos = np.random.default_rng(3).random((15, 3))
    check(soup(pos, uv), 128, 128, 32)
