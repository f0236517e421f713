"""Lassos from a camera so close to a finely textured detail that the binary32 projections of texels are off by
several pixels (csrc/select_common.cuh, lasso_w_safe): the selection is still the definition's, texel by texel,
tiles are not taken for inside or outside on the strength of their boxes, nothing off the screen is read, and a
depth map just behind the nearest texels of a tile does not hide them.  From farther away (3000) boxes decide."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import gpu_atlas, to_dev, to_np
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu

W, H, T = 512, 256, 16
WS, HS = 16384, 512


def detail(relief=20):
    """A triangle that sets the grid and a patch of 4000 x 2000 grid units that takes most of the texture."""
    s = 1.0 / (2 ** 21 - 1)
    n = 8
    u, v = np.meshgrid(np.linspace(0.01, 0.99, n + 1), np.linspace(0.02, 0.9, n + 1))
    p = np.stack([0.71 + 4000 * s * (u - 0.5), 0.63 + 2000 * s * (v - 0.5), 0.83 + relief * s * np.sin(9 * u + 7 * v)], -1)
    k = np.arange((n + 1) * n).reshape(n, n + 1)[:, :n].ravel()
    tri = np.concatenate([np.stack([k, k + 1, k + n + 2], 1), np.stack([k, k + n + 2, k + n + 1], 1)]) + 3
    pos = np.concatenate([[[0, 0, 0], [1, 0, 0], [0, 1, 1]], p.reshape(-1, 3)]).astype(np.float32)
    uv = np.concatenate([[[0.3, 0.93], [0.7, 0.93], [0.5, 0.99]], np.stack([u, v], -1).reshape(-1, 2)]).astype(np.float32)
    tri = np.concatenate([[[0, 1, 2]], tri]).astype(np.uint32)
    return synth.Mesh(pos, uv, tri, tri.copy())


@pytest.mark.parametrize("distance", [30, 100, 400, 3000])
@pytest.mark.parametrize("left", [None, 8000.25])
@pytest.mark.parametrize("batched", [False, True])
def test_closeup(distance, left, batched):
    mesh = detail()
    o, (_, a) = oracle.Atlas(mesh, W, H, tile=T), gpu_atlas(mesh, W, H, T)
    at = np.array([0.71, 0.63, 0.83]) * (2 ** 21 - 1)
    fwd = np.array([0.25, 0.15, 1.0])
    fwd /= np.linalg.norm(fwd)
    right = np.cross(fwd, [0.1, 1.0, 0.0])
    right /= np.linalg.norm(right)
    R = np.stack([0.6 * right, 0.9 * np.cross(right, fwd), 0.5 * fwd, fwd]) / 2 ** 21
    eye = at - distance * fwd
    M = np.concatenate([R, -(R @ eye)[:, None]], 1).astype(np.float32).reshape(16)
    dm = np.full((HS, WS), np.inf, np.float32)
    x0 = -1e4 if left is None else left
    poly = np.array([[x0, -1e4], [3e4, -1e4], [3e4, 1e4], [x0, 1e4]], np.float32)
    exp = np.zeros(o.tri.shape, np.uint8)
    _, amb = oracle.select_lasso(o, exp, M, dm, poly, 7)
    layer, d = to_dev(np.zeros(o.tri.shape, np.uint8)), to_dev(dm)
    if batched:
        lcl.lcl_batch_edit(lcl.Batch([(a, layer)], [[("lasso", (lcl.camera(M, WS, HS), d, poly, 7, lcl.DEFAULT_BIAS))]]))
    else:
        lcl.lcl_select_lasso(a, layer, lcl.camera(M, WS, HS), d, poly, 7)
    assert exp.any() and not ((to_np(layer, np.uint8) != exp) & (amb == 0)).any()


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("distance,seed,tile", [(600, 0, (17, 10)), (600, 1, None), (1000, 2, None), (4000, 3, None)])
def test_depth_map_just_behind(distance, seed, tile, batched):
    ws, hs, f = 64, 48, np.float32
    mesh = detail(0)
    o, (_, a) = oracle.Atlas(mesh, W, H, tile=T), gpu_atlas(mesh, W, H, T)
    rng = np.random.default_rng(seed)
    at = np.array([0.71, 0.63, 0.83]) * (2 ** 21 - 1) + rng.uniform(-300, 300, 3) * [1, 1, 0]
    fwd = np.array([0.0, 0.0, 1.0]) + rng.normal(size=3) * 0.15
    fwd /= np.linalg.norm(fwd)
    right = np.cross(fwd, [0.1, 1.0, 0.0])
    right /= np.linalg.norm(right)
    near, far = distance * 0.3 / 2 ** 21, 2.0
    R = np.stack([0.6 * right, 0.9 * np.cross(right, fwd), fwd, fwd]) / 2 ** 21
    M = np.concatenate([R, -(R @ (at - distance * fwd))[:, None]], 1)
    M[2] *= far / (far - near)
    M[2, 3] -= near * far / (far - near)
    M = M.astype(f)

    def row(k):
        x, y, z = (q.astype(f) for q in (o.px, o.py, o.pz))
        return ((M[k, 0] * x + M[k, 1] * y) + M[k, 2] * z) + M[k, 3]

    w = row(3)
    seen = (o.tri != 0xFFFFFFFF) & (w > 0) & (np.abs(row(0)) < w) & (np.abs(row(1)) < w) & (row(2) >= 0) & (row(2) <= w)
    if tile:  # of its texels in view, else of all
        seen[:tile[1] * T] = seen[(tile[1] + 1) * T:] = seen[:, :tile[0] * T] = seen[:, (tile[0] + 1) * T:] = False
    dm = np.full((hs, ws), (row(2) / w)[seen].min() + f(2.5e-5), f)
    poly = np.array([[-1e3, -1e3], [1e3, -1e3], [1e3, 1e3], [-1e3, 1e3]], f)
    exp = np.zeros(o.tri.shape, np.uint8)
    _, amb = oracle.select_lasso(o, exp, M.reshape(16), dm, poly, 7, bias=0.0)
    layer, d = to_dev(np.zeros(o.tri.shape, np.uint8)), to_dev(dm)
    cam = lcl.camera(M.reshape(16), ws, hs)
    if batched:
        lcl.lcl_batch_edit(lcl.Batch([(a, layer)], [[("lasso", (cam, d, poly, 7, 0.0))]]))
    else:
        lcl.lcl_select_lasso(a, layer, cam, d, poly, 7, bias=0.0)
    assert (exp.astype(bool) & (amb == 0)).any()
    assert not ((to_np(layer, np.uint8) != exp) & (amb == 0)).any()
