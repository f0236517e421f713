"""Zonal statistics (csrc/numeric.cu) where the integer sums change their unit or give way to binary64, and
where a warp meets more zones than it keeps: magnitudes over the whole float range within a row, values of a
single bit far below the others, subnormals, many zones per strip, sums of long runs, narrow textures.
Counts, areas and extremes are exact; the sums keep the bounds that include/lcl.h states."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, to_dev
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu


def values(kind, n, rng):
    if kind == "wide":       # every finite exponent
        v = rng.integers(0, 1 << 32, size=n, dtype=np.uint64).astype(np.uint32).view(np.float32)
        return np.where(np.isfinite(v), v, np.float32(1))
    if kind == "tiny":       # normal values with subnormals and single far smaller bits among them
        v = rng.standard_normal(n).astype(np.float32)
        v[::7] *= np.float32(2.0 ** -40)
        v[::11] = np.float32(2.0 ** -149) * rng.integers(1, 1000, size=len(v[::11])).astype(np.float32)
        return v
    if kind == "steps":      # magnitudes that rise along the texture
        return (np.float32(2.0) ** np.linspace(-100, 100, n).astype(np.float32) * rng.choice([-1, 1], n)).astype(np.float32)
    return np.full(n, 3.0, np.float32) * rng.choice([1, -1, 0], n).astype(np.float32)


@pytest.mark.parametrize("shape", [(256, 96, 16), (100, 70, 32), (4, 300, 8), (512, 512, 32)], ids=lambda s: "%dx%d" % s[:2])
@pytest.mark.parametrize("kind", ["wide", "tiny", "steps", "signs"])
@pytest.mark.parametrize("zones", [1, 3, 150])
def test_float_sums(shape, kind, zones):
    W, H, T = shape
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    o = oracle.Atlas(mesh, W, H, tile=T)
    _, a = gpu_atlas(mesh, W, H, T)
    rng = np.random.default_rng(W + zones)
    v = values(kind, W * H, rng).reshape(H, W).astype(np.float32)
    mask = (rng.random((H, W)) < 0.9).astype(np.uint8)
    z = None if zones == 1 else (rng.integers(0, zones, (H, W)) if zones > 3 else
                                 (np.add.outer(np.arange(H), np.arange(W)) // 9 % zones)).astype(np.uint8)
    layer = lcl.NumericLayer(W, H, "f32")
    layer.data.copy_(torch.from_numpy(v))
    words = np.zeros(layer.mask.numel() * 4, np.uint8)
    packed = np.packbits(mask.reshape(-1), bitorder="little")
    words[:packed.size] = packed
    layer.mask.copy_(torch.from_numpy(words.view(np.int32)))
    got = lcl.zone_stats_host(lcl.lcl_numeric_stats(a, layer, None if z is None else to_dev(z), zones))
    on = mask.astype(bool) & o.covered()
    zi = np.zeros((H, W), np.int64) if z is None else z.astype(np.int64)
    w = np.where(on, o.area_w[np.where(on, o.tri, 0)], 0).astype(np.float64)
    d = v.astype(np.float64)
    for k in range(zones):
        at = on & (zi == k)
        n = int(at.sum())
        assert got["count"][k] == n
        assert got["area"][k] == int(w[at].sum())
        if not n:
            continue
        assert got["vmin"][k] == d[at].min() and got["vmax"][k] == d[at].max()
        # against numpy's pairwise sums, whose own error is far below the stated bounds
        assert abs(got["sum"][k] - d[at].sum()) <= 2.0 ** -53 * (n + 60) * np.abs(d[at]).sum()
        assert abs(got["wsum"][k] - (d * w)[at].sum()) <= 2.0 ** -52 * (n + 60) * np.abs(d * w)[at].sum()
