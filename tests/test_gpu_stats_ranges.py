"""Zonal statistics of float layers whose values range too widely for one unit (csrc/numeric.cu): the sums keep the
bounds of include/lcl.h as they stand -- against exact integer sums, so a zone of one texel is exact -- and a few
outliers cost no more than a small factor in time."""
import os
from fractions import Fraction

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, to_dev
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu


def values(kind, n, rng):
    v = rng.standard_normal(n).astype(np.float32)
    if kind == "outliers":    # ordinary values after single huge ones: the unit has to come down again
        v[rng.integers(0, n, max(1, n // 200))] = 1e30
    elif kind == "alternating":
        v[::2] *= np.float32(2.0 ** -50)
    elif kind == "falling":   # magnitudes that fall along the texture
        v *= (np.float32(2.0) ** np.linspace(100, -100, n).astype(np.float32))
    elif kind == "log":
        v *= np.exp2(rng.uniform(-60, 60, n)).astype(np.float32)
    elif kind == "subnormal":
        v = (v * np.float32(1e-40)).astype(np.float32)
    return v


@pytest.mark.parametrize("kind", ["plain", "outliers", "alternating", "falling", "log", "subnormal"])
@pytest.mark.parametrize("shape,zones", [((256, 96, 16), 1), ((512, 256, 32), 3), ((100, 70, 32), 700), ((4, 300, 8), 1200)],
                         ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else str(s))
def test_sums_within_the_stated_bounds(shape, zones, kind):
    W, H, T = shape
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    o = oracle.Atlas(mesh, W, H, tile=T)
    _, a = gpu_atlas(mesh, W, H, T)
    rng = np.random.default_rng(W + zones)
    v = values(kind, W * H, rng).reshape(H, W)
    z = None if zones == 1 else (np.add.outer(np.arange(H), np.arange(W)) // 9 % 3 if zones == 3 else
                                 rng.integers(0, zones, (H, W))).astype(np.uint8 if zones <= 256 else np.uint16)
    layer = lcl.NumericLayer(W, H, "f32")
    layer.data.copy_(torch.from_numpy(v))
    layer.mask.fill_(-1)
    got = lcl.zone_stats_host(lcl.lcl_numeric_stats(a, layer, None if z is None else to_dev(z), zones))
    on = o.covered()
    zi = np.zeros((H, W), np.int64) if z is None else z.astype(np.int64)
    w = o.area_w[np.where(on, o.tri, 0)].astype(object)
    # every float32 is a multiple of 2^-149
    units = np.array([int(np.ldexp(x, 60)) << 89 if abs(x) >= 1 else int(Fraction(float(x)) * 2 ** 149)
                      for x in v.ravel().tolist()], object).reshape(H, W)
    ones = 0
    for k in range(zones):
        at = on & (zi == k)
        n = int(at.sum())
        assert got["count"][k] == n
        if not n:
            continue
        ones += n == 1
        for key, terms, factor in (("sum", units[at], n - 1), ("wsum", units[at] * w[at], 2 * n)):
            off = abs(Fraction(float(got[key][k])) * 2 ** 149 - int(terms.sum()))
            assert off <= Fraction(factor, 2 ** 53) * int(np.abs(terms).sum()), (key, k, n)
    assert ones or zones < 700


@pytest.mark.skipif(os.environ.get("LCL_DEBUG_BOUNDS") == "1", reason="times of the bounds-checking build")
@pytest.mark.parametrize("zones", [1, 40])
@pytest.mark.parametrize("kind", ["outliers", "log", "subnormal"])
def test_outliers_cost_little(kind, zones):
    W = H = 2048
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    _, a = gpu_atlas(mesh, W, H, 32)
    layer = lcl.NumericLayer(W, H, "f32")
    layer.mask.fill_(-1)
    z = None if zones == 1 else ((torch.arange(H, device="cuda")[:, None] // 100 * 7 + torch.arange(W, device="cuda") // 150)
                                 % zones).to(torch.uint8).contiguous()
    out = torch.empty(48 * zones, dtype=torch.uint8, device="cuda")

    def time_of(k):
        layer.data.copy_(torch.from_numpy(values(k, W * H, np.random.default_rng(1)).reshape(H, W)))
        best = float("inf")
        for _ in range(5):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(10):
                lcl.lcl_numeric_stats(a, layer, z, zones, out)
            t1.record()
            t1.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best

    time_of("plain")
    plain = time_of("plain")
    assert time_of(kind) < 4 * plain  # 8 to 50 times with an atomic per texel
