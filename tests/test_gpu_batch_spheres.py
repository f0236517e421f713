"""Batches without lassos (csrc/batch.cu), whose kernels leave out the lassos' code, against the same strokes one call
at a time: all models of one tile side, so that an item has one ticket up to sixteen, with and without texture
padding, for every split of the launch, and a texture with more units than the cull's warps draw one by one."""
import os

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import gpu_atlas, sphere_recs
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu


def check(sizes, T, n, pads, r_hi=0.4, config=None):
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    o = oracle.Atlas(mesh, 64, 64, tile=32)  # the grid only
    rng = np.random.default_rng(T + n)
    models, queues, want = [], [], []
    for i, (W, H) in enumerate(sizes):
        _, a = gpu_atlas(mesh, W, H, T)
        recs = sphere_recs(o, synth.sphere_strokes(mesh, n, 17 + i, 0.01, r_hi, 1, 255))
        if pads:
            recs["flags"][::2] = lcl.pad_flags(3, 2)
        seq = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
        for k in range(n):
            lcl.lcl_select_sphere(a, seq, recs[k:k + 1])
        models.append((a, torch.zeros((H, W), dtype=torch.uint8, device="cuda")))
        queues.append([("sphere", r) for r in recs])
        want.append(seq)
    batch = lcl.Batch(models, queues)
    if config is None:
        lcl.lcl_batch_edit(batch)
    else:
        lcl.lcl_batch_upload(batch)
        lcl.lcl_batch_launch(batch, config=config)
    for (_, layer), w in zip(models, want):
        assert torch.equal(layer, w) and int(layer.max()) > 0


@pytest.mark.parametrize("T", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("pads", [False, True])
@pytest.mark.parametrize("n", [1, 33, 64])
def test_spheres_only(T, pads, n):
    check([(64, 40), (300, 170), (524, 260)], T, n, pads)


@pytest.mark.parametrize("T", [8, 32, 128])
@pytest.mark.parametrize("split", [1, 2, 4, 8])
@pytest.mark.parametrize("threads", [64, 256])
def test_splits(T, split, threads):
    check([(300, 170)], T, 12, True, config=lcl.batch_config(threads=threads, split=split))


@pytest.mark.parametrize("pads", [False, True])
def test_more_units_than_warps_draw(pads):
    check([(4100, 4090)], 8, 5, pads, r_hi=0.2)


@pytest.mark.skipif(os.environ.get("LCL_DEBUG_BOUNDS") == "1", reason="times of the bounds-checking build")
def test_small_tiles_leave_no_tickets_empty():
    mesh = synth.vessel_cylindrical(200, 100, noise_amp=0.03, seed=5)
    o = oracle.Atlas(mesh, 64, 64, tile=32)  # the grid only
    recs = sphere_recs(o, synth.sphere_strokes(mesh, 64, 17, 0.005, 0.1, 1, 255))

    def time_of(T):
        _, a = gpu_atlas(mesh, 4096, 4096, T)
        batch = lcl.Batch([(a, torch.zeros((4096, 4096), dtype=torch.uint8, device="cuda"))], [[("sphere", r) for r in recs]])
        lcl.lcl_batch_upload(batch)
        best = float("inf")
        for _ in range(6):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(10):
                lcl.lcl_batch_launch(batch)
            t1.record()
            t1.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best

    assert time_of(8) < 4.5 * time_of(32)  # 6.5 with eight tickets per item whatever its tile
