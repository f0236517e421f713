"""The batch's cull and apply (csrc/batch.cu) at their edges, against the same strokes one call at a time: full
queues of 64 strokes with more lassos than a warp takes in one go, tiles of every side, and textures whose
tiles end inside a unit of four and inside a super-tile, with and without texture padding."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import gpu_atlas, to_dev
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu

SHAPES = [(64, 40, 8), (204, 130, 8), (300, 170, 16), (524, 260, 16), (204, 130, 32), (160, 150, 64), (384, 256, 128)]


@pytest.mark.parametrize("pads", [False, True])
@pytest.mark.parametrize("n_sphere,n_lasso", [(64, 0), (24, 40), (1, 1)])
def test_batch_equals_single_calls(n_sphere, n_lasso, pads):
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    rng = np.random.default_rng(n_sphere + pads)
    models, queues, want = [], [], []
    for i, (W, H, T) in enumerate(SHAPES):
        m, a = gpu_atlas(mesh, W, H, T)
        cams = [synth.orbit_camera(mesh, 240, 180, rng) for _ in range(2)]
        cds = []
        for c in cams:
            cam = lcl.lcl_camera_from_vp(a, c.vp, 240, 180)
            d = torch.empty((180, 240), dtype=torch.float32, device="cuda")
            lcl.lcl_depth_render(m, a, cam, d)
            cds.append((cam, d))
        flags = [lcl.pad_flags(int(rng.integers(1, 9)), int(rng.integers(1, 9))) if pads and rng.random() < 0.4 else 0
                 for _ in range(n_sphere + n_lasso)]
        queue = []
        for e in rng.permutation(n_sphere + n_lasso):
            label = int(e) * 3 + 1
            if e < n_sphere:
                st = synth.sphere_strokes(mesh, 1, 100 * i + int(e), 0.02, 0.5, 1, 255)
                rec = lcl.lcl_quantize_sphere(a, st.centre[0], st.radius[0], label)
                rec["flags"] = flags[e]
                queue.append(("sphere", rec))
            else:
                cam, d = cds[e % 2]
                poly = synth.star_lasso((float(rng.uniform(60, 180)), float(rng.uniform(40, 140))),
                                        int(rng.integers(3, 65)), float(rng.uniform(10, 90)), rng)
                queue.append(("lasso", (cam, d, poly, label, lcl.DEFAULT_BIAS, flags[e])))
        init = rng.integers(0, 5, size=(H, W)).astype(np.uint8)
        seq = to_dev(init)
        for kind, v in queue:
            if kind == "sphere":
                lcl.lcl_select_sphere(a, seq, np.array([v], lcl.SPHERE_DTYPE))
            else:
                lcl.lcl_select_lasso(a, seq, v[0], v[1], v[2], v[3], v[4], flags=v[5])
        models.append((a, to_dev(init)))
        queues.append(queue)
        want.append(seq)
    lcl.lcl_batch_edit(lcl.Batch(models, queues))
    torch.cuda.synchronize()
    for (_, layer), w, shape in zip(models, want, SHAPES):
        assert torch.equal(layer, w), shape
