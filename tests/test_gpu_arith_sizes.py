"""Arithmetic overlays of float layers, which load ahead (csrc/numeric.cu), with several chunks per thread, a partial
last mask word, results in place, and a scalar; every bit against torch."""
import pytest
import torch

import synth
from gpu_util import gpu_atlas
from paper_2501_14807_gb300 import lcl

pytestmark = pytest.mark.gpu


def bits(words, n):
    return ((words[:, None] >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).bool().reshape(-1)[:n]


@pytest.mark.parametrize("W,H", [(1500, 1001), (1764, 1763), (2500, 2501)])
@pytest.mark.parametrize("ty", ["f16", "f32"])
@pytest.mark.parametrize("form", ["layers", "in place", "scalar"])
def test_float_arith(W, H, ty, form):
    mesh = synth.vessel_charts(80, 40, 20, 10, 512, seed=6)
    _, a = gpu_atlas(mesh, W, H, 32)
    g = torch.Generator("cuda").manual_seed(W)
    A, B = lcl.NumericLayer(W, H, ty), lcl.NumericLayer(W, H, ty)
    for layer in (A, B):
        layer.data.copy_(torch.randn((H, W), device="cuda", generator=g))
        layer.mask.copy_(torch.randint(-2 ** 31, 2 ** 31, (layer.mask.numel(),), device="cuda", generator=g, dtype=torch.int64))
    n = W * H
    ok = bits(A.mask, n) & bits(a.cover(), n)
    x, y = A.data.float(), B.data.float()
    if form == "scalar":
        y = torch.full_like(x, 0.25)
    else:
        ok &= bits(B.mask, n)
    exp = torch.where(ok.view(H, W), (x - y).to(A.data.dtype), 0.0)
    out = A if form == "in place" else lcl.NumericLayer(W, H, ty)
    if form == "scalar":
        lcl.lcl_numeric_arith(a, A, None, out, "sub", int(torch.tensor(0.25, dtype=A.data.dtype).view(
            torch.int16 if ty == "f16" else torch.int32)))
    else:
        lcl.lcl_numeric_arith(a, A, B, out, "sub")
    assert torch.equal(out.data, exp.to(out.data.dtype)) and torch.equal(bits(out.mask, n), ok) and bool(ok.any())
