"""The 64 -> 64 tensor-core layers and residual blocks writing planar float32 themselves: tile
edges (128 and 126 pixels, odd heights, one row, one pixel), with and without residual and
activation, and onto a tensor that is also an input.  Layers within one rounding of the 64-bit layer
on rounded operands (and FP32 summation), blocks equal to their two layers."""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu
DT = {"bf16": torch.bfloat16, "fp16": torch.float16}
ULP = {"bf16": 2.0 ** -8, "fp16": 2.0 ** -11}


def _inputs(H, W, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rs = np.random.default_rng(H * 1000 + W)
    c = lambda a: torch.from_numpy(np.asarray(a, np.float32)).cuda()
    x, r = (c(rs.uniform(-1, 1, size=(64, H, W))) for _ in range(2))
    w = c(rs.normal(size=(64, 64, 3, 3)) * np.sqrt(2.0 / 576)).to(DT[prec]).float()
    return x, r, w, c(rs.uniform(-0.1, 0.1, size=64))


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("H,W", [(1, 1), (3, 127), (2, 128), (5, 129), (7, 253), (1, 300)])
@pytest.mark.parametrize("act,res", [(0, False), (1, True)])
def test_layer(prec, H, W, act, res):
    x, r, w, b = _inputs(H, W, prec)
    y = nv.nvisr_conv2d(prec, x, w, b, act, r if res else None)
    s = nv.nvisr_conv2d_static(prec, x, w, b, act, r if res else None)
    torch.cuda.synchronize()
    assert torch.equal(y, s) and torch.equal(y, y.to(DT[prec]).float())
    q = lambda t: t.to(DT[prec]).double().cpu()
    ref = F.conv2d(q(x)[None], q(w), b.double().cpu(), padding=1)[0]
    mag = F.conv2d(q(x).abs()[None], q(w).abs(), b.double().cpu().abs(), padding=1)[0]
    if act:
        ref = torch.where(ref >= 0, ref, 0.1 * ref)
    if res:
        ref = ref + q(r)
    # one rounding of the output, FP32 sums of 577 terms
    assert ((y.double().cpu() - ref).abs() <= ULP[prec] * ref.abs() + 1e-5 * (1 + mag)).all()


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_in_place(prec):
    x, _, w, b = _inputs(9, 200, prec)
    want = nv.nvisr_conv2d_static(prec, x, w, b, 1, x)
    got = nv.nvisr_conv2d_static(prec, x, w, b, 1, x, out=x)
    torch.cuda.synchronize()
    assert got.data_ptr() == x.data_ptr() and torch.equal(got, want)


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("H,W", [(1, 1), (2, 125), (5, 126), (4, 127), (9, 252), (3, 253), (40, 380)])
def test_block_equals_two_layers(prec, H, W):
    x, _, w, b = _inputs(H, W, prec)
    y = nv.nvisr_resblock2d(prec, x, w, b, w.flip(0).contiguous(), b)
    h = nv.nvisr_conv2d(prec, x, w, b, 1)
    want = nv.nvisr_conv2d(prec, h, w.flip(0).contiguous(), b, 0, x)
    torch.cuda.synchronize()
    assert torch.equal(y, want)
