"""The FP32 3x3 layer at the edges of its tiles (64 pixels x 2 rows; 16, 32 or 64 outputs;
slices of 8 input channels), straight on the caller's planar tensors, and in place.  Against a
64-bit convolution within the FP32 layer's tolerance (2e-5 for inputs in [-1, 1])."""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu


def _inputs(cin, cout, H, W):
    rs = np.random.default_rng(cin * 7 + cout * 3 + W)
    c = lambda a: torch.from_numpy(np.asarray(a, np.float32)).cuda()
    return (c(rs.uniform(-1, 1, size=(cin, H, W))), c(rs.normal(size=(cout, cin, 3, 3)) * np.sqrt(2.0 / (9 * cin))),
            c(rs.uniform(-0.1, 0.1, size=cout)), c(rs.uniform(-1, 1, size=(cout, H, W))))


@pytest.mark.parametrize("cin,cout,H,W,act,res", [
    (3, 16, 1, 1, 0, False), (64, 64, 1, 64, 1, True), (9, 64, 9, 65, 0, True), (8, 32, 7, 63, 1, False),
    (16, 96, 5, 66, 0, True), (64, 12, 17, 127, 1, True), (32, 48, 4, 129, 0, False), (64, 64, 150, 700, 1, True),
    (64, 64, 250, 330, 0, False)])
def test_fp32_layer_matches_64_bit(cin, cout, H, W, act, res):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x, w, b, r = _inputs(cin, cout, H, W)
    y = nv.nvisr_conv2d("fp32", x, w, b, act, r if res else None)
    torch.cuda.synchronize()
    ref = F.conv2d(x.double().cpu()[None], w.double().cpu(), b.double().cpu(), padding=1)[0]
    if act:
        ref = torch.where(ref >= 0, ref, 0.1 * ref)
    if res:
        ref = ref + r.double().cpu()
    assert (y.double().cpu() - ref).abs().max() < 2e-5


def test_fp32_layer_in_place():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x, w, b, _ = _inputs(64, 64, 21, 90)
    want = nv.nvisr_conv2d_static("fp32", x, w, b, 1, x)
    got = nv.nvisr_conv2d_static("fp32", x, w, b, 1, x, out=x)
    torch.cuda.synchronize()
    assert got.data_ptr() == x.data_ptr() and torch.equal(got, want)
