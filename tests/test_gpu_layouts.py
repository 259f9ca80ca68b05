"""The planar <-> blocked layout kernels of the layer entry points at the edges of their tiles
(32 pixels a warp, 128 a block), with planes that are and are not 16-byte aligned: a 1x1
convolution with identity weights gives its input back exactly, rounded to the precision."""
import pytest
import torch

import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("C", [64, 128, 24])
@pytest.mark.parametrize("H,W", [(1, 1), (1, 31), (4, 8), (3, 11), (1, 127), (8, 16), (3, 43), (5, 52), (20, 33)])
@pytest.mark.parametrize("shift", [0, 1])
def test_identity_layer_round_trips(prec, C, H, W, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cout = min(C, 64)
    if prec != "fp32" and C == 24:
        cout = C = 32  # the tensor-core layer's narrow form
    k = 1 if prec == "fp32" or C % 64 == 0 else 3
    g = torch.Generator(device="cuda").manual_seed(H * 1000 + W + C)
    x = torch.randn(C * H * W + shift, generator=g, device="cuda")[shift:].view(C, H, W)
    w = torch.zeros(cout, C, k, k, device="cuda")
    w[torch.arange(cout), torch.arange(cout), k // 2, k // 2] = 1.0
    y = nv.nvisr_conv2d(prec, x, w, None)
    torch.cuda.synchronize()
    dt = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[prec]
    assert torch.equal(y, x[:cout].to(dt).float())
