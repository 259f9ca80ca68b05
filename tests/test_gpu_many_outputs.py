"""A layer call with more output channels than the weights' layout launch has threads: every bias
is read, and nothing of an earlier call in the kept memory is."""
import pytest
import torch

import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cout", [311296 + 17, 700000])
@pytest.mark.parametrize("static", [False, True])
def test_every_bias_is_laid_out(cout, static):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if static and cout > 500000:
        pytest.skip("larger than the static area")
    nv.load()
    call = nv.nvisr_conv2d_static if static else nv.nvisr_conv2d
    # fills the working memory with something else
    px = 200 if static else 1024
    filled = torch.full((64, px, 300), 7.5, device="cuda")
    call("fp32", filled, torch.ones((16, 64, 1, 1), device="cuda"), torch.zeros(16, device="cuda"))
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    x = torch.full((1, 1, 1), 0.75, device="cuda")
    w = torch.randn((cout, 1, 1, 1), generator=g, device="cuda")
    b = torch.randn((cout,), generator=g, device="cuda")
    y = call("fp32", x, w, b)
    # one product and one sum, each rounded to float32
    assert torch.equal(y.flatten(), w.flatten() * 0.75 + b)
