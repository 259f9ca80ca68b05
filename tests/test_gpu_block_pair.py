"""The fused residual block where its work split has edges: the last single column tile of an odd
count cut into two halves (odd and even heights, one row), tiles that just fit or just spill
over 126 and 252 pixels, and strips of a row or two.  The same values as two single-layer
launches, bit for bit."""
import numpy as np
import pytest
import torch

import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 126), (3, 127), (1, 252), (5, 253), (7, 378), (8, 379), (33, 60), (64, 64), (19, 1300)]


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("H,W", SIZES)
def test_block_edges_equal_two_launches(prec, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rs = np.random.default_rng(1000 * H + W)
    c = lambda a: torch.from_numpy(np.asarray(a, np.float32)).cuda()
    std = np.sqrt(2.0 / 576)
    x = c(rs.uniform(-1, 1, size=(64, H, W)))
    w1, w2 = (c(rs.normal(size=(64, 64, 3, 3)) * std) for _ in range(2))
    b1, b2 = (c(rs.uniform(-0.1, 0.1, size=64)) for _ in range(2))
    fused = nv.nvisr_resblock2d(prec, x, w1, b1, w2, b2, fused=True)
    plain = nv.nvisr_resblock2d(prec, x, w1, b1, w2, b2, fused=False)
    torch.cuda.synchronize()
    assert torch.isfinite(fused).all()
    assert torch.equal(fused, plain)
