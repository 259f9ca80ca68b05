"""The tensor-core deformable convolution where its gather has edges: samples left, right, above
and below the image by whole and fractional pixels, one-pixel-wide and one-row images, row ends
inside and at the end of a warp's 32 pixels and a tile's 128, every group count.  Against the
FP64 oracle on operands rounded as the kernel stores them, within two half-ulps of the sum of
magnitudes (one rounding of the sample, one of the output)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("groups,H,W", [(8, 1, 1), (8, 9, 1), (4, 1, 33), (8, 6, 31), (2, 5, 32), (1, 4, 65), (8, 3, 127),
                                        (8, 2, 128), (4, 3, 129)])
def test_gather_edges_match_oracle(prec, groups, H, W):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rs = np.random.default_rng(100 * W + H)
    x = rs.uniform(-1, 1, size=(64, H, W)).astype(np.float32)
    # whole, half and any offsets up to past the image on every side
    off = rs.choice([-2.0, -1.5, -1.0, -0.5, 0.0, 0.25, 0.5, 1.0, 1.75, float(W), -float(H), float(H) + 0.5],
                    size=(18 * groups, H, W)).astype(np.float32)
    mask = rs.choice([0.0, 0.3, 1.0], size=(9 * groups, H, W)).astype(np.float32)
    w = (rs.normal(size=(64, 64, 3, 3)) * np.sqrt(2.0 / 576)).astype(np.float32)
    b = rs.uniform(-0.1, 0.1, size=64).astype(np.float32)
    got = nv.nvisr_dcn2d(prec, *(torch.from_numpy(a).cuda() for a in (x, off, mask, w, b)), groups)
    torch.cuda.synchronize()
    dt = torch.bfloat16 if prec == "bf16" else torch.float16
    q = lambda a: torch.from_numpy(a).to(dt).double().numpy()
    ref = oracle.dcn2d(q(x), off, mask, q(w), b, groups)
    mag = oracle.dcn2d(np.abs(q(x)), off, mask, np.abs(q(w)), None, groups)
    ulp = 2.0 ** -8 if prec == "bf16" else 2.0 ** -11
    err = np.abs(got.double().cpu().numpy() - ref)
    assert (err <= ulp * (mag + np.abs(ref)) + 1e-5).all(), err.max()
