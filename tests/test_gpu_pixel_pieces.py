"""Ingest and requantise where their warps' pieces have edges: rows that end inside, at and just
past a lane's 4 columns and a warp's 128, two-row and one-block images, sample planes whose rows
are and are not aligned to a lane's accesses, float planes of an odd pitch.  Against the FP64
oracle, within the bounds of the per-stage tests."""
import numpy as np
import pytest
import torch

import oracle
import paper_2308_03121_gb300 as nv
from gpu_util import assert_codes_match, fmt_dict, from_dev, prequant

pytestmark = pytest.mark.gpu

SIZES = [(2, 2), (4, 2), (6, 8), (126, 4), (128, 2), (130, 6), (132, 2), (254, 2), (256, 4), (258, 2), (514, 4)]
FORMS = [(8, "420", "left"), (10, "420", "left"), (8, "420", "center"), (10, "420", "center"), (12, "420", "point"),
         (8, "444", "left"), (10, "444", "left")]


def plane(H, W, bits, shift):
    """A device plane whose rows start `shift` samples into a wider buffer of an odd pitch."""
    dt = torch.uint8 if bits <= 8 else torch.int16
    return torch.full((H, W + 2 * shift + (1 if shift else 0)), 7, dtype=dt, device="cuda")[:, shift:shift + W]


@pytest.mark.parametrize("W,H", SIZES)
@pytest.mark.parametrize("bits,sub,loc", FORMS)
@pytest.mark.parametrize("shift", [0, 1])
def test_pieces(W, H, bits, sub, loc, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rs = np.random.default_rng(W * 31 + H * 7 + bits)
    cw, ch = (W // 2, H // 2) if sub == "420" else (W, H)
    dt = np.uint8 if bits <= 8 else np.uint16
    fr = {k: rs.integers(0, 1 << bits, size=(H, W) if k == "Y" else (ch, cw)).astype(dt) for k in "YUV"}
    fd, f = fmt_dict(W, H, bits, sub, "limited", loc), nv.fmt(W, H, bits, sub, "limited", loc)
    pitch = (W + 3) // 4 * 4 + 4
    dev = {}
    for k in "YUV":
        dev[k] = plane(*fr[k].shape, bits, shift)
        dev[k].copy_(torch.from_numpy(fr[k].view(np.int16) if bits > 8 else fr[k]).cuda())
    out = torch.full((3, H, pitch), float("nan"), device="cuda")
    nv.nvisr_ingest(f, dev["Y"], dev["U"], dev["V"], out)
    torch.cuda.synchronize()
    err = np.abs(out[:, :, :W].double().cpu().numpy() - oracle.ingest(fr, fd)).max()
    assert err < 8e-6, err  # values to about 2.3, FP32
    assert torch.isnan(out[:, :, W:]).all()

    rgb = rs.uniform(-0.08, 1.08, size=(3, H, W)).astype(np.float32)
    src = torch.zeros((3, H, pitch), device="cuda")
    src[:, :, :W] = torch.from_numpy(rgb).cuda()
    got = {k: plane(*fr[k].shape, bits, shift) for k in "YUV"}
    nv.nvisr_requant(f, src, got["Y"], got["U"], got["V"])
    torch.cuda.synchronize()
    assert_codes_match({k: from_dev(got[k], bits) for k in "YUV"}, prequant(rgb.astype(np.float64), fd), bits)
    if shift:  # nothing beside the rows
        for k in "YUV":
            wide = got[k].as_strided((got[k].shape[0], shift), (got[k].stride(0), 1), 0)
            assert (wide == 7).all()
