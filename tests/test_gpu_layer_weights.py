"""Layer calls in a row on the same working memory, each with other weights and biases than the call
before: every call's kernel reads its own, however short the launches around the layout are."""
import numpy as np
import pytest
import torch

import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu


def _calls(kind, rs, h, w):
    t = lambda *s, k=1.0: torch.from_numpy((rs.uniform(-1, 1, size=s) * k).astype(np.float32)).cuda()
    if kind in ("block_fused", "block_unfused"):
        x = t(64, h, w)
        return lambda p: nv.nvisr_resblock2d("bf16", x, p[0], p[1], p[2], p[3], fused=kind == "block_fused"), \
            lambda: (t(64, 64, 3, 3, k=0.1), t(64), t(64, 64, 3, 3, k=0.1), t(64))
    if kind == "dcn":
        x, off, mask = t(64, h, w), t(144, h, w, k=3.0), t(72, h, w).abs()
        return lambda p: nv.nvisr_dcn2d("bf16", x, off, mask, p[0], p[1], 8), lambda: (t(64, 64, 3, 3, k=0.1), t(64))
    name, prec, cin, cout, k = kind
    x = t(cin, h, w)
    call = nv.nvisr_conv2d_static if name == "static" else nv.nvisr_conv2d
    return lambda p: call(prec, x, p[0], p[1], 1), lambda: (t(cout, cin, k, k, k=0.1), t(cout))


@pytest.mark.parametrize("h,w", [(1, 1), (9, 131)])
@pytest.mark.parametrize("kind", [("conv", "fp32", 64, 64, 3), ("conv", "fp16", 64, 64, 3), ("conv", "bf16", 16, 48, 3),
                                  ("conv", "bf16", 128, 64, 1), ("conv", "fp8", 64, 64, 3),
                                  ("static", "fp16", 64, 64, 3), ("static", "bf16", 64, 16, 3), "block_fused",
                                  "block_unfused", "dcn"], ids=str)
def test_each_call_reads_its_own_weights(kind, h, w):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nv.load()
    run, params = _calls(kind, np.random.default_rng(7), h, w)
    sets = [params() for _ in range(3)]
    want = [run(p).clone() for p in sets]
    assert not torch.equal(want[0], want[1]) and not torch.equal(want[1], want[2])
    for i in range(60):
        assert torch.equal(run(sets[i % 3]), want[i % 3]), i
