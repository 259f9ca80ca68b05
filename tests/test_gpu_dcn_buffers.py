"""Buffers of a filter's deformable layers: their copy of the input may lie in memory that holds
nothing at that moment, whatever the order of the network's layers."""
import numpy as np
import pytest
import torch

import paper_2308_03121_gb300 as nv
import synth
from test_gpu_filter import run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nv.load()


def _first_output_first(text, blob):
    """The network with frame 0's trunk and output layer described before the alignment."""
    lines = text.splitlines()
    at = 0
    early, rest, ew, rw = [], [], [], []
    for line in lines:
        tok = line.split()
        is_layer = tok[0] in ("conv", "dcn")
        kv = dict(t.split("=") for t in tok[2:]) if is_layer else {}
        n = 0
        if is_layer and "share" not in kv:
            k = int(kv.get("k", 3))
            n = int(kv["cout"]) * int(kv["cin"]) * k * k + int(kv["cout"])
        e = not is_layer or tok[1][0] in "ft"
        if tok[0] == "out":
            e = False
        (early if e else rest).append(line)
        (ew if e else rw).append(blob[at:at + n])
        at += n
    assert at == len(blob)
    return "\n".join(early + rest) + "\n", np.concatenate(ew + rw)


def test_output_described_before_the_alignment():
    """A 4x network gives the same outputs whether its first output layer comes before the
    deformable layers or after them, bit for bit (70 x 38: ragged tiles)."""
    W, H, N = 70, 38, 4
    frames = synth.frames_textured(synth.BASE_SEED + 90, N, W, H, 8, "420", "limited")
    flags = np.zeros(N, bool)
    text, blob = synth.net_group_stvsr(synth.BASE_SEED + 91, nres=1)
    early = _first_output_first(text, blob)
    order = [line.split()[1] for line in early[0].splitlines() if line.startswith(("conv", "dcn"))]
    assert order.index("tu2") < order.index("a0")
    fi, fo = nv.fmt(W, H, 8), nv.fmt(4 * W, 4 * H, 8)
    want, _ = run_gpu(text, blob, frames, flags, fi, fo, "bf16", scale=4)
    got, _ = run_gpu(*early, frames, flags, fi, fo, "bf16", scale=4)
    assert len(want) == len(got) == 2 * N
    for t, (a, b) in enumerate(zip(want, got)):
        for k in "YUV":
            assert np.array_equal(a[k], b[k]), (t, k)
