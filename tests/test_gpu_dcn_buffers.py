"""Buffers of a filter's deformable layers: their copy of the input may lie in memory that holds
nothing at that moment, whatever the order of the network's layers."""
import numpy as np
import pytest
import torch

import oracle
import paper_2308_03121_gb300 as nv
import synth
from gpu_util import fmt_dict, lsb_stats, prequant
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


def _two_frame_net(scale, nres, dead_end=False, narrow=""):
    """Two frames -> one output: extract, offset/mask head, deformable layer, nres residual blocks,
    output layer.  dead_end adds layers after the deformable one that nothing reads: the last needs a
    buffer that is idle before.  narrow: a deformable layer's input is also concatenated with 16
    channels of frame 1, so that it is blocked by 8 channels: that of a second layer ("chain", which
    without the dead ends gathers from the input itself), or that of the only layer, at half size
    ("pool", whose pixel pairs lie in two idle buffers)."""
    rng = np.random.default_rng(synth.BASE_SEED + 92)
    C, G = 64, 8
    spec = synth.NetSpec("group", 2, scale, "bilinear", flags="extra")
    spec.conv(rng, "f0", "frame0", 3, C, act="lrelu")
    spec.conv(rng, "f1", "frame1", 3, 16 if narrow == "pool" else C, act="lrelu", share=None if narrow == "pool" else "f0")
    rows = np.ones(27 * G)
    rows[: 18 * G] = synth.OFFSET_GAIN
    if narrow == "pool":
        spec.pool("p0", "f0", C)
        spec.pool("p1", "f1", 16)
        spec.conv(rng, "mix", "p0,p1", C + 16, C)
        spec.conv(rng, "om", "mix", C, 27 * G, row_gains=rows)
        spec.dcn(rng, "al", "p0", "om", C, C, G)
        spec.up("ua", "al", C)
        prev = "ua"
    else:
        spec.conv(rng, "om", "f0,f1", 2 * C, 27 * G, row_gains=rows)
        spec.dcn(rng, "al", "f0", "om", C, C, G)
        prev = "al"
    if narrow == "chain":
        spec.conv(rng, "g1", "frame1", 3, 16, act="lrelu")
        spec.conv(rng, "mix", "al,g1", C + 16, C)
        spec.conv(rng, "om2", "mix", C, 27 * G, row_gains=rows)
        spec.dcn(rng, "al2", "al", "om2", C, C, G)
        prev = "al2"
    for i in range(nres):
        spec.conv(rng, f"r{i}a", prev, C, C, act="lrelu")
        spec.conv(rng, f"r{i}b", f"r{i}a", C, C, add=prev, gain=synth.RES_GAIN)
        prev = f"r{i}b"
    if dead_end:
        for k in range(3 if narrow else 2):
            spec.conv(np.random.default_rng(k), f"dead{k}", prev, C, C)
    spec.conv(rng, "tail", prev, C, 3 * scale * scale, ps=2 if scale == 2 else None, gain=synth.TAIL_GAIN)
    spec.out("tail", skip="frame0")
    return spec.build()


# scale, residual blocks, layers nothing reads, device memory of the 70 x 38 filter with one copy of
# the deformable layer's input (128 bytes a pixel)
FORMS = [(1, 0, False, 6632960), (1, 0, True, 7268864), (2, 1, False, 7250688), (2, 0, False, 6614784)]


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("scale,nres,dead_end,need", FORMS)
def test_deformable_layer_needs_one_copy_of_its_input(scale, nres, dead_end, need, prec):
    """Networks at scale 1 and 2, whose output images are too small for half of the pixel pairs, with
    and without an idle tensor that is not: the filter fits a budget of what it needs with one copy
    of the layer's input, and its outputs are the oracle's within one code."""
    W, H, N = 70, 38, 3
    frames = synth.frames_textured(synth.BASE_SEED + 93, N, W, H, 8, "420", "limited")
    flags = np.zeros(N, bool)
    text, blob = _two_frame_net(scale, nres, dead_end)
    fi, fo = nv.fmt(W, H, 8), nv.fmt(scale * W, scale * H, 8)
    eng = nv.Engine(hbm_budget_bytes=need)
    eng.filter(text, blob, fi, fo, prec, scale)
    eng.close()
    fdo = fmt_dict(scale * W, scale * H, 8)
    ref = oracle.run_filter(frames, flags, text, blob, fmt_dict(W, H, 8), fdo, keep_float=True)
    outs, _ = run_gpu(text, blob, frames, flags, fi, fo, prec, scale=scale, options=nv.OPT_GUARD_BANDS)
    assert len(outs) == len(ref) > 0
    for got, r in zip(outs, ref):
        pq = prequant(r, fdo)
        mx, _ = lsb_stats(got, {k: oracle.quantise(pq[k], 8) for k in "YUV"})
        assert mx <= 1, mx


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("narrow", ["", "chain", "pool"])
def test_gather_from_planes_equals_gather_from_pairs(prec, narrow):
    """The same network with and without the idle buffers that layers nothing reads bring, bit for bit:
    pixel pairs against 8-channel planes or the input itself; and the oracle's codes within one."""
    W, H, N = 70, 38, 3
    frames = synth.frames_textured(synth.BASE_SEED + 93, N, W, H, 10, "444", "full")
    flags = np.zeros(N, bool)
    fm = nv.fmt(W, H, 10, "444", "full")
    a, _ = run_gpu(*_two_frame_net(1, 0, False, narrow), frames, flags, fm, fm, prec, scale=1)
    b, _ = run_gpu(*_two_frame_net(1, 0, True, narrow), frames, flags, fm, fm, prec, scale=1)
    fd = fmt_dict(W, H, 10, "444", "full")
    ref = oracle.run_filter(frames, flags, *_two_frame_net(1, 0, False, narrow), fd, fd, keep_float=True)
    assert len(a) == len(b) == len(ref) > 0
    for x, y, r in zip(a, b, ref):
        for k in "YUV":
            assert np.array_equal(x[k], y[k]), k
        pq = prequant(r, fd)
        mx, _ = lsb_stats(x, {k: oracle.quantise(pq[k], 10) for k in "YUV"})
        assert mx <= 1, mx
