"""Frames whose width leaves a rest of 1 to 3 pixels to the groups of four that the packing of frames
works in, at the edge of a block (514 = 128 groups and two pixels) and below one group."""
import numpy as np
import pytest
import torch

import oracle
import paper_2308_03121_gb300 as nv
import synth
from gpu_util import assert_codes_match, fmt_dict, lsb_stats, prequant
from test_gpu_filter import run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nv.load()


NETS = {
    "tuple3_32ch": lambda: synth.net_tuple(synth.BASE_SEED + 94, frames=3, channels=32, nres=1),
    "tuple7_64ch": lambda: synth.net_tuple(synth.BASE_SEED + 95, frames=7, channels=64, nres=1),
    "group": lambda: synth.net_group_general(synth.BASE_SEED + 96, 1, True, False, False),
}


@pytest.mark.parametrize("net,prec,W", [("tuple3_32ch", "fp32", 514), ("tuple3_32ch", "fp32", 2),
                                        ("tuple3_32ch", "bf16", 514), ("tuple7_64ch", "bf16", 514),
                                        ("group", "bf16", 514)])
def test_every_column_is_packed(net, prec, W):
    H, N = 6, 4
    frames = synth.frames_textured(synth.BASE_SEED + 97, N, W, H, 10, "420", "limited")
    flags = np.zeros(N, bool)
    text, blob = NETS[net]()
    fdi, fdo = fmt_dict(W, H, 10), fmt_dict(2 * W, 2 * H, 10)
    ref = oracle.run_filter(frames, flags, text, blob, fdi, fdo, keep_float=True)
    outs, _ = run_gpu(text, blob, frames, flags, nv.fmt(W, H, 10), nv.fmt(2 * W, 2 * H, 10), prec)
    assert len(outs) == len(ref)
    for got, r in zip(outs, ref):
        pq = prequant(r, fdo)
        if prec == "fp32":
            assert_codes_match(got, pq, 10)
        else:
            mx, _ = lsb_stats(got, {k: oracle.quantise(pq[k], 10) for k in "YUV"})
            assert mx <= 1, mx


def test_batched_pack_equals_each_stream_alone():
    """Two streams of 514 columns through one batch, whose heads read packed tuples, against each
    stream alone, whose head reads the frames themselves."""
    W, H, N = 514, 6, 4
    text, blob = synth.net_tuple(synth.BASE_SEED + 98, frames=5, channels=64, nres=1)
    clips = [synth.frames_textured(synth.BASE_SEED + 99 + k, N, W, H, 10, "420", "limited") for k in range(2)]
    fi, fo = nv.fmt(W, H, 10), nv.fmt(2 * W, 2 * H, 10)
    want = [run_gpu(text, blob, c, np.zeros(N, bool), fi, fo, "bf16")[0] for c in clips]
    eng = nv.Engine()
    flts = [eng.filter(text, blob, fi, fo, "bf16", 2) for _ in clips]
    batch = eng.batch(flts)
    for i in range(N):
        for f, c in zip(flts, clips):
            assert f.push((c[i]["Y"], c[i]["U"], c[i]["V"])) == nv.Status.OK
    for f in flts:
        f.flush()
    for t in range(N):
        assert batch.step() == 2
        for k, f in enumerate(flts):
            out = f.alloc_out_host()
            st, _ = f.pull(out)
            assert st == nv.Status.OK
            for p, name in zip(out, "YUV"):
                assert np.array_equal(p.astype(np.int64), want[k][t][name]), (t, k, name)
    batch.close()
    eng.close()
