"""The kept working memory behind the per-call layer entry points: calls of different sizes on
several threads and streams at once give what the same calls give one after the other, and a
capturing stream is refused."""
import threading

import numpy as np
import pytest
import torch

import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu


def _job(seed):
    rs = np.random.default_rng(seed)
    c = lambda *s: torch.from_numpy(rs.uniform(-1, 1, size=s).astype(np.float32)).cuda()
    h, w = int(rs.integers(3, 60)), int(rs.integers(3, 300))
    x, wt, b = c(64, h, w), c(64, 64, 3, 3) * 0.06, c(64)
    off, mask = c(18 * 8, h, w) * 2, c(9 * 8, h, w).abs()
    kind = ("conv", "fp8", "block", "dcn")[seed % 4]
    if kind == "conv":
        return lambda st: nv.nvisr_conv2d("fp16", x, wt, b, 1, x, stream=st)
    if kind == "fp8":
        return lambda st: nv.nvisr_conv2d("fp8", x, wt, b, 0, stream=st)
    if kind == "block":
        return lambda st: nv.nvisr_resblock2d("bf16", x, wt, b, wt, None, stream=st)
    return lambda st: nv.nvisr_dcn2d("bf16", x, off, mask, wt, b, 8, stream=st)


def test_calls_on_threads_and_streams_do_not_share_memory():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nv.load()
    jobs = [_job(s) for s in range(16)]
    torch.cuda.synchronize()
    want = [j(None).clone() for j in jobs]
    got, errors = [[] for _ in range(4)], []

    def work(t):
        try:
            st = torch.cuda.Stream()
            for r in range(5):
                for k in range(t, 16, 4):
                    got[t].append((k, jobs[(k + r) % 16](st)))
                    got[t][-1] = ((k + r) % 16, got[t][-1][1])
        except Exception as e:  # noqa: BLE001 -- shown by the assertion below
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for per in got:
        assert len(per) == 20
        for k, y in per:
            assert torch.equal(y, want[k]), k


def test_capturing_stream_is_refused():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nv.load()
    job = _job(0)
    job(None)
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        g.capture_begin()
        try:
            with pytest.raises(nv.NvisrError):
                job(st)
        finally:
            g.capture_end()
    torch.cuda.synchronize()
    assert torch.equal(job(None), job(None))
