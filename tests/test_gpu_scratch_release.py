"""The device memory that the layer calls keep: how much stays, and what gives it back."""
import threading

import pytest
import torch

import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu

MB = 1 << 20
SLACK = 16 * MB  # allocation granularity


def _call(mpix):
    """A 1x1 FP32 layer of 8 -> 16 channels, whose working memory is 96 bytes a pixel."""
    n = int(mpix * 1e6)
    nv.nvisr_conv2d("fp32", torch.ones((8, 1, n), device="cuda"), torch.ones((16, 8, 1, 1), device="cuda"), None)
    return 96 * n


def _used():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.fixture
def base():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nv.load()
    _call(0.1)  # the kernels' code is loaded
    nv.nvisr_release_scratch()
    yield _used()
    nv.nvisr_release_scratch()


def test_release_gives_the_kept_memory_back(base):
    size = _call(5)
    assert size - SLACK <= _used() - base <= size + SLACK
    nv.nvisr_release_scratch()
    assert _used() - base <= SLACK
    _call(5)  # from a thread that has made no CUDA call
    t = threading.Thread(target=nv.nvisr_release_scratch)
    t.start()
    t.join()
    assert _used() - base <= SLACK


def test_an_engine_that_goes_takes_the_kept_memory_along(base):
    eng = nv.Engine()
    with_engine = _used()
    size = _call(5)
    assert _used() - with_engine >= size - SLACK
    eng.close()
    assert _used() - base <= SLACK


def test_kept_memory_is_bounded(base):
    sizes = [_call(m) for m in (4, 5, 6)]  # 384 + 480 + 576 MB: the oldest goes
    assert sum(sizes[1:]) - SLACK <= _used() - base <= 1024 * MB + SLACK
    before = _used()
    assert _call(12) > 1024 * MB  # more than what is kept at all: not kept
    assert abs(_used() - before) <= SLACK


def test_an_allocation_that_would_fail_gives_the_kept_memory_back(base):
    size = _call(5)
    assert _used() - base >= size - SLACK
    eng = nv.Engine()
    text = "nvisr-net 1\nfamily tuple\nframes 1\nscale 2\nskip none\nconv t in=tuple cin=3 cout=12 k=3 act=none ps=2\nout t\n"
    blob = torch.zeros(12 * 27 + 12).numpy()
    side = 1 << 17  # a ring of frames far larger than the device
    with pytest.raises(nv.NvisrError) as e:
        eng.filter(text, blob, nv.fmt(side, side, 8), nv.fmt(2 * side, 2 * side, 8), "fp32", 2)
    assert e.value.status == nv.Status.OUT_OF_MEMORY
    assert _used() - base <= 2 * SLACK
    eng.close()
