"""Layer calls whose output partly overlaps an input: where the kernel would read what it has
overwritten it works on copies, so the values are those of a call on memory of its own."""
import pytest
import torch

import paper_2308_03121_gb300 as nv

pytestmark = pytest.mark.gpu
H, W = 9, 131
N = H * W


@pytest.mark.parametrize("entry", ["nvisr_conv2d", "nvisr_conv2d_static"])
@pytest.mark.parametrize("prec,cin,cout,k", [("fp32", 64, 64, 3), ("fp32", 8, 16, 1), ("bf16", 64, 64, 3),
                                             ("fp16", 64, 64, 3), ("bf16", 16, 48, 3)])
@pytest.mark.parametrize("over", ["x", "res"])
@pytest.mark.parametrize("shift", [-N - 3, -1, 1, 4, N + 3])
def test_output_partly_over_an_input(entry, prec, cin, cout, k, over, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = nv.load()
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    rand = lambda *s: torch.rand(s, generator=g, device="cuda") * 2 - 1
    w, b = rand(cout, cin, k, k) * 0.1, rand(cout)
    pad = 2 * N
    buf = rand(pad + (cin + cout) * N + pad)
    other = rand(max(cin, cout) * N)
    n_in = (cin if over == "x" else cout) * N
    inside = buf[pad:pad + n_in]
    x, r = (inside, other[:cout * N]) if over == "x" else (other[:cin * N], inside)
    y = buf[pad + shift:pad + shift + cout * N]
    want = getattr(nv, entry)(prec, x.reshape(cin, H, W).clone(), w, b, 1, r.reshape(cout, H, W).clone())
    st = getattr(lib, entry)(nv.PREC[prec], x.data_ptr(), cin, H, W, w.data_ptr(), b.data_ptr(), cout, k, 1, r.data_ptr(),
                             y.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert st == nv.Status.OK
    torch.cuda.synchronize()
    assert torch.equal(y.reshape(cout, H, W), want)
