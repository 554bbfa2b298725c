"""Weights that are the output of the call before on the same stream: the
kernel-level calls read them only after that call's kernel has finished."""
import pytest

from helpers import stream_handle
from paper_2609_10018_gb300 import binding

pytestmark = pytest.mark.gpu


# (a filter of one tile of 64 columns is kept in shared memory, more tiles are streamed)
@pytest.mark.parametrize("kind,C,N,stride", [
    ("conv", 64, 64, 1),     # halo tiles, filter kept
    ("conv", 256, 256, 1),   # halo tiles, filter streamed
    ("conv", 64, 64, 2),     # box per tap, filter kept
    ("conv", 256, 256, 2),   # box per tap, filter streamed
    ("gemm", 768, 200, 0),
])
def test_weights_from_the_call_before(kind, C, N, stride):
    import torch
    g = torch.Generator(device="cuda").manual_seed(C + N + stride)

    def f16(*shape, std=1.0):
        return (torch.randn(shape, generator=g, device="cuda") * std).half()

    depth, width = 16384, 9 * C if kind == "conv" else C  # a long reduction: the producer runs for a while
    a, b = f16(N, depth), f16(width, depth, std=0.05 / depth ** 0.5)
    w = torch.empty((N, width), dtype=torch.float16, device="cuda")
    s = stream_handle()

    def produce():
        binding.elasto_op_gemm(s, a.data_ptr(), b.data_ptr(), None, w.data_ptr(), None, N, width, depth,
                               binding.EPI_BIAS_F16)

    if kind == "conv":
        assert binding.elasto_op_conv2d_tile(2, 28, 28, C, N, 3, stride, 1).fields() == (64, stride == 1, stride == 1, 0)
        x = f16(2, 28, 28, C)
        out = torch.empty((2, 28 // stride, 28 // stride, N), dtype=torch.float16, device="cuda")

        def consume():
            binding.elasto_op_conv2d(s, x.data_ptr(), 2, 28, 28, C, w.data_ptr(), N, 3, stride, 1, None, 0,
                                     out.data_ptr())
    else:
        x = f16(300, C)
        out = torch.empty((300, N), dtype=torch.float16, device="cuda")

        def consume():
            binding.elasto_op_gemm(s, x.data_ptr(), w.data_ptr(), None, out.data_ptr(), None, 300, N, C,
                                   binding.EPI_BIAS_F16)

    produce()
    torch.cuda.synchronize()
    consume()
    torch.cuda.synchronize()
    want = out.clone()
    assert torch.isfinite(want).all()
    for _ in range(5):
        w.fill_(float("nan"))
        out.zero_()
        torch.cuda.synchronize()
        produce()
        consume()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
