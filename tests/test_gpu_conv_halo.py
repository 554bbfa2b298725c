"""Stride-1 convolutions on halo tiles at the edges of their pixel blocks,
channel groups and filter tiles, against fp64."""
import numpy as np
import pytest

from helpers import dev, empty_dev, stream_handle
from oracle import resnet as orr
from paper_2609_10018_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,C,N,k,pad,relu,columns", [
    (3, 56, 56, 64, 64, 3, 1, True, 64),      # filter resident; odd number of blocks per pair
    (1, 5, 9, 40, 24, 3, 1, True, 32),        # one block: the pair's second CTA has none
    (7, 30, 57, 136, 88, 3, 1, False, 96),    # ragged blocks in both axes, three channel groups
    (5, 28, 28, 128, 200, 3, 0, True, 64),    # no padding; filter streamed, four tiles, the last 8 channels wide
    (9, 14, 14, 256, 520, 3, 1, True, 96),    # filter streamed, six tiles not a multiple of 64 wide
    (2, 17, 140, 24, 16, 5, 2, True, 16),     # 5 x 5, image wider than a block
    (4, 8, 8, 256, 64, 2, 0, False, 64),      # even kernel
    (128, 56, 56, 16, 16, 3, 1, True, 16),    # 16-wide filter taps: one K step a tap
    (128, 31, 29, 8, 24, 3, 1, False, 32),    # half a K step
])
def test_halo_convolution_matches_fp64(B, H, W, C, N, k, pad, relu, columns):
    import torch
    assert binding.elasto_op_conv2d_tile(B, H, W, C, N, k, 1, pad).fields() == (columns, 1, 1, 0)
    rng = np.random.default_rng(B * 100 + H + C + N)
    x = rng.standard_normal((B, H, W, C)).astype(np.float16)
    w = (rng.standard_normal((N, C, k, k)) * np.sqrt(2.0 / (C * k * k))).astype(np.float16)
    bias = (rng.standard_normal(N) * 0.1).astype(np.float32)
    packed = np.zeros((N, k, k, 16 if C <= 16 else (C + 63) // 64 * 64), np.float16)
    packed[..., :C] = w.transpose(0, 2, 3, 1)
    ref = orr.conv2d(x.astype(np.float64), w.astype(np.float64), 1, pad) + bias
    if relu:
        ref = np.maximum(ref, 0)
    out = empty_dev(ref.shape, torch.uint16)
    out.fill_(0x7E00)  # f16 NaN: every output must be written
    dx, dw, db = dev(x.view(np.uint16)), dev(packed.view(np.uint16)), dev(bias)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.elasto_op_conv2d(stream_handle(), dx.data_ptr(), B, H, W, C, dw.data_ptr(), N, k, 1, pad, db.data_ptr(),
                             relu, out.data_ptr(), status.data_ptr())
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = out.cpu().numpy().view(np.float16).astype(np.float64)
    assert np.all(np.isfinite(got))
    # one f16 rounding (2^-11 relative, doubled) and fp32 accumulation
    assert np.all(np.abs(got - ref) <= 2.0 ** -10 * np.abs(ref) + 1e-4 * np.max(np.abs(ref)))


@pytest.mark.parametrize("stride", [1, 2])  # halo tiles, and a box per tap
@pytest.mark.parametrize("which", ["x", "w", "out"])
def test_misaligned_pointers_are_refused(stride, which):
    """Every pointer that is not 16-byte aligned is refused before a launch."""
    import torch
    assert binding.elasto_op_conv2d_tile(2, 28, 28, 64, 64, 3, stride, 1).halo == (stride == 1)
    buf = {k: torch.zeros(1 << 20, dtype=torch.float16, device="cuda") for k in ("x", "w", "out")}
    ptr = {k: v.data_ptr() + (8 if k == which else 0) for k, v in buf.items()}
    with pytest.raises(binding.ElastoError) as e:
        binding.elasto_op_conv2d(stream_handle(), ptr["x"], 2, 28, 28, 64, ptr["w"], 64, 3, stride, 1, None, True,
                                 ptr["out"])
    assert e.value.status == binding.ERR_UNSUPPORTED
