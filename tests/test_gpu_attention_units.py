"""Attention at the edges of its work units: one query tile per item (both
softmax groups then take whole items in turn) or two, every number of whole
64-key chunks and of masked 16-key pieces after them, several items per CTA."""
import numpy as np
import pytest

from helpers import bf16_to_f64, dev, empty_dev, stream_handle
from oracle import vit as ov
from paper_2609_10018_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n,h", [
    (310, 64, 1), (153, 128, 2), (200, 100, 3), (77, 48, 4), (305, 33, 1),  # one query tile; odd items per CTA
    (160, 192, 2), (153, 193, 1), (90, 240, 2), (101, 255, 3), (3, 144, 5),  # two
])
def test_attention_units_match_fp64(B, n, h):
    import torch
    rng = np.random.default_rng(B + 1000 * n + h)
    x = rng.standard_normal((B, n, 3, h, 64), dtype=np.float32)
    x[:, n // 2, 1] *= 4.0  # one key with large scores
    qkv = synth.f32_to_bf16_bits(x)
    out = empty_dev((B, n, h * 64), torch.uint16)
    out.fill_(0x7FC0)  # bf16 NaN: every output must be written
    dq = dev(qkv)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.elasto_op_attention(stream_handle(), dq.data_ptr(), out.data_ptr(), B, n, h, status.data_ptr())
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = bf16_to_f64(out)
    assert np.all(np.isfinite(got))
    for b in np.unique(np.linspace(0, B - 1, 24).astype(int)):
        q = bf16_to_f64(qkv[b])
        ref = np.concatenate([ov.attention(q[:, 0, j], q[:, 1, j], q[:, 2, j], 64) for j in range(h)], axis=-1)
        # P and O are rounded to bf16 (2^-9 each, relative)
        assert np.max(np.abs(got[b] - ref)) <= 1e-2 * np.max(np.abs(ref)), (b, float(np.max(np.abs(got[b] - ref))))


@pytest.mark.parametrize("n", [256, 255])
def test_row_sum_keeps_small_numerators(n):
    """Four keys with numerator 1, the rest 0.98 * 2^-24 each: too small to change
    a partial sum near 1 alone, not in pairs. The values put every output at a
    bf16 rounding tie plus 24 * 2^-23 relative, between the exact denominator
    (30.9 * 2^-23 over 4) and the 15.7 * 2^-23 that is left where every second
    numerator is lost."""
    import torch
    x = np.zeros((1, n, 3, 1, 64), np.float32)
    x[..., 0, 0, :2] = 1.0
    x[..., 1, 0, :2] = (-133.0, -0.25)  # exp(-133.25 / 8) = 0.98 * 2^-24
    x[:, 0:8:2, 1] = 0.0
    for key, value in ((0, 1.0), (2, 2.0 ** -8), (4, 24 * 2.0 ** -23)):
        x[:, key, 2] = value
    dq, out = dev(synth.f32_to_bf16_bits(x)), empty_dev((1, n, 64), torch.uint16)
    binding.elasto_op_attention(stream_handle(), dq.data_ptr(), out.data_ptr(), 1, n, 1)
    torch.cuda.synchronize()
    assert np.all(bf16_to_f64(out) == 0.25)
