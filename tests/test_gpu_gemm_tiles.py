"""The GEMM's tile variants at their edges, against fp64: CTA pairs at short
reductions with ragged last rows and columns, the residual added by the store
or read ahead, CNN block outputs, and convolutions on pairs whose last pixel
block is missing. Each test first asserts that its sizes get the tile it is
meant for: (columns, pair, halo, pieces read ahead)."""
import numpy as np
import pytest

from helpers import bf16_to_f64, dev, empty_dev, stream_handle
from oracle import resnet as orr
from oracle import vit as ov
from paper_2609_10018_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def _bf16(rng, shape, scale=1.0):
    return synth.f32_to_bf16_bits(rng.standard_normal(shape, dtype=np.float32) * np.float32(scale))


@pytest.mark.parametrize("M,N,K,epi,tile", [
    (19457, 2312, 768, binding.EPI_BIAS_BF16, (256, 1, 0, 0)),       # pairs: one row, eight columns past the tiles
    (19457, 2312, 776, binding.EPI_BIAS_GELU_BF16, (256, 1, 0, 0)),  # pairs, K a remainder of a k-block
    (19713, 520, 264, binding.EPI_BIAS_GELU_BF16, (192, 0, 0, 0)),   # single CTAs, ragged in every direction
    (19713, 520, 1160, binding.EPI_BIAS_RESID_F32, (192, 1, 0, 0)),  # pairs, residual added by the store
    (25089, 776, 520, binding.EPI_BIAS_RESID_F32, (160, 1, 0, 1)),   # pairs, short reduction past the L2: read ahead
    (257, 64, 64, binding.EPI_BIAS_RESID_F32, (32, 0, 0, 2)),        # few tiles: residual read ahead
    (12289, 40, 192, binding.EPI_BIAS_RESID_F32, (64, 0, 0, 0)),     # narrow single tiles
])
def test_tile_edges_match_fp64(M, N, K, epi, tile):
    import torch
    assert binding.elasto_op_gemm_tile(M, N, K, epi).fields() == tile
    rng = np.random.default_rng(M + N + K)
    A, W = _bf16(rng, (M, K)), _bf16(rng, (N, K), 0.05)
    bias = rng.standard_normal(N).astype(np.float32)
    x0 = rng.standard_normal((M, N)).astype(np.float32)
    f32 = epi == binding.EPI_BIAS_RESID_F32
    out = dev(x0) if f32 else empty_dev((M, N), torch.uint16)
    if not f32:
        out.fill_(0x7FC0)  # bf16 NaN: every output must be written
    dA, dW, db = dev(A), dev(W), dev(bias)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.elasto_op_gemm(stream_handle(), dA.data_ptr(), dW.data_ptr(), db.data_ptr(), out.data_ptr(), None, M, N, K,
                           epi, status.data_ptr())
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = out.cpu().numpy().astype(np.float64) if f32 else bf16_to_f64(out)
    assert np.all(np.isfinite(got))
    rows = np.unique(np.concatenate([np.arange(min(M, 300)), rng.choice(M, 500), np.arange(max(0, M - 300), M)]))
    ref = bf16_to_f64(A[rows]) @ bf16_to_f64(W).T + bias
    if epi == binding.EPI_BIAS_GELU_BF16:
        ref = ov.gelu(ref)
    if f32:  # fp32 accumulation over K and one fp32 addition
        ref = ref + x0[rows]
        tol = 1e-5 * np.max(np.abs(ref))
    else:  # one bf16 rounding (2^-9 relative, doubled) and the GELU form's 2.5e-5
        tol = 2.0 ** -8 * np.abs(ref) + 3e-5 + 1e-5 * np.max(np.abs(ref))
    assert np.all(np.abs(got[rows] - ref) <= tol), float(np.max(np.abs(got[rows] - ref)))


@pytest.mark.parametrize("B,S,C,N,k,stride,tile", [
    (109, 7, 520, 512, 3, 1, (256, 1, 0, 0)),   # pairs; two images per block: 55 blocks, the last pair has one
    (99, 29, 200, 264, 3, 2, (192, 1, 0, 0)),   # pairs, strided; ragged pixel blocks and channels
    (77, 14, 136, 256, 3, 2, (128, 0, 0, 0)),   # single CTAs, strided, two images per block
    (41, 28, 256, 512, 1, 2, (192, 0, 0, 0)),   # single CTAs, strided projection
    (51, 29, 200, 264, 3, 1, (144, 1, 1, 0)),   # halo tiles, ragged pixel blocks and channels
])
def test_conv_tiles_match_fp64(B, S, C, N, k, stride, tile):
    import torch
    assert binding.elasto_op_conv2d_tile(B, S, S, C, N, k, stride, k // 2).fields() == tile
    rng = np.random.default_rng(B + S + C)
    x = rng.standard_normal((B, S, S, C)).astype(np.float16)
    w = (rng.standard_normal((N, C, k, k)) * np.sqrt(2.0 / (C * k * k))).astype(np.float16)
    bias = (rng.standard_normal(N) * 0.1).astype(np.float32)
    packed = np.zeros((N, k, k, (C + 63) // 64 * 64), np.float16)
    packed[..., :C] = w.transpose(0, 2, 3, 1)
    o = (S + 2 * (k // 2) - k) // stride + 1
    out = empty_dev((B, o, o, N), torch.uint16)
    out.fill_(0x7E00)  # f16 NaN: every output must be written
    dx, dw, db = dev(x.view(np.uint16)), dev(packed.view(np.uint16)), dev(bias)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.elasto_op_conv2d(stream_handle(), dx.data_ptr(), B, S, S, C, dw.data_ptr(), N, k, stride, k // 2,
                             db.data_ptr(), True, out.data_ptr(), status.data_ptr())
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = out.cpu().numpy().view(np.float16).astype(np.float64)
    assert np.all(np.isfinite(got))
    pick = np.array([0, 1, B // 2, B - 2, B - 1])
    ref = np.maximum(orr.conv2d(x[pick].astype(np.float64), w.astype(np.float64), stride, k // 2) + bias, 0)
    # one f16 rounding (2^-11 relative, doubled) and fp32 accumulation
    assert np.all(np.abs(got[pick] - ref) <= 2.0 ** -10 * np.abs(ref) + 1e-4 * np.max(np.abs(ref)))


@pytest.mark.parametrize("M,N,K,tile", [
    (100353, 248, 64, (128, 0, 0, 3)),    # one k-block a tile: the residual read three pieces ahead
    (100353, 264, 64, (64, 0, 0, 3)),     # the same, narrow tiles
    (25089, 1024, 200, (128, 0, 0, 2)),   # past the L2, 128 columns
    (25089, 1032, 200, (192, 0, 0, 2)),   # 192 columns
    (3137, 2056, 520, (192, 0, 0, 1)),    # 192 columns, one piece ahead
    (6273, 2056, 520, (256, 0, 0, 1)),    # 256 columns
    (129, 72, 64, (64, 0, 0, 3)),         # one wave
])
def test_block_output_tiles_match_fp64(M, N, K, tile):
    import torch
    assert binding.elasto_op_gemm_tile(M, N, K, binding.EPI_BIAS_RESID_RELU_F16).fields() == tile
    rng = np.random.default_rng(M + N + K)
    A = rng.standard_normal((M, K), dtype=np.float32).astype(np.float16)
    W = (rng.standard_normal((N, K)) * np.sqrt(2.0 / K)).astype(np.float16)
    bias = rng.standard_normal(N).astype(np.float32)
    R = rng.standard_normal((M, N), dtype=np.float32).astype(np.float16)
    out = empty_dev((M, N), torch.uint16)
    out.fill_(0x7E00)  # f16 NaN: every output must be written
    dA, dW, db, dR = dev(A.view(np.uint16)), dev(W.view(np.uint16)), dev(bias), dev(R.view(np.uint16))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.elasto_op_gemm(stream_handle(), dA.data_ptr(), dW.data_ptr(), db.data_ptr(), out.data_ptr(), dR.data_ptr(),
                           M, N, K, binding.EPI_BIAS_RESID_RELU_F16, status.data_ptr())
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = out.cpu().numpy().view(np.float16)
    assert np.all(np.isfinite(got))
    rows = np.unique(np.concatenate([np.arange(min(M, 300)), rng.choice(M, 500), np.arange(max(0, M - 300), M)]))
    ref = np.maximum(A[rows].astype(np.float64) @ W.astype(np.float64).T + bias + R[rows].astype(np.float64), 0)
    # one f16 rounding (2^-11 relative, doubled) and fp32 accumulation
    assert np.all(np.abs(got[rows].astype(np.float64) - ref) <= 2.0 ** -10 * np.abs(ref) + 1e-5 * np.max(np.abs(ref)))
