"""GPU parity of the 4-bit GEMM at the edges of its tiles (128 channels x 128 tokens, two k-blocks per hand-over to the drain)."""
import numpy as np
import pytest

from oracle import trdq_oracle as O
from paper_2503_06564_b200 import workloads as WL
from tests.util import bf16_to_f32_np, check_output, to_dev_bf16

pytestmark = pytest.mark.gpu


def _layer(N, K, seed):
    from paper_2503_06564_b200 import trdq
    rng = np.random.default_rng(seed)
    signs = (rng.integers(0, 2, (1, K)) * 2 - 1).astype(np.int8)
    rot = trdq.Rotation(K, [0, 1000], signs, None)
    w = WL.to_bf16_bits(rng.standard_normal((N, K)) * 0.02)
    bias = WL.to_bf16_bits(rng.standard_normal(N) * 0.01)
    act, wv = O.fused_vectors(signs[0], None)
    return rot, trdq.trdq_prepare_weights(rot, to_dev_bf16(w), 4), bias, act, O.prepare_w4(w, wv), rng


@pytest.mark.parametrize("M,N,K", [
    (1, 128, 256),        # one full hand-over
    (63, 144, 384),       # an odd number of k-blocks; one channel group past a tile
    (64, 112, 128),       # a single k-block; half the tokens of a tile, channels short of a tile
    (65, 256, 512),       # one token past the first drain warp
    (128, 16, 640),
    (129, 240, 768),
    (2400, 1168, 256),    # more tiles than SMs: every ring wraps from tile to tile
])
def test_tile_edges(M, N, K):
    from paper_2503_06564_b200 import trdq
    rot, wts, bias, act, (packed, sw4), rng = _layer(N, K, M + N + K)
    x = WL.to_bf16_bits(rng.standard_normal((M, K)))
    codes, scales = trdq.trdq_rotate_quantize(rot, 0, to_dev_bf16(x))
    q_ref, sx_ref = O.rotate_quantize(x, act)
    assert np.array_equal(codes.cpu().numpy(), q_ref)
    y_ref = O.linear_w4_rows(q_ref, sx_ref, packed, sw4, bias, np.arange(M))
    y = trdq.trdq_linear(wts, 0, codes, scales, to_dev_bf16(bias))
    assert check_output(bf16_to_f32_np(y), y_ref)[1] <= 1.0
    # the same rows as two segments: tiles of both in one launch, the split inside a tile of the single call
    cut = M // 3
    if cut:
        parts = trdq.trdq_linear_cfg(wts, 0, [codes[:cut].clone(), codes[cut:].clone()], [scales[:cut].clone(), scales[cut:].clone()],
                                     to_dev_bf16(bias))
        for got, want in zip(parts, (y[:cut], y[cut:])):
            assert np.array_equal(bf16_to_f32_np(got), bf16_to_f32_np(want))
    assert trdq.trdq_device_status() == 0


def test_bias_that_cancels_the_product():
    """Bias equal to minus the product up to its bf16 rounding: the part of the 64-bit sum that fp32 drops decides the result."""
    from paper_2503_06564_b200 import trdq
    M, N, K = 96, 160, 512
    rot, wts, _, act, (packed, sw4), rng = _layer(N, K, 5)
    x = np.repeat(WL.to_bf16_bits(rng.standard_normal((1, K)) * 4.0), M, axis=0)
    codes, scales = trdq.trdq_rotate_quantize(rot, 0, to_dev_bf16(x))
    q_ref, sx_ref = O.rotate_quantize(x, act)
    product = O.linear_w4_rows(q_ref[:1], sx_ref[:1], packed, sw4, None, np.arange(1))[0]
    bias = WL.to_bf16_bits(-product.astype(np.float64))
    y_ref = O.linear_w4_rows(q_ref, sx_ref, packed, sw4, bias, np.arange(M))
    y = trdq.trdq_linear(wts, 0, codes, scales, to_dev_bf16(bias))
    check_output(bf16_to_f32_np(y), y_ref)
