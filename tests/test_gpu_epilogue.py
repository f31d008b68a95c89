"""GPU parity of the dequantizing epilogue: biases that make the cancellation test fire in every chunk of 32 columns, column
counts that end inside a chunk, and special values that must stay in their own output."""
import numpy as np
import pytest

from oracle import trdq_oracle as O
from paper_2503_06564_b200 import workloads as WL
from tests.util import bf16_to_f32_np, check_output, to_dev_bf16

pytestmark = pytest.mark.gpu


def _layer(N, K, wbits, seed):
    from paper_2503_06564_b200 import trdq
    rng = np.random.default_rng(seed)
    signs = (rng.integers(0, 2, (1, K)) * 2 - 1).astype(np.int8)
    rot = trdq.Rotation(K, [0, 1000], signs, None)
    w = WL.to_bf16_bits(rng.standard_normal((N, K)) * 0.02)
    act, wv = O.fused_vectors(signs[0], None)
    return rot, trdq.trdq_prepare_weights(rot, to_dev_bf16(w), wbits), act, O.prepare_w8(w, wv) if wbits == 8 else O.prepare_w4(w, wv), rng


@pytest.mark.parametrize("M,N", [(40, 16), (40, 208), (7100, 1552), (7100, 1584)])  # one CTA per tile, then CTA pairs
def test_bias_larger_than_the_product(M, N):
    from paper_2503_06564_b200 import trdq
    K = 256
    rot, wts, act, (qw, sw), rng = _layer(N, K, 8, M + N)
    x = WL.to_bf16_bits(rng.standard_normal((M, K)))
    codes, scales = trdq.trdq_rotate_quantize(rot, 0, to_dev_bf16(x))
    q_ref, sx_ref = O.rotate_quantize(x, act)
    product = O.linear_w8_rows(q_ref, sx_ref, qw, sw, None, np.arange(M))
    bias = -product[rng.integers(0, M, N), np.arange(N)].astype(np.float64)  # cancels one row of every column
    bias[::5] = rng.standard_normal(bias[::5].shape) * 100.0
    bits = WL.to_bf16_bits(bias)
    y = trdq.trdq_linear(wts, 0, codes, scales, to_dev_bf16(bits))
    check_output(bf16_to_f32_np(y), O.linear_w8_rows(q_ref, sx_ref, qw, sw, bits, np.arange(M)))


@pytest.mark.parametrize("M,wbits", [(40, 8), (68000, 8), (70, 4)])  # one CTA per tile, CTA pairs, 4-bit weights
def test_special_values_stay_in_their_column(M, wbits):
    """GELU and the cancellation test work on several columns at once: a NaN or an infinite bias may not show in the others."""
    from paper_2503_06564_b200 import trdq
    N, K = 160, 256
    rot, wts, _, _, rng = _layer(N, K, wbits, 3)
    x = WL.to_bf16_bits(rng.standard_normal((M, K)))
    codes, scales = trdq.trdq_rotate_quantize(rot, 0, to_dev_bf16(x))
    bias = rng.standard_normal(N)
    clean = bf16_to_f32_np(trdq.trdq_linear_act(wts, 0, codes, scales, to_dev_bf16(WL.to_bf16_bits(bias))))
    bias[[1, 37]] = np.nan
    bias[70] = np.inf
    got = bf16_to_f32_np(trdq.trdq_linear_act(wts, 0, codes, scales, to_dev_bf16(WL.to_bf16_bits(bias))))
    special = [1, 37, 70]
    assert np.all(np.isnan(got[:, [1, 37]])) and np.all(got[:, 70] == np.inf)
    assert np.array_equal(np.delete(got, special, axis=1), np.delete(clean, special, axis=1))


@pytest.mark.parametrize("M,wbits", [(3, 8), (2304, 8), (3, 4)])  # one CTA per tile, CTA pairs, 4-bit weights
def test_gelu_of_every_bf16_value(M, wbits):
    """With zero weights the pre-activation is the bias, so one layer of 65536 columns meets every finite bf16 value, the ones whose
    GELU is near the bottom of the float range among them.  fp32: the exponent of 2 (up to 150) has passed five
    roundings, so the power is off by 150 * 5 * 2^-24 * ln 2 < 2^-14; then the rounding to bf16, 2^-8, and half its smallest
    subnormal, 2^-134."""
    from paper_2503_06564_b200 import trdq
    K = 128
    bits = np.arange(65536, dtype=np.uint32).astype(np.uint16)
    bits[~np.isfinite(WL.bf16_bits_to_f32(bits))] = 0
    v = WL.bf16_bits_to_f32(bits).astype(np.float64)
    rot = trdq.Rotation(K, [0, 1000], np.ones((1, K), np.int8), None)
    wts = trdq.trdq_prepare_weights(rot, to_dev_bf16(np.zeros((65536, K), np.uint16)), wbits)
    codes, scales = trdq.trdq_rotate_quantize(rot, 0, to_dev_bf16(WL.to_bf16_bits(np.random.default_rng(1).standard_normal((M, K)))))
    got = trdq.trdq_linear_act(wts, 0, codes, scales, to_dev_bf16(bits))
    with np.errstate(over="ignore"):
        want = v / (1.0 + np.exp(-2.0 * np.sqrt(2.0 / np.pi) * (v + 0.044715 * v ** 3)))
    for row in (0, M - 1):
        err = np.abs(bf16_to_f32_np(got[row]).astype(np.float64) - want)
        assert np.all(err <= (2.0 ** -8 + 2.0 ** -14) * np.abs(want) + 1.01 * 2.0 ** -134)
