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


@pytest.mark.parametrize("M,N", [(40, 16), (40, 208), (4700, 1552), (4700, 1584)])  # one CTA per tile, then CTA pairs
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


@pytest.mark.parametrize("M,wbits", [(40, 8), (46000, 8), (70, 4)])
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
