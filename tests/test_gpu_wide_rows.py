"""GPU parity of rotate + quantize on rows of more than 80 blocks: one row per CTA, two CTAs per SM up to 128 blocks, more rows than CTAs."""
import numpy as np
import pytest

from oracle import trdq_oracle as O
from paper_2503_06564_b200 import workloads as WL
from tests.util import to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,blocks", [(1, 81), (310, 81), (37, 127), (5, 128), (300, 128), (3, 129), (151, 160), (2, 161)])
def test_wide_rows_match_the_oracle(M, blocks):
    from paper_2503_06564_b200 import trdq
    K = 128 * blocks
    rng = np.random.default_rng(K + M)
    signs = (rng.integers(0, 2, (2, K)) * 2 - 1).astype(np.int8)
    smooth = rng.uniform(0.5, 2.0, (2, K)).astype(np.float32)
    rot = trdq.Rotation(K, [0, 500, 1000], signs, smooth)
    x = WL.to_bf16_bits(rng.standard_normal((M, K + 8)) * 3.0)
    x[0, :128] = 0
    if M > 1:
        x[1] = 0          # a row of zeros: scale 0, codes 0
    xd = to_dev_bf16(x)
    for t, g in ((0, 0), (700, 1)):
        act, _ = O.fused_vectors(signs[g], smooth[g])
        q_ref, sx_ref = O.rotate_quantize(np.ascontiguousarray(x[:, :K]), act)
        codes, scales = trdq.trdq_rotate_quantize(rot, t, xd[:, :K])
        assert np.array_equal(codes.cpu().numpy(), q_ref) and np.array_equal(scales.cpu().numpy(), sx_ref)


def test_weights_of_wide_rows_match_the_oracle():
    from paper_2503_06564_b200 import trdq
    N, K = 48, 128 * 133
    rng = np.random.default_rng(3)
    signs = (rng.integers(0, 2, (2, K)) * 2 - 1).astype(np.int8)
    rot = trdq.Rotation(K, [0, 500, 1000], signs, None)
    w = WL.to_bf16_bits(rng.standard_normal((N, K)) * 0.02)
    wts = trdq.trdq_prepare_weights(rot, to_dev_bf16(w), 8)
    for g in range(2):
        codes, scales = wts.view_tensors(g)
        q_ref, s_ref = O.prepare_w8(w, O.fused_vectors(signs[g], None)[1])
        assert np.array_equal(codes.cpu().numpy(), q_ref) and np.array_equal(scales.cpu().numpy(), s_ref)
