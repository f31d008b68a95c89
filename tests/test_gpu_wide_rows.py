"""GPU parity of rotate + quantize on rows of more than 80 blocks: one row per CTA, one CTA per SM, several rows after each other in a CTA; and the codes of
rows that are not all finite."""
import numpy as np
import pytest

from oracle import trdq_oracle as O
from paper_2503_06564_b200 import workloads as WL
from tests.util import launched_kernels, to_dev_bf16

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


@pytest.mark.parametrize("blocks", [129, 160])
def test_five_rows_after_each_other_in_a_cta(blocks):
    """Magnitudes fall from one row of a CTA to its next, so that a row maximum left over from an earlier one would show in scales and codes."""
    import torch
    from paper_2503_06564_b200 import trdq
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    K, M = 128 * blocks, 4 * sms + 9
    rng = np.random.default_rng(blocks)
    signs = (rng.integers(0, 2, (1, K)) * 2 - 1).astype(np.int8)
    rot = trdq.Rotation(K, [0, 1000], signs, None)
    x = WL.to_bf16_bits(rng.standard_normal((M, K)) * 2.0 ** -(np.arange(M) // sms)[:, None])
    assert trdq.trdq_kernel_choice(0, M, K) == "rotate_quantize_kernel"
    xd = to_dev_bf16(x)
    codes, scales = trdq.trdq_rotate_quantize(rot, 0, xd)
    q_ref, sx_ref = O.rotate_quantize(x, O.fused_vectors(signs[0], None)[0])
    assert np.array_equal(codes.cpu().numpy(), q_ref) and np.array_equal(scales.cpu().numpy(), sx_ref)
    (name, grid, _), = launched_kernels(lambda: trdq.trdq_rotate_quantize(rot, 0, xd, codes, scales))
    assert "wide" in name and grid[0] == sms


@pytest.mark.parametrize("blocks", [81, 129, 161])
def test_rows_that_are_not_finite(blocks):
    """A row with an infinity has an infinite scale and codes of zero; a block with a NaN has codes of zero and leaves the others as if it were zeros."""
    from paper_2503_06564_b200 import trdq
    K = 128 * blocks
    rng = np.random.default_rng(blocks)
    signs = (rng.integers(0, 2, (1, K)) * 2 - 1).astype(np.int8)
    rot = trdq.Rotation(K, [0, 1000], signs, None)
    x = WL.to_bf16_bits(rng.standard_normal((6, K)))
    clean = x.copy()
    x[1, 700] = 0x7F80            # +inf
    x[2, K - 1] = 0xFF80          # -inf
    x[3, 300] = 0x7FC0            # NaN, in block 2
    clean[3, 256:384] = 0
    x[4] = 0x7FC0                 # nothing but NaN
    clean[4] = 0
    codes, scales = (a.cpu().numpy() for a in trdq.trdq_rotate_quantize(rot, 0, to_dev_bf16(x)))
    q_ref, sx_ref = O.rotate_quantize(clean, O.fused_vectors(signs[0], None)[0])
    for row in (0, 3, 4, 5):
        assert np.array_equal(codes[row], q_ref[row]) and scales[row] == sx_ref[row], row
    for row in (1, 2):
        assert not codes[row].any() and scales[row] == np.inf, row
