"""GPU parity of the two forms of the 4-bit GEMM's sum over scale groups (two 32-bit numbers up to nine groups in large problems, 64 bits otherwise) at the
ends of their ranges: largest sums of both signs, sums that swing back, scales on either side of what the first form takes."""
import numpy as np
import pytest

from oracle import trdq_oracle as O
from paper_2503_06564_b200 import workloads as WL
from tests.util import bf16_to_f32_np, check_output, to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks", [1, 8, 9, 10])
@pytest.mark.parametrize("span", [1.0, 2.0 ** -2, 2.0 ** -9])   # smallest scale of a channel over its largest: one binade, three, too many
def test_sums_at_the_ends_of_their_range(blocks, span):
    import torch
    from paper_2503_06564_b200 import trdq
    K, N, M = 128 * blocks, 160, 72
    rng = np.random.default_rng(blocks)
    signs = np.ones((1, K), np.int8)
    rot = trdq.Rotation(K, [0, 1000], signs, None)
    # a weight block with one entry rotates to equal values: every 4-bit code is +-7, the scale is the entry's
    w = np.zeros((N, K))
    size = np.where(rng.random((N, blocks)) < 0.5, 1.0, span) * rng.uniform(1.0, 1.99, (N, blocks))
    w[:, ::128] = size * np.where(rng.random((N, blocks)) < 0.5, -1.0, 1.0)
    w[: N // 2, ::128] = np.abs(w[: N // 2, ::128])
    w[N - 32:] = rng.standard_normal((32, K)) * 0.02   # and ordinary channels, a whole warp of them
    w = WL.to_bf16_bits(w)
    wts = trdq.trdq_prepare_weights(rot, to_dev_bf16(w), 4)
    packed, sw4 = O.prepare_w4(w, O.fused_vectors(signs[0], None)[1])
    codes = rng.integers(-127, 128, (M, K)).astype(np.int8)
    codes[0], codes[1], codes[2] = 127, -127, 0
    codes[3] = np.where(np.arange(K) < K // 2, 127, -127)
    codes[4] = np.where(np.arange(K) // 128 % 2, 127, -127)
    scales = rng.uniform(0.01, 0.02, M).astype(np.float32)
    y_ref = O.linear_w4_rows(codes, scales, packed, sw4, None, np.arange(M))
    c, sx = torch.from_numpy(codes).cuda(), torch.from_numpy(scales).cuda()
    # alone, and repeated until the problem is large (200 k-blocks per SM): no row count of a tile, so every row meets many lanes and columns
    for copies in (1, 148 * 200 // (2 * blocks) * 128 // M + 4):
        y = trdq.trdq_linear(wts, 0, c.repeat(copies, 1), sx.repeat(copies))
        # one fp32 rounding of the sum and one of its product are far below a bf16 step: the result is the bf16 number next to the oracle's value
        assert check_output(bf16_to_f32_np(y[:M]), y_ref)[1] <= 1.0
        assert not bf16_to_f32_np(y[2:3]).any()
        assert bool((y.view(copies, M, N).view(torch.int16) == y[:M].view(torch.int16)).all())
    assert trdq.trdq_device_status() == 0
