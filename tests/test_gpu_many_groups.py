"""GPU test of weight preparation for more time-step groups than one grid dimension holds."""
import numpy as np
import pytest

from paper_2503_06564_b200 import workloads as WL
from tests.util import to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wbits", [4, 8])
def test_more_groups_than_a_grid_dimension_holds(wbits):
    """65537 groups of the smallest layer: the first, the last of the first 65535 and those behind it give what a rotation with that
    group alone gives, linear included (4-bit weights: its multiplier tables are made per group)."""
    import torch
    from paper_2503_06564_b200 import trdq
    N, K, G = 16, 128, 65537
    rng = np.random.default_rng(8)
    signs = (rng.integers(0, 2, (G, K), dtype=np.int8) * 2 - 1).astype(np.int8)
    w = to_dev_bf16(WL.to_bf16_bits(rng.standard_normal((N, K)) * 0.02))
    x = to_dev_bf16(WL.to_bf16_bits(rng.standard_normal((5, K))))
    wts = trdq.trdq_prepare_weights(trdq.Rotation(K, np.arange(G + 1), signs, None), w, wbits)
    for g in (0, 65534, 65535, G - 1):
        one_rot = trdq.Rotation(K, [0, 1], signs[g:g + 1], None)
        one = trdq.trdq_prepare_weights(one_rot, w, wbits)
        for got, want in zip(wts.view_tensors(g), one.view_tensors(0)):
            assert torch.equal(got, want)
        codes, scales = trdq.trdq_rotate_quantize(one_rot, 0, x)
        assert torch.equal(trdq.trdq_linear(wts, g, codes, scales), trdq.trdq_linear(one, 0, codes, scales))
    assert trdq.trdq_device_status() == 0
