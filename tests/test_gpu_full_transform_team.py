"""GPU parity of the full transform's team kernel (one thread per block) at the edges of its tiles and of its dispatch."""
import numpy as np
import pytest

from oracle import trdq_oracle as O
from paper_2503_06564_b200 import workloads as WL
from tests.util import to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,pad", [
    (444, 1152, 0),     # one-warp teams of three rows: just a tile per SM
    (445, 1152, 8),     # a last tile of one row; rows with a stride
    (3600, 128, 0),     # one block per row, many rows per warp
    (1301, 1280, 0),
    (321, 4608, 0),     # three-warp teams
    (150, 6144, 24),
    (149, 7680, 0),     # the widest rows the team kernel takes
    (149, 8192, 0),     # the next one goes to the lane-group kernel
    (2000, 1152, 0),    # several tiles per team: the input stage and the row buffer are reused
])
def test_codes_match_oracle(M, K, pad):
    from paper_2503_06564_b200 import trdq
    rng = np.random.default_rng(M + K)
    d1, d2 = ((rng.integers(0, 2, (1, K)) * 2 - 1).astype(np.int8) for _ in range(2))
    smooth = rng.uniform(0.25, 4.0, (1, K)).astype(np.float32)
    perm = rng.permutation(K).astype(np.int32)[None, :]
    x = rng.standard_normal((M, K + pad))
    x[:, rng.choice(K, max(1, K // 100), replace=False)] *= 30.0
    x[M // 2] = 0.0
    bits = WL.to_bf16_bits(x)
    rot = trdq.Rotation(K, [0, 1000], d1, smooth, perm=perm, signs2=d2)
    codes, scales = trdq.trdq_rotate_quantize(rot, 0, to_dev_bf16(bits)[:, :K])
    a1, _ = O.fused_vectors(d1[0], smooth[0])
    c_ref, s_ref = O.rotate2_quantize(np.ascontiguousarray(bits[:, :K]), a1, perm[0], O.second_vector(d2[0], K))
    assert np.array_equal(scales.cpu().numpy(), s_ref)
    assert np.array_equal(codes.cpu().numpy(), c_ref)
    assert trdq.trdq_device_status() == 0
