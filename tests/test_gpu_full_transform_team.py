"""GPU parity of the full transform's team kernel (one thread per block) at the edges of its tiles and of its dispatch."""
import ctypes

import numpy as np
import pytest

from oracle import trdq_oracle as O
from paper_2503_06564_b200 import workloads as WL
from tests.util import to_dev_bf16

pytestmark = pytest.mark.gpu


def _prefers_team(M, K):
    """The library's own choice between the team kernel and the lane-group kernel."""
    from paper_2503_06564_b200 import trdq
    f = getattr(trdq.lib(), "_ZN4trdq20rotate2_prefers_teamEii")
    f.restype, f.argtypes = ctypes.c_bool, [ctypes.c_int32, ctypes.c_int32]
    return f(M, K)


@pytest.mark.parametrize("K,last,first", [    # rows: still the lane-group kernel, already the team kernel
    (128, 8903, 8904), (384, 4704, 4705), (1024, 1438, 1439), (1152, 1470, 1471), (1536, 1953, 1954), (2048, 1302, 1303), (4096, 1627, 1628),
    (4608, 769, 770), (6144, 473, 474), (7680, 1627, 1628), (8192, 100000, None),
])
def test_dispatch_line(K, last, first):
    """Where the rule says the team kernel is ahead, on the 148 SMs it was measured on (figures at the rule)."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("row counts of 148 SMs")
    assert not _prefers_team(last, K) and (first is None or _prefers_team(first, K))


@pytest.mark.parametrize("K", [128, 384, 1152, 2048, 4608, 7680])
def test_three_tiles_per_team(K):
    """The input stage is refilled, the row buffer reused and the three row-maximum buffers turned: at most 384 / (K / 128) rows are
    under way per SM, whatever the cut into teams, so every team has two tiles and some a third, the last one ragged."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    M = 2 * sms * (384 // (K // 128)) + sms // 2 + 1
    assert _prefers_team(M, K)
    _check_codes(M, K, 8)


@pytest.mark.parametrize("M,K,pad", [
    (444, 1152, 0),     # few rows: the lane-group kernel
    (445, 1152, 8),     # rows with a stride
    (3600, 128, 0),
    (1301, 1280, 0),
    (2001, 1280, 8),    # fewer than a tile per SM: still the lane-group kernel
    (2101, 1280, 8),    # the team kernel: five-warp teams of fourteen rows, a last tile of one row
    (321, 4608, 0),
    (800, 4608, 0),     # four-warp teams of three rows
    (150, 6144, 24),
    (475, 6144, 24),    # three-warp teams of two rows, the last one alone
    (149, 7680, 0),
    (1700, 7680, 0),    # the widest rows the team kernel takes
    (149, 8192, 0),
    (2000, 1152, 0),    # three-warp teams of ten rows, most without a tile
])
def test_codes_match_oracle(M, K, pad):
    _check_codes(M, K, pad)


def _check_codes(M, K, pad):
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
