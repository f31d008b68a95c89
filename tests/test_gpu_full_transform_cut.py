"""The full transform's team kernel against the lane-group kernel, bit for bit: every kind of cut into teams, with the input tile, the rotated
rows and the codes of a team taking turns in one buffer."""
import numpy as np
import pytest

from tests.util import launched_kernels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,piece", [   # rows in all (the team kernel), row width, rows of a piece (the lane-group kernel)
    (17001, 384, 3000),    # three-warp teams of 32 rows, a last tile of nine
    (9475, 640, 1000),
    (1475, 1152, 700),     # few rows: smaller tiles, most teams with one
    (16383, 1152, 1400),   # four-warp teams of 14 rows
    (9001, 1408, 1200),    # eight rows, a last tile of one
    (5000, 2048, 1200),    # four teams' share of rows by eights
    (4099, 2560, 500),
    (6007, 3072, 500),     # two teams of six warps
    (4099, 4608, 700),     # three rows of 36 blocks in four warps
    (2701, 6144, 400),
    (2001, 7680, 800),     # the widest rows the team kernel takes
])
@pytest.mark.parametrize("pad", [0, 8])
def test_same_bits_as_lane_groups(M, K, piece, pad):
    import torch
    from paper_2503_06564_b200 import trdq
    rng = np.random.default_rng(M + K)
    signs = (rng.integers(0, 2, (2, 1, K)) * 2 - 1).astype(np.int8)
    rot = trdq.Rotation(K, [0, 1000], signs[0], rng.uniform(0.5, 2.0, (1, K)).astype(np.float32),
                        perm=rng.permutation(K).astype(np.int32)[None], signs2=signs[1])
    g = torch.Generator(device="cuda").manual_seed(M + K)
    x = torch.randn((M, K + pad), generator=g, device="cuda").to(torch.bfloat16)[:, :K]
    x[M // 2] = 0.0
    x[M - 1, ::3] = float("inf")
    codes, scales = trdq.trdq_rotate_quantize(rot, 0, x)
    (name, _, _), = launched_kernels(lambda: trdq.trdq_rotate_quantize(rot, 0, x, codes, scales))
    assert "rotate2_quantize_team_kernel" in name, name
    for a in range(0, M, piece):
        c, s = trdq.trdq_rotate_quantize(rot, 0, x[a:a + piece])
        (name, _, _), = launched_kernels(lambda: trdq.trdq_rotate_quantize(rot, 0, x[a:a + piece], c, s))
        assert "rotate2_quantize_rows_kernel" in name, (a, name)
        assert torch.equal(c, codes[a:a + piece]) and torch.equal(s.view(torch.int32), scales[a:a + piece].view(torch.int32)), a
    assert trdq.trdq_device_status() == 0
