"""The CTA-pair GEMM against the single-CTA GEMM, bit for bit, in every mode and tile width: its epilogue parameters are staged a tile
ahead by warps of their own, and with GELU a warp owns 64 columns of a tile."""
import numpy as np
import pytest

from tests.util import launched_kernels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,width", [  # K = 128: an epilogue as long as the main loop, two to five tiles per pair
    (84611, 128, 128, 128),
    (21505, 528, 128, 192),   # 16 columns past a tile, a last tile of one row
    (33000, 384, 128, 192),
    (9601, 1168, 128, 256),   # 144 columns of the last column tile
    (43009, 256, 128, 256),
    (5200, 1168, 1792, 192),  # the longest reduction with a warp per 64 columns, and the next: eight warps
    (5200, 1168, 1920, 192),
])
@pytest.mark.parametrize("with_bias", [True, False])
def test_same_bits_as_one_cta_per_tile(M, N, K, width, with_bias):
    import torch
    from paper_2503_06564_b200 import trdq
    g = torch.Generator(device="cuda").manual_seed(M + N)
    rot = trdq.Rotation(K, [0, 1000], np.ones((1, K), np.int8), None)
    wts = trdq.trdq_prepare_weights(rot, (torch.randn((N, K), generator=g, device="cuda") * 0.02).to(torch.bfloat16), 8)
    codes = torch.randint(-127, 128, (M, K), generator=g, device="cuda", dtype=torch.int8)
    scales = torch.rand((M,), generator=g, device="cuda") * 0.02
    zero = torch.randint(0, 256, (M,), generator=g, device="cuda", dtype=torch.int32)
    # outputs on both sides of the cancellation test, and pre-activations on both sides of -9.75 (subnormal powers in GELU)
    bias = (torch.randn((N,), generator=g, device="cuda") * 6.0).to(torch.bfloat16) if with_bias else None
    assert trdq.trdq_kernel_choice(1, M, K, N, 8) == f"gemm_w8a8_pair_kernel<{width}>"
    calls = [lambda c, s, z: trdq.trdq_linear(wts, 0, c, s, bias),
             lambda c, s, z: trdq.trdq_linear_act(wts, 0, c, s, bias),
             lambda c, s, z: trdq.trdq_linear_asym(wts, 0, c.view(torch.uint8), s, z, bias)]
    warps = [8, width // 16 if K <= 1792 else 8, 8]   # epilogue warps
    for call, ew in zip(calls, warps):
        whole = call(codes, scales, zero)
        (name, _, block), = launched_kernels(lambda: call(codes, scales, zero))
        assert f"gemm_w8a8_pair_kernelILi{width}E" in name and block[0] == 128 + 32 * ew, (name, block)
        for a in (0, 4000, M - 2000):
            part = slice(a, a + 2000)
            assert torch.equal(whole[part].view(torch.int16), call(codes[part].clone(), scales[part].clone(), zero[part].clone()).view(torch.int16))
    assert trdq.trdq_device_status() == 0


GELU, ASYM = "gelu", "asym"


@pytest.mark.parametrize("kind,M,N,K,pair", [
    (GELU, 1100, 4656, 1152, True), (GELU, 1999, 2576, 768, True), (GELU, 1664, 3072, 768, True), (GELU, 1400, 3680, 2176, True),
    (ASYM, 1100, 4656, 1152, True), (ASYM, 1400, 3680, 2176, True), (ASYM, 1999, 2576, 1024, True), (ASYM, 2900, 3072, 768, True),
    (ASYM, 1999, 4608, 768, False),    # below 2048 rows
    (GELU, 1999, 2416, 1152, False),   # below 78 tiles
    (GELU, 2330, 2704, 1152, False), (GELU, 1550, 4096, 1792, False), (ASYM, 1543, 4096, 1408, False),   # two wide rounds against two narrower ones
    (ASYM, 2574, 3456, 256, False), (ASYM, 2574, 3456, 384, True),     # a third round
])
def test_long_epilogues_take_pairs_from_1024_rows_on(kind, M, N, K, pair):
    """GELU and asymmetric codes change to CTA pairs earlier than the plain epilogue: the same bits as in pieces that do not."""
    import os
    import torch
    from paper_2503_06564_b200 import trdq
    g = torch.Generator(device="cuda").manual_seed(M + N)
    rot = trdq.Rotation(K, [0, 1000], np.ones((1, K), np.int8), None)
    wts = trdq.trdq_prepare_weights(rot, (torch.randn((N, K), generator=g, device="cuda") * 0.02).to(torch.bfloat16), 8)
    codes = torch.randint(-127, 128, (M, K), generator=g, device="cuda", dtype=torch.int8)
    scales = torch.rand((M,), generator=g, device="cuda") * 0.01
    zero = torch.randint(0, 256, (M,), generator=g, device="cuda", dtype=torch.int32)
    bias = torch.randn((N,), generator=g, device="cuda").to(torch.bfloat16)
    if kind == GELU:
        call = lambda c, s, z: trdq.trdq_linear_act(wts, 0, c, s, bias)
    else:
        call = lambda c, s, z: trdq.trdq_linear_asym(wts, 0, c.view(torch.uint8), s, z, bias)
    whole = call(codes, scales, zero)
    for a in range(0, M, 700):
        part = slice(a, min(a + 700, M))
        piece = [t[part].clone() for t in (codes, scales, zero)]
        assert torch.equal(whole[part].view(torch.int16), call(*piece).view(torch.int16))
    if "TRDQ_PAIR_MIN_M" not in os.environ:
        for args, expected in (((codes, scales, zero), pair), (piece, False)):
            (name, _, _), = launched_kernels(lambda: call(*args))
            assert ("gemm_w8a8_pair_kernel" if expected else "gemm_w8a8_kernel") in name, name
    assert trdq.trdq_device_status() == 0
