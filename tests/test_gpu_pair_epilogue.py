"""The CTA-pair GEMM against the single-CTA GEMM, bit for bit, in every mode and tile width: its epilogue parameters are staged a tile
ahead by warps of their own, and with GELU a warp owns 64 columns of a tile."""
import numpy as np
import pytest

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
    for call in calls:
        whole = call(codes, scales, zero)
        for a in (0, 4000, M - 2000):
            part = slice(a, a + 2000)
            assert torch.equal(whole[part].view(torch.int16), call(codes[part].clone(), scales[part].clone(), zero[part].clone()).view(torch.int16))
    assert trdq.trdq_device_status() == 0


@pytest.mark.parametrize("M,N,K", [(1100, 4656, 1152), (1999, 2576, 768), (1664, 3072, 768), (1400, 3680, 2176)])
def test_long_epilogues_take_pairs_from_1024_rows_on(M, N, K):
    """GELU and asymmetric codes change to CTA pairs earlier than the plain epilogue: the same bits as in pieces that do not."""
    import torch
    from paper_2503_06564_b200 import trdq
    g = torch.Generator(device="cuda").manual_seed(M + N)
    rot = trdq.Rotation(K, [0, 1000], np.ones((1, K), np.int8), None)
    wts = trdq.trdq_prepare_weights(rot, (torch.randn((N, K), generator=g, device="cuda") * 0.02).to(torch.bfloat16), 8)
    codes = torch.randint(-127, 128, (M, K), generator=g, device="cuda", dtype=torch.int8)
    scales = torch.rand((M,), generator=g, device="cuda") * 0.01
    zero = torch.randint(0, 256, (M,), generator=g, device="cuda", dtype=torch.int32)
    bias = torch.randn((N,), generator=g, device="cuda").to(torch.bfloat16)
    for call in (lambda c, s, z: trdq.trdq_linear_act(wts, 0, c, s, bias), lambda c, s, z: trdq.trdq_linear_asym(wts, 0, c.view(torch.uint8), s, z, bias)):
        whole = call(codes, scales, zero)
        for a in range(0, M, 700):
            part = slice(a, min(a + 700, M))
            assert torch.equal(whole[part].view(torch.int16), call(codes[part].clone(), scales[part].clone(), zero[part].clone()).view(torch.int16))
    assert trdq.trdq_device_status() == 0
