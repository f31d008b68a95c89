"""GPU test of the single-CTA GEMM with tiles of 64 columns: the same rows give the same bits as in a call that is large enough for wider tiles."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _outputs(trdq, wts, codes, u8, scales, zero, bias):
    return [trdq.trdq_linear(wts, 0, codes, scales, bias), trdq.trdq_linear_act(wts, 0, codes, scales, bias),
            trdq.trdq_linear_asym(wts, 0, u8, scales, zero, bias), trdq.trdq_gemm_i32(wts, 0, codes)]


@pytest.mark.parametrize("N", [16, 64, 80, 1040])
@pytest.mark.parametrize("K", [128, 1152])
def test_same_bits_as_in_a_larger_call(N, K):
    import torch
    from paper_2503_06564_b200 import trdq
    rows = 148 * 128 * 3   # more tiles of 64 columns than one round, whatever N
    rot = trdq.Rotation(K, [0, 1000], np.ones((1, K), np.int8), None)
    gen = torch.Generator(device="cuda").manual_seed(N + K)
    wts = trdq.trdq_prepare_weights(rot, torch.randn((N, K), generator=gen, device="cuda").bfloat16(), 8)
    codes = torch.randint(-127, 128, (rows, K), generator=gen, device="cuda", dtype=torch.int8)
    u8 = torch.randint(0, 256, (rows, K), generator=gen, device="cuda", dtype=torch.uint8)
    scales = torch.rand((rows,), generator=gen, device="cuda") * 1e-3
    zero = torch.randint(0, 256, (rows,), generator=gen, device="cuda", dtype=torch.int32)
    bias = torch.randn((N,), generator=gen, device="cuda").bfloat16()
    large = _outputs(trdq, wts, codes, u8, scales, zero, bias)
    for M in (1, 127, 129, 300):
        for a, b in zip(_outputs(trdq, wts, codes[:M], u8[:M], scales[:M], zero[:M], bias), large):
            assert torch.equal(a.view(torch.uint8), b[:M].contiguous().view(torch.uint8))
        # two row segments, the split inside what is one tile otherwise
        if M > 2:
            parts = trdq.trdq_linear_cfg(wts, 0, [codes[:M // 3].clone(), codes[M // 3:M].clone()], [scales[:M // 3].clone(), scales[M // 3:M].clone()], bias)
            assert torch.equal(torch.cat(parts).view(torch.int16), large[0][:M].contiguous().view(torch.int16))
    assert trdq.trdq_device_status() == 0


@pytest.mark.skipif("TRDQ_PAIR_MIN_M" in os.environ, reason="the rule is replaced")
@pytest.mark.parametrize("M,N,narrow", [(1, 16, True), (128, 148 * 64, True), (128, 149 * 64, False), (512, 37 * 64, True), (640, 26 * 64, True), (640, 27 * 64, False),
                                        (1408, 768, True), (1536, 768, False)])
def test_dispatch_line(M, N, narrow):
    import torch
    from paper_2503_06564_b200 import trdq
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the line is drawn for 148 SMs")
    assert (trdq.trdq_kernel_choice(1, M, 1152, N, 8) == "gemm_w8a8_kernel<64>") == narrow
