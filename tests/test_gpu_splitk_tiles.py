"""GPU test of split-K with tiles of 64 and of 128 columns (the narrow ones where they fit one round of the SMs): bit-identical to the unsplit linear."""
import numpy as np
import pytest

from tests.util import launched_kernels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,width", [
    (1, 16, 8192, 64),          # one column tile that is mostly padding
    (130, 48, 8320, 64),        # two row tiles, an uneven last range
    (128, 1152, 16384, 64),     # 144 of 148 SMs
    (128, 1200, 16384, 128),    # 19 narrow tiles of eight ranges: more than the SMs
    (512, 400, 8192, 128),
])
def test_same_as_the_unsplit_linear(M, N, K, width):
    import torch
    from paper_2503_06564_b200 import trdq
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the widths expected here are those of 148 SMs")
    rot = trdq.Rotation(K, [0, 1000], np.ones((1, K), np.int8), None)
    gen = torch.Generator(device="cuda").manual_seed(M + N)
    wts = trdq.trdq_prepare_weights(rot, torch.randn((N, K), generator=gen, device="cuda").bfloat16(), 8)
    codes = torch.randint(-127, 128, (M, K), generator=gen, device="cuda", dtype=torch.int8)
    scales = torch.rand((M,), generator=gen, device="cuda") * 1e-3
    for bias in (None, torch.randn((N,), generator=gen, device="cuda").bfloat16()):
        y = trdq.trdq_linear_splitk(wts, 0, codes, scales, bias)
        assert torch.equal(y.view(torch.int16), trdq.trdq_linear(wts, 0, codes, scales, bias).view(torch.int16))
    splits, nbytes = trdq.trdq_linear_splitk_workspace(wts, M)
    assert splits > 1
    out, workspace = torch.empty_like(y), torch.empty((nbytes,), dtype=torch.uint8, device="cuda")
    kernels = launched_kernels(lambda: trdq.trdq_linear_splitk(wts, 0, codes, scales, None, out, workspace))
    assert any(f"gemm_w8a8_kernelILi{width}ELi1" in name for name, _, _ in kernels), kernels
    assert trdq.trdq_device_status() == 0
