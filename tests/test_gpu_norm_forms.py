"""The two forms of the LayerNorm + rotation kernel (modulation requested ahead or where it is used) give the same bits: which one runs depends
on the row count, and may not show."""
import numpy as np
import pytest

from tests.util import launched_kernels

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,piece,ahead", [   # M rows take one form, pieces of them the other or another number of rows per CTA
    (4097, 640, 1110, False),    # modulation where it is used (the other form would need a round more); pieces: ahead
    (2500, 1024, 370, False),
    (7104, 384, 3552, False),    # a round more costs less than a tenth, but there are few rounds
    (4440, 1152, 1110, False),
    (5920, 1280, 1110, False),
    (2479, 1152, 407, True),
    (777, 384, 111, True),
    (300, 1536, 37, True),       # the widest rows of the form ahead
    (8192, 1408, 1110, True),    # six rounds in place of five
    (300, 1664, 37, False),
    (300, 256, 37, False),
])
@pytest.mark.parametrize("modulated", [True, False])
def test_same_bits_whatever_the_row_count(M, K, piece, ahead, modulated):
    import torch
    from paper_2503_06564_b200 import trdq
    rng = np.random.default_rng(M + K)
    rot = trdq.Rotation(K, [0, 1000], (rng.integers(0, 2, (1, K)) * 2 - 1).astype(np.int8), rng.uniform(0.5, 2.0, (1, K)).astype(np.float32))
    g = torch.Generator(device="cuda").manual_seed(M + K)
    sample = 37
    x = (torch.randn((M, K), generator=g, device="cuda") * 3.0 + 1.0).to(torch.bfloat16)
    x[M // 3] = 0.0
    mod = [(torch.randn((-(-M // sample), K), generator=g, device="cuda") * 0.2).to(torch.bfloat16) if modulated else None for _ in range(2)]
    codes, scales = trdq.trdq_norm_rotate_quantize(rot, 0, x, mod[0], mod[1], sample, 1e-6)
    (name, _, block), = launched_kernels(lambda: trdq.trdq_norm_rotate_quantize(rot, 0, x, mod[0], mod[1], sample, 1e-6, codes, scales))
    assert ("norm_rotate_quantize_rows_kernelILi256ELb1E" in name) == ahead and block[0] <= (256 if ahead else 320), (name, block)
    assert piece % sample == 0
    for a in range(0, M, piece):
        part = [m[a // sample:].contiguous() if modulated else None for m in mod]
        c, s = trdq.trdq_norm_rotate_quantize(rot, 0, x[a:a + piece].contiguous(), part[0], part[1], sample, 1e-6)
        assert torch.equal(c, codes[a:a + piece]) and torch.equal(s.view(torch.int32), scales[a:a + piece].view(torch.int32)), a
    assert trdq.trdq_device_status() == 0
