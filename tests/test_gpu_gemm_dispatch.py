"""Which 8-bit GEMM kernel a shape gets, on both sides of every line of the rule, as the library reports it (figures at the rule)."""
import os

import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.skipif("TRDQ_PAIR_MIN_M" in os.environ, reason="the rule is replaced")]


@pytest.mark.parametrize("K,N,first", [  # first: the row count from which CTA pairs run
    (128, 1024, 10560), (896, 1024, 10560), (1024, 1024, 7040), (1408, 1024, 7040), (1536, 1024, 4992), (3968, 1024, 4992),
    (4096, 1024, 3584), (4096, 256, 11776), (6016, 1024, 3584), (6144, 512, 5120), (7040, 512, 5120), (7168, 128, 2048), (12288, 4608, 2048),
])
def test_pair_kernel_from_this_row_count_on(K, N, first):
    from paper_2503_06564_b200 import trdq
    assert trdq.trdq_kernel_choice(1, first - 1, K, N, 8).startswith("gemm_w8a8_kernel<")
    assert trdq.trdq_kernel_choice(1, first, K, N, 8).startswith("gemm_w8a8_pair_kernel<")
