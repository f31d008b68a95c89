"""GPU parity of the asymmetric path at row counts that take the team kernel and the CTA-pair GEMM."""
import numpy as np
import pytest

from oracle import trdq_oracle as O
from paper_2503_06564_b200 import workloads as WL
from tests.util import bf16_to_f32_np, check_output, to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,pad", [
    (16400, 1152, 8),    # one-warp teams, three tiles each, a last tile of two rows; rows with a stride
    (2100, 4608, 0),     # four-warp teams
    (4100, 2304, 16),
    (1030, 9216, 0),     # below the rule, wide rows
    (3300, 9216, 0),     # three-warp teams of one row
    (147500, 128, 0),    # one block per row
    (8000, 1152, 0),     # below the rule: the lane-group kernel
])
def test_codes_match_oracle(M, K, pad):
    from paper_2503_06564_b200 import trdq
    rng = np.random.default_rng(M + K)
    signs = np.ones((1, K), np.int8)
    x = rng.standard_normal((M, K + pad)) + 0.7
    x[:, rng.choice(K, max(1, K // 100), replace=False)] *= 20.0
    x[3] = 0.0                          # scale 0, zero point 0, codes 0
    x[5] = 0.0
    x[5, 0:K:128], x[5, 1:K:128] = 1024.0, 2.0 ** -12   # values far from zero in a tiny range: products above 2^22
    x[M - 1] = -np.abs(x[M - 1])
    bits = WL.to_bf16_bits(x)
    rot = trdq.Rotation(K, [0, 1000], signs, None)
    codes, scales, zp = trdq.trdq_rotate_quantize_asym(rot, 0, to_dev_bf16(bits)[:, :K])
    act, _ = O.fused_vectors(signs[0], None)
    c_ref, s_ref, z_ref = O.rotate_quantize_asym(np.ascontiguousarray(bits[:, :K]), act)
    assert np.array_equal(scales.cpu().numpy(), s_ref)
    assert np.array_equal(zp.cpu().numpy(), z_ref)
    assert np.array_equal(codes.cpu().numpy(), c_ref)
    assert trdq.trdq_device_status() == 0


@pytest.mark.parametrize("K,first", [(128, 147456), (1152, 16384), (2048, 4608), (4608, 2048), (6144, 1536), (6912, 2428), (8192, 2048), (9216, 3186)])
def test_dispatch_line(K, first):
    """From this row count on the team kernel is ahead (figures at the rule)."""
    import ctypes
    from paper_2503_06564_b200 import trdq
    prefers = getattr(trdq.lib(), "_ZN4trdq33rotate_quantize_asym_prefers_teamEii")
    prefers.restype, prefers.argtypes = ctypes.c_bool, [ctypes.c_int32, ctypes.c_int32]
    assert prefers(first, K) and not prefers(first - 1, K)


@pytest.mark.parametrize("M,N,K", [
    (3073, 3536, 256),   # CTA pairs; columns that end inside a tile
    (10500, 1040, 128),
    (2048, 208, 256),    # too small an output for them: one CTA per tile
])
def test_linear_matches_oracle(M, N, K):
    from paper_2503_06564_b200 import trdq
    rng = np.random.default_rng(M + N)
    signs = (rng.integers(0, 2, (1, K)) * 2 - 1).astype(np.int8)
    rot = trdq.Rotation(K, [0, 1000], signs, None)
    w, bias = WL.to_bf16_bits(rng.standard_normal((N, K)) * 0.02), WL.to_bf16_bits(rng.standard_normal(N) * 0.01)
    wts = trdq.trdq_prepare_weights(rot, to_dev_bf16(w), 8)
    x = WL.to_bf16_bits(rng.standard_normal((M, K)) + 0.7)
    codes, scales, zp = trdq.trdq_rotate_quantize_asym(rot, 0, to_dev_bf16(x))
    y = trdq.trdq_linear_asym(wts, 0, codes, scales, zp, to_dev_bf16(bias))
    act, wv = O.fused_vectors(signs[0], None)
    qw, sw = O.prepare_w8(w, wv)
    c_ref, s_ref, z_ref = O.rotate_quantize_asym(x, act)
    y_ref = O.linear_asym_rows(c_ref, s_ref, z_ref, qw, sw, bias, np.arange(M))
    assert check_output(bf16_to_f32_np(y), y_ref)[1] <= 1.0
    assert trdq.trdq_device_status() == 0


@pytest.mark.parametrize("M,K,part", [(16400, 1152, 4100), (2100, 4608, 700)])
def test_special_rows_do_not_depend_on_the_row_count(M, K, part):
    """Rows of infinities, NaN, overflowing sums and ranges so narrow that 255 / range overflows: the call over all rows (team kernel)
    gives what calls over a part of them (lane-group kernel) give."""
    import torch
    from paper_2503_06564_b200 import trdq
    rng = np.random.default_rng(K)
    x = rng.standard_normal((M, K)) * 3.0
    at = rng.permutation(M)[:16]
    x[at[0], 3] = x[at[1], K - 1] = np.nan
    x[at[2], 5], x[at[3], 5] = np.inf, -np.inf
    x[at[4], 1:3] = np.inf
    x[at[5], 1], x[at[5], 2] = np.inf, -np.inf
    x[at[6]], x[at[7], 0] = 3e38, 3.3e38
    x[at[8:12]] = 0.0
    x[at[8]], x[at[9], K - 1], x[at[10], 130] = 1e-39, 1e-38, 2e-36
    x[at[12:]] *= np.float64(2.0) ** np.array([-100, -126, -60, 100])[:, None]
    xd = torch.from_numpy(x).cuda().to(torch.bfloat16)
    rot = trdq.Rotation(K, [0, 1000], (rng.integers(0, 2, (1, K)) * 2 - 1).astype(np.int8), None)
    whole = trdq.trdq_rotate_quantize_asym(rot, 0, xd)
    parts = [trdq.trdq_rotate_quantize_asym(rot, 0, xd[i:i + part]) for i in range(0, M, part)]
    for got, want in zip(whole, zip(*parts)):
        assert torch.equal(got.view(torch.int32 if got.element_size() == 4 else torch.uint8),
                           torch.cat(want).view(torch.int32 if got.element_size() == 4 else torch.uint8))
    assert trdq.trdq_device_status() == 0
