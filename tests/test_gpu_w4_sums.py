"""GPU parity of the 4-bit GEMM's sum over scale groups at the ends of its range: largest sums of both signs, sums that swing back, scales of one binade and of
many; the exact sum becomes a float by one rounding, in small and in large problems alike."""
import numpy as np
import pytest

from oracle import trdq_oracle as O
from paper_2503_06564_b200 import workloads as WL
from tests.util import bf16_to_f32_np, check_output, to_dev_bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks", [1, 8, 9, 10])
@pytest.mark.parametrize("span", [1.0, 2.0 ** -2, 2.0 ** -9])   # smallest scale of a channel over its largest: one binade, three, ten
def test_sums_at_the_ends_of_their_range(blocks, span):
    import torch
    from paper_2503_06564_b200 import trdq
    K, N, M = 128 * blocks, 160, 72
    rng = np.random.default_rng(blocks)
    signs = np.ones((1, K), np.int8)
    rot = trdq.Rotation(K, [0, 1000], signs, None)
    # a weight block with one entry rotates to equal values: every 4-bit code is +-7, the scale is the entry's
    w = np.zeros((N, K))
    size = np.where(rng.random((N, blocks)) < 0.5, 1.0, span) * rng.uniform(1.0, 1.99, (N, blocks))
    w[:, ::128] = size * np.where(rng.random((N, blocks)) < 0.5, -1.0, 1.0)
    w[: N // 2, ::128] = np.abs(w[: N // 2, ::128])
    w[N - 32:] = rng.standard_normal((32, K)) * 0.02   # and ordinary channels, a whole warp of them
    w = WL.to_bf16_bits(w)
    wts = trdq.trdq_prepare_weights(rot, to_dev_bf16(w), 4)
    packed, sw4 = O.prepare_w4(w, O.fused_vectors(signs[0], None)[1])
    codes = rng.integers(-127, 128, (M, K)).astype(np.int8)
    codes[0], codes[1], codes[2] = 127, -127, 0
    codes[3] = np.where(np.arange(K) < K // 2, 127, -127)
    codes[4] = np.where(np.arange(K) // 128 % 2, 127, -127)
    scales = rng.uniform(0.01, 0.02, M).astype(np.float32)
    y_ref = O.linear_w4_rows(codes, scales, packed, sw4, None, np.arange(M))
    c, sx = torch.from_numpy(codes).cuda(), torch.from_numpy(scales).cuda()
    # alone, and repeated until there are 200 k-blocks per SM: no row count of a tile, so every row meets many lanes and columns
    for copies in (1, 148 * 200 // (2 * blocks) * 128 // M + 4):
        y = trdq.trdq_linear(wts, 0, c.repeat(copies, 1), sx.repeat(copies))
        # one fp32 rounding of the sum and one of its product are far below a bf16 step: the result is the bf16 number next to the oracle's value
        assert check_output(bf16_to_f32_np(y[:M]), y_ref)[1] <= 1.0
        assert not bf16_to_f32_np(y[2:3]).any()
        assert bool((y.view(copies, M, N).view(torch.int16) == y[:M].view(torch.int16)).all())
    assert trdq.trdq_device_status() == 0


def _to_bf16(v):
    """fp32 -> bf16 bits, round to nearest even"""
    return WL.f32_to_bf16_bits(np.asarray(v, np.float32))


def _rows_where_the_sum_is_near_a_tie(codes, packed, sw4):
    """Row scales with which one rounding of the sum shows in a bf16 output.  For every row: the scale that puts the product of one of its sums just on either
    side of a boundary between two bf16 numbers, depending on whether the sum is rounded to fp32 at once or in two steps (the multiple of 2^28 and
    the rest of it by themselves).  Returns (scales, the outputs with one rounding, rows where such a sum was found)."""
    M, K = codes.shape
    groups, N = K // 128, packed.shape[0]
    q4 = O.unpack_w4(packed).astype(np.int64).reshape(N, groups, 128)
    e = np.frexp(sw4.max(axis=1))[1]
    mult = np.rint(np.ldexp(sw4.astype(np.float64), 30 - e[:, None])).astype(np.int64)
    assert not (mult & 15).any(), "the weights should need 26 bits"
    mult >>= 4
    unit = np.ldexp(1.0, e - 30).astype(np.float32)   # of the sums of 16 q4 x codes x mult / 16
    S = np.zeros((M, N), np.int64)
    F = np.full((M, N), 1.5 * 2.0 ** 51, np.float32)
    for g in range(groups):
        p = 16 * (codes[:, 128 * g:128 * (g + 1)].astype(np.int64) @ q4[:, g].T) * mult[:, g]
        S += p
        F = (F.astype(np.float64) + p.astype(np.float64)).astype(np.float32)   # both exact in fp64: one rounding
    whole = F.astype(np.float64) - 1.5 * 2.0 ** 51
    once = S.astype(np.longdouble).astype(np.float32)
    twice = (whole + (S - whole.astype(np.int64)).astype(np.float32).astype(np.float64)).astype(np.float32)
    scales = np.full(M, 1e-3, np.float32)
    found = []
    for m in range(M):
        for n in np.flatnonzero((once[m] != twice[m]) & (np.abs(S[m]) >= 2 ** 30)):
            a, b = once[m, n], twice[m, n]
            near = np.float32(min(abs(a), abs(b))) * unit[n]
            middle = ((near * np.float32(1e-3)).view(np.uint32) & np.uint32(0xFFFF0000) | np.uint32(0x8000)).view(np.float32)   # of two bf16 numbers
            s = np.float32(float(middle) / float(near))
            for _ in range(8):
                s = np.nextafter(s, np.float32(0))
            for _ in range(16):
                if _to_bf16(a * (s * unit[n])) != _to_bf16(b * (s * unit[n])):
                    scales[m] = s
                    found.append(m)
                    break
                s = np.nextafter(s, np.float32(1))
            if found and found[-1] == m:
                break
    return scales, _to_bf16(once * (scales[:, None] * unit[None, :])), found


def test_sums_are_rounded_once():
    """The exact sum becomes a float by one rounding: a row gives the same bits whatever the size of the call."""
    import torch
    from paper_2503_06564_b200 import trdq
    K, N, M = 1152, 160, 1024
    rng = np.random.default_rng(5)
    rot = trdq.Rotation(K, [0, 1000], np.ones((1, K), np.int8), None)
    w = WL.to_bf16_bits(rng.standard_normal((N, K)) * 0.02)
    wts = trdq.trdq_prepare_weights(rot, to_dev_bf16(w), 4)
    packed, sw4 = O.prepare_w4(w, O.fused_vectors(np.ones(K, np.int8), None)[1])
    codes = np.zeros((M, K), np.int8)
    codes[np.arange(M)[:, None], 128 * np.arange(K // 128) + rng.integers(0, 128, (M, K // 128))] = rng.choice([-1, 1], (M, K // 128))
    scales, y_ref, found = _rows_where_the_sum_is_near_a_tie(codes, packed, sw4)
    assert len(found) >= 20
    c, sx = torch.from_numpy(codes).cuda(), torch.from_numpy(scales).cuda()
    k_blocks = (M // 128) * (-(-N // 128)) * (K // 128)
    copies = 200 * torch.cuda.get_device_properties(0).multi_processor_count // k_blocks + 1   # 200 k-blocks per SM
    for n in (1, copies):
        y = trdq.trdq_linear(wts, 0, c.repeat(n, 1), sx.repeat(n)).view(torch.int16).cpu().numpy().view(np.uint16)
        assert np.array_equal(y.reshape(n, M, N), np.broadcast_to(y_ref, (n, M, N))), n
    assert trdq.trdq_device_status() == 0
