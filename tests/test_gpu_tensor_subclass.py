"""GPU test of the binding's outputs for inputs that are a subclass of torch.Tensor: plain tensors, as for plain inputs."""
import numpy as np
import pytest

from paper_2503_06564_b200 import workloads as WL
from tests.util import to_dev_bf16

pytestmark = pytest.mark.gpu


def test_outputs_are_plain_tensors():
    import torch
    from paper_2503_06564_b200 import trdq

    class Tagged(torch.Tensor):
        pass

    K, N, M = 256, 32, 8
    rng = np.random.default_rng(2)
    rot = trdq.Rotation(K, [0, 1000], np.ones((1, K), np.int8), None)
    wts = trdq.trdq_prepare_weights(rot, to_dev_bf16(WL.to_bf16_bits(rng.standard_normal((N, K)) * 0.02)), 8)
    plain = to_dev_bf16(WL.to_bf16_bits(rng.standard_normal((M, K))))
    for x in (plain.as_subclass(Tagged), torch.nn.Parameter(plain)):
        codes, scales = trdq.trdq_rotate_quantize(rot, 0, x)
        u8, s8, zp = trdq.trdq_rotate_quantize_asym(rot, 0, x)
        outs = [codes, scales, u8, s8, zp, *trdq.trdq_norm_rotate_quantize(rot, 0, x)]
        tagged = codes.as_subclass(Tagged)
        outs += [trdq.trdq_linear(wts, 0, tagged, scales), trdq.trdq_linear_act(wts, 0, tagged, scales), trdq.trdq_gemm_i32(wts, 0, tagged),
                 trdq.trdq_linear_asym(wts, 0, u8.as_subclass(Tagged), s8, zp), trdq.trdq_linear_splitk(wts, 0, tagged, scales),
                 *trdq.trdq_linear_cfg(wts, 0, [tagged, tagged], [scales, scales])]
        assert all(type(o) is torch.Tensor for o in outs)
        assert torch.equal(outs[7], trdq.trdq_linear(wts, 0, codes, scales))
