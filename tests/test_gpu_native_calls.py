"""The native form of the binding's hot calls against the general way: same outputs, same errors, and what it does not handle it leaves alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture
def layer():
    import torch
    from paper_2503_06564_b200 import trdq
    K, N = 256, 48
    rng = np.random.default_rng(0)
    rot = trdq.Rotation(K, [0, 500, 1000], (rng.integers(0, 2, (2, K)) * 2 - 1).astype(np.int8), None)
    gen = torch.Generator(device="cuda").manual_seed(1)
    w = torch.randn((N, K), generator=gen, device="cuda").bfloat16()
    x = torch.randn((40, K + 64), generator=gen, device="cuda").bfloat16()
    bias = torch.randn((N,), generator=gen, device="cuda").bfloat16()
    return rot, trdq.trdq_prepare_weights(rot, w, 8), x, bias


def _calls(rot, wts, t, x, bias):
    """Every call that has a native form, outputs in a list; twice with given outputs."""
    import torch
    from paper_2503_06564_b200 import trdq
    M, K, N = x.shape[0], rot.K, wts.N
    codes, scales = trdq.trdq_rotate_quantize(rot, t, x)
    u8, su, zp = trdq.trdq_rotate_quantize_asym(rot, t, x)
    wide = torch.zeros((M, N + 16), dtype=torch.bfloat16, device="cuda")[:, :N]
    mod = x[:2, :K].contiguous()
    out = [codes, scales, u8, su, zp, *trdq.trdq_rotate_quantize(rot, t, x, torch.empty_like(codes), torch.empty_like(scales)),
           *trdq.trdq_norm_rotate_quantize(rot, t, x, mod, mod, max(1, (M + 1) // 2)), *trdq.trdq_norm_rotate_quantize(rot, t, x),
           trdq.trdq_linear(wts, t, codes, scales), trdq.trdq_linear(wts, t, codes, scales, bias, wide), trdq.trdq_linear_act(wts, t, codes, scales, bias),
           trdq.trdq_linear_asym(wts, t, u8, su, zp, bias), trdq.trdq_linear_splitk(wts, t, codes, scales, bias)]
    cfg = trdq.trdq_linear_cfg(wts, t, [codes, codes], (scales, scales), bias)
    assert type(cfg) is list and len(cfg) == 2
    return out + cfg


@pytest.mark.parametrize("rows", [0, 1, 2, 40])
def test_same_outputs_as_the_general_way(layer, rows, monkeypatch):
    import torch
    from paper_2503_06564_b200 import trdq
    rot, wts, x, bias = layer
    taken = []

    class Declines:
        def __getattr__(self, name):
            return lambda *a: taken.append(name)

    for t in (100, 700):
        for view in (x[:rows, :rot.K], x[:rows, 64:], x[:rows, :rot.K].contiguous()):
            native = _calls(rot, wts, t, view, bias)
            with monkeypatch.context() as m:
                m.setattr(trdq, "_native", Declines())
                general = _calls(rot, wts, t, view, bias)
            assert len(native) == len(general)
            for a, b in zip(native, general):
                assert type(a) is torch.Tensor and a.dtype == b.dtype and a.shape == b.shape and a.stride() == b.stride() and torch.equal(a, b)
    assert set(taken) == {"rotate_quantize", "norm_rotate_quantize", "rotate_quantize_asym", "linear", "linear_asym", "linear_splitk", "linear_cfg"}


def test_errors_and_what_is_left_alone(layer):
    import torch
    from paper_2503_06564_b200 import trdq
    rot, wts, x, bias = layer
    x = x[:, :rot.K]
    codes, scales = trdq.trdq_rotate_quantize(rot, 3, x)
    native = trdq._calls()
    for call in (lambda: trdq.trdq_rotate_quantize(rot, 1000, x), lambda: trdq.trdq_linear(wts, -1, codes, scales), lambda: trdq.trdq_linear_act(wts, 0, codes, scales, act=7),
                 lambda: trdq.trdq_linear_cfg(wts, 2000, [codes, codes], [scales, scales])):
        with pytest.raises(trdq.TrdqError):
            call()
    with pytest.raises(AssertionError):
        trdq.trdq_rotate_quantize(rot, 0, x.float())
    with pytest.raises(AssertionError):
        trdq.trdq_rotate_quantize(rot, 0, x.cpu())

    class Tagged(torch.Tensor):
        pass

    class Mode(torch.overrides.TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            return func(*args, **(kwargs or {}))

    args = (rot._h.value, rot.K)
    assert native.rotate_quantize(*args, 3, x, None, None) is not None
    assert native.rotate_quantize(*args, 3, torch.nn.Parameter(x), None, None) is not None
    for t, left in ((3, x.as_subclass(Tagged)), (3, x.cpu()), (3, x.float()), (3, x.t()), (3.0, x), (np.int64(3), x), (2 ** 40, x), (3, None), (3, "x")):
        assert native.rotate_quantize(*args, t, left, None, None) is None
    assert native.rotate_quantize(None, rot.K, 3, x, None, None) is None
    with Mode():
        assert native.rotate_quantize(*args, 3, x, None, None) is None
    assert torch.func.vmap(lambda row: torch.tensor(native.rotate_quantize(*args, 3, row, None, None) is None))(x[None].repeat(2, 1, 1)).all()
    # the general way takes them as before
    for t in (3.0, np.int64(3)):
        assert all(torch.equal(a, b) for a, b in zip(trdq.trdq_rotate_quantize(rot, t, x), (codes, scales)))
    other = torch.cuda.Stream()
    other.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(other):
        again = trdq.trdq_rotate_quantize(rot, 3, x)
    other.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(again, (codes, scales)))
    closed = trdq.trdq_prepare_weights(rot, bias.new_zeros((48, rot.K)), 8)
    closed.close()
    with pytest.raises(trdq.TrdqError):
        trdq.trdq_linear(closed, 3, codes, scales)
