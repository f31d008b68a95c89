"""What the library is timed on: the calls a diffusion denoiser makes, over the range of sizes it makes them at.

Every case goes through the public entry points of ``paper_2503_06564_b200.trdq`` on synthetic tensors with the shapes and
the outlier structure of the paper's image and video models (``workloads.py``): a bf16 Gaussian bulk in which one channel in a
hundred is heavy tailed, a per-group smoothing vector formed from the channel maxima, weights of standard deviation 0.02.

Kinds of case
  linear   one quantized linear: rotate + quantize, then the integer GEMM with its epilogue (outputs allocated by the calls)
  cfg      the conditional and the unconditional half of a batch as two row segments of one GEMM launch, inputs with a row stride
  block    the quantized linears of one transformer block through trdq_run_layers: qkv, proj, fc1 with GELU, fc2 reading
           fc1's output, and on request the two cross-attention projections of the text tokens
  adaln    the same block with the LayerNorm + modulation in front of qkv and fc1 folded into the rotation
  asym     one linear with the literal asymmetric activation quantizer (zero points)
  splitk   one linear with few rows and a long reduction
  prepare  the weights of one layer rotated and quantized for every time-step group, as when a model is loaded
"""
import math

import numpy as np
import torch

from paper_2503_06564_b200 import trdq
from paper_2503_06564_b200 import workloads as WL

BLOCK = 128


# --------------------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call in use: one layer of a small batch, where launches and host work are what is paid for
        {"name": "linear_256", "kind": "linear", "M": 256, "K": 1024, "N": 1024, "wbits": 8, "act": 0, "groups": 2},
        # a DiT-XL/2 block at 256 px, batch 8 with both guidance halves: the ordinary image-sampling step
        {"name": "block_4096", "kind": "block", "M": 4096, "width": 1152, "wbits": 8, "rotation": "hadamard", "text": 0, "groups": 5},
        # a PixArt-style block at 1024 px with cross-attention on 960 text tokens: the largest single-GPU step
        {"name": "block_32768_text", "kind": "block", "M": 32768, "width": 1152, "wbits": 8, "rotation": "hadamard", "text": 960, "groups": 4},
        # a video DiT block with 4-bit weights, 16 frames, batch 2 with guidance
        {"name": "block_w4_16384", "kind": "block", "M": 16384, "width": 1152, "wbits": 4, "rotation": "hadamard", "text": 0, "groups": 3},
        # one 4-bit layer at a row count that fills no tile evenly (one image of an odd size)
        {"name": "linear_w4_1037", "kind": "linear", "M": 1037, "K": 1152, "N": 3456, "wbits": 4, "act": 0, "groups": 3},
        # guidance halves of different length kept in a wider buffer, output width not a multiple of a tile
        {"name": "cfg_ragged", "kind": "cfg", "M": 1155, "M2": 1930, "K": 1152, "N": 3472, "wbits": 8, "pad": 64, "groups": 5},
        # a block whose rotations are dense calibrated 128 x 128 blocks, 512 px
        {"name": "block_dense_16384", "kind": "block", "M": 16384, "width": 1152, "wbits": 8, "rotation": "dense", "text": 0, "groups": 2},
        # a block with the full balancing transform (rotation, zigzag permutation, second rotation)
        {"name": "block_full_4096", "kind": "block", "M": 4096, "width": 1152, "wbits": 8, "rotation": "full", "text": 0, "groups": 2},
        # a block that hands the residual stream to the library: LayerNorm and adaLN modulation folded in, 32 samples of 256 tokens
        {"name": "adaln_8192", "kind": "adaln", "M": 8192, "width": 1152, "sample": 256, "groups": 5},
        # the asymmetric quantizer of the paper's Eq. 1-3 on an ordinary layer
        {"name": "asym_4096", "kind": "asym", "M": 4096, "K": 1152, "N": 4608, "groups": 2},
        # few rows against a very long reduction
        {"name": "splitk_128", "kind": "splitk", "M": 128, "K": 16384, "N": 1152, "groups": 1},
        # model loading: the widest layer of a block prepared for five groups
        {"name": "prepare_w8", "kind": "prepare", "K": 1152, "N": 4608, "wbits": 8, "rotation": "hadamard", "groups": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng):
    return BLOCK * rng.randint(3, 12)             # 384 ... 1536: the widths of small to large DiT models


def draw(rng):
    kind = rng.choice(["linear", "linear", "cfg", "block", "block", "block", "adaln", "asym", "splitk", "prepare"])
    groups = rng.randint(1, 5)
    if kind == "linear":
        return {"kind": kind, "M": _log_int(rng, 16, 16384), "K": BLOCK * _log_int(rng, 3, 36), "N": 16 * _log_int(rng, 24, 288),
                "wbits": rng.choice([8, 8, 4]), "act": rng.choice([0, 1]), "groups": groups}
    if kind == "cfg":
        return {"kind": kind, "M": _log_int(rng, 64, 8192), "M2": _log_int(rng, 64, 8192), "K": BLOCK * _log_int(rng, 3, 36),
                "N": 16 * _log_int(rng, 24, 288), "wbits": rng.choice([8, 8, 4]), "pad": 8 * rng.randint(0, 16), "groups": groups}
    if kind == "block":
        rotation = rng.choice(["hadamard", "hadamard", "full", "dense"])
        return {"kind": kind, "M": _log_int(rng, 256, 16384), "width": _width(rng), "wbits": rng.choice([8, 8, 4]), "rotation": rotation,
                "text": rng.choice([0, rng.randint(77, 960)]), "groups": min(groups, 2) if rotation == "dense" else groups}
    if kind == "adaln":
        return {"kind": kind, "M": _log_int(rng, 256, 16384), "width": _width(rng), "sample": _log_int(rng, 64, 1024), "groups": groups}
    if kind == "asym":
        return {"kind": kind, "M": _log_int(rng, 256, 16384), "K": BLOCK * _log_int(rng, 3, 36), "N": 16 * _log_int(rng, 24, 288), "groups": groups}
    if kind == "splitk":
        return {"kind": kind, "M": _log_int(rng, 16, 512), "K": BLOCK * _log_int(rng, 64, 160), "N": 16 * _log_int(rng, 24, 96), "groups": min(groups, 2)}
    return {"kind": kind, "K": BLOCK * _log_int(rng, 3, 36), "N": 16 * _log_int(rng, 24, 288), "wbits": rng.choice([8, 8, 4]),
            "rotation": rng.choice(["hadamard", "hadamard", "full"]), "groups": groups}


# ------------------------------------------------------------------------------------------------------------ inputs
class _Inputs:
    """Tensors drawn on the device, and small host tables, from one seed."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed))
        self.rng = np.random.default_rng(int(seed))

    def randn(self, *shape):
        return torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.float32)

    def activations(self, M, K, pad=0):
        """bf16 [M, K] (row stride K + pad): N(0, 1), one channel in a hundred Student-t with three degrees of freedom."""
        x = self.randn(M, K + pad)
        n = max(1, K // 100)
        ch = torch.randperm(K, generator=self.gen, device="cuda")[:n]
        x[:, ch] = self.randn(M, n) / torch.sqrt((self.randn(M, n, 3) ** 2).sum(-1) / 3.0)
        return x.to(torch.bfloat16)[:, :K]

    def weight(self, N, K):
        return (self.randn(N, K) * 0.02).to(torch.bfloat16)

    def bias(self, N):
        return (self.randn(N) * 0.01).to(torch.bfloat16)

    def timestep(self):
        return int(self.rng.integers(0, WL.T_RANGE))

    def rotation(self, kind, w, x, groups):
        """A rotation of x's width with the smoothing of every group from the channel maxima of x and w."""
        K = w.shape[1]
        ax = x.float().abs().amax(dim=0).double().clamp_min(1e-5).cpu().numpy()
        aw = w.float().abs().amax(dim=0).double().clamp_min(1e-5).cpu().numpy()
        smooth = np.stack([aw ** (1.0 - a) / ax ** a for a in WL.group_alphas(groups)]).astype(np.float32)
        bounds = WL.group_bounds(groups)
        signs = (self.rng.integers(0, 2, (groups, K)) * 2 - 1).astype(np.int8)
        if kind == "dense":
            return trdq.DenseRotation(K, bounds, self._orthogonal_blocks(groups, K // BLOCK), smooth)
        if kind == "full":
            perm = np.stack([trdq.trdq_zigzag_permutation(ax * s) for s in smooth])
            signs2 = (self.rng.integers(0, 2, (groups, K)) * 2 - 1).astype(np.int8)
            return trdq.Rotation(K, bounds, signs, smooth, perm=perm, signs2=signs2)
        return trdq.Rotation(K, bounds, signs, smooth)

    def _orthogonal_blocks(self, groups, nb):
        """Dense orthogonal blocks [groups, nb, 128, 128]: two Walsh-Hadamard matrices between random signs and a permutation."""
        h = torch.ones((1, 1), device="cuda", dtype=torch.float64)
        while h.shape[0] < BLOCK:
            h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
        h = h / math.sqrt(BLOCK)
        sign = torch.where(self.randn(3, groups * nb, BLOCK) < 0, -1.0, 1.0).double()
        order = torch.argsort(self.randn(groups * nb, BLOCK), dim=1)
        first = torch.gather(h * sign[0][:, None, :], 2, order[:, None, :].expand(-1, BLOCK, -1)) * sign[2][:, :, None]
        return (first @ (h * sign[1][:, None, :])).float().view(groups, nb, BLOCK, BLOCK).cpu().numpy()


def _quantized_layer(inp, kind, x, N, wbits, groups):
    w = inp.weight(N, x.shape[1])
    rot = inp.rotation(kind, w, x, groups)
    return rot, trdq.trdq_prepare_weights(rot, w, wbits), inp.bias(N), w


def _empty(shape, dtype):
    return torch.empty(shape, dtype=dtype, device="cuda")


def _buffers(M, K, N):
    return _empty((M, K), torch.int8), _empty((M,), torch.float32), _empty((M, N), torch.bfloat16)


def _block_layers(case):
    """(name, K, N) of the block's linears on the image or video tokens."""
    w = case["width"]
    return (("qkv", w, 3 * w), ("proj", w, w), ("fc1", w, 4 * w), ("fc2", 4 * w, w))


def _block_inputs(inp, case, kind):
    """Per linear (rot, weights, x, codes, scales, bias, y); fc2's x is fc1's y, as in the model."""
    M, out = case["M"], {}
    for name, K, N in _block_layers(case):
        if name == "fc2":
            x = out["fc1"][-1]
            _, _, xc, _, _, bc, _ = out["fc1"]
            sample = torch.nn.functional.gelu(xc[:1024].float() @ fc1_w.float().T + bc.float(), approximate="tanh")
        else:
            x = sample = inp.activations(M, K)
        w = inp.weight(N, K)
        rot = inp.rotation(kind, w, sample, case["groups"])
        wts = trdq.trdq_prepare_weights(rot, w, case.get("wbits", 8))
        codes, scales, y = _buffers(M, K, N)
        out[name] = (rot, wts, x, codes, scales, inp.bias(N), y)
        if name == "fc1":
            fc1_w = w
    return out


# -------------------------------------------------------------------------------------------------- prepare, run, work
def prepare(case, seed):
    inp = _Inputs(seed)
    kind, s = case["kind"], {"case": case}
    s["t"] = inp.timestep()
    if kind == "block":
        parts = _block_inputs(inp, case, case["rotation"])
        layers, outs = trdq.LayerList(), []

        def add(rot, wts, x, codes, scales, bias, y, act):
            ws = None
            if case["rotation"] == "dense":
                ws = _empty((trdq.trdq_rotate_dense_workspace(rot, x.shape[0]),), torch.uint8)
            layers.add(rot, wts, x, codes, scales, bias, y, act=act, workspace=ws)
            outs.extend((codes, scales, y))

        for name, part in parts.items():
            add(*part, trdq.ACT_GELU_TANH if name == "fc1" else trdq.ACT_NONE)
        if case["text"]:
            text = inp.randn(case["text"], 4096).to(torch.bfloat16)
            for _ in range(2):
                rot, wts, bias, _ = _quantized_layer(inp, case["rotation"], text, case["width"], case["wbits"], case["groups"])
                add(rot, wts, text, *_buffers(case["text"], 4096, case["width"])[:2], bias,
                    _empty((case["text"], case["width"]), torch.bfloat16), trdq.ACT_NONE)
        s.update(layers=layers, outs=outs)
    elif kind == "adaln":
        samples = -(-case["M"] // case["sample"])
        s["mod"] = {n: tuple((inp.randn(samples, case["width"]) * 0.2).to(torch.bfloat16) for _ in range(2)) for n in ("qkv", "fc1")}
        s["parts"] = _block_inputs(inp, case, "hadamard")
    elif kind == "prepare":
        s["w"] = inp.weight(case["N"], case["K"])
        s["rot"] = inp.rotation(case["rotation"], s["w"], inp.activations(256, case["K"]), case["groups"])
    else:
        rows = [case["M"], case["M2"]] if kind == "cfg" else [case["M"]]
        x = inp.activations(sum(rows), case["K"], case.get("pad", 0))
        s["rot"], s["wts"], s["bias"], _ = _quantized_layer(inp, "hadamard", x, case["N"], case.get("wbits", 8), case["groups"])
        s["x"] = list(torch.split(x, rows))
        if kind == "splitk":
            _, nbytes = trdq.trdq_linear_splitk_workspace(s["wts"], case["M"])
            s["workspace"] = _empty((max(nbytes, 16),), torch.uint8)
    return s


def run(s):
    case, t = s["case"], s["t"]
    kind = case["kind"]
    if kind == "block":
        trdq.trdq_run_layers(s["layers"], t)
        return s["outs"]
    if kind == "adaln":
        outs = []
        for name, (rot, wts, x, codes, scales, bias, y) in s["parts"].items():
            if name in s["mod"]:
                shift, scale = s["mod"][name]
                trdq.trdq_norm_rotate_quantize(rot, t, x, shift, scale, case["sample"], 1e-6, codes, scales)
            else:
                trdq.trdq_rotate_quantize(rot, t, x, codes, scales)
            if name == "fc1":
                trdq.trdq_linear_act(wts, t, codes, scales, bias, y)
            else:
                trdq.trdq_linear(wts, t, codes, scales, bias, y)
            outs.extend((codes, scales, y))
        return outs
    if kind == "prepare":
        wts = trdq.trdq_prepare_weights(s["rot"], s["w"], case["wbits"])
        return [wts.view_tensors(g) for g in range(case["groups"])]
    if kind == "cfg":
        quantized = [trdq.trdq_rotate_quantize(s["rot"], t, x) for x in s["x"]]
        codes, scales = [q[0] for q in quantized], [q[1] for q in quantized]
        return codes + scales + list(trdq.trdq_linear_cfg(s["wts"], t, codes, scales, s["bias"]))
    x = s["x"][0]
    if kind == "asym":
        codes, scales, zero = trdq.trdq_rotate_quantize_asym(s["rot"], t, x)
        return codes, scales, zero, trdq.trdq_linear_asym(s["wts"], t, codes, scales, zero, s["bias"])
    codes, scales = trdq.trdq_rotate_quantize(s["rot"], t, x)
    if kind == "splitk":
        return codes, scales, trdq.trdq_linear_splitk(s["wts"], t, codes, scales, s["bias"], workspace=s["workspace"])
    if case["act"]:
        return codes, scales, trdq.trdq_linear_act(s["wts"], t, codes, scales, s["bias"])
    return codes, scales, trdq.trdq_linear(s["wts"], t, codes, scales, s["bias"])


def _linear_work(M, K, N, wbits):
    """One linear: x, the weights, bias and scales read once; codes, scales and y written once."""
    weights = N * K * wbits / 8 + (4 * N if wbits == 8 else 4 * N * K / BLOCK) + 2 * N
    return 2 * M * K + weights + M * K + 4 * M + 2 * M * N, 2.0 * M * N * K


def work(case):
    kind = case["kind"]
    if kind == "prepare":
        N, K, G = case["N"], case["K"], case["groups"]
        out = N * K * case["wbits"] / 8 + 4 * N * (1 if case["wbits"] == 8 else K / BLOCK)
        # a butterfly is seven additions an element, and the scaling, the maximum and the quantizer one operation each
        return {"bytes": 2.0 * N * K + G * out, "flops": 10.0 * G * N * K * (2 if case["rotation"] == "full" else 1)}
    if kind in ("block", "adaln"):
        parts = [_linear_work(case["M"], K, N, case.get("wbits", 8)) for _, K, N in _block_layers(case)]
        if kind == "block" and case["text"]:
            parts += [_linear_work(case["text"], 4096, case["width"], case["wbits"])] * 2
        if kind == "adaln":
            parts.append((2 * 4 * -(-case["M"] // case["sample"]) * case["width"], 0.0))
    else:
        parts = [_linear_work(case["M"] + case.get("M2", 0), case["K"], case["N"], case.get("wbits", 8))]
    return {"bytes": float(sum(p[0] for p in parts)), "flops": float(sum(p[1] for p in parts))}


def tolerance(case):
    """Codes and the integer sums are exact.  Outputs against a float64 epilogue on the same codes: the bf16 rounding of one in
    10^5 goes the other way (relative 2-norm up to 2.3e-5, one bf16 step = 7.8e-3 at most).  With dense blocks (tensor-core
    sums) and with the folded LayerNorm (fp32 statistics) a float64 evaluation moves a few codes in a million."""
    if case["kind"] == "adaln" or case.get("rotation") == "dense":
        return {"rel": 2e-4, "max": 1.6e-2, "differ": 1e-5}
    return {"rel": 1e-4, "max": 1.6e-2, "differ": 0.0}
