"""The work that users of this library have it do, as measurable cases.

A case is one training pass (forward and backward, every gradient) of a ConvBN, Linear-BN or TransposedConv-BN block, or
of a whole ResNet-50 body, through the public calls: `harness.Block`, the `convbn` binding, `backbone.BackboneReplay`.
Layer shapes are those of the benchmark configurations (`inputs.CONFIGS`), of the tests, or generic.
"""
import math

import torch

from paper_2305_11624_b200 import convbn as C
from paper_2305_11624_b200 import inputs as I
from paper_2305_11624_b200.backbone import BackboneReplay, resnet50_plan
from paper_2305_11624_b200.dataparallel import GradientBucket
from paper_2305_11624_b200.harness import Block

DEVICE = "cuda:0"
ELEMENT_BYTES = {"f32": 4, "bf16": 2, "f16": 2}


# ---- cases -------------------------------------------------------------------------------------------------------
def _block(kind, n, c_in, h, w, c_out, k, stride=1, pad=0, groups=1, dtype="bf16", bias=False, mode="tune"):
    """One block.  kind: "conv", "linear" (n rows) or "tconv" (h, w: the extent of its input)."""
    return dict(kind=kind, mode=mode, n=n, c_in=c_in, h=h, w=w, c_out=c_out, k=k, stride=stride, pad=pad, groups=groups,
                dtype=dtype, bias=bias)


def _backbone(batch, size, dtype="bf16", deferred=True):
    return dict(kind="backbone", batch=batch, size=size, dtype=dtype, deferred=deferred)


def listed():
    named = lambda name, case: dict(case, name=name)
    return [
        # a few images through one small fp32 block with a conv bias: what a unit of a small network or a gradient check
        # does; launches and host work count
        named("block_f32", _block("conv", 2, 16, 16, 16, 32, 3, pad=1, dtype="f32", bias=True)),
        # the Linear-BN block of a classifier or projection head on one batch of features
        named("linear_head", _block("linear", 1000, 256, 1, 1, 64, 1)),
        # the first 1x1 convolution of a stage-2 bottleneck at a large training batch: the largest activations
        named("pointwise_large", _block("conv", 256, 256, 56, 56, 64, 1)),
        # the 3x3 convolution of a stage-2 bottleneck at an ordinary batch
        named("conv3x3_stage2", _block("conv", 32, 64, 56, 56, 64, 3, pad=1)),
        # the 3-channel stem of a residual network
        named("stem", _block("conv", 64, 3, 224, 224, 64, 7, stride=2, pad=3)),
        # the 3x3 convolution of the last stage under half-precision training: few pixels, many weights
        named("conv3x3_stage5_f16", _block("conv", 64, 512, 7, 7, 512, 3, pad=1, dtype="f16")),
        # the down-sampling convolution of a detection backbone: two large images, odd extents
        named("detection_stride2", _block("conv", 2, 128, 200, 334, 128, 3, stride=2, pad=1)),
        # the depthwise convolution of an inverted-residual block
        named("depthwise", _block("conv", 64, 96, 112, 112, 96, 3, pad=1, groups=96)),
        # the grouped convolution (8 channels per group) of an aggregated-transform block
        named("grouped", _block("conv", 64, 256, 28, 28, 256, 3, pad=1, groups=32)),
        # the up-sampling block of an encoder-decoder network
        named("tconv_up", _block("tconv", 8, 256, 56, 56, 128, 2, stride=2)),
        # the Eval-mode block a user compares Tune mode with: the last 1x1 convolution of a stage-2 bottleneck
        named("eval_expand", _block("conv", 32, 64, 56, 56, 256, 1, mode="eval")),
        # a fine-tuning iteration of a whole ResNet-50 body in Tune mode, half-precision storage
        named("resnet50_iteration", _backbone(32, 224, "f16")),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


MAX_ELEMENTS = 1.5e8    # of X and of Z in a drawn block
MAX_FLOPS = 2.4e11      # of a drawn block's pass


def draw(rng):
    """One more case: the kinds of the listed ones at sizes spread over their logarithm, odd ones among them."""
    kind = rng.choice(("f32", "linear", "conv1", "conv3", "conv3", "stride2", "stem", "depthwise", "grouped", "tconv",
                       "comparator", "backbone"))
    dtype = rng.choice(("bf16", "bf16", "f16"))
    if kind == "backbone":
        return _backbone(_log_int(rng, 1, 31), 32 * rng.randint(2, 7), dtype, rng.random() < 0.5)
    while True:
        h = _log_int(rng, 7, 224)
        w = max(7, min(334, int(h * rng.uniform(0.75, 1.7))))
        n = _log_int(rng, 1, 256)
        wide = (64, 128, 256, 512, 1024, 2048)
        if kind == "f32":
            k = rng.choice((1, 3))
            case = _block("conv", _log_int(rng, 1, 16), _log_int(rng, 3, 64), min(h, 56), min(w, 56), _log_int(rng, 8, 64), k,
                          pad=k // 2, dtype="f32", bias=rng.random() < 0.5)
        elif kind == "linear":
            case = _block("linear", _log_int(rng, 128, 100000), rng.choice(wide), 1, 1, rng.choice(wide), 1, dtype=dtype)
        elif kind == "conv1":
            case = _block("conv", n, rng.choice(wide), h, w, rng.choice(wide), 1, dtype=dtype)
        elif kind == "conv3":
            c = rng.choice(wide[:4])
            case = _block("conv", n, c, h, w, c, 3, pad=1, dtype=dtype)
        elif kind == "stride2":
            c, k = rng.choice(wide[:4]), rng.choice((1, 3, 3))
            case = _block("conv", n, c, h, w, c if k == 3 else 2 * c, k, stride=2, pad=k // 2, dtype=dtype)
        elif kind == "stem":
            case = _block("conv", _log_int(rng, 1, 64), 3, max(h, 32), max(w, 32), 64, 7, stride=2, pad=3, dtype=dtype)
        elif kind == "depthwise":
            c = 32 * rng.randint(1, 12)
            case = _block("conv", n, c, h, w, c, 3, pad=1, groups=c, dtype=dtype)
        elif kind == "grouped":
            c = rng.choice((128, 256, 512))
            case = _block("conv", n, c, h, w, c, 3, pad=1, groups=c // 8, dtype=dtype)
        elif kind == "tconv":
            c = rng.choice(wide[1:4])
            case = _block("tconv", _log_int(rng, 1, 32), c, h, w, c // 2, 2, stride=2, dtype=dtype)
        else:
            k = rng.choice((1, 3))
            case = _block("conv", n, rng.choice(wide[:4]), h, w, rng.choice(wide[:4]), k, pad=k // 2, dtype=dtype,
                          mode=rng.choice(("eval", "deploy")))
        ho, wo = _out_hw(case)
        if max(case["n"] * case["c_in"] * case["h"] * case["w"], case["n"] * case["c_out"] * ho * wo) <= MAX_ELEMENTS and \
                _block_flops(case) <= MAX_FLOPS:
            return case


# ---- one pass ----------------------------------------------------------------------------------------------------
def _out_hw(c):
    if c["kind"] == "tconv":
        return tuple((e - 1) * c["stride"] - 2 * c["pad"] + c["k"] for e in (c["h"], c["w"]))
    return tuple((e + 2 * c["pad"] - c["k"]) // c["stride"] + 1 for e in (c["h"], c["w"]))


class _TransposedBlock:
    """Buffers of one TransposedConv-BN block."""

    def __init__(self, case, seed):
        n, ci, co, k, st, pad = (case[key] for key in ("n", "c_in", "c_out", "k", "stride", "pad"))
        self.desc = C.Desc.make(n, ci, case["h"], case["w"], co, k, k, st, st, pad, pad,
                                dtype={"bf16": C.BF16, "f16": C.F16}[case["dtype"]], layout=C.NHWC)
        dtype = {"bf16": torch.bfloat16, "f16": torch.float16}[case["dtype"]]
        ho, wo = C.convbn_tconv_out_shape(self.desc)
        g = torch.Generator(device=DEVICE)
        g.manual_seed(seed)
        normal = lambda count, std, dt=torch.float32: (torch.randn(count, generator=g, device=DEVICE) * std).to(dt)
        uniform = lambda lo, hi: torch.rand(co, generator=g, device=DEVICE) * (hi - lo) + lo
        vector = lambda: torch.empty(co, device=DEVICE)
        self.x, self.dz = normal(n * ci * case["h"] * case["w"], 1.0, dtype), normal(n * co * ho * wo, 1.0, dtype)
        self.w = normal(ci * co * k * k, math.sqrt(2.0 / (ci * k * k)), dtype)
        self.mean, self.beta, self.var, self.gamma = normal(co, 0.1), normal(co, 0.1), uniform(0.5, 2.0), uniform(0.5, 1.5)
        self.z, self.dx = torch.empty_like(self.dz), torch.empty_like(self.x)
        self.dw = torch.empty(self.w.numel(), device=DEVICE)
        self.dgamma, self.dbeta, self.saved = vector(), vector(), torch.empty(3 * co, device=DEVICE)
        self.workspace = torch.empty(max(256, C.convbn_tconv_workspace_bytes(self.desc)), dtype=torch.uint8, device=DEVICE)

    def step(self):
        C.convbn_tconv_tune_fwd(self.desc, self.x, self.w, None, self.gamma, self.beta, self.mean, self.var, self.z,
                                self.saved, self.workspace)
        C.convbn_tconv_tune_bwd(self.desc, self.dz, self.x, self.w, None, self.mean, self.saved, self.dx, self.dw, None,
                                self.dgamma, self.dbeta, self.workspace)


def _spec(case):
    return I.LayerSpec("case", case["n"], case["c_in"], case["h"], case["w"], case["c_out"], case["k"], case["k"],
                       stride=case["stride"], pad=case["pad"], groups=case["groups"], dtype=case["dtype"],
                       layout="nchw" if case["dtype"] == "f32" else "nhwc", bias=case["bias"])


def prepare(case, seed):
    if case["kind"] == "backbone":
        net = BackboneReplay(case["batch"], resnet50_plan(case["size"])[1], "tune", stem_hw=(case["size"], case["size"]),
                             device=DEVICE, seed=seed % (1 << 30), async_param_grads=case["deferred"], dtype=case["dtype"])
        # the parameter gradients of all layers in one flat buffer, as data-parallel training keeps them
        parts = ("dw", "dgamma", "dbeta")
        bucket = GradientBucket({"%d.%s" % (i, p): getattr(l.blk, p).numel() for i, l in enumerate(net.layers) for p in parts},
                                device=DEVICE)
        for i, l in enumerate(net.layers):
            for p in parts:
                setattr(l.blk, p, bucket.views["%d.%s" % (i, p)])
        return case, net, (net.make_inputs(seed=seed + 1), bucket)
    if case["kind"] == "tconv":
        return case, _TransposedBlock(case, seed), None
    blk = Block(_spec(case), device=DEVICE, modes=(case["mode"],))      # Linear-BN is the 1x1 block on 1 x 1 images
    blk.randomize(seed)
    if case["mode"] == "deploy":
        blk.deploy_prepare()
    return case, blk, None


def run(state):
    case, blk, inputs = state
    if case["kind"] == "backbone":
        ins, bucket = inputs
        return blk.forward_backward(ins), bucket.flat
    if case["kind"] == "tconv":
        blk.step()
    elif case["mode"] == "eval":
        blk.eval_fwd()
        blk.eval_bwd()
    elif case["mode"] == "deploy":
        blk.deploy_fwd()
        blk.deploy_bwd()
        return blk.z, blk.dx, blk.dw_fused, blk.db_fused
    else:
        blk.tune_step()
    out = [blk.z, blk.dx, blk.dw, blk.dgamma, blk.dbeta]
    return out + [blk.db] if case["bias"] else out


# ---- what a pass cannot do without --------------------------------------------------------------------------------
def _block_flops(c):
    ho, wo = _out_hw(c)
    pixels = c["h"] * c["w"] if c["kind"] == "tconv" else ho * wo
    return 3 * 2.0 * c["n"] * pixels * c["c_out"] * (c["c_in"] // c["groups"]) * c["k"] ** 2


def _block_bytes(c):
    """X and dZ in, Z and dX out, omega in and its fp32 gradient out, the per-channel vectors; Eval mode keeps Y too."""
    es, (ho, wo) = ELEMENT_BYTES[c["dtype"]], _out_hw(c)
    x, z = c["n"] * c["c_in"] * c["h"] * c["w"], c["n"] * c["c_out"] * ho * wo
    weights = c["c_out"] * (c["c_in"] // c["groups"]) * c["k"] ** 2
    kept = z if c["mode"] == "eval" else 0
    return es * (2 * x + 2 * z + kept + weights) + 4 * (weights + 10 * c["c_out"])


def _backbone_blocks(case):
    size = case["size"]
    blocks = [_block("conv", case["batch"], 3, size, size, 64, 7, stride=2, pad=3)]
    for b in resnet50_plan(size)[1]:
        (h, w), s = b.hw, b.stride
        blocks += [_block("conv", case["batch"], b.c_in, h, w, b.width, 1),
                   _block("conv", case["batch"], b.width, h, w, b.width, 3, stride=s, pad=1),
                   _block("conv", case["batch"], b.width, h // s, w // s, b.c_out, 1)]
        if s > 1 or b.c_in != b.c_out:
            blocks.append(_block("conv", case["batch"], b.c_in, h, w, b.c_out, 1, stride=s))
    return blocks


def work(case):
    blocks = _backbone_blocks(case) if case["kind"] == "backbone" else [case]
    return {"bytes": float(sum(_block_bytes(b) for b in blocks)), "flops": float(sum(_block_flops(b) for b in blocks))}


def tolerance(case):
    """About four times the largest error seen over listed and drawn cases against the same pass in fp64 (fp32 for the
    whole body), as rel / max.  Blocks: bf16 2.9e-3 / 1.7e-2, half 3.6e-4 / 2.4e-3, fp32 5.7e-7 / 2.8e-6.  In the body every
    ReLU whose argument is within rounding of zero may be decided either way, and a flipped one moves a whole gradient
    element: rel 0.15 in half and 0.48 in bf16, so half is stated at 0.5 and bf16 at 0.9 (unrelated results give 1.4)."""
    if case["kind"] == "backbone":
        return {"rel": {"bf16": 0.9, "f16": 0.5}[case["dtype"]]}
    return {"bf16": {"rel": 1e-2, "max": 6e-2}, "f16": {"rel": 1.5e-3, "max": 9.5e-3},
            "f32": {"rel": 2.5e-6, "max": 1.2e-5}}[case["dtype"]]
