"""Whole-backbone replay: forward + backward of a ResNet-50-shaped chain of ConvBN blocks in Tune, Eval or Deploy mode.

This is the shape of the paper's efficiency experiment (Sec. 3.4, Fig. 3, App. D: time per iteration and peak
memory of a ResNet-50 under the three modes) with synthetic weights and inputs: the 53 ConvBN blocks of the
network (stem, 16 bottlenecks of three convolutions, four projection shortcuts), ReLU after every block but the
last of a bottleneck, the skip connection and its ReLU at the end of each bottleneck.  Every ConvBN block, every
ReLU and every add runs through `libconvbn.so`; this module only owns buffers and the order of the calls.

What is kept from forward to backward is what a framework would keep: each convolution's input (the previous
ReLU's output), the mode's extra state (Tune: three vectors per block; Eval: the pre-normalisation tensor Y of
every block; Deploy: nothing), and nothing else.  Buffers are allocated with torch inside the pass and dropped
as soon as the backward pass has used them, so `torch.cuda.max_memory_allocated` sees the peak a training
framework would see.

The max-pool between the stem and the first stage is not a ConvBN block and has no counterpart in the library:
the first stage is fed with a synthetic tensor of the pooled shape and the stem's backward pass with a synthetic
gradient (one cheap operator out of ~170 is missing from the timed pass).
"""
import math
from dataclasses import dataclass
from typing import List, Optional, Tuple

import torch

from . import convbn as C
from . import inputs as I
from .harness import Block


@dataclass
class Bottleneck:
    c_in: int
    width: int
    c_out: int
    stride: int          # of the 3x3 convolution (and of the projection shortcut)
    hw: Tuple[int, int]  # input extent


def resnet50_plan(size: int = 224) -> Tuple[Optional[Tuple[int, int]], List[Bottleneck]]:
    """(stem input extent, bottlenecks) of a ResNet-50 for `size` x `size` images."""
    h = size // 4                     # after the stride-2 stem and the stride-2 max-pool
    plan, c_in = [], 64
    for width, blocks, stride in ((64, 3, 1), (128, 4, 2), (256, 6, 2), (512, 3, 2)):
        for b in range(blocks):
            s = stride if b == 0 else 1
            plan.append(Bottleneck(c_in, width, 4 * width, s, (h, h)))
            h //= s
            c_in = 4 * width
    return (size, size), plan


class _Layer:
    """One ConvBN block of the chain: parameters, gradients, the calls of the chosen mode."""

    def __init__(self, name, n, c_in, hw, c_out, k, stride, mode, device, seed, dtype="bf16"):
        spec = I.LayerSpec(name, n, c_in, hw[0], hw[1], c_out, k, k, stride=stride, pad=k // 2, dtype=dtype)
        self.blk = Block(spec, device=device, modes=(mode,), allocate="params")
        self.blk.randomize_params(seed)
        self.mode = mode
        if mode == "tune":          # sizes of what the passes allocate (functions of the descriptor and the device)
            with torch.cuda.device(self.blk.device):
                self.saved_bytes = max(16, C.convbn_saved_bytes(self.blk.desc, C.MODE_TUNE))
                self.fwd_bytes = max(256, C.convbn_workspace_bytes(self.blk.desc, C.PHASE_TUNE_FWD))
                self.bwd_bytes = max(256, C.convbn_workspace_bytes(self.blk.desc, C.PHASE_TUNE_BWD))
        if mode == "deploy":
            b = self.blk
            b.w_fused = torch.empty_like(b.w)
            b.b_fused = torch.empty(spec.c_out, dtype=torch.float32, device=device)
            b.dw_fused = torch.empty_like(b.dw)
            b.db_fused = torch.empty(spec.c_out, dtype=torch.float32, device=device)
            b.deploy_prepare()
        self.out_elems = n * c_out * self.blk.h_out * self.blk.w_out
        self.in_elems = n * c_in * hw[0] * hw[1]

    def forward(self, x, add=None, relu=False, saved=None, scratch=None):
        """The block's output, or max(output + add, 0): in Tune mode the addend and the ReLU are part of the block's own
        kernel, otherwise they are passes of their own.  saved, scratch (Tune mode): addresses of saved_bytes, which the
        caller keeps for the backward pass, and of fwd_bytes for this call."""
        b = self.blk
        b.x = x
        z = torch.empty(self.out_elems, dtype=b.tdtype, device=b.device)
        if self.mode == "tune":
            C.convbn_tune_fwd_glue(b.desc, x, b.w, b.b, b.gamma, b.beta, b.mu_hat, b.var_hat, z, saved, add, relu, scratch,
                                   self.fwd_bytes)
            return z
        b.z = z
        if self.mode == "eval":
            b.y_saved = torch.empty(C.convbn_saved_bytes(b.desc, C.MODE_EVAL), dtype=torch.uint8, device=b.device)
            b.with_scratch(C.PHASE_EVAL_FWD, b.eval_fwd)
        else:
            b.with_scratch(C.PHASE_DEPLOY_FWD, b.deploy_fwd)
        b.z = None
        if add is not None:
            (C.convbn_add_relu if relu else C.convbn_add)(z, add, z)
        elif relu:
            C.convbn_relu(z, z)
        return z

    def backward(self, dz, held=None, add=None, relu_mask=False, saved=None, scratch=None):
        """Gradient with respect to the block's input, plus `add`, and with `relu_mask` zero where the input (the output
        of a ReLU) is not positive; drops what the block kept for it.  With `held` (a list, Tune mode) the
        parameter-gradient pass stays on the library's side stream: what it still reads of the tensors allocated here (dZ, X)
        is parked in `held` until the caller has joined.  saved, scratch (Tune mode): addresses of the forward pass's
        vectors and of bwd_bytes, both in use until the pass is joined."""
        b = self.blk
        dx = torch.empty(self.in_elems, dtype=b.tdtype, device=b.device)
        x, b.x = b.x, None
        if self.mode == "tune":
            C.convbn_tune_bwd_glue(b.desc, dz, x, b.w, b.b, b.mu_hat, saved, dx, b.dw, b.db, b.dgamma, b.dbeta, add,
                                   relu_mask, held is not None, scratch, self.bwd_bytes)
            if held is not None:
                held.append((x, dz))
            return dx
        b.dz, b.dx, b.x = dz, dx, x
        if self.mode == "eval":
            b.with_scratch(C.PHASE_EVAL_BWD, b.eval_bwd)
            b.y_saved = None
        else:
            b.with_scratch(C.PHASE_DEPLOY_BWD, b.deploy_bwd)
        b.dx = b.dz = b.x = None
        if add is not None:
            C.convbn_add(dx, add, dx)
        if relu_mask:
            C.convbn_relu_bwd(dx, x, dx)
        return dx


def _aligned(n):
    return (n + 255) // 256 * 256


class BackboneReplay:
    def __init__(self, batch: int, plan: List[Bottleneck], mode: str, stem_hw: Optional[Tuple[int, int]] = None,
                 device="cuda:0", seed: int = 0, async_param_grads: bool = False, dtype: str = "bf16"):
        assert mode in ("tune", "eval", "deploy") and dtype in ("bf16", "f16")
        self.async_param_grads = async_param_grads
        self.mode, self.batch, self.device = mode, batch, torch.device(device)
        self.dtype = torch.bfloat16 if dtype == "bf16" else torch.float16
        n, k = batch, seed
        self.stem = None
        if stem_hw is not None:
            self.stem = _Layer("stem", n, 3, stem_hw, 64, 7, 2, mode, device, k, dtype)
            k += 1
        self.blocks = []
        for i, bt in enumerate(plan):
            hw2 = bt.hw
            hw3 = (bt.hw[0] // bt.stride, bt.hw[1] // bt.stride) if bt.stride > 1 else bt.hw
            if bt.stride > 1:      # floor convention of a 3x3 stride-2 pad-1 convolution
                hw3 = ((bt.hw[0] - 1) // bt.stride + 1, (bt.hw[1] - 1) // bt.stride + 1)
            c1 = _Layer("b%d.c1" % i, n, bt.c_in, bt.hw, bt.width, 1, 1, mode, device, k, dtype)
            c2 = _Layer("b%d.c2" % i, n, bt.width, hw2, bt.width, 3, bt.stride, mode, device, k + 1, dtype)
            c3 = _Layer("b%d.c3" % i, n, bt.width, hw3, bt.c_out, 1, 1, mode, device, k + 2, dtype)
            ds = None
            if bt.stride > 1 or bt.c_in != bt.c_out:
                ds = _Layer("b%d.ds" % i, n, bt.c_in, bt.hw, bt.c_out, 1, bt.stride, mode, device, k + 3, dtype)
            k += 4
            self.blocks.append((c1, c2, c3, ds))
        self.first = plan[0]
        self.layers = ([self.stem] if self.stem else []) + [l for blk in self.blocks for l in blk if l is not None]
        self.flops = sum(3 * l.blk.flops_per_phase() for l in self.layers)
        if mode == "tune":
            # The vectors kept from forward to backward lie in one buffer per iteration, the forward calls share one scratch
            # (one after the other on a stream), and a bottleneck's backward calls share one: with deferred gradients each
            # has its part until the join, otherwise they take turns.  An allocation per call (265 of an iteration) took
            # 1.8 us of host time each.
            self.saved_at, at = {}, 0
            for l in self.layers:
                self.saved_at[l], at = at, at + _aligned(l.saved_bytes)
            self.saved_total = at
            self.fwd_scratch = max(l.fwd_bytes for l in self.layers)
            self.bwd_at, self.bwd_total = [], []
            for blk in self.blocks:
                off, at = [], 0
                for l in blk:
                    off.append(at)
                    if l is not None and async_param_grads:
                        at += _aligned(l.bwd_bytes)
                self.bwd_at.append(off)
                self.bwd_total.append(at or max(l.bwd_bytes for l in blk if l is not None))

    # ---- one iteration ---------------------------------------------------------------------------------
    def make_inputs(self, seed: int = 1):
        g = torch.Generator(device=self.device)
        g.manual_seed(seed)
        rn = lambda n: torch.randn(n, generator=g, device=self.device).to(self.dtype)
        bt = self.first
        ins = {"x": rn(self.batch * bt.c_in * bt.hw[0] * bt.hw[1]).abs_()}      # a ReLU output feeds the first stage
        last = self.blocks[-1][2]
        ins["g"] = rn(last.out_elems)
        if self.stem:
            ins["image"] = rn(self.stem.in_elems)
            ins["g_stem"] = rn(self.stem.out_elems)
        return ins

    def forward_backward(self, ins, keep=None):
        """One training iteration.  `keep` (a dict) receives the network output, the input gradient and copies of
        every ReLU output (whose signs are the decisions a comparison has to share)."""
        relu_outs = []
        tune = self.mode == "tune"
        fwd = {}
        if tune:
            raw = lambda n: torch.empty(n, dtype=torch.uint8, device=self.device)
            saved, scratch = raw(self.saved_total), raw(self.fwd_scratch)
            base, at = saved.data_ptr(), scratch.data_ptr()
            fwd = {l: (base + o, at) for l, o in self.saved_at.items()}
        none = (None, None)
        if self.stem:
            s = self.stem.forward(ins["image"], None, True, *fwd.get(self.stem, none))
        x = ins["x"]
        for c1, c2, c3, ds in self.blocks:
            a = c1.forward(x, None, True, *fwd.get(c1, none))
            b = c2.forward(a, None, True, *fwd.get(c2, none))
            # out = relu(c3(b) + identity)
            c = c3.forward(b, ds.forward(x, None, False, *fwd.get(ds, none)) if ds is not None else x, True, *fwd.get(c3, none))
            relu_outs.append((x, a, b, c))
            if keep is not None:
                keep.setdefault("relu_outputs", []).append((a.clone(), b.clone(), c.clone()))
            x = c
        if keep is not None:
            keep["out"] = x.clone()
        scratch = None
        g = torch.empty_like(ins["g"])
        C.convbn_relu_bwd(ins["g"], x, g)                      # through the last block's ReLU
        del x, a, b, c
        # Tune mode: the parameter gradients of a bottleneck's blocks run beside its input-gradient chain and are
        # joined once per bottleneck, after which what they were reading can be released
        held = [] if self.mode == "tune" and self.async_param_grads else None
        for i in range(len(self.blocks) - 1, -1, -1):
            c1, c2, c3, ds = self.blocks[i]
            relu_outs.pop()
            at = none * 2
            if tune:
                scratch = raw(self.bwd_total[i])
                base = scratch.data_ptr()
                at = [base + o for o in self.bwd_at[i]]
            kept = lambda l: fwd.get(l, none)[0]
            gb = c3.backward(g, held, None, True, kept(c3), at[2])
            ga = c2.backward(gb, held, None, True, kept(c2), at[1])
            del gb
            gs = ds.backward(g, held, None, False, kept(ds), at[3]) if ds is not None else g
            # the two branches meet; the input of every block but the first is the ReLU output of the block below
            g = c1.backward(ga, held, gs, i > 0, kept(c1), at[0])
            del ga, gs
            if held is not None:
                C.convbn_tune_bwd_join()
                held.clear()
        if keep is not None:
            keep["dx"] = g.clone()
        if self.stem:
            gs = torch.empty_like(ins["g_stem"])
            C.convbn_relu_bwd(ins["g_stem"], s, gs)
            scratch = raw(self.stem.bwd_bytes) if tune else None
            gi = self.stem.backward(gs, None, None, False, fwd.get(self.stem, none)[0], scratch.data_ptr() if tune else None)
            if keep is not None:
                keep["d_image"] = gi.clone()
        return g

    # ---- measurements ------------------------------------------------------------------------------------
    def measure(self, iters: int = 5, warmup: int = 2):
        """(milliseconds per iteration from a CUDA-graph replay, peak bytes of one eager iteration above the
        bytes held before it: parameters, gradients and inputs)."""
        dev = self.device
        ins = self.make_inputs()
        for _ in range(warmup):
            self.forward_backward(ins)
        C.convbn_check()
        torch.cuda.synchronize(dev)
        torch.cuda.reset_peak_memory_stats(dev)
        base = torch.cuda.memory_allocated(dev)
        self.forward_backward(ins)
        torch.cuda.synchronize(dev)
        peak = torch.cuda.max_memory_allocated(dev) - base
        mode = "CUDA graph replay"
        try:
            gr = torch.cuda.CUDAGraph()
            with torch.cuda.graph(gr):
                self.forward_backward(ins)
            run = gr.replay
            run(); torch.cuda.synchronize(dev)
        except Exception as exc:          # capture unsupported: time eager calls and say so
            run, mode = (lambda: self.forward_backward(ins)), "eager calls (graph capture failed: %r)" % (exc,)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(iters):
            run()
        e1.record()
        torch.cuda.synchronize(dev)
        C.convbn_check()
        return e0.elapsed_time(e1) / iters, int(peak), mode
