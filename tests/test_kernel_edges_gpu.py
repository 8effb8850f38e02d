"""Sizes at which the tiling, the remainders or the dispatch of a kernel change, against the fp64 oracle."""
import pytest

import parity
from paper_2305_11624_b200 import inputs as I

pytestmark = pytest.mark.gpu

L = I.LayerSpec
SPECS = [
    # 8 channels per group: more chunks of channels than the grid has slots left over (the grid is rounded to chunks),
    # the widest row one box takes, a last band of one row
    L("g8_chunks", 13, 704, 9, 10, 704, 3, 3, pad=1, groups=88, bias=True),
    L("g8_wide", 1, 64, 5, 254, 64, 3, 3, pad=1, groups=8, dtype="f16"),
    # more partial slots than one batch of every thread (512 threads finish), many channels with few slots (256)
    L("g8_slots", 31, 64, 20, 16, 64, 3, 3, pad=1, groups=8), L("g8_few_slots", 2, 768, 9, 12, 768, 3, 3, pad=1, groups=96, dtype="f16"),
    L("g8_last_row", 9, 128, 17, 29, 128, 3, 3, pad=1, groups=16),
    # fp32 NCHW: one channel and one pixel row, 128 channels (nothing left for pixel groups), a plane of 64 pixels and one
    # more, more bands than blocks of a cluster, output channels that end inside a block and inside a cluster
    L("f32_tiny", 1, 1, 1, 5, 3, 3, 3, pad=1, dtype="f32", layout="nchw", bias=True),
    L("f32_c128", 2, 128, 5, 13, 128, 3, 3, pad=1, dtype="f32", layout="nchw"),
    L("f32_65", 3, 5, 13, 5, 9, 1, 1, dtype="f32", layout="nchw", bias=True),
    L("f32_many", 16, 33, 40, 37, 35, 3, 3, pad=1, dtype="f32", layout="nchw"),
    L("f32_nopad", 1, 20, 9, 30, 34, 3, 3, pad=0, dtype="f32", layout="nchw", bias=True),
    L("f32_pad2", 1, 7, 6, 9, 6, 3, 3, pad=2, dtype="f32", layout="nchw"),
    # ... several clusters for the same output channels: a share without a whole band for every block, bands that end early,
    # one output channel; 32-channel blocks and 4-channel ones that split the inputs; pixel tiles across images
    L("f32_shares", 9, 40, 19, 23, 7, 3, 3, pad=1, dtype="f32", layout="nchw", bias=True),
    L("f32_one_out", 12, 93, 48, 47, 1, 1, 1, dtype="f32", layout="nchw"),
    L("f32_shares_8", 16, 8, 56, 50, 8, 3, 3, pad=1, dtype="f32", layout="nchw"),
    L("f32_planes", 130, 17, 3, 5, 41, 3, 3, pad=1, dtype="f32", layout="nchw", bias=True),
    # rows of features: parameter gradients by the direct kernels, the rest by these
    L("f32_rows", 3001, 24, 1, 1, 37, 1, 1, dtype="f32", layout="nchw", bias=True),
    # dense GEMM by CTA pairs: an odd number of pixel tiles (the last has no partner) at 64 columns a pair; several rounds
    # at 128; 256 with a ragged last tile.  Channel chunks outermost: two chunks, weights resident and streamed
    L("pair_64", 7, 512, 7, 7, 192, 3, 3, pad=1, bias=True),
    L("pair_128", 25, 512, 7, 7, 2048, 3, 3, pad=1, dtype="f16"),
    L("pair_256", 3, 512, 112, 112, 1024, 1, 1),
    L("chunks_first", 5, 128, 24, 22, 192, 3, 3, pad=1), L("chunks_resident", 30, 128, 30, 31, 64, 2, 2, dtype="f16"),
    # weight gradient: C_out that ends inside the box of a 128-wide tile, fewer pixels than a stage
    L("wgrad_c192", 3, 64, 5, 4, 192, 3, 3, pad=1),
    # ... rows of features and one pixel-row images (two CTAs per SM), the same pixels in rows of four (one)
    L("wgrad_rows", 9001, 192, 1, 1, 64, 1, 1), L("wgrad_w3", 701, 64, 4, 3, 128, 3, 3, pad=1, dtype="f16"), L("wgrad_w4", 701, 64, 3, 4, 128, 3, 3, pad=1),
]


@pytest.mark.parametrize("spec", SPECS, ids=lambda s: s.name)
def test_tune_block(spec):
    t = parity.make_inputs(spec, 77)
    ref = parity.oracle_tune(spec, t)
    for deferred in (False, True):
        got = parity.run_tune_gpu(spec, t, deferred=deferred)
        parity.compare(got, ref, parity.TOL[spec.dtype], parity.TUNE_OUTPUTS, spec.name, dtype=spec.dtype)


EVAL = [  # Eval mode
    # more than 2048 output channels: the backward's sums by the kernel that takes any channel count, which writes no s dZ here
    L("eval_c2112", 3, 64, 5, 7, 2112, 1, 1, bias=True), L("eval_c2112_f16", 2, 128, 4, 9, 2112, 1, 1, dtype="f16"),
    # output channels that fill no 64-wide tile, strides, and the shapes of the one-launch 1x1 backward with a last tile of
    # pixels that is not full
    # (stride 2 with 1x1 in half: most of dX is zeros there, so that an exact sum of the dY that bf16 stores is already
    # 1.09 of the bound for bf16 away from the oracle in one element; in half it is 0.46)
    L("eval_o72", 3, 64, 9, 11, 72, 1, 1, bias=True), L("eval_o200_k3", 2, 64, 13, 7, 200, 3, 3, pad=1),
    L("eval_s2_k1_f16", 3, 128, 9, 9, 72, 1, 1, stride=2, dtype="f16"),
    L("eval_s2_k3", 2, 64, 11, 13, 128, 3, 3, stride=2, pad=1, bias=True),
    L("eval_64_256", 3, 64, 9, 11, 256, 1, 1, bias=True), L("eval_256_64_f16", 3, 256, 9, 11, 64, 1, 1, dtype="f16"),
    L("eval_128_64", 1, 128, 17, 19, 64, 1, 1), L("eval_64_128_f16", 5, 64, 7, 5, 128, 1, 1, bias=True, dtype="f16"),
]


@pytest.mark.parametrize("spec", EVAL, ids=lambda s: s.name)
def test_eval_block(spec):
    import test_parity_gpu
    test_parity_gpu.test_eval_and_deploy_comparators(spec)


@pytest.mark.parametrize("spec", [L("f32_inf", 2, 5, 9, 11, 6, 3, 3, pad=1, dtype="f32", layout="nchw"),
                                  L("f32_inf_wide", 40, 18, 20, 21, 40, 3, 3, pad=1, dtype="f32", layout="nchw")], ids=lambda s: s.name)
def test_fp32_block_does_not_multiply_by_its_padding(spec):
    """Infinite values: the taps that lie outside the image are left out, as the definition of the convolution has it, and do
    not add 0 x inf.  Against fp64 sums over the pixels inside the image: where those are finite, infinite, NaN."""
    import numpy as np
    from paper_2305_11624_b200 import convbn as C
    from paper_2305_11624_b200.harness import Block
    t = parity.make_inputs(spec, 21)
    t["w"][1, 2, 0, 0] = np.inf                     # no tap (0, 0) at the first row and column
    t["w"][3, 0, 2, 2] = -np.inf
    t["x"][0, 1, 0, spec.w_in - 1] = np.inf
    t["x"][1, 3, spec.h_in - 1, 4] = -np.inf
    t["dz"][0, 2, spec.h_in - 1, 0] = np.inf
    blk = Block(spec)
    blk.load(t)
    blk.tune_fwd()
    blk.tune_bwd()
    C.convbn_check()
    n, h, w, k, p = spec.n, spec.h_in, spec.w_in, spec.kh, spec.pad
    s = t["gamma"] / np.sqrt(t["var_hat"] + spec.eps)
    sw = t["w"] * s[:, None, None, None]
    z, dx, dw = np.zeros((n, spec.c_out, h, w)), np.zeros((n, spec.c_in, h, w)), np.zeros(t["w"].shape)
    with np.errstate(invalid="ignore"):
        for r in range(k):
            for q in range(k):
                o = tuple(slice(max(0, p - a), min(e, e + p - a)) for a, e in ((r, h), (q, w)))      # outputs with this tap inside
                i = tuple(slice(v.start + a - p, v.stop + a - p) for v, a in zip(o, (r, q)))
                xs, zs = t["x"][(slice(None), slice(None)) + i], t["dz"][(slice(None), slice(None)) + o]
                each = lambda a, b, eq: sum(np.multiply(*np.broadcast_arrays(a(c), b(c))) for c in range(eq))
                z[(slice(None), slice(None)) + o] += each(lambda c: xs[:, c, None], lambda c: t["w"][None, :, c, r, q, None, None], spec.c_in)
                dx[(slice(None), slice(None)) + i] += each(lambda c: zs[:, c, None], lambda c: sw[c][None, :, r, q, None, None], spec.c_out)
                for co in range(spec.c_out):
                    dw[co, :, r, q] = (zs[:, co, None] * xs).sum(axis=(0, 2, 3))
        z = z * s[None, :, None, None] + (-t["mu_hat"] * s + t["beta"])[None, :, None, None]
        dw *= s[:, None, None, None]
    for name, ref in (("z", z), ("dx", dx), ("dw", dw)):
        got, ref = blk.fetch(name), ref.reshape(blk.fetch(name).shape)
        assert np.array_equal(np.isnan(got), np.isnan(ref)), name
        assert np.array_equal(np.isinf(got), np.isinf(ref)) and np.array_equal(np.sign(got[np.isinf(got)]), np.sign(ref[np.isinf(ref)])), name
        fin = np.isfinite(ref)
        assert fin.any() and not fin.all() and np.allclose(got[fin], ref[fin], rtol=1e-4, atol=1e-4 * np.abs(ref[fin]).max()), name


TCONV = [  # (dtype, n, c_in, h, w, c_out, k, stride, pad, dil, groups, bias): kernel = stride, the GEMM on omega as it is
    ("bf16", 3, 64, 5, 7, 192, 2, 2, 0, 1, 1, True),        # tiles of 64 columns, fewer pixels than a tile
    ("f16", 1, 192, 13, 11, 64, 3, 3, 0, 1, 1, False),      # nine taps, a last tile of 15 pixels
    ("bf16", 2, 256, 21, 24, 256, 2, 2, 0, 1, 1, True),     # a tap of 256 columns
]


@pytest.mark.parametrize("case", TCONV, ids=lambda c: "%s_c%d_o%d_k%d" % (c[0], c[2], c[5], c[6]))
def test_tconv_block(case):
    import test_tconv
    test_tconv.test_library_matches_the_oracle(case)


def test_tconv_gradients_of_a_kernel_with_many_taps():
    """More than 65535 blocks of 32 weight columns: one input pixel, whose weight gradient is an outer product."""
    import torch
    from paper_2305_11624_b200 import convbn as C
    ci, co, k = 64, 128, 129
    dev = "cuda:0"
    desc = C.Desc.make(1, ci, 1, 1, co, k, k, dtype=C.BF16, layout=C.NHWC)
    assert C.convbn_tconv_out_shape(desc) == (k, k) and k * k * co // 32 > 65535
    gen = torch.Generator(device=dev)
    gen.manual_seed(6)
    rn = lambda *s: torch.randn(*s, generator=gen, device=dev)
    x, w, dz = rn(ci).bfloat16(), rn(ci, k * k, co).bfloat16(), rn(k * k, co).bfloat16()
    saved, mean = rn(3 * co), rn(co)
    dx, dw, dgamma, dbeta = torch.empty_like(x), torch.empty(ci, k * k, co, device=dev), rn(co), rn(co)
    ws = torch.empty(C.convbn_tconv_workspace_bytes(desc), dtype=torch.uint8, device=dev)
    C.convbn_tconv_tune_bwd(desc, dz, x, w, None, mean, saved, dx, dw, None, dgamma, dbeta, ws)
    C.convbn_check()
    s, r, sums = saved[:co].double(), saved[2 * co:].double(), dz.double().sum(0)
    close = lambda got, want, tol: assert_close(got.double(), want, tol)

    def assert_close(got, want, tol):
        assert bool(((got - want).norm() <= tol * want.norm()).item()), float((got - want).norm() / want.norm())

    for i in range(0, ci, 16):
        close(dw[i:i + 16], s * (x[i:i + 16, None, None].double() * dz.double()), 1e-6)      # one rounding of the product, one of s
    dot = sum((x[i].double() * dz.double() * w[i].double()).sum(0) for i in range(ci))
    close(dbeta, sums, 1e-5)
    close(dgamma, r * (dot - sums * mean.double()), 1e-5)
    close(dx, torch.stack([(w[i].double() * s * dz.double()).sum() for i in range(ci)]), parity.TOL["bf16"])


GLUE = [  # every kernel whose epilogue does the glue, and one that leaves it to passes of its own
    L("glue_1x1", 3, 128, 9, 13, 320, 1, 1, dtype="f16"),                     # GEMM, a last tile of 64 columns
    L("glue_strided", 2, 64, 11, 9, 128, 3, 3, stride=2, pad=1),              # a GEMM per parity class
    L("glue_empty", 2, 64, 10, 9, 64, 1, 1, stride=2),                        # positions without a class
    L("glue_strip", 2, 64, 21, 30, 192, 3, 3, pad=1), L("glue_strip_small", 2, 64, 21, 30, 128, 3, 3, pad=1, dtype="f16"),
    L("glue_pair", 7, 512, 7, 7, 512, 3, 3, pad=1, dtype="f16"),              # CTA pairs, an odd number of pixel tiles
    L("glue_subpixel", 1, 128, 33, 34, 128, 3, 3, stride=2, pad=1, dtype="f16"),
    L("glue_fused", 3, 256, 17, 15, 64, 1, 1), L("glue_fused_wide", 3, 64, 17, 15, 128, 1, 1, dtype="f16"),
    L("glue_stem", 2, 3, 37, 40, 64, 7, 7, stride=2, pad=3),
    L("glue_dw", 2, 32, 9, 21, 32, 3, 3, pad=1, groups=32),
    L("glue_f32", 2, 6, 9, 7, 10, 3, 3, pad=1, dtype="f32", layout="nchw"),
]


@pytest.mark.parametrize("spec", GLUE, ids=lambda s: s.name)
def test_glue_in_the_epilogue_equals_the_passes(spec):
    """convbn_tune_fwd_glue / _bwd_glue against the plain calls followed by the elementwise ones: the same bits."""
    import torch
    from paper_2305_11624_b200 import convbn as C
    from paper_2305_11624_b200.harness import Block
    blk = Block(spec)
    blk.randomize(3)
    blk.x.relu_()                                       # the mask's tensor is a ReLU output
    add_z, add_x = torch.randn_like(blk.z.normal_()), torch.randn_like(blk.x)
    blk.tune_fwd(); blk.tune_bwd()
    z, dx = blk.z.clone(), blk.dx.clone()
    grads = [t.clone() for t in (blk.dw, blk.dgamma, blk.dbeta)]
    C.convbn_check()
    for add, relu in ((None, True), (add_z, True), (add_z, False)):
        want = torch.empty_like(z)
        (C.convbn_add_relu if relu else C.convbn_add)(z, add, want) if add is not None else C.convbn_relu(z, want)
        blk.z.fill_(float("nan"))
        C.convbn_tune_fwd_glue(blk.desc, blk.x, blk.w, blk.b, blk.gamma, blk.beta, blk.mu_hat, blk.var_hat, blk.z, blk.saved,
                               add, relu, blk.workspace)
        assert torch.equal(blk.z, want), (add is not None, relu)
    for add, mask, begin in ((None, True, False), (add_x, True, True), (add_x, False, False)):
        want = dx.clone()
        if add is not None:
            C.convbn_add(want, add, want)
        if mask:
            C.convbn_relu_bwd(want, blk.x, want)
        for t in (blk.dx, blk.dw, blk.dgamma, blk.dbeta):
            t.fill_(float("nan"))
        C.convbn_tune_bwd_glue(blk.desc, blk.dz, blk.x, blk.w, blk.b, blk.mu_hat, blk.saved, blk.dx, blk.dw, blk.db,
                               blk.dgamma, blk.dbeta, add, mask, begin, blk.workspace)
        C.convbn_tune_bwd_join()
        assert torch.equal(blk.dx, want), (add is not None, mask)
        assert all(torch.equal(a, b) for a, b in zip((blk.dw, blk.dgamma, blk.dbeta), grads))
    C.convbn_check()


@pytest.mark.parametrize("spec", [s for s in GLUE if s.name in ("glue_stem", "glue_1x1", "glue_strip_small", "glue_pair", "glue_dw", "glue_f32")],
                         ids=lambda s: s.name)
def test_fused_relu_of_non_finite_values(spec):
    """NaN becomes 0 in every kernel's ReLU, as in convbn_relu; infinities and the other values are those of the passes."""
    import torch
    from paper_2305_11624_b200 import convbn as C
    from paper_2305_11624_b200.harness import Block
    blk = Block(spec)
    blk.randomize(4)
    for at, v in ((7, float("nan")), (blk.x.numel() // 2, float("inf")), (blk.x.numel() - 3, -float("inf"))):
        blk.x[at] = v
    blk.tune_fwd()
    want = torch.empty_like(blk.z)
    C.convbn_relu(blk.z, want)
    assert bool(blk.z.isnan().any()) and not bool(want.isnan().any())
    blk.z.fill_(float("nan"))
    C.convbn_tune_fwd_glue(blk.desc, blk.x, blk.w, blk.b, blk.gamma, blk.beta, blk.mu_hat, blk.var_hat, blk.z, blk.saved, None,
                           True, blk.workspace)
    C.convbn_check()
    assert torch.equal(blk.z, want)


@pytest.mark.parametrize("spec", [L("cap_3x3", 2, 64, 20, 24, 64, 3, 3, pad=1), L("cap_grouped", 2, 64, 12, 13, 64, 3, 3, pad=1, groups=8),
                                  L("cap_f32", 9, 40, 19, 23, 7, 3, 3, pad=1, dtype="f32", layout="nchw")], ids=lambda s: s.name)
def test_captured_backward_equals_the_plain_call(spec):
    """A captured backward call puts its passes on the other streams: the same bits."""
    import torch
    from paper_2305_11624_b200 import convbn as C
    from paper_2305_11624_b200.harness import Block
    blk = Block(spec)
    blk.randomize(5)
    blk.tune_fwd(); blk.tune_bwd()
    outs = (blk.dx, blk.dw, blk.dgamma, blk.dbeta)
    want = [t.clone() for t in outs]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        blk.tune_bwd()
    for t in outs:
        t.fill_(float("nan"))
    graph.replay()
    C.convbn_check()
    assert all(torch.equal(a, b) for a, b in zip(outs, want))


def test_no_allocation_call_in_fewer_slices():
    """A layer whose parameter-gradient scratch exceeds the built-in array: the call cuts it into fewer slices."""
    from paper_2305_11624_b200 import convbn as C
    from paper_2305_11624_b200.harness import Block
    spec = L("few_slices", 2, 384, 33, 4, 640, 3, 3, pad=1, bias=True)
    t = parity.make_inputs(spec, 12)
    ref = parity.oracle_tune(spec, t)
    blk = Block(spec)
    assert C.convbn_workspace_bytes(blk.desc, C.PHASE_TUNE_BWD_WEIGHT) > 16 << 20
    blk.load(t)
    blk.tune_fwd()
    for o in (blk.dw, blk.db, blk.dgamma, blk.dbeta):
        o.fill_(float("nan"))
    C.convbn_tune_bwd_weight_noalloc(blk.desc, blk.dz, blk.x, blk.w, blk.b, blk.mu_hat, blk.saved, blk.dw, blk.db, blk.dgamma,
                                     blk.dbeta)
    C.convbn_check()
    parity.compare({k: blk.fetch(k) for k in ("dw", "db", "dgamma", "dbeta")}, ref, parity.TOL["bf16"],
                   ("dw", "db", "dgamma", "dbeta"), spec.name, dtype=spec.dtype)
