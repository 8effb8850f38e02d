"""Sizes at which the splits of the depthwise, stem, adding and transposed kernels change, against the fp64 oracle with the
tolerances and per-element bounds of parity.py."""
import ctypes

import numpy as np
import pytest

import parity
from paper_2305_11624_b200 import inputs as I

pytestmark = pytest.mark.gpu

L = I.LayerSpec
SPECS = [
    # depthwise above 256 channels: two parts of different sizes, parts that end inside a sector, more parts than row strips,
    # the widest multiple of 8, a strip that ends inside a thread's columns
    L("dw_264", 2, 264, 9, 11, 264, 3, 3, pad=1, groups=264, bias=True),
    L("dw_320", 3, 320, 13, 37, 320, 3, 3, pad=1, groups=320, dtype="f16"),
    L("dw_520", 1, 520, 6, 10, 520, 3, 3, pad=0, groups=520), L("dw_1032", 1, 1032, 5, 9, 1032, 3, 3, pad=2, groups=1032),
    # stem rows that start anywhere: odd and even widths off a multiple of 8, one to four channels, 128 output channels, images
    # smaller than a chunk of rows (STEM_DATA: which kernel forms their input gradient)
    L("stem_36", 8, 3, 46, 36, 64, 7, 7, stride=2, pad=3), L("stem_35", 3, 3, 33, 35, 64, 7, 7, stride=2, pad=3, dtype="f16"),
    L("stem_253", 1, 3, 15, 253, 64, 7, 7, stride=2, pad=3, bias=True), L("stem_255", 1, 3, 14, 255, 64, 7, 7, stride=2, pad=3),
    L("stem_c1", 7, 1, 21, 19, 64, 7, 7, stride=2, pad=3), L("stem_c2_k5", 8, 2, 22, 23, 64, 5, 5, stride=2, pad=2, dtype="f16"),
    L("stem_c4", 5, 4, 25, 27, 64, 7, 7, stride=2, pad=3), L("stem_o128", 2, 3, 19, 21, 128, 7, 7, stride=2, pad=3),
    L("stem_small", 70, 3, 9, 10, 64, 7, 7, stride=2, pad=3, dtype="f16"),
    # ... the window kernel where the sub-pixel kernel would take them too: three and four channels, the widest rows it takes; and one
    # pixel wider, and more rows than pay
    L("dx_c3", 8, 3, 46, 45, 64, 7, 7, stride=2, pad=3, bias=True), L("dx_c4", 8, 4, 46, 45, 64, 7, 7, stride=2, pad=3),
    L("dx_253", 9, 3, 31, 253, 64, 7, 7, stride=2, pad=3), L("dx_253_f16", 9, 3, 32, 253, 64, 6, 6, stride=2, pad=2, dtype="f16"),
    L("dx_254", 9, 3, 31, 254, 64, 7, 7, stride=2, pad=3), L("dx_rows", 17, 3, 62, 62, 64, 7, 7, stride=2, pad=3),
    # more than 32 taps on the strip kernel: dense and block-diagonal layers
    L("taps_49", 2, 64, 20, 24, 64, 7, 7, pad=3), L("taps_81", 1, 64, 21, 20, 128, 9, 9, pad=4, dtype="f16"),
    L("taps_49_groups", 2, 128, 19, 23, 128, 7, 7, pad=3, groups=8),
    # odd widths on both sides of the forward choice: short rows by the packed GEMM, long ones and few by the window kernel
    L("fwd_packed", 260, 3, 18, 21, 64, 7, 7, stride=2, pad=3, bias=True), L("fwd_packed_o128", 90, 4, 18, 21, 128, 5, 5, stride=2, pad=2),
    L("fwd_window", 3, 3, 24, 157, 64, 7, 7, stride=2, pad=3, dtype="f16"), L("fwd_window_o128", 2, 3, 14, 301, 128, 3, 3, stride=2, pad=1),
    L("fwd_window_c4", 3, 4, 24, 157, 64, 5, 5, stride=2, pad=2), L("fwd_window_c2", 3, 2, 24, 93, 64, 8, 8, stride=2, pad=2),
    # stem filters of 257 to 512 weights per output channel, more than the window kernel's table holds, at both kinds of width; and the
    # largest that it takes
    L("stem_16x8", 2, 4, 31, 37, 64, 16, 8, stride=2, pad=3), L("stem_16x8_w40", 2, 4, 31, 40, 64, 16, 8, stride=2, pad=3),
    L("stem_13x7", 2, 3, 30, 33, 64, 13, 7, stride=2, pad=3, dtype="f16"), L("stem_16x8_c2", 2, 2, 31, 37, 64, 16, 8, stride=2, pad=3),
    # adding the slices of a weight gradient: one block per channel, in one turn and several, clusters of two and four; spans that
    # end early; a slice group per thread and many
    L("rows_64", 2, 64, 6, 7, 2048, 1, 1), L("rows_192", 2, 192, 9, 9, 320, 1, 1, bias=True),
    L("rows_128", 3, 128, 14, 15, 192, 1, 1, dtype="f16"), L("rows_slices", 9, 64, 30, 31, 64, 3, 3, pad=1),
    L("rows_k5", 4, 64, 12, 13, 64, 5, 5, pad=2), L("rows_turns", 2, 640, 9, 8, 320, 3, 3, pad=1),
    L("rows_pairs", 4, 64, 30, 31, 128, 3, 3, pad=1, bias=True), L("rows_fours", 5, 64, 28, 29, 64, 3, 3, pad=1, dtype="f16"),
    # dense epilogue: output channels that end inside a 64-column chunk, a last tile of one pixel
    L("epi_72", 3, 64, 7, 19, 72, 3, 3, pad=1, bias=True), L("epi_200", 43, 64, 3, 1, 200, 1, 1, dtype="f16"),
]


STEM_DATA = dict.fromkeys(("stem_c1", "stem_c2_k5", "stem_small", "dx_c3", "dx_c4", "dx_253", "dx_253_f16"), "umma-stem")
STEM_DATA.update(dict.fromkeys(("stem_36", "stem_35", "stem_253", "stem_255", "stem_c4", "stem_16x8", "dx_254", "dx_rows"), "umma-subpixel"))
STEM_DATA["stem_o128"] = "stem-mma"


@pytest.mark.parametrize("spec", SPECS, ids=lambda s: s.name)
def test_tune_block(spec):
    t = parity.make_inputs(spec, 78)
    ref = parity.oracle_tune(spec, t)
    got = parity.run_tune_gpu(spec, t, deferred=True)
    parity.compare(got, ref, parity.TOL[spec.dtype], parity.TUNE_OUTPUTS, spec.name, dtype=spec.dtype)
    assert got["_kernels"][1] == STEM_DATA.get(spec.name, got["_kernels"][1])


@pytest.mark.parametrize("c_out,n,h,w", [(128, 700, 18, 24), (128, 260, 30, 32), (64, 900, 9, 16)], ids=["o128", "o128_w32", "o64"])
def test_stem_forward_of_many_short_rows(c_out, n, h, w):
    """Rows shorter than a quarter of an accumulator, thousands of them: three of a group's four warps have nothing to store and
    pass by.  No wait expires, and every image of a batch of equal images comes out the same."""
    import torch
    from paper_2305_11624_b200 import convbn as C
    from paper_2305_11624_b200.harness import Block
    blk = Block(L("rows", n, 3, h, w, c_out, 7, 7, stride=2, pad=3), modes=("tune",))
    blk.randomize(83)
    x = blk.x.view(n, -1)
    x.copy_(x[:1].expand(n, -1).clone())
    for _ in range(5):
        blk.z.fill_(float("nan"))
        blk.tune_fwd()
        C.convbn_check()
        z = blk.z.view(n, -1)
        assert bool((z == z[:1]).all())
    one = Block(L("rows", 1, 3, h, w, c_out, 7, 7, stride=2, pad=3), modes=("tune",))
    one.randomize(83)
    one.x.copy_(x[0])
    one.tune_fwd()
    assert torch.equal(one.z, z[0])


# rows of 48, 80 and 144 vectors in clusters of four: with 48 the last block has no columns and goes straight to the exchange of the
# dot products
@pytest.mark.parametrize("n,c_in,k", [(10, 192, 1), (14, 320, 1), (9, 64, 3)], ids=["row192", "row320", "row576"])
def test_clusters_with_blocks_beyond_the_row(n, c_in, k):
    """Every block's part of the dot product arrives: dgamma matches the oracle, and is the same in every one of many runs."""
    import torch
    from paper_2305_11624_b200 import convbn as C
    from paper_2305_11624_b200.harness import Block
    spec = L("clusters", n, c_in, 30, 31, 64, k, k, pad=k // 2)
    t = parity.make_inputs(spec, 79)
    parity.compare(parity.run_tune_gpu(spec, t, deferred=True), parity.oracle_tune(spec, t), parity.TOL["bf16"],
                   parity.TUNE_OUTPUTS, spec.name, dtype="bf16")
    blk = Block(spec, modes=("tune",))
    blk.load(t)
    blk.tune_fwd()
    seen = torch.empty(200, 64, device=blk.device)
    for i in range(200):
        blk.dgamma.fill_(float("nan"))
        blk.tune_bwd_weight()
        seen[i].copy_(blk.dgamma)
    C.convbn_check()
    assert bool((seen == seen[0]).all())


def weight_gradient(spec, x, dz):
    """fp64 sums of dZ X over the pixels inside the image, tap by tap: nothing is multiplied that is not in the sum."""
    dw = np.zeros((spec.c_out, spec.c_in // spec.groups, spec.kh, spec.kw))
    (ho, wo), st, p = dz.shape[2:], spec.stride, spec.pad
    for r in range(spec.kh):
        for q in range(spec.kw):
            h = [i for i in range(ho) if 0 <= i * st + r - p < spec.h_in]
            w = [i for i in range(wo) if 0 <= i * st + q - p < spec.w_in]
            if h and w:
                xs = x[:, :, h[0] * st + r - p:h[-1] * st + r - p + 1:st, w[0] * st + q - p:w[-1] * st + q - p + 1:st]
                ds = dz[:, :, h[0]:h[-1] + 1, w[0]:w[-1] + 1]
                dw[:, :, r, q] = (np.einsum("nohw,nchw->oc", ds, xs) if spec.groups == 1 else (ds * xs).sum((0, 2, 3))[:, None])
    return dw


def same_kind(got, ref, name):
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref)), name
    assert np.array_equal(np.sign(got[np.isinf(got)]), np.sign(ref[np.isinf(ref)])), name


def test_depthwise_rows_beyond_a_band_are_not_multiplied():
    """An infinite X, in every row of the image and so at every edge of a band: domega is infinite where the pixel is in its
    sum, and finite elsewhere."""
    from paper_2305_11624_b200 import convbn as C
    spec = L("inf_dw", 2, 264, 11, 12, 264, 3, 3, pad=1, groups=264)
    t = parity.make_inputs(spec, 80)
    for c in range(0, 264, 2):
        t["x"][c % 4 // 2, c, c % 11, c % 12] = -np.inf if c % 3 else np.inf
    with np.errstate(invalid="ignore"):
        ref = weight_gradient(spec, t["x"], t["dz"])
        got = parity.run_tune_gpu(spec, t)["dw"]
    C.convbn_check()
    assert np.isinf(ref).any() and not np.isnan(ref).any()
    s = t["gamma"] / np.sqrt(t["var_hat"] + spec.eps)
    same_kind(got, s[:, None, None, None] * ref, spec.name)


@pytest.mark.parametrize("kh,kw", [(7, 7), (4, 5), (2, 1), (8, 8)])
def test_stem_input_gradient_of_infinite_values(kh, kw):
    """dX is infinite or NaN exactly where an infinite dZ meets a weight (window kernel, an odd width)."""
    from paper_2305_11624_b200 import convbn as C
    spec = L("inf_stem_dx", 40, 3, 18, 21, 64, kh, kw, stride=2, pad=1)
    t = parity.make_inputs(spec, 81)
    t["dz"][0, 3, 2, 1] = t["dz"][5, 60, 0, 0] = t["dz"][39, 0, -1, -1] = np.inf
    got = parity.run_tune_gpu(spec, t)
    C.convbn_check()
    assert got["_kernels"][1] == "umma-stem"
    met = np.zeros(t["x"].shape, dtype=bool)
    for n, _, i, j in np.argwhere(np.isinf(t["dz"])):
        rows, cols = np.arange(2 * i - 1, 2 * i - 1 + kh), np.arange(2 * j - 1, 2 * j - 1 + kw)
        met[n][np.ix_(range(3), rows[(rows >= 0) & (rows < 18)], cols[(cols >= 0) & (cols < 21)])] = True
    assert np.array_equal(~np.isfinite(got["dx"]), met)


@pytest.mark.parametrize("n,h,w,k", [(3, 17, 33, 7), (1, 35, 33, 3), (41, 15, 38, 5), (2, 40, 94, 7)])
def test_stem_weight_gradient_of_infinite_values(n, h, w, k):
    """domega is infinite exactly in the taps whose sums an infinite X is part of (widths off a multiple of 8); sum dZ does not see
    X at all."""
    from paper_2305_11624_b200 import convbn as C
    spec = L("inf_stem_dw", n, 3, h, w, 64, k, k, stride=2, pad=k // 2)
    t = parity.make_inputs(spec, 82)
    t["x"][0, 0, 0, 0], t["x"][n - 1, 0, h // 2, 3], t["x"][0, 1, h - 1, w - 1] = np.inf, np.inf, -np.inf
    with np.errstate(invalid="ignore"):
        got, ref = parity.run_tune_gpu(spec, t), weight_gradient(spec, t["x"], t["dz"])
    C.convbn_check()
    assert got["_kernels"][2] == "umma-stem"
    s = t["gamma"] / np.sqrt(t["var_hat"] + spec.eps)
    same_kind(got["dw"], s[:, None, None, None] * ref, spec.name)
    np.testing.assert_allclose(got["dbeta"], t["dz"].sum((0, 2, 3)), rtol=1e-4, atol=1e-3)


def test_stem_weight_gradient_without_room_for_a_packed_copy():
    """At an odd width and 17.9 MB of scratch for the packed form, the no-allocation call goes to the window kernel."""
    from paper_2305_11624_b200 import convbn as C
    from paper_2305_11624_b200.harness import Block
    spec = L("stem_noalloc", 64, 1, 239, 99, 64, 4, 3, stride=2, pad=2)
    t = parity.make_inputs(spec, 84)
    ref = parity.oracle_tune(spec, t)
    blk = Block(spec, modes=("tune",))
    assert C.convbn_workspace_bytes(blk.desc, C.PHASE_TUNE_BWD_WEIGHT) > 16 << 20
    blk.load(t)
    blk.tune_fwd()
    C.convbn_tune_bwd_weight_noalloc(blk.desc, blk.dz, blk.x, blk.w, blk.b, blk.mu_hat, blk.saved, blk.dw, blk.db, blk.dgamma, blk.dbeta)
    C.convbn_check()
    got = {k: blk.fetch(k) for k in ("dw", "dgamma", "dbeta")}
    parity.compare(got, ref, parity.TOL["f32"], ("dw", "dgamma", "dbeta"), spec.name, dtype="bf16")


# (dtype, n, c_in, h, w, c_out, k, stride, pad): dZ summed inside the weight gradient where the kernel is the stride (one tile of
# channels and several that take turns, more than eight of them, slices shorter than the turns, 3 x 3, 1 x 1), by the kernel of
# its own where the windows overlap
TCONV = [("bf16", 3, 64, 5, 7, 64, 2, 2, 0), ("f16", 2, 256, 20, 13, 128, 2, 2, 0), ("bf16", 1, 1216, 3, 5, 64, 2, 2, 0),
         ("bf16", 2, 128, 7, 9, 64, 3, 3, 0), ("f16", 2, 192, 9, 8, 64, 1, 1, 0), ("bf16", 2, 128, 9, 7, 64, 3, 2, 1),
         # the finish with one group of slices (three slices, many weights), two (six slices) and eight (more than 16)
         ("bf16", 1, 512, 20, 31, 512, 2, 2, 0), ("f16", 1, 192, 38, 39, 512, 2, 2, 0), ("bf16", 5, 64, 33, 30, 64, 2, 2, 0)]


@pytest.mark.parametrize("case", TCONV, ids=lambda c: "%s_c%d_k%d_s%d" % (c[0], c[2], c[6], c[7]))
def test_transposed_block(case):
    import test_tconv
    dtype, n, ci, h, w, co, k, st, pad = case
    test_tconv.test_library_matches_the_oracle((dtype, n, ci, h, w, co, k, st, pad, 1, 1, True))


def test_descriptors_by_reference():
    """The calls take a descriptor as it is, by reference and by pointer, and refuse anything else."""
    import torch
    from paper_2305_11624_b200 import convbn as C
    from paper_2305_11624_b200.harness import Block
    blk = Block(L("ref", 2, 64, 6, 7, 64, 1, 1), modes=("tune",))
    blk.randomize(5)
    outs = []
    for desc in (blk.desc, ctypes.byref(blk.desc), ctypes.pointer(blk.desc)):
        blk.z.fill_(0)
        C.convbn_tune_fwd(desc, blk.x, blk.w, None, blk.gamma, blk.beta, blk.mu_hat, blk.var_hat, blk.z, blk.saved,
                          blk.workspace.data_ptr(), blk.workspace.nbytes, torch.cuda.current_stream())
        outs.append(blk.z.clone())
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
    with pytest.raises(TypeError):
        C.convbn_tune_fwd(b"short", blk.x, blk.w, None, blk.gamma, blk.beta, blk.mu_hat, blk.var_hat, blk.z, blk.saved, blk.workspace)
    with pytest.raises(C.ConvBNError):
        C.convbn_tune_fwd(None, blk.x, blk.w, None, blk.gamma, blk.beta, blk.mu_hat, blk.var_hat, blk.z, blk.saved, blk.workspace)
