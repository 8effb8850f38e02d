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
    L("g8_last_row", 9, 128, 17, 29, 128, 3, 3, pad=1, groups=16),
    # fp32 NCHW: one channel and one pixel row, 128 channels (nothing left for pixel groups), a plane of 64 pixels and one
    # more, more bands than blocks of a cluster, output channels that end inside a block and inside a cluster
    L("f32_tiny", 1, 1, 1, 5, 3, 3, 3, pad=1, dtype="f32", layout="nchw", bias=True),
    L("f32_c128", 2, 128, 5, 13, 128, 3, 3, pad=1, dtype="f32", layout="nchw"),
    L("f32_65", 3, 5, 13, 5, 9, 1, 1, dtype="f32", layout="nchw", bias=True),
    L("f32_many", 16, 33, 40, 37, 35, 3, 3, pad=1, dtype="f32", layout="nchw"),
    L("f32_nopad", 1, 20, 9, 30, 34, 3, 3, pad=0, dtype="f32", layout="nchw", bias=True),
    L("f32_pad2", 1, 7, 6, 9, 6, 3, 3, pad=2, dtype="f32", layout="nchw"),
]


@pytest.mark.parametrize("spec", SPECS, ids=lambda s: s.name)
def test_tune_block(spec):
    t = parity.make_inputs(spec, 77)
    ref = parity.oracle_tune(spec, t)
    for deferred in (False, True):
        got = parity.run_tune_gpu(spec, t, deferred=deferred)
        parity.compare(got, ref, parity.TOL[spec.dtype], parity.TUNE_OUTPUTS, spec.name, dtype=spec.dtype)


TCONV = [  # (dtype, n, c_in, h, w, c_out, k, stride, pad, dil, groups, bias): kernel = stride, the GEMM on omega as it is
    ("bf16", 3, 64, 5, 7, 192, 2, 2, 0, 1, 1, True),        # tiles of 64 columns, fewer pixels than a tile
    ("f16", 1, 192, 13, 11, 64, 3, 3, 0, 1, 1, False),      # nine taps, a last tile of 15 pixels
    ("bf16", 2, 256, 21, 24, 256, 2, 2, 0, 1, 1, True),     # a tap of 256 columns
]


@pytest.mark.parametrize("case", TCONV, ids=lambda c: "%s_c%d_o%d_k%d" % (c[0], c[2], c[5], c[6]))
def test_tconv_block(case):
    import test_tconv
    test_tconv.test_library_matches_the_oracle(case)
