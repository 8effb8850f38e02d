"""Host-side contract of the C ABI: the library loads without a GPU, exports every symbol the
header declares, computes shapes and sizes, and rejects bad arguments before any launch."""
import ctypes
import os
import re

import pytest

import __graft_entry__ as G
from paper_2305_11624_b200 import convbn as C

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def built():
    G.build()


def good(**kw):
    base = dict(n=2, c_in=16, h_in=16, w_in=16, c_out=32, kh=3, kw=3, pad_h=1, pad_w=1,
                dtype=C.F32, layout=C.NCHW)
    base.update(kw)
    return C.Desc.make(**base)


def test_every_declared_symbol_is_exported():
    header = open(os.path.join(ROOT, "include", "convbn.h")).read()
    declared = set(re.findall(r"\b(convbn_[a-z_]+)\s*\(", header))
    assert declared == set(C.EXPORTS)
    lib = C.lib()
    for name in declared:
        assert getattr(lib, name) is not None


def test_out_shape_and_sizes():
    assert C.convbn_out_shape(good()) == (16, 16)
    assert C.convbn_out_shape(good(h_in=224, w_in=224, kh=7, kw=7, stride_h=2, stride_w=2, pad_h=3, pad_w=3)) == (112, 112)
    assert C.convbn_out_shape(good(h_in=200, w_in=334, stride_h=2, stride_w=2)) == (100, 167)
    assert C.convbn_out_shape(good(h_in=9, w_in=9, dil_h=2, dil_w=2, pad_h=0, pad_w=0)) == (5, 5)
    d = good()
    assert C.convbn_saved_bytes(d, C.MODE_TUNE) == 3 * 32 * 4          # s, b', r: no feature map
    assert C.convbn_saved_bytes(d, C.MODE_EVAL) == 2 * 32 * 16 * 16 * 4  # the pre-normalisation Y
    assert C.convbn_saved_bytes(d, C.MODE_DEPLOY) == 0
    b = good(dtype=C.BF16, layout=C.NHWC)
    assert C.convbn_saved_bytes(b, C.MODE_EVAL) == 2 * 32 * 16 * 16 * 2
    for ph in range(7):
        assert C.convbn_workspace_bytes(d, ph) % 256 == 0
    assert C.convbn_workspace_bytes(d, C.PHASE_TUNE_FWD) >= 32 * 16 * 9 * 4
    assert C.convbn_workspace_bytes(d, 99) == 0


def test_workspace_sizes_of_the_benchmark_layers():
    """Every phase of every benchmark layer asks for a 256-byte multiple; the parameter-gradient scratch
    (partial tiles per pixel slice) stays within a few tens of MiB, and that of the headline configuration's
    layers within the 16 MiB of the no-allocation entry point."""
    from paper_2305_11624_b200 import inputs as I
    from paper_2305_11624_b200.harness import make_desc
    for ci, layers in I.CONFIGS.items():
        for sp in layers:
            d = make_desc(sp)
            for ph in (C.PHASE_TUNE_FWD, C.PHASE_TUNE_BWD_DATA, C.PHASE_TUNE_BWD_WEIGHT):
                ws = C.convbn_workspace_bytes(d, ph)
                assert ws % 256 == 0 and ws < 64 << 20, (sp.name, ph, ws)
            wsw = C.convbn_workspace_bytes(d, C.PHASE_TUNE_BWD_WEIGHT)
            assert wsw > 0, sp.name
            if ci == 1:
                assert wsw <= 16 << 20, (sp.name, wsw)


def test_stems_read_as_they_are_ask_for_no_packed_copy():
    """3 -> 64, 7 x 7, 224 x 224, N = 32: the packed copy of X is 13.5 MB, which the forward pass asked for without a use, and
    partial sums are all that the weight gradient writes."""
    d = good(n=32, c_in=3, h_in=224, w_in=224, c_out=64, kh=7, kw=7, stride_h=2, stride_w=2, pad_h=3, pad_w=3, dtype=C.BF16,
             layout=C.NHWC)
    assert all(C.convbn_workspace_bytes(d, ph) < 1 << 18 for ph in (C.PHASE_TUNE_FWD, C.PHASE_EVAL_FWD, C.PHASE_DEPLOY_FWD))
    assert C.convbn_workspace_bytes(d, C.PHASE_TUNE_BWD_WEIGHT) < 8 << 20
    d.w_in = 31                                                       # short rows, many of them: packed
    d.n = 512
    assert C.convbn_workspace_bytes(d, C.PHASE_TUNE_FWD) > 1 << 20 and C.convbn_workspace_bytes(d, C.PHASE_TUNE_BWD_WEIGHT) > 1 << 20


def test_which_layers_the_no_allocation_call_takes():
    """Decided by the layer alone, on the host, before any pointer is looked at: a scratch of up to 16 MiB, or one that fewer
    slices bring down to that (the second and third layer)."""
    one = dict(dtype=C.BF16, layout=C.NHWC)
    taken = [good(n=2, c_in=64, h_in=20, w_in=24, c_out=128, kh=3, kw=3, pad_h=1, pad_w=1, **one),
             good(n=12, c_in=768, h_in=13, w_in=13, c_out=384, kh=3, kw=3, pad_h=1, pad_w=1, **one),
             good(n=2, c_in=1600, h_in=25, w_in=25, c_out=1856, kh=1, kw=1, pad_h=0, pad_w=0, **one)]
    refused = [good(n=8, c_in=1024, h_in=7, w_in=7, c_out=1024, kh=3, kw=3, pad_h=1, pad_w=1, **one),
               good(n=16, c_in=512, h_in=56, w_in=56, c_out=512, kh=3, kw=3, pad_h=1, pad_w=1, **one)]
    assert C.convbn_workspace_bytes(taken[0], C.PHASE_TUNE_BWD_WEIGHT) <= 16 << 20
    assert all(C.convbn_workspace_bytes(d, C.PHASE_TUNE_BWD_WEIGHT) > 16 << 20 for d in taken[1:])

    def status(d):                     # dz = NULL: a layer that is taken gets as far as the pointer checks
        with pytest.raises(C.ConvBNError) as e:
            C.convbn_tune_bwd_weight_noalloc(d, None, 4096, 4096, None, 4096, 4096, 4096, None, 4096, 4096, stream=0)
        return e.value.status

    assert [status(d) for d in refused] == [C.ECAPACITY] * 2
    assert all(status(d) != C.ECAPACITY for d in taken)


@pytest.mark.parametrize("kw", [
    dict(n=0), dict(c_in=-1), dict(kh=0), dict(stride_h=0), dict(dil_w=0), dict(pad_h=-1),
    dict(groups=3), dict(groups=0), dict(h_in=1, w_in=1, pad_h=0, pad_w=0), dict(dtype=7),
    dict(layout=5), dict(eps=-1.0),
])
def test_bad_descriptors_are_rejected_on_the_host(kw):
    d = good(**kw)
    ho, wo = ctypes.c_int(), ctypes.c_int()
    assert C.lib().convbn_out_shape(ctypes.byref(d), ctypes.byref(ho), ctypes.byref(wo)) == C.EINVAL
    assert C.convbn_saved_bytes(d, C.MODE_EVAL) == 0
    assert C.convbn_workspace_bytes(d, C.PHASE_TUNE_FWD) == 0
    with pytest.raises(C.ConvBNError) as e:
        C.convbn_tune_fwd(d, 256, 256, None, 256, 256, 256, 256, 256, 256, 256, 1 << 30, stream=0)
    assert e.value.status == C.EINVAL


def test_largest_problems():
    """The documented size limits: 2^40 elements per tensor, 2^30 weights per output channel.  One element below is
    accepted (sizes come back, nothing overflows into a small or negative number), one above is CONVBN_EINVAL."""
    ho, wo = ctypes.c_int(), ctypes.c_int()
    shape = lambda d: C.lib().convbn_out_shape(ctypes.byref(d), ctypes.byref(ho), ctypes.byref(wo))
    one = dict(kh=1, kw=1, pad_h=0, pad_w=0, dtype=C.BF16, layout=C.NHWC)
    # 2^40 activation elements exactly: 2^15 images of 2^7 x 2^8 pixels and 2^10 channels
    at_limit = good(n=1 << 15, c_in=1 << 10, h_in=1 << 7, w_in=1 << 8, c_out=1 << 10, **one)
    assert shape(at_limit) == C.OK and (ho.value, wo.value) == (1 << 7, 1 << 8)
    assert C.convbn_saved_bytes(at_limit, C.MODE_EVAL) == 2 << 40
    assert C.convbn_saved_bytes(at_limit, C.MODE_TUNE) == 3 * 4 * (1 << 10)
    for ph in (C.PHASE_TUNE_FWD, C.PHASE_TUNE_BWD, C.PHASE_EVAL_BWD):
        ws = C.convbn_workspace_bytes(at_limit, ph)
        assert 0 < ws < 3 << 40 and ws % 256 == 0, (ph, ws)      # Eval backward holds dY, a tensor of the size of Z
    assert shape(good(n=(1 << 15) + 1, c_in=1 << 10, h_in=1 << 7, w_in=1 << 8, c_out=1 << 10, **one)) == C.EINVAL   # input
    assert shape(good(n=(1 << 15) + 1, c_in=8, h_in=1 << 7, w_in=1 << 8, c_out=1 << 10, **one)) == C.EINVAL         # output
    # weights per output channel: C_in kh kw <= 2^30
    wide = dict(n=1, h_in=64, w_in=64, c_out=8, pad_h=0, pad_w=0, dtype=C.BF16, layout=C.NHWC)
    assert shape(good(c_in=1 << 18, kh=64, kw=64, **wide)) == C.OK and (ho.value, wo.value) == (1, 1)
    assert shape(good(c_in=(1 << 18) + 8, kh=64, kw=64, **wide)) == C.EINVAL
    # extents that no int holds are rejected, not wrapped
    assert shape(good(n=1, c_in=1, h_in=(1 << 31) - 1, w_in=(1 << 31) - 1, c_out=1, **one)) == C.EINVAL
    assert shape(good(h_in=16, w_in=16, pad_h=(1 << 31) - 1, pad_w=1)) == C.EINVAL


def test_argument_checks_before_any_launch():
    d = good()
    ws = C.convbn_workspace_bytes(d, C.PHASE_TUNE_FWD)
    ok = 4096
    args = lambda **o: {**dict(x=ok, w=ok, b=None, gamma=ok, beta=ok, run_mean=ok, run_var=ok, z=ok,
                               saved=ok, workspace=ok, workspace_bytes=ws, stream=0), **o}

    def status(**o):
        with pytest.raises(C.ConvBNError) as e:
            C.convbn_tune_fwd(d, **args(**o))
        return e.value.status

    assert status(x=None) == C.EINVAL
    assert status(saved=None) == C.EINVAL
    assert status(x=ok + 8) == C.EALIGN
    assert status(gamma=ok + 2) == C.EALIGN
    assert status(workspace=None) == C.EWORKSPACE
    assert status(workspace_bytes=ws - 1) == C.EWORKSPACE
    assert status(workspace=ok + 16) == C.EALIGN
    mixed = good(dtype=C.BF16, layout=C.NCHW)
    with pytest.raises(C.ConvBNError) as e:
        C.convbn_tune_fwd(mixed, **args())
    assert e.value.status == C.EUNSUPPORTED
    # db must be given exactly when b is
    with pytest.raises(C.ConvBNError) as e:
        C.convbn_tune_bwd_weight(d, ok, ok, ok, ok, ok, ok, ok, None, ok, ok, ok, 1 << 30, stream=0)
    assert e.value.status == C.EINVAL


def test_addresses_may_be_integers_of_any_kind():
    """Pointers, sizes and streams as plain integers or as subclasses of int (an address type of another package)."""
    class Address(int):
        pass
    with pytest.raises(C.ConvBNError) as e:
        C.convbn_tune_fwd(good(), Address(4096), 4096, None, 4096, 4096, 4096, 4096, 4096, Address(4096 + 8), Address(4096),
                          Address(1 << 30), stream=Address(0))
    assert e.value.status == C.EALIGN                       # `saved` is the one that is off


def test_the_library_takes_plain_addresses_in_full_width():
    """lib() itself, with descriptors and integer addresses as they are: an address whose lower half is zero is no NULL."""
    d, ok, high = good(), 4096, 1 << 32
    two = C.Desc.make(1, 8, 4, 4, 8, 3, 3, 2, 2, 1, 1)
    lib = C.lib()
    assert lib.convbn_tune_fwd(d, high, ok + 8, None, ok, ok, ok, ok, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_tune_bwd_data(d, high, ok + 8, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_tune_bwd_weight(d, high, ok, ok + 8, None, ok, ok, ok, None, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_tune_bwd(d, high, ok, ok + 8, None, ok, ok, ok, ok, None, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_tune_bwd_begin(d, high, ok, ok + 8, None, ok, ok, ok, ok, None, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_tune_fwd_glue(d, high, ok + 8, None, ok, ok, ok, ok, ok, ok, None, 0, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_tune_bwd_glue(d, high, ok, ok + 8, None, ok, ok, ok, ok, None, ok, ok, None, 0, 0, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_eval_fwd(d, high, ok + 8, None, ok, ok, ok, ok, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_eval_bwd(d, high, ok, ok, ok + 8, ok, ok, ok, ok, ok, None, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_deploy_fwd(d, high, ok + 8, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_deploy_bwd(d, high, ok, ok + 8, ok, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_tconv_tune_fwd(two, high, ok + 8, None, ok, ok, ok, ok, ok, ok, ok, 1 << 33, 0) == C.EALIGN
    assert lib.convbn_tconv_tune_bwd(two, high, ok, ok + 8, None, ok, ok, ok, ok, None, ok, ok, ok, 1 << 33, 0) == C.EALIGN


def test_descriptors_in_every_form():
    """The forms a C parameter `const convbn_desc *` takes are taken, with the bytes that they point at; others are refused."""
    class Longer(C.Desc):
        _fields_ = [("more", ctypes.c_int)]

    bad, d = good(n=0), good()
    longer = Longer(*[getattr(d, f) for f, _ in C.Desc._fields_], 7)
    args = (4096, 4096, None, 4096, 4096, 4096, 4096, 4096, 4096 + 8, 4096)

    def status(desc, size=1 << 30):
        with pytest.raises(C.ConvBNError) as e:
            C.convbn_tune_fwd(desc, *args, size, stream=0)
        return e.value.status

    good_forms = [d, ctypes.byref(d), ctypes.pointer(d), (C.Desc * 1)(d), (C.Desc * 2)(d, bad), longer, ctypes.byref(longer)]
    assert [status(f) for f in good_forms] == [C.EALIGN] * len(good_forms)          # `saved` is off
    second = (C.Desc * 2)(bad, d)
    assert status(second) == C.EINVAL and status(ctypes.byref(second[0])) == C.EINVAL
    assert status(ctypes.byref(second[0], ctypes.sizeof(C.Desc))) == C.EALIGN
    assert status(None) == C.EINVAL and status(ctypes.POINTER(C.Desc)()) == C.EINVAL
    for other in (bytes(d), bytearray(d), 4096, 1.0, "desc", ctypes.byref(ctypes.c_int(1))):
        with pytest.raises(TypeError):
            C.convbn_tune_fwd(other, *args, 1 << 30, stream=0)
    assert status(d, (1 << 64) - 1) == C.EALIGN                                     # the largest size_t
    for size in (1.5, "1"):
        with pytest.raises(TypeError):
            C.convbn_tune_fwd(d, *args, size, stream=0)


def test_the_binding_is_built_per_interpreter_and_only_with_its_headers(monkeypatch, tmp_path, capsys):
    """A library that is up to date stays, a binding of another interpreter is not this one's, and without Python's headers the
    library is there alone."""
    import importlib.machinery
    from paper_2305_11624_b200 import build as B
    assert os.path.basename(B.BINDING) == "_binding" + importlib.machinery.EXTENSION_SUFFIXES[0]
    made = []
    monkeypatch.setattr(B, "LIBRARY", str(tmp_path / "lib.so"))
    monkeypatch.setattr(B, "BINDING", str(tmp_path / "_binding.here.so"))
    monkeypatch.setattr(B, "_build_library", lambda verbose: (made.append("library"), open(B.LIBRARY, "w").close()))
    monkeypatch.setattr(B, "_build_binding", lambda: (made.append("binding"), open(B.BINDING, "w").close()))
    (tmp_path / "_binding.other.so").write_text("")
    monkeypatch.setattr(B, "_headers", lambda: False)
    assert B.build() == B.LIBRARY and made == ["library"] and "Python.h" in capsys.readouterr().err
    monkeypatch.setattr(B, "_headers", lambda: True)
    B.build()
    B.build()
    assert made == ["library", "binding"]


def test_plans_kept_per_thread():
    """More layers than a thread keeps plans of, asked for in changing order, in both 16-bit types in turn, by two threads at
    once: every size is the one that a thread asked for nothing else gives."""
    import random
    import threading
    rng, asked = random.Random(3), []
    for i in range(300):
        kind = i % 4
        kw = dict(n=rng.randint(1, 40), h_in=rng.randint(8, 60), w_in=rng.randint(8, 60), dtype=C.BF16 if i % 2 else C.F16, layout=C.NHWC)
        c = 64 * rng.randint(1, 6)
        if kind == 0:
            d = good(c_in=c, c_out=64 * rng.randint(1, 6), **kw)
        elif kind == 1:
            d = good(c_in=3, c_out=64, kh=7, kw=7, stride_h=2, stride_w=2, pad_h=3, pad_w=3, **kw)
        elif kind == 2:
            d = good(c_in=c, c_out=c, groups=rng.choice((c, c // 8)), **kw)
        else:
            d = good(c_in=c, c_out=64, kh=2, kw=2, stride_h=2, stride_w=2, pad_h=0, pad_w=0, **kw)
        asked += [(d, ph) for ph in range(7)] + ([(d, "transposed")] if kind == 3 else [])
    size = lambda d, ph: C.convbn_tconv_workspace_bytes(d) if ph == "transposed" else C.convbn_workspace_bytes(d, ph)
    alone = {}

    def one(i):
        alone[i] = size(*asked[i])

    def many(order, out):
        out.extend((i, size(*asked[i])) for i in order)

    def run(*targets):
        threads = [threading.Thread(target=f, args=a) for f, a in targets]
        for t in threads:
            t.start()
        for t in threads:
            t.join()

    for i in range(len(asked)):
        run((one, (i,)))
    orders = [rng.sample(range(len(asked)), len(asked)) for _ in range(3)]
    got = [[], [], []]
    many(orders[0] + orders[0][:700], got[0])
    run((many, (orders[1], got[1])), (many, (orders[2], got[2])))
    assert len(alone) == len(asked) and len(set(alone.values())) > 500
    assert all(alone[i] == v for g in got for i, v in g)


def test_status_strings():
    assert C.status_string(C.OK) == "ok"
    assert "workspace" in C.status_string(C.EWORKSPACE)
    assert C.status_string(1234) == "unknown status"
    assert C.convbn_last_kernel(99) == "none"
