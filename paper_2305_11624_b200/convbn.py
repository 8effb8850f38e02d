"""Thin binding of ``libconvbn.so`` (declared in ``include/convbn.h``): ctypes, and the extension module ``_binding`` for the calls that a
training step makes.

Argument marshalling only: every function has the name and argument order of its C entry point,
takes torch CUDA tensors (or raw integer device addresses, or None for NULL) and returns nothing;
a non-zero status raises ``ConvBNError``.  There is no fallback: if the compiled library is
missing, importing succeeds but the first call raises.
"""
import ctypes
import importlib.machinery
import importlib.util
import os
from typing import Optional

_HERE = os.path.dirname(os.path.abspath(__file__))
LIBRARY = os.path.join(_HERE, "libconvbn.so")

OK, EINVAL, EUNSUPPORTED, EWORKSPACE, EALIGN, ECUDA, ETIMEOUT, ECAPACITY = range(8)
F32, BF16, F16 = 0, 1, 2
NCHW, NHWC = 0, 1
MODE_TUNE, MODE_EVAL, MODE_DEPLOY = 0, 1, 2
(PHASE_TUNE_FWD, PHASE_TUNE_BWD_DATA, PHASE_TUNE_BWD_WEIGHT, PHASE_EVAL_FWD, PHASE_EVAL_BWD,
 PHASE_DEPLOY_FWD, PHASE_DEPLOY_BWD, PHASE_TUNE_BWD) = range(8)

EXPORTS = (
    "convbn_out_shape", "convbn_saved_bytes", "convbn_workspace_bytes", "convbn_tune_fwd",
    "convbn_tune_bwd_data", "convbn_tune_bwd_weight", "convbn_eval_fwd", "convbn_eval_bwd",
    "convbn_deploy_prepare", "convbn_deploy_fwd", "convbn_deploy_bwd", "convbn_check",
    "convbn_status_string", "convbn_last_kernel", "convbn_host_step_arena_bytes",
    "convbn_tune_step_host", "convbn_tune_step_host_begin", "convbn_tune_step_host_join", "convbn_profile_begin", "convbn_profile_end",
    "convbn_tune_bwd_weight_noalloc", "convbn_selftest_wait_timeout", "convbn_tune_bwd", "convbn_linear_desc", "convbn_relu", "convbn_add_relu", "convbn_relu_bwd", "convbn_add",
    "convbn_tune_bwd_begin", "convbn_tune_bwd_join", "convbn_tune_fwd_glue", "convbn_tune_bwd_glue",
    "convbn_tconv_out_shape", "convbn_tconv_workspace_bytes", "convbn_tconv_tune_fwd", "convbn_tconv_tune_bwd",
)


class ConvBNError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__("%s: %s (status %d)" % (where, status_string(status), status))


class Desc(ctypes.Structure):
    """Mirror of ``convbn_desc``."""
    _fields_ = [(k, ctypes.c_int) for k in (
        "n", "c_in", "h_in", "w_in", "c_out", "kh", "kw", "stride_h", "stride_w", "pad_h", "pad_w",
        "dil_h", "dil_w", "groups", "dtype", "layout")] + [("eps", ctypes.c_double)]

    @classmethod
    def make(cls, n, c_in, h_in, w_in, c_out, kh, kw, stride_h=1, stride_w=1, pad_h=0, pad_w=0,
             dil_h=1, dil_w=1, groups=1, dtype=BF16, layout=NHWC, eps=1e-5):
        return cls(n, c_in, h_in, w_in, c_out, kh, kw, stride_h, stride_w, pad_h, pad_w, dil_h,
                   dil_w, groups, dtype, layout, float(eps))


_lib = None


def _signatures():
    """argtypes of the entry points that take pointers: ctypes then converts plain integers itself, without an object per
    argument, and to their full width (d: descriptor, p: pointer or stream, z: size, i: int, q: long long, f: double).  The
    calls of a training step go through _binding here; whoever takes them from lib() gets them typed all the same."""
    kinds = {"d": ctypes.POINTER(Desc), "p": ctypes.c_void_p, "z": ctypes.c_size_t, "i": ctypes.c_int,
             "q": ctypes.c_longlong, "f": ctypes.c_double}
    table = {
        "convbn_tune_fwd": "dppppppppppzp", "convbn_tune_bwd_data": "dpppppzp", "convbn_tune_bwd_weight": "dppppppppppp" "zp",
        "convbn_tune_bwd": "dppppppppppppzp", "convbn_tune_bwd_begin": "dppppppppppppzp", "convbn_tune_bwd_join": "p",
        "convbn_tune_fwd_glue": "dppppppppppipzp", "convbn_tune_bwd_glue": "dppppppppppppiipzp",
        "convbn_tconv_tune_fwd": "dppppppppppzp", "convbn_tconv_tune_bwd": "dppppppppppppzp",
        "convbn_eval_fwd": "dppppppppppzp", "convbn_eval_bwd": "dpppppppppppppzp",
        "convbn_deploy_fwd": "dpppppzp", "convbn_deploy_bwd": "dpppppppzp",
        "convbn_tune_bwd_weight_noalloc": "dppppppppppp", "convbn_deploy_prepare": "dppppppppp",
        "convbn_relu": "ippqp", "convbn_add_relu": "ipppqp", "convbn_relu_bwd": "ipppqp",
        "convbn_add": "ipppqp", "convbn_workspace_bytes": "di", "convbn_saved_bytes": "di", "convbn_check": "p",
    }
    return {name: [kinds[k] for k in sig] for name, sig in table.items()}


def lib():
    """Load the compiled library (raises OSError with the build hint if it is absent)."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIBRARY):
            raise OSError("%s not found: run `python -m paper_2305_11624_b200.build` "
                          "(there is no CPU fallback)" % LIBRARY)
        L = ctypes.CDLL(LIBRARY)
        L.convbn_saved_bytes.restype = ctypes.c_size_t
        L.convbn_workspace_bytes.restype = ctypes.c_size_t
        L.convbn_host_step_arena_bytes.restype = ctypes.c_size_t
        L.convbn_status_string.restype = ctypes.c_char_p
        L.convbn_last_kernel.restype = ctypes.c_char_p
        for name in EXPORTS:
            getattr(L, name)
        for name, types in _signatures().items():
            getattr(L, name).argtypes = types
        _lib = L
    return _lib


_native = None


def _calls():
    """The entry points of csrc/binding.cpp."""
    global _native
    if _native is None:
        lib()
        path = os.path.join(_HERE, "_binding" + importlib.machinery.EXTENSION_SUFFIXES[0])
        if not os.path.exists(path):
            raise OSError("%s not found: run `python -m paper_2305_11624_b200.build`" % path)
        spec = importlib.util.spec_from_file_location(__package__ + "._binding", path)
        module = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(module)
        _native = module
    return _native


def _desc(desc):
    """A descriptor given in another form that a `const convbn_desc *` takes (by reference, by pointer, an array's first, a
    structure derived from it, None), as a Desc at that address; anything else is a TypeError."""
    if desc is None:
        return None
    address = ctypes.cast(ctypes.POINTER(Desc).from_param(desc), ctypes.c_void_p).value
    if address is None:
        return None
    view = Desc.from_address(address)
    view.given = desc                    # (keeps what it points into)
    return view


def _ptr(t):
    """Address for a c_void_p parameter: a tensor's, an integer as it is, None for NULL."""
    if t is None or type(t) is int:
        return t
    try:                        # twenty of these per call: isinstance first took 20 ns more for each tensor
        return t.data_ptr()
    except AttributeError:
        if isinstance(t, int):
            return t
        raise


def _vp(t) -> ctypes.c_void_p:
    """The same as an object, for entry points without declared argument types."""
    return ctypes.c_void_p(_ptr(t))


def _stream(stream):
    if stream is None:
        import torch
        return torch._C._cuda_getCurrentRawStream(torch._C._cuda_getDevice())
    if isinstance(stream, int):
        return stream
    return stream.cuda_stream


def _nbytes(t) -> int:
    return 0 if t is None else t.nbytes


def _raise(status: int, where: str):
    if status != OK:
        raise ConvBNError(status, where)


def status_string(status: int) -> str:
    return lib().convbn_status_string(ctypes.c_int(status)).decode()


def convbn_last_kernel(phase: int) -> str:
    return lib().convbn_last_kernel(ctypes.c_int(phase)).decode()


def convbn_out_shape(desc: Desc):
    ho, wo = ctypes.c_int(0), ctypes.c_int(0)
    _raise(lib().convbn_out_shape(ctypes.byref(desc), ctypes.byref(ho), ctypes.byref(wo)),
           "convbn_out_shape")
    return ho.value, wo.value


def convbn_linear_desc(rows: int, in_features: int, out_features: int, dtype: int = BF16, eps: float = 1e-5) -> Desc:
    """Descriptor under which the convolution entry points compute a Linear-BN block on a [rows, in] matrix."""
    d = Desc()
    _raise(lib().convbn_linear_desc(ctypes.c_int(rows), ctypes.c_int(in_features), ctypes.c_int(out_features),
                                    ctypes.c_int(dtype), ctypes.c_double(eps), ctypes.byref(d)), "convbn_linear_desc")
    return d


def convbn_saved_bytes(desc: Desc, mode: int) -> int:
    return int(lib().convbn_saved_bytes(desc, mode))


def convbn_workspace_bytes(desc: Desc, phase: int) -> int:
    return int(lib().convbn_workspace_bytes(desc, phase))


def convbn_tune_fwd(desc, x, w, b, gamma, beta, run_mean, run_var, z, saved, workspace=None,
                    workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_tune_fwd(desc, x, w, b, gamma, beta, run_mean, run_var, z, saved,
                                                   workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_tune_fwd")


def convbn_tune_bwd_data(desc, dz, w, saved, dx, workspace=None,
                         workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_tune_bwd_data(desc, dz, w, saved, dx, workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_tune_bwd_data")


def convbn_tune_bwd_weight(desc, dz, x, w, b, run_mean, saved, dw, db, dgamma, dbeta,
                           workspace=None, workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_tune_bwd_weight(desc, dz, x, w, b, run_mean, saved, dw, db, dgamma, dbeta,
                                                          workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_tune_bwd_weight")


def convbn_tune_bwd(desc, dz, x, w, b, run_mean, saved, dx, dw, db, dgamma, dbeta, workspace=None,
                    workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_tune_bwd(desc, dz, x, w, b, run_mean, saved, dx, dw, db, dgamma, dbeta,
                                                   workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_tune_bwd")


def convbn_tune_bwd_begin(desc, dz, x, w, b, run_mean, saved, dx, dw, db, dgamma, dbeta, workspace=None,
                          workspace_bytes: Optional[int] = None, stream=None):
    """convbn_tune_bwd that returns with the parameter-gradient pass still running on the library's side lane."""
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_tune_bwd_begin(desc, dz, x, w, b, run_mean, saved, dx, dw, db, dgamma,
                                                         dbeta, workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_tune_bwd_begin")


def convbn_tune_bwd_join(stream=None) -> None:
    """Make `stream` wait for every parameter-gradient pass begun by this thread on the current device."""
    status = (_native or _calls()).convbn_tune_bwd_join(stream)
    if status:
        _raise(status, "convbn_tune_bwd_join")


def convbn_tune_fwd_glue(desc, x, w, b, gamma, beta, run_mean, run_var, z, saved, add, relu, workspace=None,
                         workspace_bytes: Optional[int] = None, stream=None):
    """convbn_tune_fwd with the addend and the ReLU of a residual network in its epilogue."""
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_tune_fwd_glue(desc, x, w, b, gamma, beta, run_mean, run_var, z, saved, add,
                                                        1 if relu else 0, workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_tune_fwd_glue")


def convbn_tune_bwd_glue(desc, dz, x, w, b, run_mean, saved, dx, dw, db, dgamma, dbeta, add, relu_mask, begin,
                         workspace=None, workspace_bytes: Optional[int] = None, stream=None):
    """convbn_tune_bwd (or, with `begin`, convbn_tune_bwd_begin) with dx += add and the mask x > 0 in its epilogue."""
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_tune_bwd_glue(desc, dz, x, w, b, run_mean, saved, dx, dw, db, dgamma,
                                                        dbeta, add, 1 if relu_mask else 0, 1 if begin else 0, workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_tune_bwd_glue")


def convbn_tconv_out_shape(desc):
    h, w = ctypes.c_int(0), ctypes.c_int(0)
    _raise(lib().convbn_tconv_out_shape(ctypes.byref(desc), ctypes.byref(h), ctypes.byref(w)), "convbn_tconv_out_shape")
    return h.value, w.value


def convbn_tconv_workspace_bytes(desc) -> int:
    f = lib().convbn_tconv_workspace_bytes
    f.restype = ctypes.c_size_t
    return int(f(ctypes.byref(desc)))


def convbn_tconv_tune_fwd(desc, x, w, b, gamma, beta, run_mean, run_var, z, saved, workspace=None,
                          workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_tconv_tune_fwd(desc, x, w, b, gamma, beta, run_mean, run_var, z, saved,
                                                         workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_tconv_tune_fwd")


def convbn_tconv_tune_bwd(desc, dz, x, w, b, run_mean, saved, dx, dw, db, dgamma, dbeta, workspace=None,
                          workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_tconv_tune_bwd(desc, dz, x, w, b, run_mean, saved, dx, dw, db, dgamma,
                                                         dbeta, workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_tconv_tune_bwd")


def convbn_tune_bwd_weight_noalloc(desc, dz, x, w, b, run_mean, saved, dw, db, dgamma, dbeta,
                                   stream=None):
    """Same results as convbn_tune_bwd_weight for callers that must not allocate device memory:
    no workspace argument, the library's built-in 16 MiB scratch array is used instead.  Raises
    ConvBNError(ECAPACITY) when the layer needs more scratch than that.  Calls sharing a device
    must not overlap on it."""
    _raise(lib().convbn_tune_bwd_weight_noalloc(desc, _ptr(dz), _ptr(x), _ptr(w),
                                                _ptr(b), _ptr(run_mean), _ptr(saved), _ptr(dw),
                                                _ptr(db), _ptr(dgamma), _ptr(dbeta), _stream(stream)),
           "convbn_tune_bwd_weight_noalloc")


def convbn_eval_fwd(desc, x, w, b, gamma, beta, run_mean, run_var, z, y_saved, workspace=None,
                    workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_eval_fwd(desc, x, w, b, gamma, beta, run_mean, run_var, z, y_saved,
                                                   workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_eval_fwd")


def convbn_eval_bwd(desc, dz, x, y_saved, w, gamma, run_mean, run_var, dx, dw, db, dgamma, dbeta,
                    workspace=None, workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_eval_bwd(desc, dz, x, y_saved, w, gamma, run_mean, run_var, dx, dw, db,
                                                   dgamma, dbeta, workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_eval_bwd")


def convbn_deploy_prepare(desc, w, b, gamma, beta, run_mean, run_var, w_fused, b_fused, stream=None):
    _raise(lib().convbn_deploy_prepare(desc, _ptr(w), _ptr(b), _ptr(gamma), _ptr(beta),
                                       _ptr(run_mean), _ptr(run_var), _ptr(w_fused), _ptr(b_fused),
                                       _stream(stream)),
           "convbn_deploy_prepare")


def convbn_deploy_fwd(desc, x, w_fused, b_fused, z, workspace=None,
                      workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_deploy_fwd(desc, x, w_fused, b_fused, z, workspace, workspace_bytes, stream)
    if status:
        _raise(status, "convbn_deploy_fwd")


def convbn_deploy_bwd(desc, dz, x, w_fused, dx, dw_fused, db_fused, workspace=None,
                      workspace_bytes: Optional[int] = None, stream=None):
    if type(desc) is not Desc:
        desc = _desc(desc)
    status = (_native or _calls()).convbn_deploy_bwd(desc, dz, x, w_fused, dx, dw_fused, db_fused, workspace,
                                                     workspace_bytes, stream)
    if status:
        _raise(status, "convbn_deploy_bwd")


def _dtype_of(t) -> int:
    import torch
    return {torch.bfloat16: BF16, torch.float16: F16}.get(t.dtype, F32)


def convbn_relu(a, out, stream=None):
    _raise(lib().convbn_relu(_dtype_of(a), _ptr(a), _ptr(out), a.numel(), _stream(stream)),
           "convbn_relu")


def convbn_add_relu(a, b, out, stream=None):
    _raise(lib().convbn_add_relu(_dtype_of(a), _ptr(a), _ptr(b), _ptr(out), a.numel(),
                                 _stream(stream)), "convbn_add_relu")


def convbn_relu_bwd(a, y, out, stream=None):
    _raise(lib().convbn_relu_bwd(_dtype_of(a), _ptr(a), _ptr(y), _ptr(out), a.numel(),
                                 _stream(stream)), "convbn_relu_bwd")


def convbn_add(a, b, out, stream=None):
    _raise(lib().convbn_add(_dtype_of(a), _ptr(a), _ptr(b), _ptr(out), a.numel(),
                            _stream(stream)), "convbn_add")


def convbn_check(stream=None) -> None:
    _raise(lib().convbn_check(_stream(stream)), "convbn_check")


def convbn_selftest_wait_timeout(stream=None) -> None:
    """Queue the failure-path self-test: the next convbn_check() raises ConvBNError(ETIMEOUT)."""
    _raise(lib().convbn_selftest_wait_timeout(ctypes.c_void_p(_stream(stream))), "convbn_selftest_wait_timeout")


def convbn_host_step_arena_bytes(desc: Desc) -> int:
    return int(lib().convbn_host_step_arena_bytes(ctypes.byref(desc)))


def convbn_tune_step_host(desc, x, dz, w, b, gamma, beta, run_mean, run_var, z, dx, dw, db, dgamma,
                          dbeta, device_arena, arena_bytes: Optional[int] = None, stream=None):
    """All tensors but ``device_arena`` are HOST tensors (page-locked for asynchronous copies)."""
    ab = _nbytes(device_arena) if arena_bytes is None else arena_bytes
    _raise(lib().convbn_tune_step_host(ctypes.byref(desc), _vp(x), _vp(dz), _vp(w), _vp(b),
                                       _vp(gamma), _vp(beta), _vp(run_mean), _vp(run_var),
                                       _vp(z), _vp(dx), _vp(dw), _vp(db), _vp(dgamma),
                                       _vp(dbeta), _vp(device_arena), ctypes.c_size_t(ab),
                                       ctypes.c_void_p(_stream(stream))),
           "convbn_tune_step_host")


def convbn_tune_step_host_begin(desc, x, dz, w, b, gamma, beta, run_mean, run_var, z, dx, dw, db, dgamma,
                          dbeta, device_arena, arena_bytes: Optional[int] = None, stream=None):
    """All tensors but ``device_arena`` are HOST tensors (page-locked for asynchronous copies)."""
    ab = _nbytes(device_arena) if arena_bytes is None else arena_bytes
    _raise(lib().convbn_tune_step_host_begin(ctypes.byref(desc), _vp(x), _vp(dz), _vp(w), _vp(b),
                                       _vp(gamma), _vp(beta), _vp(run_mean), _vp(run_var),
                                       _vp(z), _vp(dx), _vp(dw), _vp(db), _vp(dgamma),
                                       _vp(dbeta), _vp(device_arena), ctypes.c_size_t(ab),
                                       ctypes.c_void_p(_stream(stream))),
           "convbn_tune_step_host_begin")


def convbn_tune_step_host_join(stream=None) -> None:
    """Make `stream` wait for the downloads of every convbn_tune_step_host_begin call of this thread on this device."""
    _raise(lib().convbn_tune_step_host_join(ctypes.c_void_p(_stream(stream))), "convbn_tune_step_host_join")


def convbn_profile_begin() -> None:
    _raise(lib().convbn_profile_begin(), "convbn_profile_begin")


def convbn_profile_end() -> dict:
    """{kernel family: (launches, total milliseconds)} since convbn_profile_begin()."""
    buf = ctypes.create_string_buffer(1 << 16)
    _raise(lib().convbn_profile_end(buf, ctypes.c_size_t(len(buf))), "convbn_profile_end")
    out = {}
    for line in buf.value.decode().splitlines():
        name, count, ms = line.split()
        out[name] = (int(count), float(ms))
    return out
