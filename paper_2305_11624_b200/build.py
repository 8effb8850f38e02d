"""Compile ``csrc/*.cu`` for sm_100a into ``paper_2305_11624_b200/libconvbn.so`` with nvcc.

``csrc/binding.cpp``, the Python entry to the calls of a training step, becomes ``_binding`` with this interpreter's extension
suffix beside it (g++); without Python's C headers the library is built alone, for use from C.
Sources are compiled in parallel to objects under ``_build/`` and linked with the static CUDA
runtime; the driver API (tensor-map encoding) is resolved at run time through the runtime's
entry-point query, so the library loads on a machine without a GPU driver.
"""
import importlib.machinery
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
BUILD_DIR = os.path.join(_HERE, "_build")
LIBRARY = os.path.join(_HERE, "libconvbn.so")
BINDING = os.path.join(_HERE, "_binding" + importlib.machinery.EXTENSION_SUFFIXES[0])    # (an interpreter loads its own only)
CXX = os.environ.get("CXX", "g++")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
ARCH = ["-gencode", "arch=compute_100a,code=sm_100a"]
CFLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xptxas", "-v",
          "--expt-relaxed-constexpr", "-Wno-deprecated-gpu-targets"]


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps_mtime():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(_HERE, "..", "include", "convbn.h"))
    return max(os.path.getmtime(f) for f in files)


def _compile(src: str, verbose: bool) -> str:
    obj = os.path.join(BUILD_DIR, os.path.basename(src)[:-3] + ".o")
    cmd = [NVCC] + ARCH + CFLAGS + ["-c", src, "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    log = os.path.join(BUILD_DIR, os.path.basename(src)[:-3] + ".ptxas.log")
    with open(log, "w") as f:
        f.write(r.stderr)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("nvcc failed on %s" % src)
    if verbose:
        sys.stderr.write(r.stderr)
    return obj


def _build_binding():
    tmp = BINDING + ".tmp.%d" % os.getpid()
    cmd = [CXX, "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-Wall",
           "-I" + sysconfig.get_paths()["include"], os.path.join(CSRC, "binding.cpp"), "-o", tmp,
           "-L" + _HERE, "-l:libconvbn.so", "-Wl,-rpath,$ORIGIN"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, BINDING)


def _headers() -> bool:
    return os.path.exists(os.path.join(sysconfig.get_paths()["include"], "Python.h"))


def build(force: bool = False, verbose: bool = False) -> str:
    """Build the library and the binding if missing or older than any source; return the library's path."""
    fresh = lambda f: not force and os.path.exists(f) and os.path.getmtime(f) >= _deps_mtime()
    if not fresh(LIBRARY):
        _build_library(verbose)
    if not fresh(BINDING) and _headers():
        _build_binding()
    elif not os.path.exists(BINDING):
        print("no Python.h in %s: %s is not built" % (sysconfig.get_paths()["include"], os.path.basename(BINDING)), file=sys.stderr)
    return LIBRARY


def _build_library(verbose: bool):
    os.makedirs(BUILD_DIR, exist_ok=True)
    with ThreadPoolExecutor(max_workers=8) as ex:
        objs = list(ex.map(lambda s: _compile(s, verbose), sources()))
    tmp = LIBRARY + ".tmp.%d" % os.getpid()
    cmd = [NVCC] + ARCH + ["-shared", "-cudart", "static", "-o", tmp] + objs
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIBRARY)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
