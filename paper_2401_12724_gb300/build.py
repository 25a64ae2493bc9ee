"""Builds libbysdf.so in-tree with nvcc for sm_103a (no CMake, no torch), and
the call path of api.py against torch's headers (one host translation unit)."""
from __future__ import annotations

import os
import subprocess
import sys
import threading
import warnings
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD_DIR = os.path.join(PKG, "_build")
LIB_PATH = os.path.join(PKG, "libbysdf.so")
# The index-checking build (-DBYSDF_DEBUG_BOUNDS): every checked index that
# falls out of range sets bit 2 of the launch's error word and is clamped;
# a separate library, built on demand by the tests that use it.
BOUNDS_BUILD_DIR = os.path.join(BUILD_DIR, "bounds")
BOUNDS_LIB_PATH = os.path.join(PKG, "libbysdf_bounds.so")
# The native call path of api.py (csrc/bysdf_torch.cpp); both libraries use it.
BINDING_SRC = os.path.join(CSRC, "bysdf_torch.cpp")
BINDING_PATH = os.path.join(PKG, "_bysdf_torch.so")
SOURCES = ["bysdf_api.cu", "bysdf_fwd.cu", "bysdf_fwd_eval.cu", "bysdf_fwd_sample.cu",
           "bysdf_fwd_pdf.cu", "bysdf_fwd_fused.cu", "bysdf_fwd_stoch.cu", "bysdf_bwd.cu",
           "bysdf_trace.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
NVCC_FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
              "--expt-relaxed-constexpr", "-I", INCLUDE, "-I", CSRC]
# The forward, backward and ray-yarn kernels divide and take square roots
# with the hardware's approximate instructions (a few ulp: far inside the
# 1e-4 tolerance of values and gradients, and inside the margins of the
# tracer's conservative culling bounds), and flush single-precision
# denormals (below 2^-126) to zero, which spares those instructions their
# denormal scaling.
FAST_FLAGS = {s: ["-prec-div=false", "-prec-sqrt=false", "-ftz=true"]
              for s in ("bysdf_fwd_eval.cu", "bysdf_fwd_sample.cu", "bysdf_fwd_pdf.cu",
                        "bysdf_fwd_fused.cu", "bysdf_fwd_stoch.cu", "bysdf_fwd.cu",
                        "bysdf_bwd.cu", "bysdf_trace.cu")}
_lock = threading.Lock()


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _deps():
    hdrs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))]
    return [os.path.join(CSRC, s) for s in SOURCES] + hdrs + [os.path.join(INCLUDE, "bysdf.h")]


def _stale(lib: str, deps=None) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(p) > t for p in deps or _deps())


def _build_binding(force: bool) -> None:
    """Builds the native call path of api.py.  The library does not need it (its
    calls then go through ctypes), so a failure is a warning."""
    try:
        if force or _stale(BINDING_PATH, [BINDING_SRC, os.path.join(INCLUDE, "bysdf.h")]) \
                or not binding_matches():
            _compile_binding()
    except Exception as e:  # no compiler, no headers, no torch
        warnings.warn(f"the native call path was not built, calls go through ctypes: {e}")


def _abi() -> str:
    """What the binding's object layouts and symbols follow beside its source."""
    import sysconfig

    import torch

    return " ".join((torch.__version__, str(sysconfig.get_config_var("SOABI")),
                     f"cxx11={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"))


def binding_matches() -> bool:
    """The built binding is this Python's and this torch's (its stamp says so)."""
    try:
        with open(BINDING_PATH + ".abi") as f:
            return f.read() == _abi()
    except OSError:
        return False


def _compile_binding() -> None:
    import sysconfig

    import torch
    from torch.utils import cpp_extension as X

    inc = [*X.include_paths(), sysconfig.get_paths()["include"],
           os.path.join(os.path.dirname(os.path.dirname(_nvcc())), "include")]
    tmp = BINDING_PATH + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-w",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           *(f"-I{p}" for p in [INCLUDE, *inc]), BINDING_SRC, "-o", tmp]
    for d in X.library_paths():
        cmd += [f"-L{d}", f"-Wl,-rpath,{d}"]
    cmd += ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for bysdf_torch.cpp:\n{r.stderr}")
    with open(tmp + ".abi", "w") as f:
        f.write(_abi())
    # the binary goes first: one without its stamp is built again, never loaded
    if os.path.exists(BINDING_PATH + ".abi"):
        os.remove(BINDING_PATH + ".abi")
    os.replace(tmp, BINDING_PATH)
    os.replace(tmp + ".abi", BINDING_PATH + ".abi")


def build(force: bool = False, verbose: bool = False, ptxas_info: bool = False,
          bounds: bool = False) -> str:
    """Compile the CUDA sources in parallel and link libbysdf.so (static
    cudart), or with bounds the index-checking libbysdf_bounds.so."""
    lib = BOUNDS_LIB_PATH if bounds else LIB_PATH
    bdir = BOUNDS_BUILD_DIR if bounds else BUILD_DIR
    defs = ["-DBYSDF_DEBUG_BOUNDS"] if bounds else []
    with _lock:
        if not force and not _stale(lib):
            _build_binding(False)
            return lib
        os.makedirs(bdir, exist_ok=True)
        nvcc = _nvcc()
        extra = ["-Xptxas", "-v"] if ptxas_info else []

        def compile_one(src):
            obj = os.path.join(bdir, src.replace(".cu", ".o"))
            cmd = [nvcc, *ARCH, *NVCC_FLAGS, *defs, *FAST_FLAGS.get(src, []), *extra, "-c",
                   os.path.join(CSRC, src), "-o", obj]
            r = subprocess.run(cmd, capture_output=True, text=True)
            if r.returncode != 0:
                raise RuntimeError(f"nvcc failed for {src}:\n{r.stderr}")
            if verbose or ptxas_info:
                sys.stderr.write(r.stderr)
            return obj

        with ThreadPoolExecutor(max_workers=len(SOURCES) + 1) as ex:
            binding = ex.submit(_build_binding, force and not bounds)
            objs = list(ex.map(compile_one, SOURCES))
            binding.result()
        tmp = lib + f".tmp{os.getpid()}"
        cmd = [nvcc, *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stderr}")
        os.replace(tmp, lib)
        return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_info="--ptxas" in sys.argv,
                bounds="--bounds" in sys.argv))
