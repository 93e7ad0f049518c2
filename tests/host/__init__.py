"""The library's host code on a CUDA runtime that a test controls (fake_cuda.cc): no GPU."""
import ctypes as ct
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(os.path.dirname(HERE)), "paper_2007_12266_gb300", "csrc")


def cuda_include():
    from paper_2007_12266_gb300 import _build
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")


def build(folder):
    """Compile and load it; the library's entry points have their argument types. (-Bsymbolic:
    its own runtime, not one that the process has loaded already.)"""
    from paper_2007_12266_gb300 import _lib
    out = os.path.join(str(folder), "libhost.so")
    src = [os.path.join(CSRC, f) for f in ("api.cu", "batch_api.cu", "server.cu")] + [os.path.join(HERE, "fake_cuda.cc")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-w", "-I", cuda_include(), "-x", "c++", *src, "-o", out],
                   check=True)
    lib = ct.CDLL(out)
    for name, (res, args) in _lib.SIGNATURES.items():
        fn = getattr(lib, name, None)
        if fn is not None:
            fn.restype, fn.argtypes = res, args
    for name, res, args in (("fake_fail", None, [ct.c_int, ct.c_int]), ("fake_memory_limit", None, [ct.c_size_t]),
                            ("fake_reset_peak", None, []), ("fake_peak", ct.c_size_t, []), ("fake_live", ct.c_size_t, []),
                            ("fake_launches", ct.c_longlong, []), ("fake_refused", ct.c_longlong, []),
                            ("fake_uploads", ct.c_longlong, [])):
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = res, args
    return lib
