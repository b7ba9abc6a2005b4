"""The library's host code (gm_api.cu) on the CPU: linked with a CUDA runtime on
host memory (host_cuda.cpp) instead of the CUDA runtime and the kernels."""
import ctypes as C
import functools
import os
import subprocess
import tempfile

import paper_1101_1245_gb300 as g
from paper_1101_1245_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))


@functools.lru_cache(None)
def library() -> C.CDLL:
    with tempfile.TemporaryDirectory() as d:
        out = os.path.join(d, "host_cuda.so")
        subprocess.run([b.nvcc(), "-std=c++17", "-O1", *b.ARCH, "-Xcompiler", "-fPIC", "-I", b.INCLUDE, "-I", b.CSRC,
                        "-x", "cu", "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", out,
                        os.path.join(b.CSRC, "gm_api.cu"), os.path.join(HERE, "host_cuda.cpp")], check=True)
        L = C.CDLL(out)
    for name, (res, args) in g.SIGNATURES.items():
        f = getattr(L, name)
        f.restype, f.argtypes = res, args
    for f in (L.host_cuda_calls, L.host_cuda_pending, L.host_cuda_launched, L.host_cuda_misfits):
        f.restype = C.c_long
    L.host_cuda_calls.argtypes = [C.c_char_p]
    L.host_cuda_fail.argtypes = [C.c_char_p, C.c_int]
    L.host_cuda_launched.argtypes = [C.c_void_p, C.c_long]
    return L
