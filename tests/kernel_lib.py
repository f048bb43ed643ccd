"""ctypes access to internal kernels (tests/kernel_entry.cu), linked against
the built library."""
import ctypes
import functools
import os
import subprocess
import tempfile

from gpu_util import require_lib

HERE = os.path.dirname(os.path.abspath(__file__))


@functools.lru_cache(None)
def kernels():
    M = require_lib()
    M.lib()
    from paper_2509_11424_gb300 import build as b
    out = os.path.join(tempfile.mkdtemp(), 'kernel_entry.so')
    cmd = [b.nvcc()] + b.ARCH + b.FLAGS + ['-shared', os.path.join(HERE, 'kernel_entry.cu'), '-o', out, b.LIB,
                                           '-Xlinker', '-rpath=' + os.path.dirname(b.LIB)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(out)
    P, i64, i32, f64 = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, ctypes.c_double
    L.k_dot.argtypes = [i32, P, P, i64, i32, P]
    L.k_multi_dot.argtypes = [i32, P, i64, i32, P, i64, i32, P]
    L.k_basis.argtypes = [P, i32, P, i64, i32, P, f64, P]
    L.k_dot_qr.argtypes = [i32, P, P, i64, i32, P, P]
    L.k_multi_axpy.argtypes = [i32, P, i64, i32, P, i64, i32, P, f64, P]
    L.k_wgrad_f32.argtypes = [P, P, P, P, i32, i32, i32, P]
    L.k_site_dots.argtypes = [P, P, ctypes.c_float, i32, i32, P, P]
    L.k_alloc_failures.argtypes = [i32, i64]
    L.k_alloc_failures.restype = None
    return L


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())
