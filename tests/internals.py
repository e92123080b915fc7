"""Builds and loads tests/internals.cu: the library with a few more entry points."""
import ctypes as C
import os
import subprocess
import tempfile

from paper_2605_22269_b200 import binding as B
from paper_2605_22269_b200 import build as BUILD

HERE = os.path.dirname(os.path.abspath(__file__))
_LIB = None


def build():
    """Path of the built library; in the tree where that can be written."""
    src, (main, deps) = os.path.join(HERE, "internals.cu"), BUILD.TARGETS["libmukv.so"]
    out = os.path.join(HERE, "_build", "libinternals.so")
    if BUILD._stale(out, [src, main] + deps):
        try:
            os.makedirs(os.path.dirname(out), exist_ok=True)
            writable = os.access(os.path.dirname(out), os.W_OK)
        except OSError:
            writable = False
        if not writable:
            out = os.path.join(tempfile.mkdtemp(prefix="internals"), "libinternals.so")
        r = subprocess.run([os.environ.get("NVCC", "nvcc")] + BUILD.NVCC_FLAGS + ["-o", out, src], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    return out


def load():
    global _LIB
    if _LIB is None:
        out = build()
        _LIB = B.load_library(out)
        _LIB.internals_wait_limit.restype = None
        _LIB.internals_wait_limit.argtypes = [C.c_void_p, C.c_ulonglong]
        _LIB.internals_scan_shape.restype = _LIB.internals_scores.restype = None
        _LIB.internals_scan_shape.argtypes = [C.c_longlong, C.c_int, C.c_int, C.POINTER(C.c_int)]
        _LIB.internals_scan_by_rows.restype = C.c_int
        _LIB.internals_scan_by_rows.argtypes = [C.c_longlong, C.c_int, C.c_int]
        _LIB.internals_scores.argtypes = [C.c_void_p, C.POINTER(C.c_longlong)]
        _LIB.internals_on_tensor_cores.restype = C.c_int
        _LIB.internals_on_tensor_cores.argtypes = [C.POINTER(B.MukvConfig)]
        _LIB.internals_score_noalloc.restype = C.c_int32
        _LIB.internals_score_noalloc.argtypes = _LIB.mukv_score_frames_noalloc.argtypes + [C.c_ulonglong]
    return _LIB


def scan_shape(rows, nq, n_sms=148):
    """(question tiles of a warp, question groups, row tiles of a block)"""
    out = (C.c_int * 3)()
    load().internals_scan_shape(rows, nq, n_sms, out)
    return tuple(out)
