"""Builds and loads tests/native/helper.cu (on a machine with a GPU only)."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np

from paper_2607_23115_gb300 import binding as B
from paper_2607_23115_gb300 import build as G

SRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native", "helper.cu")
OUT = os.path.join(G.BUILD, "libtesthelper.so")
_lib = None


def helper() -> ctypes.CDLL:
    global _lib
    if _lib is None:
        B.lib()
        if not os.path.exists(OUT) or os.path.getmtime(OUT) < max(
                os.path.getmtime(p) for p in (SRC, B.LIB_PATH)):
            os.makedirs(G.BUILD, exist_ok=True)
            tmp = "%s.tmp%d" % (OUT, os.getpid())
            subprocess.check_call([G.NVCC, *G.ARCH, "-O2", "-std=c++17", "-Xcompiler", "-fPIC",
                                   "-shared", "-I", G.INCLUDE, "-I", G.CSRC, "-o", tmp, SRC,
                                   B.LIB_PATH])
            os.replace(tmp, OUT)
        _lib = ctypes.CDLL(OUT)
    return _lib


def hold(smem: int, ns: int, stream) -> None:
    """A block that holds smem bytes of shared memory for ns, on every SM if two do not fit one."""
    f = helper().helper_hold
    f.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_void_p]
    rc = f(smem, ns, stream.cuda_stream)
    assert rc == 0, rc


class HitsOut(ctypes.Structure):
    _fields_ = [("status", ctypes.c_int64), ("hits", ctypes.c_int64), ("calls", ctypes.c_int64),
                ("mask0", ctypes.c_uint64), ("slots_ok", ctypes.c_uint64),
                ("uses_old", ctypes.c_uint64), ("uses_new", ctypes.c_uint64),
                ("ctl_left", ctypes.c_uint64)]


def all_hits(grid: int, nch: int, bar_count: int = 0, err: int = 0,
             wait_ns: int = 4_000_000_000) -> HitsOut:
    """A call of hits alone in an evicting cache (helper_all_hits)."""
    f = helper().helper_all_hits
    f.argtypes = [ctypes.c_uint32, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int,
                  ctypes.c_uint64, ctypes.c_void_p]
    out = HitsOut()
    rc = f(grid, nch, bar_count, err, wait_ns, ctypes.byref(out))
    assert rc == 0, rc
    return out


def hash_alone(buf, C: int, probe: bool, wait_ns: int):
    """(fingerprints, error recorded) of the hash kernel by itself (helper_hash)."""
    f = helper().helper_hash
    f.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_uint64, ctypes.c_int,
                  ctypes.c_uint64, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    n = buf.numel()
    fp = np.zeros(-(-n // C), dtype=np.uint64)
    err, lone = ctypes.c_int(), ctypes.c_int()
    rc = f(buf.data_ptr(), n, C, int(probe), wait_ns, fp.ctypes.data, ctypes.byref(err),
           ctypes.byref(lone))
    assert rc == 0 and lone.value == 1, (rc, lone.value)
    return fp, err.value
