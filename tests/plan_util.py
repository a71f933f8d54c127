"""Builds and loads plan_probe.cpp (see there)."""
import ctypes
import os
import subprocess

import numpy as np

import paper_2507_15230_gb300 as gale
from paper_2507_15230_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
_lib = None


def probe():
    global _lib
    if _lib is None:
        gale.load_library()
        src = os.path.join(HERE, "plan_probe.cpp")
        out = os.path.join(_build.BUILD, "libplanprobe.so")
        if not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(src), os.path.getmtime(_build.LIB)):
            tmp = f"{out}.tmp{os.getpid()}"
            subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", _build.CSRC, "-I",
                            os.path.join(_build.CUDA_HOME, "include"), src, "-o", tmp, _build.LIB,
                            f"-Wl,-rpath,{_build.BUILD}"], check=True, capture_output=True)
            os.replace(tmp, out)
        _lib = ctypes.CDLL(out)
    return _lib


FIELDS = ("nv_own", "n_own", "n_vt", "max_deg", "class", "total", "mode")


def item_plans(ctx, threads):
    """Every work item's planning figures (a host-only context)."""
    lib = probe()
    n = lib.probe_items(ctx._h)
    out = np.zeros((n, len(FIELDS)), np.int64)
    lib.probe_plans(ctx._h, threads, out.ctypes.data_as(ctypes.c_void_p))
    return {f: out[:, i] for i, f in enumerate(FIELDS)}


def merged_total(ctx, ids, threads):
    """Shared memory of one plan over the listed items, as a size bin's."""
    ids = np.ascontiguousarray(ids, np.int32)
    f = probe().probe_merged
    f.restype = ctypes.c_int64
    return int(f(ctx._h, ids.ctypes.data_as(ctypes.c_void_p), len(ids), threads))
