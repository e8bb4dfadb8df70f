"""Builds and binds the host-only check of the tree builder (tests/_build/libwalk_grid_host.so)."""
import ctypes as C
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(os.path.dirname(HERE)), "paper_2203_14354_gb300", "csrc")
OUT = os.path.join(os.path.dirname(HERE), "_build")


def build():
    os.makedirs(OUT, exist_ok=True)
    src = [os.path.join(HERE, "walk_grid_host.cpp"), os.path.join(CSRC, "bvh_build.cpp")]
    lib = os.path.join(OUT, "libwalk_grid_host.so")
    newest = max(os.path.getmtime(f) for f in src + [os.path.join(CSRC, "lxo_internal.h")])
    if not os.path.exists(lib) or os.path.getmtime(lib) < newest:
        tmp = lib + f".tmp{os.getpid()}"
        cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
        subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-pthread", f"-I{cuda}/include", *src, "-o",
                        tmp], check=True)
        os.replace(tmp, lib)
    return lib


def walk_grid_check(det, points, ids, leaf_size=0, n_threads=0):
    """(status, points lost, points seen); see walk_grid_host.cpp."""
    L = C.CDLL(build())
    tri = np.ascontiguousarray(det.verts[det.tris].reshape(-1, 9), np.float32)
    pts, ids = np.ascontiguousarray(points, np.float32), np.ascontiguousarray(ids, np.uint32)
    lost, seen = C.c_uint32(), C.c_uint32()
    status = L.walk_grid_check(C.c_void_p(tri.ctypes.data), C.c_uint32(len(tri)), C.c_uint32(leaf_size),
                               C.c_uint32(n_threads), C.c_void_p(pts.ctypes.data), C.c_void_p(ids.ctypes.data),
                               C.c_uint32(len(ids)), C.byref(lost), C.byref(seen))
    return status, lost.value, seen.value
