"""Builds tests/native/parts.cu against the library and loads it; builds variants of
the library."""
import ctypes
import os
import subprocess

from paper_2305_13380_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def _run(cmd):
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def load(tmp_dir, lib=None):
    """parts.so, linked with lib (default: the library)."""
    build.build()
    lib = lib or build.LIB
    so = os.path.join(str(tmp_dir), "parts.so")
    _run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", os.path.join(HERE, "native", "parts.cu"), "-o", so, lib,
          "-Xlinker", "-rpath=" + os.path.dirname(lib)])
    L = ctypes.CDLL(so)
    L.part_scan_words.restype = ctypes.c_long
    L.part_scan_words.argtypes = [ctypes.c_long]
    return L


def variant(tmp_dir, defines, files):
    """The library with the given files of csrc/ compiled with -D defines; its path."""
    build.build()
    obj = os.path.join(build.OUT_DIR, "obj")
    objs = {f: os.path.join(obj, os.path.basename(f) + ".o") for f in build._sources()}
    if not all(os.path.exists(o) for o in objs.values()):
        build.build(force=True)
    for src in objs:
        if os.path.basename(src) in files:
            objs[src] = os.path.join(str(tmp_dir), os.path.basename(src) + ".o")
            _run([build.nvcc(), *build.ARCH, *build.FLAGS, *("-D" + d for d in defines), "-c", src, "-o", objs[src]])
    lib = os.path.join(str(tmp_dir), "libsph.so")
    _run([build.nvcc(), *build.ARCH, "-shared", "-Xlinker", "-soname=" + lib, "-o", lib, *objs.values()])
    return lib


def ptr(t):
    return ctypes.c_void_p(0 if t is None else t.data_ptr())


def stream():
    import torch
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
