"""Builds tests/native/parts.cu against the library and loads it."""
import ctypes
import os
import subprocess

from paper_2305_13380_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def load(tmp_dir):
    build.build()
    so = os.path.join(str(tmp_dir), "parts.so")
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", os.path.join(HERE, "native", "parts.cu"), "-o", so,
           "-L" + build.OUT_DIR, "-lsph", "-Xlinker", "-rpath=" + build.OUT_DIR]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(so)
    L.part_scan_words.restype = ctypes.c_long
    L.part_scan_words.argtypes = [ctypes.c_long]
    return L


def ptr(t):
    return ctypes.c_void_p(0 if t is None else t.data_ptr())


def stream():
    import torch
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
