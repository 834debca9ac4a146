"""Kernels that need more shared memory than the default, on every device of a
process: the launchers linked against a stand-in for the CUDA runtime (no GPU)."""
import os
import subprocess

from paper_2305_13380_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_opt_in_on_every_device(tmp_path):
    build.build()
    exe = tmp_path / "two_devices"
    objs = [os.path.join(build.OUT_DIR, "obj", f + ".cu.o") for f in ("radix", "density", "force", "sym", "tree_loops")]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    srcs = [os.path.join(HERE, "native", f) for f in ("two_devices.cu", "fake_cuda.cpp")]
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-cudart", "none", *srcs, *objs, "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
    lines = [line.split() for line in r.stdout.splitlines()]
    assert len(lines) == 7 * (3 + 8 * 3 + 1)
    assert [line for line in lines if line[2] != "0"] == []
