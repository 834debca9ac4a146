"""Look-back waits that run out: a tile then counts what lies before it itself.  A
variant of the library whose waits all run out (no published word is ever seen)
gives the same cells, nested grids, masks, reverse pairs and groups as the library,
bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

import native_parts
from paper_2305_13380_gb300 import build, inputs

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def variant(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    return native_parts.variant(tmp_path_factory.mktemp("expired"), ["SPH_POLL_LIMIT=-1"], ["radix.cu", "tree.cu"])


def _calls(lib, out):
    """Runs in a process of its own, on the library at `lib`."""
    import torch
    from paper_2305_13380_gb300 import sph
    sph.LIB = lib
    got = {}
    for n in (8193, 30011):
        p = inputs.clustered(n, n_spheres=4, seed=n)
        t = sph.to_device(p)
        part = sph.particles(t)
        ctx = sph.Context(sph.sph_default_params(box_size=float(p["L"])))
        cells = sph.sph_build_cells(ctx, t["x"], t["y"], t["z"], t["h0"])
        got[f"cells{n}"], got[f"perm{n}"] = sph.sph_cells_copy(ctx, cells)
        group = torch.empty(n, dtype=torch.int32, device="cuda")
        sph.sph_fof(ctx, t["x"], t["y"], t["z"], 0.2 * n ** (-1.0 / 3.0), group)
        got[f"group{n}"] = group.cpu().numpy()
        ctx = sph.Context(sph.sph_default_params(box_size=float(p["L"]), flags=sph.SPH_FLAG_TREE))
        on = torch.as_tensor((np.arange(n) % 3 == 0).astype(np.uint8), device="cuda")
        h, d, f = t["h0"], sph.alloc_density(n), sph.alloc_force(n)
        for k in range(4):
            cells = sph.sph_build_cells(ctx, t["x"], t["y"], t["z"], h)
            sph.sph_density(ctx, cells, part, h, sph.density_out(d))
            if not sph.sph_status(ctx) & sph.SPH_ST_REBUILD:
                break
            h = d["h"].clone()
        assert sph.sph_status(ctx) == 0
        sph.sph_force(ctx, cells, part, sph.density_out(d), sph.force_out(f))
        got.update({f"{k}{n}": v.cpu().numpy() for k, v in {**d, **f}.items()})
        h = d["h"].clone()
        cells = sph.sph_build_cells(ctx, t["x"], t["y"], t["z"], h)
        sph.sph_density_active(ctx, cells, part, h, on, sph.density_out(d))
        sph.sph_force_active(ctx, cells, part, sph.density_out(d), on, sph.force_out(f))
        assert sph.sph_status(ctx) == 0
        got.update({f"masked_{k}{n}": v.cpu().numpy() for k, v in {**d, **f}.items()})
    np.savez(out, **got)


def test_same_results(variant, tmp_path):
    got = []
    for name, lib in (("library", build.LIB), ("expired", variant)):
        out = str(tmp_path / (name + ".npz"))
        code = "import test_gpu_expired_waits as t; t._calls(%r, %r)" % (lib, out)
        env = dict(os.environ, PYTHONPATH=os.pathsep.join([HERE, os.path.dirname(HERE)]))
        r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr
        got.append(np.load(out))
    assert len(got[0].files) > 50
    for k in got[0].files:
        assert np.array_equal(got[0][k], got[1][k]), k


@pytest.mark.parametrize("n", [1, 4096, 4097, 100000])
def test_scan(variant, tmp_path, n):
    import test_gpu_scan
    v = np.random.default_rng(n).integers(0, 256, n)
    parts = native_parts.load(tmp_path, variant)
    for dtype in ("int32", "uint8"):
        assert np.array_equal(test_gpu_scan._scan(parts, v, dtype), np.concatenate([[0], np.cumsum(v)]))
