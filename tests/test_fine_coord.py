"""The fixed-point estimate of the nested grids' fine coordinate: wherever it
decides, it gives floor(1024 fl(fl(x n_c) / L)); and positions on sub-cell faces,
where the exact path decides, against the FP64 oracle."""
import math
import struct

import numpy as np
import pytest

from paper_2305_13380_gb300 import inputs


def _bits(v):
    return struct.unpack("<Q", struct.pack("<d", v))[0]


def _estimate(x, scale):
    """tree.cu's fine_coord_fast before the clamp; None: the exact path."""
    xb, cb = _bits(x), _bits(scale)
    ex, ec = xb >> 52, cb >> 52
    sh = 2108 - ex - ec
    if not (0 < ex < 2047 and 33 <= sh <= 63):
        return None
    one = 1 << 52
    P = ((((xb & (one - 1)) | one) << 11) * (((cb & (one - 1)) | one) << 11)) >> 64
    frac = (P >> (sh - 32)) & 0xffffffff
    if not ((frac - (1 << 14)) & 0xffffffff) < (1 << 32) - (1 << 15):
        return None
    return P >> sh


@pytest.mark.parametrize("L", [1.0, 0.7, 3.3e-9, 1.0e12, 142.25])
@pytest.mark.parametrize("n_c", [1, 3, 54, 127, 1000, 60000])
def test_estimate_matches_definition(L, n_c):
    rng = np.random.default_rng(n_c)
    faces = rng.integers(0, 1024 * n_c, 1000) * L / (1024.0 * n_c)
    x = np.concatenate([rng.random(4000) * L, faces, np.nextafter(faces, np.inf), np.nextafter(faces, -np.inf),
                        rng.random(500) * L * 2.0 ** -rng.integers(0, 60, 500), [-0.1 * L, 0.0, 5e-324]])
    scale = n_c * 1024.0 / L
    decided = 0
    for v in x.tolist():
        g = _estimate(v, scale)
        if g is not None:
            decided += 1
            assert g == math.floor(((v * n_c) / L) * 1024.0)
    assert decided > 3900


@pytest.mark.gpu
@pytest.mark.parametrize("L", [1.0, 0.7])
def test_positions_on_sub_cell_faces(orc, L):
    import torch
    from gpu_common import as_f32, compare, run_gpu
    from paper_2305_13380_gb300 import build
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    build.build()
    p = dict(inputs.clustered(4000, n_spheres=3, seed=5))
    rng = np.random.default_rng(3)
    for k in "xyz":
        # on the sub-cell faces of a 16^3 top grid (and so of its divisors), or
        # an ulp beside them
        q = np.round(np.asarray(p[k]) * 16384) % 16384 / 16384 * L
        s = rng.integers(-1, 2, len(q))
        q = np.where(s < 0, np.nextafter(q, -np.inf), np.where(s > 0, np.nextafter(q, np.inf), q))
        p[k] = np.where(q < 0, 0.0, q)
    pos = np.stack([p[k] for k in "xyz"], 1)
    keep = np.sort(np.unique(np.round(pos / L * 16384), axis=0, return_index=True)[1])  # no two on one spot
    p = {k: (np.asarray(v)[keep] if np.ndim(v) else v) for k, v in p.items()}
    p["L"], p["h0"] = L, p["h0"] * L
    q = as_f32(p)
    g = run_gpu(p, tree=True, n_leaf=8)
    od, of = orc.density_force(q, q["h0"])
    compare(g, od, of)
