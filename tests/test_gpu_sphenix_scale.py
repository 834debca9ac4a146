"""SPHENIX conduction of gas at rest in units where the kernel gradients (H^-5) are
subnormal floats: du/dt goes as 1 / length, so lengths and masses scaled by powers of
two give the scaled result but for the rounding of the subnormal factors; and
pressures that are subnormal weight the conduction as others do."""
import numpy as np
import pytest

from paper_2305_13380_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


def _conduction(side, scale, tree, u_scale=1.0):
    """du/dt of the conduction alone (no velocities), alpha_c = 1, in a box of side scale."""
    import torch
    from paper_2305_13380_gb300 import sph
    p = dict(inputs.lattice(side, seed=side, sigma_v=0.0))
    n = side ** 3
    rng = np.random.default_rng(side)
    for k in "xyz":
        p[k] = np.asarray(p[k]) * scale
    p["h0"], p["m"], p["L"] = np.asarray(p["h0"]) * scale, np.full(n, scale ** 3 / n), scale
    p["u"] = rng.uniform(0.5, 1.5, n) * u_scale
    for k in ("vx", "vy", "vz"):
        p[k] = np.zeros(n)
    ctx = sph.Context(sph.sph_default_params(box_size=scale, flags=sph.SPH_FLAG_TREE if tree else 0))
    t = sph.to_device(p)
    part, d, f = sph.particles(t), sph.alloc_density(n), sph.alloc_force(n)
    h = t["h0"]
    for _ in range(6):
        cells = sph.sph_build_cells(ctx, t["x"], t["y"], t["z"], h)
        sph.sph_density(ctx, cells, part, h, sph.density_out(d))
        if not sph.sph_status(ctx) & sph.SPH_ST_REBUILD:
            break
        h = d["h"].clone()
    one = torch.ones(n, dtype=torch.float32, device="cuda")
    sph.sph_force_sphenix(ctx, cells, part, sph.density_out(d), one, one, sph.force_out(f))
    assert sph.sph_status(ctx) == 0
    return f["du_dt"].double().cpu().numpy(), d["h"].double().cpu().numpy()


# side 8: the blocks' kernel; 16: the overflow kernel too (cells just past the staging)
@pytest.mark.parametrize("tree", [False, True])
@pytest.mark.parametrize("side,power", [(8, 28), (16, 29)])
def test_subnormal_gradients(side, power, tree):
    ref, h1 = _conduction(side, 1.0, tree)
    scale = 2.0 ** power
    got, h = _conduction(side, scale, tree)
    assert np.array_equal(h, h1 * scale)
    H5 = (1.825742 * h.max()) ** -5
    assert H5 < 2.0 ** -126
    # a factor H^-5 is off by at most half a step of 2^-149, of its two in a pair's
    # visc; and so the sum, by that part of its terms' absolute sum, which is some
    # tens of the result's rms (some fifty terms of either sign)
    tol = 100 * 2 * 2.0 ** -150 / H5
    assert tol < 0.02
    rms = np.sqrt(np.mean(ref ** 2))
    assert np.abs(got * scale - ref).max() <= tol * rms


@pytest.mark.parametrize("tree", [False, True])
def test_subnormal_pressures(tree):
    # u of 1e-39: P and P_i + P_j subnormal, their quotient of one order; conduction
    # goes as u^1.5, below the smallest float here: only its finiteness is seen
    got, _ = _conduction(8, 1.0, tree, u_scale=1e-39)
    assert np.isfinite(got).all()
