"""The uniform grid's overflow kernels in the SPHENIX force and gradient pass, the
time-step limiter and the masked loops: cells whose sources are staged and listed
(lattices of side 11, 14, 16) and cells that are streamed (side 9), against the FP64
oracle."""
import numpy as np
import pytest

from paper_2305_13380_gb300 import inputs

import test_gpu_active as active
import test_gpu_sphenix as sphenix
import test_gpu_timebins as timebins
from gpu_common import GAMMA_K, as_f32, compare, coord_floor, expected_nc

pytestmark = pytest.mark.gpu

STAGING = 1216   # sources of a block's 64 cells that the blocks' kernels stage
LISTED = 640     # sources of a cell's 27 that the overflow force stages


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


def _lattice(side):
    """The lattice, checked to overflow the staging and to be listed or streamed."""
    p = inputs.lattice(side, seed=side, sigma_v=0.05)
    per = side ** 3 / expected_nc(p["h0"], float(p["L"])) ** 3
    assert side == 16 or 64 * per > 1.05 * STAGING
    assert (27 * per > 1.05 * LISTED) if side == 9 else (27 * per < 0.95 * LISTED)
    return p


@pytest.mark.parametrize("side", [9, 11, 14, 16])
def test_sphenix(orc, side):
    # the bounds of test_gpu_sphenix.py (its own inputs also take every branch of the
    # parameters' updates, which these small ones need not)
    p = _lattice(side)
    q, _, st, dt = sphenix._setup(orc, p, seed=side)
    g = sphenix._run_gpu(p, st, dt)
    X = orc.Sphenix()
    f64 = {k: v.astype(np.float64) for k, v in st.items()}
    od, av, og, of = orc.sphenix_evaluate(q, q["h0"], f64["alpha_v"], f64["alpha_c"], f64["div_v_prev"], f64["v_sig"],
                                          dt, X)
    vmax = float(np.sqrt(q["vx"] ** 2 + q["vy"] ** 2 + q["vz"] ** 2).max())
    compare(g, od, of, cell=g["_cell"], vmax=vmax)
    H = GAMMA_K * od["h"]
    du = np.maximum(np.abs(q["u"] - q["u"].min()), np.abs(q["u"] - q["u"].max()))
    lim = 1e-4 * np.sqrt(np.mean(og["lap_u"] ** 2)) + 5e-5 * np.abs(og["lap_u"]) + \
        2.0 * coord_floor(g["_cell"], od["h"]) * 12.0 * du / H ** 2
    assert (np.abs(g["lap_u"] - og["lap_u"]) / lim).max() <= 1.0
    e_vc = 1e-5 * og["v_c"] + np.sqrt(8e-5 * np.max(od["P"] / od["rho"]))
    lim = dt * (X.beta_c * H * lim / np.sqrt(q["u"]) + f64["alpha_c"] * e_vc / H) + \
        X.alpha_c_max * np.abs(g["alpha_v"] - av).max() / X.alpha_v_max + 2e-6
    assert (np.abs(g["alpha_c"] - og["alpha_c"]) / lim).max() <= 1.0
    assert np.abs(of["du_cond"]).max() > 1e-3 * np.abs(of["du_dt"]).max()


@pytest.mark.parametrize("share", [0.02, 0.3])
@pytest.mark.parametrize("side", [9, 11, 14, 16])
def test_masked(orc, side, share):
    p = _lattice(side)
    m = active._blob(p, share, seed=side)
    base, (g,) = active._run(p, [m])
    idx = np.where(m)[0]
    q = as_f32(p)
    od_all = orc.density(q, q["h0"])
    compare(g, {k: v[idx] for k, v in od_all.items()}, orc.force(q, od_all, targets=idx), idx=idx,
            cell=1.0 / expected_nc(p["h0"], 1.0), vmax=float(np.abs(q["vx"]).max() * 2))
    for k in ("ax", "ay", "az", "du_dt", "v_sig"):
        assert np.all(g[k][~m] == active.SENTINEL), k


@pytest.mark.parametrize("side", [9, 11, 14])
def test_limiter(orc, side):
    p = _lattice(side)
    rng = np.random.default_rng(side)
    h = np.asarray(p["h0"]).astype(np.float32)
    v = np.exp(rng.uniform(np.log(0.5), np.log(500.0), len(h))).astype(np.float32)
    g = timebins._gpu_bins(p, h, v)
    b0, edge, lo, hi = timebins._bounds(orc, p, h, v)
    assert np.all(g >= lo) and np.all(g <= hi)
    assert np.mean(g == orc.limit_time_bins(p, h, b0)) > 0.99
    assert np.sum(g > b0) > 50   # the limiter acted
