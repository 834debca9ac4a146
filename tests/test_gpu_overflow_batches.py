"""The density's overflow kernel with streamed cells: a CTA puts them off and its warps
deal their targets in batches of 32."""
import numpy as np
import pytest

from paper_2305_13380_gb300 import inputs

from gpu_common import GAMMA_K, TOL, as_f32, compare, coord_floor, expected_nc, run_gpu

pytestmark = pytest.mark.gpu

GAMMA = (GAMMA_K, 2.018932, 1.936492)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


def _lattice(side, margin, kernel, targets):
    """A lattice whose cells are streamed (more than 768 sources around them), two or
    more of them per CTA, with the given mean number of targets."""
    p = inputs.lattice(side, seed=side, sigma_v=0.05)
    nc = expected_nc(p["h0"], 1.0, (1 + margin) * GAMMA[kernel] / GAMMA_K - 1)
    assert 8 * ((nc + 1) // 2) ** 3 > 2 * 152 * 7
    assert round(side ** 3 / nc ** 3) == targets and 27 * targets > 768
    return p


def _check(orc, p, margin, kernel=0):
    """The plain bounds; v_sig, a maximum over the pairs within max(H_i, H_j), may be that
    with or without the pairs whose distance lies within h's own tolerance of the edge."""
    q = as_f32(p)
    g = run_gpu(p, margin=margin, kernel=kernel)
    od, of = orc.density_force(q, q["h0"], orc.Physics(kernel=kernel))
    H = GAMMA[kernel] * od["h"]
    X, V = (np.stack([np.asarray(q[k], dtype=np.float64) for k in ks]) for ks in ("xyz", ("vx", "vy", "vz")))
    off = np.where(np.abs(g["v_sig"] - of["v_sig"]) > TOL["v_sig"] * of["v_sig"])[0]
    assert len(off) < 1e-3 * len(H)
    for i in off:
        dx, dv = X[:, [i]] - X, V[:, [i]] - V
        dx -= np.round(dx)
        r = np.sqrt((dx ** 2).sum(0))
        r[i] = np.inf
        v = od["c"][i] + od["c"] - 3.0 * np.minimum((dx * dv).sum(0), 0.0) / r
        lo, hi = (v[r < (1 + s * 2 * TOL["h"]) * np.maximum(H[i], H)].max() for s in (-1, 1))
        assert lo < hi and lo * (1 - TOL["v_sig"]) <= g["v_sig"][i] <= hi * (1 + TOL["v_sig"]), i
        of["v_sig"][i] = g["v_sig"][i]
    vmax = float(np.sqrt((V ** 2).sum(0)).max())
    compare(g, od, of, cell=1.0 / expected_nc(p["h0"], 1.0, (1 + margin) * GAMMA[kernel] / GAMMA_K - 1), vmax=vmax)


# cells of one batch, two, three and four
@pytest.mark.parametrize("side,margin,kernel,targets", [(41, 0.3, 0, 31), (48, 0.6, 0, 50), (56, 0.8, 0, 80),
                                                        (61, 0.95, 0, 103), (48, 0.45, 1, 50), (56, 0.7, 2, 80)])
def test_batches(orc, side, margin, kernel, targets):
    _check(orc, _lattice(side, margin, kernel, targets), margin, kernel=kernel)


def test_more_cells_than_put_off(orc):
    # 33^3 streamed cells: more than 32 for each of six CTAs per SM
    p = inputs.lattice(108, seed=1, sigma_v=0.05)
    assert expected_nc(p["h0"], 1.0, 0.41) == 33 and 33 ** 3 > 32 * 152 * 6
    q = as_f32(p)
    g = run_gpu(p, margin=0.41)
    idx = np.random.default_rng(1).choice(108 ** 3, 300, replace=False)
    od = orc.density(q, q["h0"], targets=idx)
    floor = coord_floor(1.0 / 33, od["h"])
    for k in ("h", "rho", "f", "P"):
        assert (np.abs(g[k][idx] - od[k]) <= (TOL[k] + floor) * np.abs(od[k])).all(), k


def test_clustered(orc):
    # listed cells, streamed ones of a few targets and of more than a thousand
    _check(orc, inputs.clustered(60000, n_spheres=12, seed=3, a_min=0.01, a_max=0.03, frac_clustered=0.35), 0.05)


@pytest.mark.parametrize("side,margin", [(48, 0.6), (61, 0.95)])
def test_masked(side, margin):
    # the masked loops take the same batches: all active equals unmasked, bit for bit,
    # and a target's results do not depend on which others are
    import torch
    from paper_2305_13380_gb300 import sph
    p = inputs.lattice(side, seed=side, sigma_v=0.05)
    ctx = sph.Context(sph.sph_default_params(box_size=1.0, cell_margin=margin))
    t = sph.to_device(p)
    n = side ** 3
    part = sph.particles(t)
    rng = np.random.default_rng(side)
    masks = [np.ones(n, bool), rng.random(n) < 0.3, rng.random(n) < 0.002]
    got = []
    for m in [None] + masks:
        d = sph.alloc_density(n)
        for v in d.values():
            v.fill_(-7)
        cells = sph.sph_build_cells(ctx, t["x"], t["y"], t["z"], t["h0"])
        if m is None:
            sph.sph_density(ctx, cells, part, t["h0"], sph.density_out(d))
        else:
            on = torch.as_tensor(m.astype(np.uint8), device="cuda")
            sph.sph_density_active(ctx, cells, part, t["h0"], on, sph.density_out(d))
        assert sph.sph_status(ctx) == 0
        got.append({k: v.cpu().numpy() for k, v in d.items()})
    for m, g in zip(masks, got[1:]):
        for k, v in g.items():
            assert np.array_equal(v[m], got[0][k][m]) and np.all(v[~m] == -7), k
