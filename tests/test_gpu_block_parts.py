"""Blocks of small uniform grids are shared between several CTAs: a box alone
(few blocks) gives bit for bit what it gives within a pool (many blocks, one CTA
each)."""
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


@pytest.mark.parametrize("kernel", [0, 1, 2])
@pytest.mark.parametrize("lanes", [0, 2, 4])
@pytest.mark.parametrize("side", [8, 13, 16])
def test_alone_and_in_a_pool(side, lanes, kernel):
    from paper_2305_13380_gb300 import sph
    from paper_2305_13380_gb300.pool import Pool
    box = inputs.lattice(side, seed=side, sigma_v=0.05)
    filler = inputs.lattice(16, seed=1, sigma_v=0.05)
    params = sph.sph_default_params(kernel=kernel, lanes_per_target=lanes)
    out = []
    for sims in ([box], [box] + [filler] * 40):
        P = Pool(sims, params=params)
        P.start()
        P.step()
        P.stream.synchronize()
        assert P.status() == 0
        s = P.sim_slice(0)
        out.append({k: v[s].copy() for k, v in P.host().items()})
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k
