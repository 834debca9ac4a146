"""The masked nested force on a million particles, whose windows hold four rounds: every
particle active gives the unmasked results bit for bit, and a few active ones theirs,
up to the order of the sums, with nothing written elsewhere."""
import numpy as np
import pytest

from paper_2305_13380_gb300 import inputs

import test_gpu_active as active

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


def test_million():
    n = 1000003  # a last window of three targets
    p = inputs.clustered(n, n_spheres=64, seed=4)
    few = np.random.default_rng(2).random(n) < 0.001
    few[-3:] = True
    base, (every, some) = active._run(p, [np.ones(n, bool), few], grid="nested")
    for k in ("h", "rho", "ax", "ay", "az", "du_dt", "v_sig"):
        assert np.array_equal(every[k], base[k]), k
    # an FP32 sum of some hundred terms of either sign, in another order
    for k in ("ax", "ay", "az", "du_dt"):
        rms = np.sqrt(np.mean(base[k][few].astype(np.float64) ** 2))
        assert np.abs(some[k][few].astype(np.float64) - base[k][few]).max() <= 1e-4 * rms, k
        assert np.all(some[k][~few] == active.SENTINEL), k
