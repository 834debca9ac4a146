"""Blocks of a small uniform grid of which some need more than one round a warp (more
than 128 targets, or 64 at four lanes) and are shared between CTAs, and some do not:
the box alone gives bit for bit what it gives within a pool (one CTA per block), and
masked loops on every particle what the unmasked ones give."""
import numpy as np
import pytest

from paper_2305_13380_gb300 import inputs

import test_gpu_active as active
import test_gpu_block_parts as parts

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


@pytest.mark.parametrize("kernel,lanes", [(0, 0), (0, 4), (1, 0), (2, 0)])
@pytest.mark.parametrize("side", [20, 22, 30])
def test_alone_and_in_a_pool(side, lanes, kernel):
    parts.test_alone_and_in_a_pool(side, lanes, kernel)


@pytest.mark.parametrize("side", [20, 22, 30])
def test_all_active(side):
    p = inputs.lattice(side, seed=side, sigma_v=0.05)
    base, (g,) = active._run(p, [np.ones(side ** 3, bool)])
    for k in ("h", "rho", "f", "div_v", "curl_v", "P", "c", "balsara", "ax", "ay", "az", "du_dt", "v_sig"):
        assert np.array_equal(g[k], base[k]), k
