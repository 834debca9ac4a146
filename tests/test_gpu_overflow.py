"""The uniform grid's overflow kernels: cells just past the blocks' staging,
cells whose 27-cell neighbourhood is staged and listed or streamed, cells of
more than 32 and more than 128 targets, and more cells than resident CTAs,
against the FP64 oracle."""
import numpy as np
import pytest

from paper_2305_13380_gb300 import inputs

from gpu_common import as_f32, compare, expected_nc, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


def _check(orc, p, margin, kernel=0):
    q = as_f32(p)
    g = run_gpu(p, margin=margin, kernel=kernel)
    od, of = orc.density_force(q, q["h0"], orc.Physics(kernel=kernel))
    vmax = float(np.sqrt(max(np.max(q["vx"] ** 2 + q["vy"] ** 2 + q["vz"] ** 2), 0.0)))
    compare(g, od, of, cell=float(p["L"]) / expected_nc(p["h0"], float(p["L"]), margin), vmax=vmax)


@pytest.mark.parametrize("side,margin", [(8, 0.05), (9, 0.05), (11, 0.3), (14, 0.05), (16, 0.05), (16, 0.25),
                                         (16, 0.6), (19, 0.05), (20, 1.4), (56, 0.3)])
def test_lattice_cells(orc, side, margin):
    _check(orc, inputs.lattice(side, seed=side, sigma_v=0.05), margin)


@pytest.mark.parametrize("kernel", [1, 2])
@pytest.mark.parametrize("side,margin", [(16, 0.05), (19, 0.3)])
def test_lattice_cells_other_kernels(orc, kernel, side, margin):
    _check(orc, inputs.lattice(side, seed=side, sigma_v=0.05), margin, kernel=kernel)
