"""The cell and key sorts at the sizes where their route or their tiles change:
one block up to 8192 items (warps of 256), tiles of 2048 beyond, digits that all
keys share."""
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


@pytest.mark.parametrize("h_scale", [0.4, 1.0, 4.0])
@pytest.mark.parametrize("n", [1, 31, 256, 257, 2047, 2049, 8191, 8192, 8193, 10240, 40961])
def test_cells_bit_exact(orc, n, h_scale):
    import torch
    from paper_2305_13380_gb300 import sph
    x = np.random.default_rng(n).random((3, n))
    h = np.full(n, min(h_scale * 1.2348 * n ** (-1.0 / 3.0), 0.15), dtype=np.float32)
    ctx = sph.Context(sph.sph_default_params(box_size=1.0))
    t = [torch.as_tensor(v, device="cuda") for v in x]
    cells = sph.sph_build_cells(ctx, *t, torch.as_tensor(h, device="cuda"))
    cs, perm = sph.sph_cells_copy(ctx, cells)
    assert sph.sph_status(ctx) == 0
    nc = expected_nc(h, 1.0, n=n)
    assert cells.n_c == nc
    ocs, operm = orc.build_cells(x[0], x[1], x[2], 1.0, nc)
    assert np.array_equal(cs, ocs)
    assert np.array_equal(perm, operm)


@pytest.mark.parametrize("n", [8191, 8192, 8193, 12289])
def test_nested_grids(orc, n):
    p = inputs.clustered(n, n_spheres=5, seed=n)
    q = as_f32(p)
    g = run_gpu(p, tree=True, n_leaf=16)
    od, of = orc.density_force(q, q["h0"])
    compare(g, od, of)
