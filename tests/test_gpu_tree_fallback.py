"""The nested grids' per-target kernels: targets beside a dense core whose
reach holds about as many sources as a row (32), a staged chunk (320) and the
streamed batches (128 and 256) end at, in children of one source and of many,
against the FP64 oracle."""
import pytest

from gpu_common import as_f32, compare, run_gpu
from test_gpu_tree_rounds import _core_and_shell

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


@pytest.mark.parametrize("n_leaf", [1, 64])
@pytest.mark.parametrize("n_core", [255, 288, 319, 320, 321, 512, 1025])
def test_targets_beside_a_core(orc, n_core, n_leaf):
    p = _core_and_shell(n_core, 150, 3500, seed=n_core)
    q = as_f32(p)
    g = run_gpu(p, tree=True, n_leaf=n_leaf)
    g = run_gpu(p, tree=True, n_leaf=n_leaf, h_start=g["h"])
    od, of = orc.density_force(q, q["h0"])
    compare(g, od, of)


@pytest.mark.parametrize("factor", [0.3, 3.0])
def test_starting_supports_far_off(orc, factor):
    # every support grows or shrinks a lot from its start: selections again at
    # a larger radius, at a coarser level, and sources far beyond the support
    p = _core_and_shell(700, 200, 3500, seed=7)
    q = as_f32(p)
    g = run_gpu(p, tree=True, n_leaf=16)
    g = run_gpu(p, tree=True, n_leaf=16, h_start=(factor * g["h"]).clip(max=0.12))
    od, of = orc.density_force(q, q["h0"])
    compare(g, od, of)
