"""Friends-of-friends in dense cells, whose particles are taken by octants:
labels equal to the oracle's bit for bit where cells hold about as many
particles as the rule asks for, where blobs sit on cell corners and on the
periodic boundary, and where two blobs are just within or just beyond the
linking length."""
import numpy as np
import pytest

from test_gpu_fof import _gpu_fof

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


def _blobs(sizes, b, spread, seed):
    rng = np.random.default_rng(seed)
    cen = rng.random((len(sizes), 3))
    cen[0] = 0.0  # the box corner: eight cells, all wrapped
    cen[1] = np.round(cen[1] / b) * b  # near a cell corner
    # a chain of blobs: the next one within 0.9 .. 2.1 linking lengths
    for k in range(2, len(sizes)):
        d = rng.normal(size=3)
        cen[k] = cen[k - 1] + d / np.linalg.norm(d) * b * rng.uniform(0.9, 2.1)
    p = np.concatenate([cen[k] + spread * b * rng.normal(size=(m, 3)) for k, m in enumerate(sizes)])
    return np.mod(np.concatenate([p, rng.random((2000, 3))]), 1.0)


@pytest.mark.parametrize("nc", [7, 12, 30])
@pytest.mark.parametrize("spread", [0.05, 0.3, 1.0])
def test_blobs(orc, nc, spread):
    b = 1.0 / (nc + 0.3)
    p = _blobs([15, 16, 17, 40, 300, 900, 31, 33, 128, 2500, 64, 16], b, spread, seed=nc)
    rng = np.random.default_rng(1)
    x, y, z = (np.ascontiguousarray(v) for v in p[rng.permutation(len(p))].T)
    assert np.array_equal(_gpu_fof(x, y, z, 1.0, b), orc.fof(x, y, z, 1.0, b))


def test_just_within_and_beyond(orc):
    # two dense blobs whose nearest particles are one linking length apart, less
    # or more by a part in 1e9, and wide cells that are not taken by octants
    b = 0.0313
    for eps, nb in ((-1e-9, 1), (1e-9, 2)):
        rng = np.random.default_rng(7)
        blob = 0.002 * rng.random((400, 3))
        blob[0] = (0.002, 0.001, 0.001)
        other = blob * (-1.0, 1.0, 1.0) + (0.004 + b * (1 + eps), 0.0, 0.0)
        p = np.concatenate([blob, other]) + (0.2, 0.3, 0.4)
        x, y, z = (np.ascontiguousarray(v) for v in p.T)
        got = _gpu_fof(x, y, z, 1.0, b)
        assert np.array_equal(got, orc.fof(x, y, z, 1.0, b)) and len(np.unique(got)) == nb
    p = np.concatenate([0.02 * rng.random((500, 3)) + 0.5, rng.random((300, 3))])
    x, y, z = (np.ascontiguousarray(v) for v in p.T)
    assert np.array_equal(_gpu_fof(x, y, z, 1.0, 0.3), orc.fof(x, y, z, 1.0, 0.3))
