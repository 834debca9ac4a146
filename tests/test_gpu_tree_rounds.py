"""The nested-grid density's rounds of four targets: windows that cut leaves,
rounds that keep more sources than their buffer holds, and leaves that are
taken whole or by children, against the FP64 oracle."""
import numpy as np
import pytest

from paper_2305_13380_gb300 import inputs

from gpu_common import as_f32, compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


def _core_and_shell(n_core, n_shell, n_bg, seed):
    """A dense core, a shell of targets around it whose lists each take in a
    part of the core (different parts, so that a round's lists hold more
    sources together than its buffer), and a uniform background."""
    rng = np.random.default_rng(seed)
    def ball(n, lo, hi):
        d = rng.normal(size=(n, 3))
        r = rng.uniform(lo ** 3, hi ** 3, n) ** (1.0 / 3.0)
        return 0.5 + d / np.linalg.norm(d, axis=1)[:, None] * r[:, None]
    p = np.concatenate([ball(n_core, 0.0, 0.01), ball(n_shell, 0.012, 0.05), rng.random((n_bg, 3))])
    n = len(p)
    nd = np.concatenate([np.full(n_core, n_core / 4.2e-6), np.full(n_shell, n_shell / 5.2e-4 + n_bg),
                         np.full(n_bg, float(n_bg))])
    v = rng.normal(0.0, 0.05, (n, 3))
    return dict(L=1.0, x=p[:, 0], y=p[:, 1], z=p[:, 2], vx=v[:, 0], vy=v[:, 1], vz=v[:, 2], m=np.full(n, 1.0 / n),
                u=np.exp(rng.normal(size=n)), h0=np.minimum(1.2348 * nd ** (-1.0 / 3.0), 0.1))


@pytest.mark.parametrize("kernel", [0, 1, 2])
@pytest.mark.parametrize("sizes", [(600, 300, 4000), (2500, 1000, 4003), (5000, 61, 4502)])
def test_core_and_shell(orc, kernel, sizes):
    p = _core_and_shell(*sizes, seed=sum(sizes))
    q = as_f32(p)
    # the second call starts from the converged h, so that lists are built for it
    g = run_gpu(p, tree=True, kernel=kernel, n_leaf=32)
    g = run_gpu(p, tree=True, kernel=kernel, n_leaf=32, h_start=g["h"])
    od, of = orc.density_force(q, q["h0"], orc.Physics(kernel=kernel))
    compare(g, od, of)


@pytest.mark.parametrize("n_leaf", [1, 2, 3, 4, 5, 8, 9, 33])
def test_leaves_across_windows(orc, n_leaf):
    # groups of every small size, cut by windows at every offset
    p = inputs.clustered(2500 + n_leaf, n_spheres=3, seed=n_leaf, frac_clustered=0.6)
    q = as_f32(p)
    g = run_gpu(p, tree=True, n_leaf=n_leaf)
    od, of = orc.density_force(q, q["h0"])
    compare(g, od, of)


@pytest.mark.parametrize("case", ["short", "mid", "long"])
def test_reverse_pairs_sorted(case):
    # the force adds a receiver's reverse pairs in order of their source, which
    # atomics had put in any order: segments sorted by a thread (up to 32), a
    # warp (up to 512) or a block give the same bits in every run
    if case == "short":
        p = inputs.clustered(5000, n_spheres=4, seed=2, a_min=0.02, a_max=0.05)
    elif case == "mid":
        p = inputs.clustered(20000, n_spheres=4, seed=43)
    else:
        p = _core_and_shell(20000, 3000, 6000, seed=5)
    runs = [run_gpu(p, tree=True, n_leaf=32) for _ in range(3)]
    for r in runs[1:]:
        for k in ("h", "rho", "ax", "ay", "az", "du_dt", "v_sig"):
            assert np.array_equal(runs[0][k], r[k]), k
