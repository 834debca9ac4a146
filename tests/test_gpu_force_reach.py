"""The force on given density results whose supports exceed the cells: every pair of
the 27 cells within max(H_i, H_j) counts, in the blocks' kernel and in the overflow
kernel alike."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
GAMMA_K = 1.825742


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2305_13380_gb300 import build
    build.build()


# three cells a side: a block stages 64 / 27 of the particles, at most 1216; the
# overflow kernel lists up to 640 sources
@pytest.mark.parametrize("n", [400, 513, 520, 600, 640, 700])
def test_supports_beyond_the_cells(n):
    import torch
    from paper_2305_13380_gb300 import sph
    rng = np.random.default_rng(n)
    X = rng.random((3, n))
    H = np.where(np.arange(n) % 20 == 0, 0.4, 0.3)
    h = (H / GAMMA_K).astype(np.float32)
    P = rng.uniform(0.5, 1.5, n).astype(np.float32)
    dev = lambda v, t=torch.float32: torch.as_tensor(np.asarray(v), device="cuda").to(t)  # noqa: E731
    zero, one = np.zeros(n), np.ones(n)
    t = {k: dev(X[i], torch.float64) for i, k in enumerate("xyz")}
    t.update({k: dev(zero) for k in ("vx", "vy", "vz")}, m=dev(one / n), u=dev(one))
    ctx = sph.Context(sph.sph_default_params(box_size=1.0))
    cells = sph.sph_build_cells(ctx, t["x"], t["y"], t["z"], dev(np.full(n, 0.17)))
    assert sph.sph_cells_sync(ctx, cells) == 3
    d = sph.alloc_density(n)
    for k, v in dict(h=h, rho=one, f=one, P=P, c=one, balsara=zero, div_v=zero, curl_v=zero).items():
        d[k].copy_(dev(v))
    f = sph.alloc_force(n)
    sph.sph_force(ctx, cells, sph.particles(t), sph.density_out(d), sph.force_out(f))
    a = np.stack([f[k].double().cpu().numpy() for k in ("ax", "ay", "az")])
    # the same in 64 bits: the image of j in the cell beside i's
    H = GAMMA_K * h.astype(np.float64)
    cell = np.floor(X * 3).astype(int)
    ref = np.zeros((3, n))
    for i in range(n):
        dc = cell - cell[:, i:i + 1]
        shift = np.where(dc == 2, -1, np.where(dc == -2, 1, 0))
        dx = X[:, i:i + 1] - (X + shift)
        r = np.sqrt((dx ** 2).sum(0))
        r[i] = np.inf
        near = r < np.maximum(H[i], H)

        def grad(Hk):  # W'(r) / r of the cubic spline
            q = r / Hk
            w = -48 / np.pi * (np.maximum(1 - q, 0) ** 2 - np.maximum(1 - 2 * q, 0) ** 2)
            return w / (Hk ** 4 * r)

        s = np.where(near, -(P[i].astype(float) * grad(H[i]) + P * grad(H)) / n, 0.0)
        s[i] = 0.0
        ref[:, i] = np.nansum(np.where(near, s * dx, 0.0), axis=1)
    rms = np.sqrt((ref ** 2).sum(0).mean())
    assert np.abs(a - ref).max() <= 1e-4 * rms
