"""The nested grids' fine coordinate on the device: the fixed-point estimate with the
exact path behind it against the definition, floor(1024 fl(fl(x n_c) / L)) clamped to
the top cell, on random positions, on sub-cell faces and an ulp beside them, and on
positions that only the exact path takes."""
import ctypes

import numpy as np
import pytest

import native_parts

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def parts(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    return native_parts.load(tmp_path_factory.mktemp("parts"))


@pytest.mark.parametrize("L", [1.0, 0.7, 3.3e-9, 1.0e12, 142.25])
@pytest.mark.parametrize("n_c", [1, 3, 54, 127, 1000, 60000])
def test_matches_definition(parts, L, n_c):
    import torch
    rng = np.random.default_rng(n_c)
    faces = rng.integers(0, 1024 * n_c, 200000) * L / (1024.0 * n_c)
    x = np.concatenate([rng.random(400000) * L, faces, np.nextafter(faces, np.inf), np.nextafter(faces, -np.inf),
                        rng.random(20000) * L * 2.0 ** -rng.integers(0, 60, 20000),
                        [0.0, 5e-324, -5e-324, -0.1 * L, L, np.nextafter(L, 0.0), 1.5 * L]])
    xd = torch.as_tensor(x, device="cuda")
    got = torch.zeros((2, len(x)), dtype=torch.int32, device="cuda")
    rc = parts.part_fine_coords(ctypes.c_long(len(x)), native_parts.ptr(xd), ctypes.c_double(L), ctypes.c_int(n_c),
                                native_parts.ptr(got[0]), native_parts.ptr(got[1]), native_parts.stream())
    torch.cuda.synchronize()
    assert rc == 0
    fast, exact = got.cpu().numpy()
    assert np.array_equal(fast, exact)
    s = x * n_c / L
    k = np.clip(np.floor(s), 0, n_c - 1)
    ref = np.clip(np.floor(s * 1024.0), k * 1024, k * 1024 + 1023)
    assert np.array_equal(exact, ref)
