"""The exclusive scan over look-back tiles: lengths around its tiles of 4096, and
sums up to 2^31 - 1 (the reverse pairs that a context may hold)."""
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


def _scan(parts, v, dtype="int32"):
    import torch
    n = len(v)
    a = torch.as_tensor(v, device="cuda").to(getattr(torch, dtype))
    out = torch.full((n + 1,), -1, dtype=torch.int32, device="cuda")
    scratch = torch.empty(parts.part_scan_words(n), dtype=torch.int32, device="cuda")
    f = parts.part_scan if dtype == "int32" else parts.part_scan_bytes
    rc = f(native_parts.ptr(a), native_parts.ptr(out), ctypes.c_long(n), native_parts.ptr(scratch),
           native_parts.stream())
    torch.cuda.synchronize()
    assert rc == 0
    return out.cpu().numpy()


@pytest.mark.parametrize("dtype", ["int32", "uint8"])
@pytest.mark.parametrize("n", [1, 15, 16, 4095, 4096, 4097, 100000, 4096 * 1100 + 3])
def test_lengths(parts, n, dtype):
    v = np.random.default_rng(n).integers(0, 256, n)
    assert np.array_equal(_scan(parts, v, dtype), np.concatenate([[0], np.cumsum(v)]))


@pytest.mark.parametrize("total", [2 ** 30 - 1, 2 ** 30, 2 ** 30 + 1, 2 ** 31 - 1])
@pytest.mark.parametrize("n", [4096, 20000, 4096 * 300])
def test_large_sums(parts, n, total):
    rng = np.random.default_rng(n)
    v = np.zeros(n, dtype=np.int64)
    v[rng.integers(0, n, 5)] = total // 7
    v[0] += total - v.sum() - 1
    v[n - 1] += 1
    assert np.array_equal(_scan(parts, v), np.concatenate([[0], np.cumsum(v)]))
