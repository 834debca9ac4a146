"""The sort of the reverse pairs on synthetic segments of every length class: sorted
by a thread (up to 8, 16, 32), by a warp in registers (64, 128, 256) or in shared
memory (512), by a block in shared memory (6144) or in place; in blocks of receivers
that fit the staging and in others; against numpy."""
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


EDGES = [0, 1, 2, 7, 8, 9, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1000, 4095,
         4096, 4097, 6143, 6144, 6145, 10000, 70001]


def _lengths(case):
    rng = np.random.default_rng(len(case))
    if case == "every class":
        return np.array(EDGES)
    if case == "one receiver":
        return np.array([300])
    if case == "short":
        return rng.integers(0, 33, 5000)
    if case == "mid":
        return rng.integers(33, 513, 3000)
    if case == "long":
        return rng.integers(513, 9000, 700)
    # blocks of 256 receivers just within and just past the staging of 6144 entries
    v = np.full(1024, 24)
    v[300], v[600], v[601] = 25, 23, 26
    v[768:] = rng.choice(EDGES[:24], 256)
    return v


@pytest.mark.parametrize("case", ["every class", "one receiver", "short", "mid", "long", "staging edge"])
def test_segments(parts, case):
    import torch
    lens = _lengths(case)
    n = len(lens)
    start = np.concatenate([[0], np.cumsum(lens)])
    rng = np.random.default_rng(n)
    # packed sources: 26 bits of index under a shift code up to 42; few distinct ones
    # in every third segment
    rev = ((rng.integers(0, 43, start[-1]) << 26) | rng.integers(0, 1 << 26, start[-1])).astype(np.int64)
    for i in range(0, n, 3):
        rev[start[i]:start[i + 1]] &= 0x3
    dev = {k: torch.as_tensor(v, device="cuda").to(torch.int32) for k, v in
           dict(start=start, queue=np.zeros(n), counts=np.zeros(2)).items()}
    r = torch.as_tensor(rev.astype(np.uint32).view(np.int32), device="cuda")
    rc = parts.part_sort_reverse_pairs(ctypes.c_long(n), native_parts.ptr(dev["start"]), native_parts.ptr(r),
                                       native_parts.ptr(dev["queue"]), native_parts.ptr(dev["counts"]),
                                       native_parts.stream())
    torch.cuda.synchronize()
    assert rc == 0
    # the length classes went where they belong
    assert dev["counts"].cpu().tolist() == [int(((lens > 32) & (lens <= 512)).sum()), int((lens > 512).sum())]
    got = r.cpu().numpy().view(np.uint32)
    ref = np.concatenate([np.sort(rev[a:b]) for a, b in zip(start[:-1], start[1:])]).astype(np.uint32)
    assert np.array_equal(got, ref)
