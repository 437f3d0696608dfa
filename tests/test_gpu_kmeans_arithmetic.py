"""The arithmetic of the centroids in the one-kernel k-means run, beside that of the separate passes: a group's mean is the one that a float64 division
gives, to the bit, and the squared norms are rounded once."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2608_18484_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("kmeans_arithmetic") / "lib.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "kmeans_arithmetic.cu")
    subprocess.run([build.NVCC] + build.FLAGS + ["-shared", "-o", out, src], check=True)
    L = C.CDLL(out)
    L.group_means.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_int, C.c_void_p, C.c_void_p]
    L.row_norms.argtypes = [C.c_void_p, C.c_int, C.c_void_p]
    return L


def _means_equal(lib, sums, counts, shift):
    sums, counts = np.broadcast_arrays(np.asarray(sums, np.int64), np.asarray(counts, np.int64))
    s, c = torch.from_numpy(sums.ravel().copy()).cuda(), torch.from_numpy(counts.ravel().astype(np.int32)).cuda()
    quick, divided = [torch.empty(s.numel(), dtype=torch.float32, device="cuda") for _ in range(2)]
    assert lib.group_means(s.data_ptr(), c.data_ptr(), s.numel(), shift, quick.data_ptr(), divided.data_ptr()) == 0
    assert torch.equal(quick.view(torch.int32), divided.view(torch.int32))
    ref = sums.ravel() * 2.0 ** -shift / counts.ravel()          # (float64 as above: the cast of the sum, a power of two, the division)
    assert np.array_equal(divided.cpu().numpy(), ref.astype(np.float32))


@pytest.mark.parametrize("shift", [24, 45, -3])
def test_means_are_those_of_a_division(lib, shift):
    rng = np.random.default_rng(7)
    powers = 2 ** np.arange(1, 31, dtype=np.int64)
    counts = np.unique(np.concatenate([[1, 2, 3, 2 ** 31 - 1], powers, powers - 1, powers + 1, rng.integers(1, 2 ** 31, 400)]))
    edge = np.array([0, 1, 2, 3, 2 ** 24 - 1, 2 ** 24 + 1, 2 ** 53 - 1, 2 ** 53 + 1, 2 ** 62 - 1, 2 ** 62 + 1, 2 ** 63 - 1], np.int64)
    sums = np.concatenate([edge, -edge, (rng.integers(1, 2 ** 62, 400) >> rng.integers(0, 61, 400)) * rng.choice([-1, 1], 400)])
    _means_equal(lib, sums[None, :], counts[:, None], shift)
    # quotients at and beside the midpoints of two float32
    mid = 2 * rng.integers(2 ** 23, 2 ** 24, 3000) + 1
    n = np.concatenate([rng.choice(counts, 2000), rng.integers(1, 50000, 1000)])
    for delta in (-8, -1, 0, 1, 8):
        _means_equal(lib, mid * n + delta, n, shift)


@pytest.mark.parametrize("n,size", [(1, 1.0), (5, 1e-3), (4096, 1.0), (4099, 1e3)])
def test_norms_are_rounded_once(lib, n, size):
    rows = (np.random.default_rng(n).standard_normal((n, 64)) * size).astype(np.float32)
    rows[:, 48:] *= n % 2                                        # (columns beyond the rank hold zeros)
    x, out = torch.from_numpy(rows).cuda(), torch.empty(n, dtype=torch.float32, device="cuda")
    assert lib.row_norms(x.data_ptr(), n, out.data_ptr()) == 0
    ref = (rows.astype(np.float64) ** 2).sum(1)
    # half a unit in the last place of a float32, and 64 float64 roundings
    assert (np.abs(out.cpu().numpy() - ref) <= ref * (2.0 ** -24 + 64 * 2.0 ** -53)).all()
