"""The arithmetic of the centroids in the one-kernel k-means run: their squared norms are rounded once, as in the separate passes."""
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
    L.row_norms.argtypes = [C.c_void_p, C.c_int, C.c_void_p]
    return L


@pytest.mark.parametrize("n,size", [(1, 1.0), (5, 1e-3), (4096, 1.0), (4099, 1e3)])
def test_norms_are_rounded_once(lib, n, size):
    rows = (np.random.default_rng(n).standard_normal((n, 64)) * size).astype(np.float32)
    rows[:, 48:] *= n % 2                                        # (columns beyond the rank hold zeros)
    x, out = torch.from_numpy(rows).cuda(), torch.empty(n, dtype=torch.float32, device="cuda")
    assert lib.row_norms(x.data_ptr(), n, out.data_ptr()) == 0
    ref = (rows.astype(np.float64) ** 2).sum(1)
    # half a unit in the last place of a float32, and 64 float64 roundings
    assert (np.abs(out.cpu().numpy() - ref) <= ref * (2.0 ** -24 + 64 * 2.0 ** -53)).all()
