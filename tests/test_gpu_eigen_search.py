"""The search for eigenvalues in float64 by itself.  Of a diagonal matrix the counts are exact and the eigenvalues are known to the bit, so what
is left is the width of the last interval: below 4.7e-16 of the largest entry, half of it between its middle and the eigenvalue, and a rounding."""
import ctypes as C
import os
import subprocess

import pytest
import torch

from paper_2608_18484_b200 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("eigen_search") / "lib.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "eigen_search.cu")
    subprocess.run([build.NVCC] + build.FLAGS + ["-shared", "-o", out, src], check=True)
    L = C.CDLL(out)
    L.largest_eigenvalues.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_int, C.c_void_p]
    return L


@pytest.mark.parametrize("n,r", [(128, 64), (128, 48), (64, 64), (64, 1)])
def test_width_of_the_last_interval(lib, n, r):
    batch = 6
    gen = torch.Generator(device="cuda").manual_seed(n + r)
    d = torch.rand(batch, n, dtype=torch.float64, device="cuda", generator=gen)
    d[:, 5] = 1.0
    d[3:, ::2] *= -1.0                                          # signs of both kinds
    M = torch.diag_embed(d).contiguous()
    lam = torch.empty(batch, r, dtype=torch.float64, device="cuda")
    assert lib.largest_eigenvalues(M.data_ptr(), batch, n, r, lam.data_ptr()) == 0
    err = (lam - d.sort(1, descending=True).values[:, :r]).abs().max().item()
    assert err <= 0.5 * 4.7e-16 + 2.0 ** -53, err
