"""Block-sparse float32 attention on group sizes at the edges of its row counts (8 rows per thread step, 64 rows per tile) and
of its key tiles, with tiles whose keys are cut into parts (one head) and tiles that are not (40 heads)."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B
from tests.gpu_util import to_np

pytestmark = pytest.mark.gpu

SIZES = [1, 7, 8, 9, 16, 17, 25, 33, 0, 41, 49, 57, 63, 64, 65, 127, 128, 129, 0, 200, 3]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("heads", [1, 40], ids=["split", "whole"])
def test_row_and_key_counts(heads, d):
    rng = np.random.default_rng(10 * heads + d)
    N, C = sum(SIZES), len(SIZES)
    block = -(-N // C)
    assert -(-N // block) == C
    gen = torch.Generator(device="cuda").manual_seed(d)
    Q, K, V = [torch.randn(1, heads, N, d, device="cuda", generator=gen) for _ in range(3)]
    aQ, aK, ptr, idx = [], [], [], []
    for _ in range(heads):
        aQ.append(rng.permutation(np.repeat(np.arange(C), rng.permutation(SIZES))))
        aK.append(rng.permutation(np.repeat(np.arange(C), rng.permutation(SIZES))))
        routes = [np.sort(rng.choice(C, size=n, replace=False)) for n in rng.permutation([C, C] + list(range(1, C - 1)))]
        # every group is routed to at least one group with keys
        full = int(np.argmax(np.bincount(aK[-1], minlength=C)))
        routes = [np.unique(np.append(r, full)) for r in routes]
        ptr.append(np.concatenate([[0], np.cumsum([len(r) for r in routes])]))
        idx.append(np.concatenate(routes))
    kw = dict(block=block, density=0.5, n_sample=64, n_probe=0, mode=1, softmax_scale=d ** -0.5)
    plan = B.sparsepr_plan_import(Q, K, V, dict(kv_assign=np.stack(aK), q_assign=np.stack(aQ), route_ptr=np.stack(ptr), route_idx=idx), **kw)
    O = B.sparsepr_attend(plan, Q, K, V)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    for i in sorted({0, heads // 2, heads - 1}):
        ref = orc.sparse_attention(to_np(Q[0, i]), to_np(K[0, i]), to_np(V[0, i]), aQ[i], aK[i], ptr[i], idx[i], d ** -0.5)
        # float32 sums of at most 1102 terms of mixed sign: 2^-24 sqrt(1102) = 2e-6 of their size
        assert orc.rel_l2(to_np(O[0, i]), ref) < 2e-6


@pytest.mark.parametrize("H,N", [(8, 7161), (24, 32760)])
def test_workspace_is_that_of_the_copies(H, N):
    """The attend workspace of a large call: the group-major copies of Q, K and V, less than half as much again for
    the probe rows and the fit, and a fixed number of partial states of cut tiles."""
    s = B.Shape(B=1, H=H, N=N, d=128, dv=128, dtype=B.F32, Hkv=H)
    for f in ("q_stride", "k_stride", "v_stride", "o_stride"):
        getattr(s, f)[:] = [H * N * 128, N * 128, 128]
    p = B.make_params(block=64, density=0.25, n_sample=128, n_probe=64)
    copies = 3 * 4 * H * N * 128
    need = B.lib().sparsepr_attend_workspace_bytes(ctypes.byref(s), ctypes.byref(p))
    assert copies < need <= 1.4 * copies + 16 * 148 * 64 * 130 * 4     # (sixteen states of 64 rows per SM)
