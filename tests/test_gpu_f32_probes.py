"""Exact and hard-drop rows of the probes in float32 (32 rows per CTA, key slices of whole tiles of 64, states that change hands
where a K/V group ends): probe counts at the edges of the row tiles, token counts at those of the key tiles and slices."""
import numpy as np
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B
from paper_2608_18484_b200 import workloads as W
from tests.gpu_util import heads_to_device, to_np
from tests.test_gpu_attend import oracle_plans, plans_to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("M,grid", [(1, (1, 16, 16)), (31, (1, 31, 37)), (32, (1, 8, 8)), (33, (1, 9, 57)), (65, (3, 31, 29)), (128, (1, 32, 36))])
def test_probe_rows(M, grid, d):
    wl = W.TINY.scaled(grid=grid, H=1, d=d, n_probe=M)
    host, (Qd, Kd, Vd) = heads_to_device(wl, [0])
    junk = torch.full((8 << 20,), float("nan"), device="cuda")   # what is read before it is written shows
    del junk
    kw = dict(density=0.3, block=24, n_sample=64, n_probe=M, softmax_scale=wl.softmax_scale, lam=10.0)
    prm = orc.default_params(**kw)
    plans = oracle_plans(host, prm)
    C = -(-wl.N // 24)
    plan = B.sparsepr_plan_import(Qd, Kd, Vd, plans_to_host(plans, C, C), **kw)
    O = to_np(B.sparsepr_attend(plan, Qd, Kd, Vd)[0, 0])
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    Q, K, V = host[0]
    P = plans[0]["probe_idx"]
    # float32 sums with a 2-ulp exp2: the bound of the attention path; the other rows carry the fit to both states
    assert orc.rel_l2(O[P], orc.dense_attention(Q, K, V, plans[0]["scale"], rows=P)) <= 1e-5
    assert orc.rel_l2(O, orc.attend_head(Q, K, V, plans[0], prm)[0]) <= 1e-5
