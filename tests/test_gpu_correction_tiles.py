"""The residual correction over runs of tiles: more tiles than CTAs, so that a CTA works on several and changes heads between or
within them; last tiles of one row, of a part and full."""
import pytest

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B
from paper_2608_18484_b200 import workloads as W
from tests.gpu_util import assert_bf16_close, heads_to_device, to_np
from tests.test_gpu_attend import oracle_plans, plans_to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("heads,grid", [(80, (1, 3, 43)), (60, (2, 16, 12)), (50, (1, 23, 22))], ids=["129", "384", "506"])
def test_runs_of_tiles(heads, grid, d):
    wl = W.VIDEO_480P.scaled(grid=grid, H=heads, d=d, n_probe=48)
    host, (Qd, Kd, Vd) = heads_to_device(wl, list(range(heads)))
    # 48 probes for up to 128 output dimensions: at a ridge of 1 the fitted map has a norm of several units and multiplies the error of
    # the probe rows (2^-9, bf16 probabilities) by it; at 10 its norm is below one and the bound of a single bf16 output holds
    kw = dict(density=0.4, block=wl.block, n_sample=64, n_probe=wl.n_probe, softmax_scale=1.0, mode=0, lam=10.0)
    prm = orc.default_params(**kw)
    plans = oracle_plans(host, prm)
    C = -(-wl.N // wl.block)
    plan = B.sparsepr_plan_import(Qd, Kd, Vd, plans_to_host(plans, C, C), **kw)
    O = B.sparsepr_attend(plan, Qd, Kd, Vd)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    for i in sorted({0, 1, heads // 2, heads - 1}):
        Q, K, V = host[i]
        assert_bf16_close(to_np(O[0, i]), orc.attend_head(Q, K, V, plans[i], prm)[0])      # as for the other bf16 outputs
