"""The fit at the edges of its kernels' splits (8 probe slices, chunks of 32 probes, 32- and 64-wide Gram tiles, 64 or 32
right-hand sides per elimination): a single probe, a chunk and one, several chunks with a remainder, for both head
dimensions and data types, against the oracle on the oracle's own plan."""
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B
from paper_2608_18484_b200 import workloads as W
from tests.gpu_util import heads_to_device, to_np
from tests.test_gpu_attend import check, oracle_plans, plans_to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r_out", [16, 128], ids=["rank16", "full"])
@pytest.mark.parametrize("M", [1, 33, 200])
@pytest.mark.parametrize("dtype,d", [("f32", 64), ("f32", 128), ("bf16", 64), ("bf16", 128)])
def test_fit_sizes(dtype, d, M, r_out):
    wl = W.TINY.scaled(grid=(1, 32, 33), dtype=dtype, d=d)
    host, (Qd, Kd, Vd) = heads_to_device(wl, [0, 1])
    # a ridge of 10 keeps the system well conditioned whatever M is against d, so the bounds of `check` apply to the output
    kw = dict(density=0.5, block=64, n_sample=64, n_probe=M, softmax_scale=1.0, r_out=r_out, lam=10.0)
    prm = orc.default_params(**kw)
    plans = oracle_plans(host, prm)
    C = -(-wl.N // 64)
    plan = B.sparsepr_plan_import(Qd, Kd, Vd, plans_to_host(plans, C, C), **kw)
    O = B.sparsepr_attend(plan, Qd, Kd, Vd)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0 and torch.isfinite(O).all()
    for i, (Q, K, V) in enumerate(host):
        check(to_np(O[0, i]), orc.attend_head(Q, K, V, plans[i], prm)[0], dtype == "f32")


@pytest.mark.parametrize("what", ["weights", "pivot"])
@pytest.mark.parametrize("dtype,d", [("f32", 128), ("bf16", 64)])
def test_no_fit_is_reported(dtype, d, what):
    """Probes of no weight at all, and a single probe without a ridge (a zero matrix), more heads than run at once: the error word
    says so and the output is that of hard drop outside the probe rows."""
    H, N = 80, 256
    gen = torch.Generator(device="cuda").manual_seed(1)
    Q, K, V = [torch.randn(1, H, N, d, device="cuda", generator=gen).mul_(d ** -0.25).to(torch.float32 if dtype == "f32" else torch.bfloat16) for _ in range(3)]
    kw = dict(density=0.5, block=64, n_sample=64, n_probe=16 if what == "weights" else 1, softmax_scale=1.0, lam=10.0 if what == "weights" else 0.0)
    host = B.sparsepr_plan_export(B.sparsepr_plan(Q, K, V, **kw))
    if what == "weights":
        host["probe_w"][:] = 0.0
    plan = B.sparsepr_plan_import(Q, K, V, host, **kw)
    O = B.sparsepr_attend(plan, Q, K, V)
    hard = B.sparsepr_attend(B.sparsepr_plan_import(Q, K, V, host, **dict(kw, mode=1)), Q, K, V)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 5
    keep = torch.ones(H, N, dtype=torch.bool, device="cuda")
    keep.scatter_(1, torch.from_numpy(host["probe_idx"]).long().cuda(), False)
    assert torch.equal(O[0][keep], hard[0][keep])
