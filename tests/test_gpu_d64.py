"""bf16 tensors with head dimension 64 on the tensor-core kernels: full tiles, doubled and packed group remainders, probe
slices, the two-word correction and the projections, against the oracle on the oracle's own plan (outputs) and through the
GPU's own plan (links); tolerances as for d = 128 where the output is bf16.  Probabilities, sums and features are float32 here."""
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B
from paper_2608_18484_b200 import workloads as W
from tests.gpu_util import assert_bf16_close, heads_to_device, to_np
from tests.test_gpu_attend import oracle_plans, plans_to_host
from tests.test_gpu_plan_parity import check_links, plan_links

pytestmark = pytest.mark.gpu

CASES = [("480p-like", W.VIDEO_480P.scaled(grid=(3, 30, 52), H=2, d=64, n_probe=64)),
         ("ragged", W.WORLD.scaled(grid=(1, 31, 43), H=2, d=64, n_probe=130)),
         ("720p-like", W.VIDEO_720P.scaled(grid=(1, 45, 80), H=2, d=64, n_probe=33))]


@pytest.mark.parametrize("mode", [0, 1], ids=["fitted", "hard"])
@pytest.mark.parametrize("name,wl", CASES, ids=[c[0] for c in CASES])
def test_attend_d64(name, wl, mode):
    host, (Qd, Kd, Vd) = heads_to_device(wl, [0, 1])
    junk = torch.full((64 << 20,), float("nan"), device="cuda")   # anything read before it is written shows
    del junk
    kw = dict(density=wl.density, block=wl.block, n_sample=wl.n_sample, n_probe=wl.n_probe, softmax_scale=1.0, mode=mode, lam=1.0)
    prm = orc.default_params(**kw)
    plans = oracle_plans(host, prm)
    C = -(-wl.N // wl.block)
    plan = B.sparsepr_plan_import(Qd, Kd, Vd, plans_to_host(plans, C, C), **kw)
    O, Osp = B.sparsepr_attend(plan, Qd, Kd, Vd, return_sparse=True)
    O2 = B.sparsepr_attend(plan, Qd, Kd, Vd)                       # (without the float32 copy the output goes another way)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    for i, (Q, K, V) in enumerate(host):
        O_hat, O_sp, _ = orc.attend_head(Q, K, V, plans[i], prm)
        assert_bf16_close(to_np(Osp[0, i]), O_sp)
        assert_bf16_close(to_np(O[0, i]), O_hat)
        assert_bf16_close(to_np(O2[0, i]), O_hat)


@pytest.mark.parametrize("name,wl", CASES, ids=[c[0] for c in CASES])
def test_float32_inside_d64(name, wl):
    """Hard-drop rows and features before any rounding to bf16.  Rows: probabilities in two bf16 words (2^-18) of exponentials good to
    2^-22, sums in float32: 2e-6 (one bf16 word: 2e-4).  Features: three words of F, float32 sums: 2^-23 in the 2-norm, and a fifth."""
    host, (Qd, Kd, Vd) = heads_to_device(wl, [0, 1])
    kw = dict(density=wl.density, block=wl.block, n_sample=wl.n_sample, n_probe=wl.n_probe, softmax_scale=1.0, mode=1)
    prm = orc.default_params(**kw)
    plans = oracle_plans(host, prm)
    C = -(-wl.N // wl.block)
    _, Osp = B.sparsepr_attend(B.sparsepr_plan_import(Qd, Kd, Vd, plans_to_host(plans, C, C), **kw), Qd, Kd, Vd, return_sparse=True)
    feat = B.sparsepr_plan_export_features(B.sparsepr_plan(Qd, Kd, Vd, **kw), fields=("F_Q", "phi_Q"))
    for i, (Q, K, V) in enumerate(host):
        _, O_sp, _ = orc.attend_head(Q, K, V, plans[i], prm)
        assert orc.rel_l2(to_np(Osp[0, i]), O_sp) <= 2e-6
        assert orc.rel_l2(feat["phi_Q"][i], orc.query_response(Q, feat["F_Q"][i])) <= 1.4e-7


@pytest.mark.parametrize("name,wl", CASES, ids=[c[0] for c in CASES])
def test_one_rounding_d64(name, wl):
    """The corrected output is the float64 value rounded to bf16 once: float32 errors of about 2e-6 before the rounding, whose steps are
    2^-8, turn it another way for one element in a thousand, small differences of larger terms for some more: 5e-3."""
    host, (Qd, Kd, Vd) = heads_to_device(wl, [0, 1])
    kw = dict(density=wl.density, block=wl.block, n_sample=wl.n_sample, n_probe=wl.n_probe, softmax_scale=1.0, lam=10.0)
    prm = orc.default_params(**kw)
    plans = oracle_plans(host, prm)
    C = -(-wl.N // wl.block)
    plan = B.sparsepr_plan_import(Qd, Kd, Vd, plans_to_host(plans, C, C), **kw)
    O, _ = B.sparsepr_attend(plan, Qd, Kd, Vd, return_sparse=True)
    O2 = B.sparsepr_attend(plan, Qd, Kd, Vd)
    assert torch.equal(O, O2)
    for i, (Q, K, V) in enumerate(host):
        ref = torch.from_numpy(orc.attend_head(Q, K, V, plans[i], prm)[0]).to(torch.bfloat16)
        assert (O2[0, i].cpu() != ref).double().mean() <= 5e-3


def test_plan_d64():
    wl = CASES[0][1]
    host, (Qd, Kd, Vd) = heads_to_device(wl, [0, 1])
    kw = dict(density=wl.density, block=wl.block, n_sample=wl.n_sample, n_probe=wl.n_probe, softmax_scale=1.0)
    plan = B.sparsepr_plan(Qd, Kd, Vd, **kw)
    exp, feat = B.sparsepr_plan_export(plan), B.sparsepr_plan_export_features(plan)
    prm = orc.default_params(**kw)
    check_links(wl, [plan_links(wl, i, Q, K, exp, feat, prm) for i, (Q, K, V) in enumerate(host)])


@pytest.mark.parametrize("N", [1, 127, 129, 1000])
def test_dense_d64_strided(N):
    gen = torch.Generator(device="cuda").manual_seed(N)
    Q, K, V = [torch.randn(2, N, 3, 64, device="cuda", generator=gen).bfloat16().permute(0, 2, 1, 3) for _ in range(3)]
    O = B.sparsepr_dense(Q, K, V, 0.125)
    for b in range(2):
        for h in range(3):
            assert_bf16_close(to_np(O[b, h]), orc.dense_attention(to_np(Q[b, h]), to_np(K[b, h]), to_np(V[b, h]), 0.125))
