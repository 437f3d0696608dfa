"""Block-sparse bf16 attention on group sizes at the edges of its query tiles (remainders of at most 32 rows, at most 64 rows, one
tile, two tiles and what is left of them) and of its key boxes and tiles (16 and 128 keys)."""
import numpy as np
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B
from tests.gpu_util import assert_bf16_close, to_np

pytestmark = pytest.mark.gpu

SIZES = [1, 15, 16, 17, 32, 33, 0, 64, 65, 127, 128, 129, 160, 161, 255, 256, 257, 0, 288, 289, 384, 513, 2]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("heads", [3, 20], ids=["few", "many"])
def test_row_and_key_counts(heads, d):
    rng = np.random.default_rng(d)
    N, C = sum(SIZES), len(SIZES)
    block = -(-N // C)
    assert -(-N // block) == C
    gen = torch.Generator(device="cuda").manual_seed(d)
    Q, K, V = [torch.randn(1, heads, N, d, device="cuda", generator=gen).bfloat16() for _ in range(3)]
    aQ, aK, ptr, idx = [], [], [], []
    for _ in range(heads):
        aQ.append(rng.permutation(np.repeat(np.arange(C), rng.permutation(SIZES))))
        aK.append(rng.permutation(np.repeat(np.arange(C), rng.permutation(SIZES))))
        full = int(np.argmax(np.bincount(aK[-1], minlength=C)))   # every group is routed to at least one group with keys
        routes = [np.unique(np.append(rng.choice(C, size=n, replace=False), full)) for n in rng.permutation([C] + list(range(1, C)))]
        ptr.append(np.concatenate([[0], np.cumsum([len(r) for r in routes])]))
        idx.append(np.concatenate(routes))
    kw = dict(block=block, density=0.5, n_sample=64, n_probe=0, mode=1, softmax_scale=d ** -0.5)
    plan = B.sparsepr_plan_import(Q, K, V, dict(kv_assign=np.stack(aK), q_assign=np.stack(aQ), route_ptr=np.stack(ptr), route_idx=idx), **kw)
    O, Osp = B.sparsepr_attend(plan, Q, K, V, return_sparse=True)
    O2 = B.sparsepr_attend(plan, Q, K, V)                          # (without the float32 copy the output goes another way)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    for i in sorted({0, 1, heads - 1}):
        ref = orc.sparse_attention(to_np(Q[0, i]), to_np(K[0, i]), to_np(V[0, i]), aQ[i], aK[i], ptr[i], idx[i], d ** -0.5)
        for out in (O[0, i], Osp[0, i], O2[0, i]):
            assert_bf16_close(to_np(out), ref)                      # probabilities and output in bf16, sums in float32


@pytest.mark.parametrize("heads,N", [(1, 257), (148, 129), (74, 384), (37, 1000)])
def test_dense_pairs(heads, N):
    """One and two query tiles per CTA, the second one full, ragged (one row) and empty: two where one per CTA
    would make two rounds on 148 SMs and two make one."""
    gen = torch.Generator(device="cuda").manual_seed(N)
    Q, K, V = [torch.randn(1, heads, N, 128, device="cuda", generator=gen).bfloat16() for _ in range(3)]
    O = B.sparsepr_dense(Q, K, V, 128 ** -0.5)
    for i in sorted({0, heads - 1}):
        assert_bf16_close(to_np(O[0, i]), orc.dense_attention(to_np(Q[0, i]), to_np(K[0, i]), to_np(V[0, i]), 128 ** -0.5))


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def bnhd(gen, B_, H, N, d):
    return torch.randn(B_, N, H, d, device="cuda", generator=gen).bfloat16().transpose(1, 2)


@pytest.mark.parametrize("d,group", [(64, 1), (128, 1), (128, 4)])
@pytest.mark.parametrize("N", [129, 384, 1000])
def test_dense_pairs_batched(N, d, group):
    """Two query tiles per CTA with two batch entries, tensors stored as [B, N, H, d] and several query heads to a K/V head, on as
    many heads as make more than one round of single tiles on this GPU."""
    tiles = -(-N // 128)
    H = -(-2 * sms() // (2 * tiles) // 4) * 4                        # two rounds of tiles (or a little more), one of pairs
    gen = torch.Generator(device="cuda").manual_seed(N + d)
    Q, K, V = bnhd(gen, 2, H, N, d), bnhd(gen, 2, H // group, N, d), bnhd(gen, 2, H // group, N, d)
    O = B.sparsepr_dense(Q, K, V, d ** -0.5)
    assert O.stride() == Q.stride()
    for b, h in [(0, 0), (0, H - 1), (1, 1), (1, H // 2), (1, H - 1)]:
        assert_bf16_close(to_np(O[b, h]), orc.dense_attention(to_np(Q[b, h]), to_np(K[b, h // group]), to_np(V[b, h // group]), d ** -0.5))


@pytest.mark.parametrize("d,group", [(64, 1), (128, 1), (128, 4)])
def test_pairs_batched(d, group):
    """The list of pairs with two batch entries, [B, N, H, d] and grouped queries: enough rows for it on this GPU, 20 rounds of tiles
    (40 at d = 64)."""
    rng = np.random.default_rng(group)
    N, C = sum(SIZES), len(SIZES)
    H = -(-(20 if d == 128 else 40) * sms() * 128 // (2 * N) // 4) * 4 + 4
    gen = torch.Generator(device="cuda").manual_seed(group)
    Q, K, V = bnhd(gen, 2, H, N, d), bnhd(gen, 2, H // group, N, d), bnhd(gen, 2, H // group, N, d)
    aK = [rng.permutation(np.repeat(np.arange(C), rng.permutation(SIZES))) for _ in range(2 * H // group)]
    aQ, ptr, idx = [], [], []
    for i in range(2 * H):
        aQ.append(rng.permutation(np.repeat(np.arange(C), rng.permutation(SIZES))))
        full = int(np.argmax(np.bincount(aK[i // group], minlength=C)))
        routes = [np.unique(np.append(rng.choice(C, size=n, replace=False), full)) for n in rng.permutation([C] + list(range(1, C)))]
        ptr.append(np.concatenate([[0], np.cumsum([len(r) for r in routes])]))
        idx.append(np.concatenate(routes))
    kw = dict(block=-(-N // C), density=0.5, n_sample=64, n_probe=0, mode=1, softmax_scale=d ** -0.5)
    plan = B.sparsepr_plan_import(Q, K, V, dict(kv_assign=np.stack(aK), q_assign=np.stack(aQ), route_ptr=np.stack(ptr), route_idx=idx), **kw)
    O, Osp = B.sparsepr_attend(plan, Q, K, V, return_sparse=True)
    O2 = B.sparsepr_attend(plan, Q, K, V)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    for i in [0, 1, H - 1, H, 2 * H - 1]:
        b, h = divmod(i, H)
        kv = (K[b, h // group], V[b, h // group])
        ref = orc.sparse_attention(to_np(Q[b, h]), to_np(kv[0]), to_np(kv[1]), aQ[i], aK[i // group], ptr[i], idx[i], d ** -0.5)
        for out in (O[b, h], Osp[b, h], O2[b, h]):
            assert_bf16_close(to_np(out), ref)


@pytest.mark.parametrize("d", [64, 128])
def test_pairs_with_correction(d):
    """A fitted call whose tiles come in pairs, which hand their rows to the correction in two words, against calls on two heads of
    it, whose tiles come alone.  d = 64: float32 up to the rounding, which then differs for few elements; d = 128: bf16 probabilities."""
    N = 3100
    H = -(-(20 if d == 128 else 40) * sms() * 128 // N) + 1
    gen = torch.Generator(device="cuda").manual_seed(d)
    Q, K, V = [torch.randn(1, H, N, d, device="cuda", generator=gen).mul_(d ** -0.25).bfloat16() for _ in range(3)]
    kw = dict(Ck=8, Cq=8, density=0.5, n_sample=64, n_probe=16, softmax_scale=1.0, lam=10.0)     # groups of three tiles
    plan = B.sparsepr_plan(Q, K, V, **kw)
    O = B.sparsepr_attend(plan, Q, K, V)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    host = B.sparsepr_plan_export(plan)
    for hs in ([0, 1], [H // 2, H - 1]):
        q, k, v = [x[:, hs].contiguous() for x in (Q, K, V)]
        O2 = B.sparsepr_attend(B.sparsepr_plan_import(q, k, v, {n: a[hs] for n, a in host.items()}, **kw), q, k, v)
        assert_bf16_close(to_np(O[:, hs]), to_np(O2))
        if d == 64:
            assert (O[:, hs] != O2).double().mean() <= 5e-3
