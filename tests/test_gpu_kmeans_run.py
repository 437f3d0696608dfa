"""k-means runs whose passes are one kernel (few rows and centroids per head): a head's row tiles over a cluster of CTAs, tiles kept in shared memory or
fetched again, one and two chunks of centroids, more moved rows than its list holds, first sums in several windows, and rows that are all undecided.
The query partition against Lloyd's iteration in float64 on the features that the plan exports; as in the other k-means tests the centroids of the two
differ by a float32 rounding (6e-8), and one row in about a million is that near a tie: at most one row per head differs."""
import numpy as np
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B

pytestmark = pytest.mark.gpu


def _check(plan, C, iters, heads, N, init=None):
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    a = B.sparsepr_plan_export(plan)["q_assign"]
    phi = B.sparsepr_plan_export_features(plan, fields=("phi_Q",))["phi_Q"]
    for h in heads:
        ref, _ = orc.kmeans(phi[h], C, orc.stride_sample(C, N, 0, orc.TAG_Q_INIT, h), iters, None if init is None else init[h])
        assert (a[h] != ref).sum() <= 1, (h, int((a[h] != ref).sum()))
    return a


@pytest.mark.parametrize("H,N,C,iters,rQ", [
    (1, 40, 3, 6, 64),            # less than a row tile
    (2, 127, 16, 5, 17), (1, 129, 17, 1, 48), (3, 385, 1, 3, 64),
    (2, 4097, 128, 8, 48),        # one chunk of centroids, three tiles per CTA
    (1, 8193, 64, 4, 64),         # 65 tiles, five per CTA: fetched again in every pass
    (2, 2049, 129, 5, 64),        # a second chunk of one centroid
    (15, 6001, 256, 3, 33),       # two full chunks
    (22, 16384, 128, 3, 16),      # 22 tiles per CTA: first sums in two windows
])
def test_runs_of_all_shapes(H, N, C, iters, rQ):
    gen = torch.Generator(device="cuda").manual_seed(N)
    Q, K = [torch.randn(1, H, N, 128, device="cuda", generator=gen).mul_(128 ** -0.25).bfloat16() for _ in range(2)]
    plan = B.sparsepr_plan(Q, K, K, density=0.5, Ck=C, Cq=C, rQ=rQ, n_sample=64, n_probe=16, softmax_scale=1.0, kmeans_iters=iters)
    _check(plan, C, iters, sorted({0, H - 1}), N)


@pytest.mark.parametrize("H,N,C", [(2, 3000, 48), (22, 16384, 128)])
def test_a_warm_run_from_a_foreign_partition_moves_most_rows(H, N, C):
    gen = torch.Generator(device="cuda").manual_seed(N)
    Q0, Q, K = [torch.randn(1, H, N, 64, device="cuda", generator=gen).mul_(64 ** -0.25).bfloat16() for _ in range(3)]
    kw = dict(density=0.5, Ck=C, Cq=C, n_sample=64, n_probe=16, softmax_scale=1.0)
    prev = B.sparsepr_plan(Q0, K, K, kmeans_iters=2, **kw)
    init = B.sparsepr_plan_export(prev)["q_assign"]
    plan = B.sparsepr_plan(Q, K, K, params=B.make_params(kmeans_iters=3, **kw), warm_from=prev)
    _check(plan, C, 3, sorted({0, H - 1}), N, init)


def test_rows_between_equal_centroids_and_the_fixed_point():
    """Five distinct rows, sixteen initial centroids among them: rows have several nearest centroids, the lowest one takes them all, and the run ends
    once a pass changes nothing."""
    N, C = 2003, 16
    gen = torch.Generator(device="cuda").manual_seed(5)
    rows = torch.randn(5, 128, device="cuda", generator=gen)
    Q = rows[torch.arange(N, device="cuda") % 5][None, None].bfloat16()
    K = torch.randn(1, 1, N, 128, device="cuda", generator=gen).bfloat16()
    plan = B.sparsepr_plan(Q, K, K, density=0.5, Ck=C, Cq=C, n_sample=64, n_probe=16, softmax_scale=0.1, kmeans_iters=8)
    a = _check(plan, C, 8, [0], N)
    assert len(np.unique(a[0])) <= 5 and B.sparsepr_plan_stats(plan)["kmeans_passes_q"] < 8
