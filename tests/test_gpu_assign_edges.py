"""Assignment at the edges of the tensor-core kernel's splits: groups of 16 columns, chunks of 128 centroids (two of them
resident, more of them streamed), row tiles of 128 in pairs, feature widths of 16 to 64; and a k-means run whose sums are
formed once and then updated, which must follow the definition pass by pass."""
import numpy as np
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,C,r", [(1, 1, 1), (127, 15, 16), (129, 16, 17), (385, 17, 48), (257, 33, 48), (640, 127, 64), (2049, 128, 64),
                                   (2050, 129, 33), (3000, 255, 64), (3001, 256, 48), (3100, 257, 64), (3333, 385, 64),
                                   (5000, 1000, 32), (9000, 2048, 64)])
def test_assign_at_the_edges(n, C, r):
    rng = np.random.default_rng(n * 7 + C)
    X = rng.normal(size=(n, r)).astype(np.float32)
    mu = (X[rng.integers(0, n, C)] + 0.2 * rng.normal(size=(C, r))).astype(np.float32)
    if C > 4:
        mu[C // 2] = mu[1]                                   # a tie: the lowest id wins
    a = B.sparsepr_stage_assign(torch.from_numpy(X).cuda(), torch.from_numpy(mu).cuda()).cpu().numpy()
    assert np.array_equal(a, orc.kmeans_assign(X, mu))


@pytest.mark.parametrize("r", [16, 48, 64])
def test_assign_where_the_scores_are_least_exact(r):
    """Decisions against float64 on rows whose scores lose most: large norms with small differences, terms that cancel, words of the
    split at their worst, terms just below the last place of a large one, and centroid pairs that lie nearly alike about the rows."""
    rng = np.random.default_rng(r)
    n, C = 3000, 150
    N = lambda *s: rng.normal(size=s)
    worst = 1 + 2.0 ** -8 - 2.0 ** -17
    small = lambda k: np.concatenate([np.ones((k, 1)), 2.0 ** -11 * (1 + rng.random((k, r - 1)))], 1)
    mid = N(C // 2, r)
    off = 1e-4 * N(C // 2, r)
    cases = [(N(n, r) + 100 / r ** 0.5, N(C, r) + 100 / r ** 0.5),
             (np.sign(N(n, r)) * worst * 2.0 ** rng.integers(-6, 7, (n, r)), np.sign(N(C, r)) * worst * 2.0 ** rng.integers(-6, 7, (C, r))),
             (small(n), -small(C)), (100 * N(n, r), 1e-3 * N(C, r)), (1e-3 * N(n, r), 100 * N(C, r)),
             (mid[rng.integers(0, C // 2, n)] + 1e-3 * N(n, r), np.concatenate([mid + off, mid - off]))]
    for X, mu in cases:
        X, mu = X.astype(np.float32), mu.astype(np.float32)
        a = B.sparsepr_stage_assign(torch.from_numpy(X).cuda(), torch.from_numpy(mu).cuda()).cpu().numpy()
        assert np.array_equal(a, orc.kmeans_assign(X, mu))


@pytest.mark.parametrize("N,C,iters", [(1000, 130, 8), (2047, 128, 5), (4100, 300, 8)])
def test_updated_sums_follow_the_definition(N, C, iters):
    """Query partition of a plan against Lloyd's iteration in float64 on the features the plan exports.  The centroids of the
    two differ by a float32 rounding (6e-8), and one row in about a million is that near a tie: at most one row differs."""
    gen = torch.Generator(device="cuda").manual_seed(N)
    Q, K = [torch.randn(1, 2, N, 128, device="cuda", generator=gen).mul_(128 ** -0.25).bfloat16() for _ in range(2)]
    kw = dict(density=0.5, Ck=C, Cq=C, n_sample=64, n_probe=16, softmax_scale=1.0, kmeans_iters=iters)
    plan = B.sparsepr_plan(Q, K, K, **kw)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    a = B.sparsepr_plan_export(plan)["q_assign"]
    phi = B.sparsepr_plan_export_features(plan, fields=("phi_Q",))["phi_Q"]
    for h in range(2):
        ref, _ = orc.kmeans(phi[h], C, orc.stride_sample(C, N, 0, orc.TAG_Q_INIT, h), iters)
        assert (a[h] != ref).sum() <= 1, (a[h] != ref).sum()
