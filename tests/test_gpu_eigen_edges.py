"""Feature maps of metrics at the edges of the Householder reduction: nothing to reduce (a diagonal metric: every step is skipped), steps that
are skipped now and then (2 x 2 blocks), and a metric of low rank beside a diagonal.  F F^T against the eigen-decomposition in float64."""
import numpy as np
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B
from tests.gpu_util import to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["diagonal", "blocks", "low-rank"])
@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 128), (torch.float32, 64)])
def test_feature_map_of_special_metrics(kind, dtype, d):
    N, r = 4 * d, 48
    n = np.arange(N)
    X = np.zeros((N, d))
    X[n, n % d] = 0.5 + (d - n % d) / 16                        # the retained eigenvalues lie apart from the others
    if kind == "blocks":
        X[n, (n % d) ^ 1] = 0.25 * (n // d)
    if kind == "low-rank":
        X[::2] += 2.0 * np.sin(np.outer(n[::2] % 3 + 1, np.arange(d)))
    gen = torch.Generator(device="cuda").manual_seed(d)
    K, V = [torch.randn(1, 1, N, d, device="cuda", generator=gen).to(dtype) for _ in range(2)]
    Q = torch.from_numpy(X)[None, None].to("cuda", dtype)
    plan = B.sparsepr_plan(Q, K, V, density=0.5, block=64, n_sample=N, n_probe=16, rK=r, softmax_scale=1.0)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    F = B.sparsepr_plan_export_features(plan, fields=("F_K",))["F_K"][0].astype(np.float64)
    ref = orc.eig_feature_map(orc.key_response_metric(to_np(Q[0, 0])), r)[0]
    err = np.linalg.norm(F @ F.T - ref @ ref.T) / np.linalg.norm(ref @ ref.T)
    assert err <= (1e-4 if dtype == torch.bfloat16 else 1e-5), err
