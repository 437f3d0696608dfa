"""Feature maps of metrics whose rank is below the number of retained directions: their null vectors are one group of equal eigenvalues for the
orthogonalisation, and a matrix whose group does not come out orthogonal is left to the Jacobi kernel (in float32: some of rank 1
at d = 128, of several ranks at d = 64).  F F^T against the decomposition in float64."""
import numpy as np
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B
from tests.gpu_util import to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rank,r", [(1, 2), (1, 64), (2, 64), (25, 48), (40, 64), (63, 64)])
@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 128), (torch.float32, 64)])
def test_rank_below_the_retained_directions(dtype, d, rank, r):
    H, N = 3, 512
    gen = torch.Generator(device="cuda").manual_seed(100 * rank + d)
    rows = torch.randn(H, rank, d, device="cuda", generator=gen).to(dtype)
    Q = rows[:, torch.arange(N, device="cuda") % rank][None].contiguous()
    K = torch.randn(1, H, N, d, device="cuda", generator=gen).to(dtype)
    plan = B.sparsepr_plan(Q, K, K, density=0.5, block=64, n_sample=N, n_probe=16, rK=r, softmax_scale=1.0)
    assert B.sparsepr_plan_stats(plan)["device_error"] == 0
    got = B.sparsepr_plan_export_features(plan, fields=("F_K",))["F_K"].astype(np.float64)
    for h in range(H):
        F, ref = got[h], orc.eig_feature_map(orc.key_response_metric(to_np(Q[0, h])), r)[0]
        err = np.linalg.norm(F @ F.T - ref @ ref.T) / np.linalg.norm(ref @ ref.T)
        # float32 tensors (float64 solver): 1e-5, the bound of their metrics of full rank.  bf16 tensors: a column of a matrix that is left to the Jacobi
        # kernel goes through at most 20 sweeps of d - 1 rotations in float32, each off by up to 2^-23
        assert err <= (20 * (d - 1) * 2.0 ** -23 if dtype == torch.bfloat16 else 1e-5), (h, err)
