"""Route selection of heads whose score matrix fits the registers of one CTA (up to 128 and 160 groups) and the first sizes beyond, against the
oracle: no, few and many equal scores at the cut, empty groups, budgets of nothing and of everything, costs beyond 32 bits."""
import numpy as np
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Cq,Ck", [(1, 1), (16, 33), (17, 128), (128, 128), (129, 5), (3, 160), (160, 160), (161, 160)])
@pytest.mark.parametrize("levels,size", [(0, 300), (64, 300), (2, 40), (0, 200000)])
def test_selection_in_registers(Cq, Ck, levels, size):
    rng = np.random.default_rng(1000 * Cq + Ck + levels)
    score = rng.random((Cq, Ck)) ** 4
    if levels:
        score = np.round(score * levels) / levels                # cells of score 0 among them
    score = score.astype(np.float32)
    n_q, n_k = [(rng.integers(0, size, c) * (rng.random(c) > 0.2)).astype(np.int32) for c in (Cq, Ck)]
    total = int(n_q.astype(np.int64).sum() * n_k.astype(np.int64).sum())
    for budget, everything in [(0, False), (total // 7, False), (total // 2, False), (total - 1, False), (total, False), (0, True)]:
        ptr, idx, pairs = B.sparsepr_stage_route(torch.from_numpy(score).cuda(), torch.from_numpy(n_q).cuda(), torch.from_numpy(n_k).cuda(),
                                                 max(budget, 0), select_all=everything)
        p0, i0, pr0 = orc.route_select(score, n_q, n_k, max(budget, 0), select_all=everything)
        ptr, idx = ptr.cpu().numpy(), idx.cpu().numpy()
        assert np.array_equal(ptr, p0) and np.array_equal(idx[:ptr[-1]], i0) and int(pairs.item()) == pr0
