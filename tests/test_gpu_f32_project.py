"""float32 response projections with one row per thread (few rows in the call) and two (many): the plan of a head is the same
whole numbers whichever of them its call takes, at row counts off the 64 and 256 rows of their CTAs."""
import numpy as np
import pytest
import torch

from paper_2608_18484_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("N", [577, 701, 1025])
def test_head_alone_and_among_many(N, d):
    heads = 4 * 148 * 64 // N + 2
    gen = torch.Generator(device="cuda").manual_seed(N + d)
    Q, K, V = [torch.randn(1, heads, N, d, device="cuda", generator=gen) for _ in range(3)]
    kw = dict(density=0.3, block=32, n_sample=64, n_probe=16, softmax_scale=d ** -0.5)
    one = [x[:, :1].contiguous() for x in (Q, K, V)]
    few, many = [B.sparsepr_plan_export(B.sparsepr_plan(*x, **kw)) for x in (one, (Q, K, V))]
    for k in ("kv_assign", "q_assign", "route_ptr", "probe_idx"):
        assert np.array_equal(few[k][0], many[k][0]), k
    n = few["route_ptr"][0][-1]
    assert np.array_equal(few["route_idx"][0][:n], many["route_idx"][0][:n])
