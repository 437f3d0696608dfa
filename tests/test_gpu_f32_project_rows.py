"""float32 response projections: the rows per thread that a call takes follow from the CTAs that one SM gets of either kind, on any number of SMs,
and the plan of a head is the same whole numbers whichever it is."""
import re

import numpy as np
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

from paper_2608_18484_b200 import binding as B

pytestmark = pytest.mark.gpu


def _plan(Q, K, **kw):
    """The exported plan and the rows per thread of its projections (the kernel's last template argument), keys first."""
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        plan = B.sparsepr_plan(Q, K, K, block=32, density=0.3, n_sample=64, n_probe=16, softmax_scale=Q.shape[-1] ** -0.5, **kw)
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA]
    return B.sparsepr_plan_export(plan), [int(m.group(1)) for n in names for m in [re.search(r"\bk_project<[^>]*?(\d)>", n)] if m]


def _inputs(heads, N, d):
    gen = torch.Generator(device="cuda").manual_seed(N + d)
    return [torch.randn(1, heads, N, d, device="cuda", generator=gen) for _ in range(2)]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("per_sm,rows", [(4, 2), (5, 1)])       # CTAs of 64 rows on an SM: four beside one of 256, five beside two
def test_rows_per_thread_of_two_heads(per_sm, rows, d):
    N = 32 * per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    Q, K = _inputs(2, N, d)
    assert _plan(Q, K, Ck=32, Cq=32, kmeans_iters=1)[1] == [rows, rows]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("N", [577, 701, 1025])
def test_one_row_alone_and_two_among_many(N, d):
    heads = 8 * torch.cuda.get_device_properties(0).multi_processor_count * 64 // N + 2
    Q, K = _inputs(heads, N, d)
    many, rows = _plan(Q, K)
    assert rows == [2, 2]
    few, rows = _plan(Q[:, :1].contiguous(), K[:, :1].contiguous())
    assert rows == [1, 1]
    for k in ("kv_assign", "q_assign", "route_ptr", "probe_idx"):
        assert np.array_equal(few[k][0], many[k][0]), k
    n = few["route_ptr"][0][-1]
    assert np.array_equal(few["route_idx"][0][:n], many["route_idx"][0][:n])
