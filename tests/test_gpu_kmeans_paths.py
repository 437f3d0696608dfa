"""Which kernels a plan's k-means takes, and that the partition of a head does not depend on it: a head alone goes through one kernel for the whole run,
among more heads than there are SMs through separate passes."""
import numpy as np
import pytest
import torch
from torch.profiler import ProfilerActivity, profile

import tests.test_gpu_kmeans_run as runs
from paper_2608_18484_b200 import binding as B

pytestmark = pytest.mark.gpu

SHAPES = next(m.args[1] for m in runs.test_runs_of_all_shapes.pytestmark if m.name == "parametrize")


def _plan(*args, **kw):
    """The plan and the numbers of its launches of the run kernel and of separate assignment passes."""
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        plan = B.sparsepr_plan(*args, **kw)
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA]
    return plan, [sum(k in n for n in names) for k in ("k_kmeans_run", "k_kmeans_assign_tc")]


@pytest.mark.parametrize("H,N,C,iters,rQ", SHAPES)
def test_the_shapes_of_the_run_kernel_take_it(H, N, C, iters, rQ):
    x = torch.randn(1, H, N, 128, device="cuda").bfloat16()
    launched = _plan(x, x, x, density=0.5, Ck=C, Cq=C, rQ=rQ, n_sample=64, n_probe=16, softmax_scale=1.0, kmeans_iters=iters)[1]
    assert launched == [2, 0]                                    # keys and queries


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 128)])
@pytest.mark.parametrize("N,C", [(1003, 33), (2049, 129), (700, 256)])
def test_head_alone_and_among_many(N, C, dtype, d):
    heads = torch.cuda.get_device_properties(0).multi_processor_count + 2
    gen = torch.Generator(device="cuda").manual_seed(N + d)
    Q, K = [torch.randn(1, heads, N, d, device="cuda", generator=gen).mul_(d ** -0.25).to(dtype) for _ in range(2)]
    kw = dict(density=0.5, Ck=C, Cq=C, n_sample=64, n_probe=16, softmax_scale=1.0)
    many, launched = _plan(Q, K, K, **kw)
    assert launched[0] == 0 and launched[1] > 2
    many = B.sparsepr_plan_export(many)
    for h in (0, heads - 1):
        one = [x[:, h:h + 1].contiguous() for x in (Q, K, K)]
        alone, launched = _plan(*one, head_offset=h, **kw)
        assert launched == [2, 0]
        alone = B.sparsepr_plan_export(alone)
        for k in ("kv_assign", "q_assign"):
            assert np.array_equal(alone[k][0], many[k][h]), (h, k, int((alone[k][0] != many[k][h]).sum()))
