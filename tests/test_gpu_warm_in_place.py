"""A warm plan made in the workspace of the plan that seeds it (destroyed before), with another number of k-means passes: the partition lies where the
seed lay, and it is the one that a workspace of its own gives."""
import ctypes as C

import pytest
import torch

from paper_2608_18484_b200 import binding as B

pytestmark = pytest.mark.gpu


def _plan(ws, Q, K, iters, seed=None):
    shape, params = B.make_shape(Q, K, K, Q), B.make_params(density=0.3, block=64, n_probe=32, kmeans_iters=iters, softmax_scale=1.0)
    assert B.lib().sparsepr_plan_workspace_bytes(C.byref(shape), C.byref(params)) <= ws.numel()
    h, a_k, a_q = C.c_void_p(), C.c_void_p(), C.c_void_p()
    args = (C.byref(shape), C.byref(params), Q.data_ptr(), K.data_ptr(), None)
    tail = (ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream, C.byref(h))
    code = B.lib().sparsepr_plan(*args, *tail) if seed is None else B.lib().sparsepr_plan_warm(*args, *seed, *tail)
    assert code == 0
    assert B.lib().sparsepr_plan_assignments(h, C.byref(a_k), C.byref(a_q)) == 0
    return h, (a_k, a_q)


def _partition(ws, ptrs, n):
    torch.cuda.synchronize()
    at = [p.value - ws.data_ptr() for p in ptrs]
    return [ws[o:o + 4 * n].view(torch.int32).clone() for o in at]


@pytest.mark.parametrize("iters", [2, 1, 40])
@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 128)])
def test_warm_plan_in_the_workspace_of_its_seed(dtype, d, iters):
    H, N = 24, 1411
    gen = torch.Generator(device="cuda").manual_seed(d)
    Q, K, Q2, K2 = [torch.randn(1, H, N, d, device="cuda", generator=gen).to(dtype) for _ in range(4)]
    size = max(B.lib().sparsepr_plan_workspace_bytes(C.byref(B.make_shape(Q, K, K, Q)), C.byref(B.make_params(block=64, n_probe=32, kmeans_iters=t)))
               for t in (8, iters))
    ws, other = [torch.zeros(size, dtype=torch.uint8, device="cuda") for _ in range(2)]
    cold, seed = _plan(ws, Q, K, 8)
    own, ptrs = _plan(other, Q2, K2, iters, seed)
    want = _partition(other, ptrs, H * N)
    B.lib().sparsepr_plan_destroy(own)
    torch.cuda.synchronize()
    B.lib().sparsepr_plan_destroy(cold)
    warm, ptrs = _plan(ws, Q2, K2, iters, seed)
    got = _partition(ws, ptrs, H * N)
    B.lib().sparsepr_plan_destroy(warm)
    assert [p.value for p in ptrs] == [p.value for p in seed]
    for g, w in zip(got, want):
        assert torch.equal(g, w)
