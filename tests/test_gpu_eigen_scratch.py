"""Feature maps of several heads whose scratch holds what other solves left there: NaN, then a plan whose spectra have other means.  The maps,
their scale included, against the eigen-decomposition in float64; the bounds are those of the metrics at the edges of the reduction."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import sparsepr_oracle as orc
from paper_2608_18484_b200 import binding as B
from tests.gpu_util import to_np

pytestmark = pytest.mark.gpu


def _plan(ws, Q, K, params):
    shape, h = B.make_shape(Q, K, K, Q), C.c_void_p()
    size = B.lib().sparsepr_plan_workspace_bytes(C.byref(shape), C.byref(params))
    assert size <= ws.numel()
    assert B.lib().sparsepr_plan(C.byref(shape), C.byref(params), Q.data_ptr(), K.data_ptr(), None, ws.data_ptr(), ws.numel(),
                                 torch.cuda.current_stream().cuda_stream, C.byref(h)) == 0
    return B.Plan(h, ws, shape, params, 0)


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 128), (torch.float32, 64)])
def test_maps_do_not_depend_on_what_the_scratch_held(dtype, d):
    H, N, r = 5, 8 * d, 48
    gen = torch.Generator(device="cuda").manual_seed(d)
    params = B.make_params(density=0.5, Ck=160, Cq=32, n_sample=N, n_probe=16, rK=r, rQ=r, softmax_scale=1.0)
    shape_of = torch.empty(1, H, N, d, device="cuda", dtype=dtype)
    shape = B.make_shape(shape_of, shape_of, shape_of, shape_of)
    ws = torch.full((B.lib().sparsepr_plan_workspace_bytes(C.byref(shape), C.byref(params)),), 0xFF, dtype=torch.uint8, device="cuda")
    for decay in (0.97, 0.9, 0.99):                             # spectra of different shapes, so of different means
        columns = decay ** torch.arange(d, device="cuda")
        columns[r:] *= 0.25                                     # the retained eigenvalues lie apart from the others
        Q, K = [(torch.randn(1, H, N, d, device="cuda", generator=gen) * columns).to(dtype) for _ in range(2)]
        plan = _plan(ws, Q, K, params)
        assert B.sparsepr_plan_stats(plan)["device_error"] == 0
        got = B.sparsepr_plan_export_features(plan, fields=("F_K", "F_Q", "kappa"))
        assign = B.sparsepr_plan_export(plan)["kv_assign"]
        for h in range(H):
            n_k = np.bincount(assign[h], minlength=got["kappa"][h].shape[0])
            for name, metric in (("F_K", orc.key_response_metric(to_np(Q[0, h]))), ("F_Q", orc.query_response_metric(got["kappa"][h], n_k))):
                F, ref = got[name][h].astype(np.float64), orc.eig_feature_map(metric, r)[0]
                err = np.linalg.norm(F @ F.T - ref @ ref.T) / np.linalg.norm(ref @ ref.T)
                assert err <= (1e-4 if dtype == torch.bfloat16 else 1e-5), (name, decay, h, err)
        del plan
