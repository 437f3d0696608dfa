"""Several threads with streams and workspaces of their own on one kept plan: the plan's auxiliary streams and events are shared."""
import ctypes as C
import threading

import pytest
import torch

from paper_2608_18484_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [(torch.float32, 64), (torch.bfloat16, 64), (torch.bfloat16, 128)], ids=["f32", "bf16-64", "bf16-128"])
def test_attend_from_threads(dtype, d):
    gen = torch.Generator(device="cuda").manual_seed(3)
    sets = [[(torch.randn(1, 2, 2048, d, generator=gen, device="cuda") * d ** -0.25).to(dtype) for _ in range(3)] for _ in range(2)]
    plan = B.sparsepr_plan(*sets[0], block=64, density=0.3, n_sample=64, n_probe=64, softmax_scale=1.0)
    refs = [B.sparsepr_attend(plan, *s) for s in sets]
    torch.cuda.synchronize()
    L, wrong = B.lib(), []

    def work(k):
        stream = torch.cuda.Stream()
        ws = torch.empty(plan.attend_bytes, dtype=torch.uint8, device="cuda")
        outs = [torch.empty_like(refs[0]) for _ in range(60)]
        torch.cuda.synchronize()
        for n, out in enumerate(outs):                           # inputs that change from call to call
            q, k_, v = sets[(n + k) % 2]
            if L.sparsepr_attend(plan.handle, q.data_ptr(), k_.data_ptr(), v.data_ptr(), out.data_ptr(), None, ws.data_ptr(), C.c_size_t(ws.numel()),
                                 C.c_void_p(stream.cuda_stream)) != 0:
                wrong.append("status")
        stream.synchronize()
        wrong.extend(n for n, out in enumerate(outs) if not torch.equal(out, refs[(n + k) % 2]))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong and B.sparsepr_plan_stats(plan)["device_error"] == 0
