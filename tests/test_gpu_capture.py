"""Calls recorded into a CUDA graph: attend on a plan that was made before the capture (kept over several steps, the plan call just
queued or long complete), plan and attend in one graph, and attend outside the graph that made its plan."""
import pytest
import torch

from paper_2608_18484_b200 import binding as B

pytestmark = pytest.mark.gpu

KINDS = [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 64)]


@pytest.mark.parametrize("M,mode", [(64, 0), (0, 0), (64, 1)], ids=["fitted", "no-probes", "hard"])
@pytest.mark.parametrize("dtype,d", KINDS, ids=["bf16-128", "bf16-64", "f32-64"])
def test_attend_under_capture(dtype, d, M, mode):
    gen = torch.Generator(device="cuda").manual_seed(d)
    Q, K, V = [(torch.randn(1, 2, 4096, d, generator=gen, device="cuda") * d ** -0.25).to(dtype) for _ in range(3)]
    kw = dict(block=64, density=0.3, n_sample=64, n_probe=M, mode=mode, softmax_scale=1.0)
    ref = B.sparsepr_attend(B.sparsepr_plan(Q, K, V, **kw), Q, K, V)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        for attended in (False, True):
            plan = B.sparsepr_plan(Q, K, V, **kw)
            out = torch.zeros_like(Q)
            plan.attend_workspace = torch.empty(plan.attend_bytes, dtype=torch.uint8, device="cuda")
            if attended:
                B.sparsepr_attend(plan, Q, K, V, out=out)
                out.zero_()
            graph = torch.cuda.CUDAGraph()
            graph.capture_begin()                              # (unlike torch.cuda.graph without waiting for the GPU)
            B.sparsepr_attend(plan, Q, K, V, out=out)
            graph.capture_end()
            for _ in range(2):
                out.zero_()
                graph.replay()
                assert torch.equal(out, ref)
            out.zero_()
            B.sparsepr_attend(plan, Q, K, V, out=out)          # and outside again
            assert torch.equal(out, ref) and B.sparsepr_plan_stats(plan)["device_error"] == 0
            del graph

        out = torch.zeros_like(Q)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            plan = B.sparsepr_plan(Q, K, V, **kw)
            B.sparsepr_attend(plan, Q, K, V, out=out)
        graph.replay()
        assert torch.equal(out, ref)
        out.zero_()
        B.sparsepr_attend(plan, Q, K, V, out=out)
        assert torch.equal(out, ref)
        second = torch.cuda.CUDAGraph()
        with torch.cuda.graph(second, stream=stream):
            B.sparsepr_attend(plan, Q, K, V, out=out)
        out.zero_()
        second.replay()
        assert torch.equal(out, ref)
        torch.cuda.synchronize()
