"""Steps inside a caller's stream capture: the replayed graph gives the direct call's field, bit for bit."""
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP32, GP_FP64, Plan, field_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,dtype", [(GP_FP64, torch.complex128), (GP_FP32, torch.complex64)])
@pytest.mark.parametrize("n,steps", [(16, 1), (32, 8), (96, 5)])
def test_captured_steps(prec, dtype, n, steps):
    stream = torch.cuda.Stream()
    plan = Plan(field_params(n, 0.004, xi_over_dx=1.5, precision=prec), stream=stream)
    g = torch.Generator(device="cuda").manual_seed(n)
    start = torch.view_as_complex(torch.randn(n, n, n, 2, generator=g, device="cuda", dtype=dtype.to_real())).contiguous()
    ref, x, before = start.clone(), start.clone(), start.clone()
    torch.cuda.synchronize()
    plan.step([ref], steps)           # tables and kernel attributes are set up outside the capture
    plan.sync()
    for _ in range(2):                # the second capture finds the same field and step count as the first
        x.copy_(start)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            plan.step([x], steps)
        assert torch.equal(x, start)  # captured, not run
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(x, ref)
    for _ in range(3):                # the plan's own graphs as before
        before.copy_(start)
        torch.cuda.synchronize()
        plan.step([before], steps)
        plan.sync()
        assert torch.equal(before, ref)
