"""An adjoint call that cannot get its kinetic tables leaves the cotangent as it was.

cudaMalloc is refused while the calling thread captures another stream (a host error, nothing is launched into
the capture): the tables of a step back do not exist then, those of the forward steps do.
"""
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP32, GP_FP64, GP_SPLIT_KNK, GP_SPLIT_NKN, GPError, Plan, field_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,dtype", [(GP_FP32, torch.complex64), (GP_FP64, torch.complex128)])
@pytest.mark.parametrize("split", [GP_SPLIT_NKN, GP_SPLIT_KNK])
def test_cotangent_kept_when_tables_are_missing(prec, dtype, split):
    n = 32
    mine = torch.cuda.Stream()
    plan = Plan([field_params(n, dt, xi_over_dx=1.5, precision=prec, split=split) for dt in (0.004, 0.002)], stream=mine)
    psi = torch.ones(n, n, n, dtype=dtype, device="cuda")
    lam = torch.full_like(psi, 0.5 + 0.25j)
    torch.cuda.synchronize()
    plan.adjoint_step(0, psi, lam, 3)                       # workspace and kernels of the other field
    plan.step([psi.clone(), psi.clone()], 2)                # this field's forward tables
    plan.sync()
    keep = lam.clone()
    torch.cuda.synchronize()
    graph, other = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    status = None
    with torch.cuda.stream(other):
        graph.capture_begin()
        try:
            plan.adjoint_step(1, psi, lam, 3)
        except GPError as e:
            status = e.status
        try:
            graph.capture_end()
        except Exception:  # noqa: BLE001 -- the refused call may have ended the capture
            pass
    torch.cuda.synchronize()
    kept = torch.equal(lam, keep)
    try:
        plan.step([psi.clone(), psi.clone()], 1)            # reports the refused allocation's pending error
    except GPError:
        pass
    plan.step([psi.clone(), psi.clone()], 1)
    plan.sync()
    assert status == 3 and kept                             # GP_ERR_OOM


def test_shared_float64_fields_kept_when_tables_are_missing():
    """The same for float64 fields that share memory: the second field's tables cannot be had, the first has its own."""
    n = 32
    plan = Plan([field_params(n, dt, xi_over_dx=1.5, precision=GP_FP64) for dt in (0.004, 0.002)], stream=torch.cuda.Stream())
    x = torch.full((n, n, n), 0.5 + 0.25j, dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    plan.adjoint_step(0, x.clone(), x.clone(), 1)           # the first field's tables
    plan.sync()
    keep = x.clone()
    torch.cuda.synchronize()
    graph, other = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    status = None
    with torch.cuda.stream(other):
        graph.capture_begin()
        try:
            plan.step([x, x], 2)
        except GPError as e:
            status = e.status
        try:
            graph.capture_end()
        except Exception:  # noqa: BLE001
            pass
    torch.cuda.synchronize()
    kept = torch.equal(x, keep)
    try:
        plan.step([x, x], 1)                                # reports the refused allocation's pending error
    except GPError:
        pass
    plan.step([x, x], 1)
    plan.sync()
    assert status == 3 and kept
