"""The float32 adjoint and imaginary-time steps at 512 and 1024 points (kernels with capped registers of their own)
against the float64 ones.

Tolerance: the 2e-5 of the shorter lengths (a handful of steps of about 3e-7 each; energies are sums over N^3 points).
"""
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP32, GP_FP64, GP_SPLIT_KNK, GP_SPLIT_NKN, Plan, field_params

pytestmark = pytest.mark.gpu
TOL = 2e-5


def _field(n, seed, mean=1.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.empty(n, n, n, dtype=torch.complex64, device="cuda")
    torch.view_as_real(x).normal_(0.0, 0.2, generator=g)
    return x.add_(mean)


def _err(a, b):
    d = torch.linalg.vector_norm(b).item()
    return torch.linalg.vector_norm(b.sub_(a)).item() / d     # b is overwritten


@pytest.mark.parametrize("n,split,m", [(512, GP_SPLIT_NKN, 3), (512, GP_SPLIT_KNK, 3), (1024, GP_SPLIT_NKN, 2), (1024, GP_SPLIT_KNK, 1)])
def test_adjoint(n, split, m):
    psi, lam0 = _field(n, 1), _field(n, 2, 0.0)
    out = []
    for prec, dt in ((GP_FP32, torch.complex64), (GP_FP64, torch.complex128)):
        plan = Plan(field_params(n, 0.0005, xi_over_dx=1.5, precision=prec, split=split))
        lam = lam0.to(dt, copy=True)
        plan.adjoint_step(0, psi.to(dt), lam, m)
        plan.sync()
        out.append(lam)
        del plan, lam
    err = _err(*out)
    del out
    torch.cuda.empty_cache()
    assert err < TOL, err


@pytest.mark.parametrize("flow", [0, 1, 2])
def test_imaginary_time_at_1024(flow):
    n = 1024
    start, out, energy = _field(n, 3), [], []
    for prec, dt in ((GP_FP32, torch.complex64), (GP_FP64, torch.complex128)):
        plan = Plan(field_params(n, 0.01, alpha=0.05, beta=20.0, precision=prec))
        x = start.to(dt, copy=True)
        energy.append(plan.argle(0, x, flow, 1e-3, 2))
        out.append(x)
        del plan, x
    err = _err(*out)
    del out
    torch.cuda.empty_cache()
    assert err < TOL and abs(energy[0] - energy[1]) < TOL * abs(energy[1]), (err, energy)
