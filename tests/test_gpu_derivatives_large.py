"""Float32 diagnostics and structure functions at 512 and 1024 points against the float64 ones.

Tolerance: the 2e-5 of the shorter lengths.  A gradient's float32 rounding, 1e-7 of the field, is amplified by up to
N / 2 over the field's scale (here modes up to 6 and white noise): 1e-5 of the smooth gradient at a point, and the
sums average over N^3 points.
"""
import numpy as np
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP32, GP_FP64, Plan, field_params

pytestmark = pytest.mark.gpu
TOL = 2e-5


@pytest.mark.parametrize("n,white", [(512, True), (512, False), (1024, True)])
def test_float32_against_float64(n, white):
    g = torch.Generator(device="cuda").manual_seed(n + white)
    psi = torch.empty(n, n, n, dtype=torch.complex64, device="cuda")
    if white:
        torch.view_as_real(psi).normal_(0.0, 0.2, generator=g)
        psi += 1.0
    else:
        x = 2 * np.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n
        cx, cy, cz = torch.cos(2 * x)[None, None, :], torch.sin(3 * x)[None, :, None], torch.cos(x)[:, None, None]
        ph = 2.0 * cx * cy + cz * torch.sin(6 * x)[None, None, :] + x[None, None, :]
        psi.copy_(torch.polar((1.0 + 0.3 * cy * cz).expand_as(ph), ph))
        del ph
    got, ref = [], []
    for out, prec in ((got, GP_FP32), (ref, GP_FP64)):
        plan = Plan(field_params(n, 0.001, xi_over_dx=1.5, precision=prec))
        f = psi if prec == GP_FP32 else psi.to(torch.complex128)
        d, spec = plan.diagnostics(0, f)
        out += [d, spec, plan.structure_function(0, f, order=2)]
        del plan, f
    torch.cuda.empty_cache()
    for k, v in ref[0].items():
        assert abs(got[0][k] - v) <= TOL * max(abs(v), 1e-3 * abs(ref[0]["E"])), k
    for k, v in ref[1].items():
        assert np.max(np.abs(got[1][k] - v)) <= 10 * TOL * max(np.max(np.abs(v)), 1e-3 * abs(ref[0]["E"])), k
    assert np.max(np.abs(got[2] - ref[2])) <= 10 * TOL * np.max(np.abs(ref[2]))
