"""The ring field of a float32 plan (formed in twofold float32) against that of a float64 plan.

Tolerance: the field's components are at most 1 and rounded to float32 once (6e-8); the product of 40
factors of about 2^-40 relative error each adds less than 1e-10.  1.2e-7 is one unit in the last place.
"""
import math

import pytest
import torch

from paper_2003_03590_gb300 import GP_FP32, GP_FP64, Plan, field_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 12, 64, 96])
@pytest.mark.parametrize("count,r0,r1,xi_dx", [(0, 1.0, 2.0, 1.5), (1, 0.0, 0.0, 1.5), (40, 4.0, 12.0, 1.5), (7, 1.0, 60.0, 0.05),
                                               (5, 2.0, 3.0, 40.0), (3, 1e7, 2e7, 1.5)])
def test_float32_ring_field_is_the_rounded_float64_one(n, count, r0, r1, xi_dx):
    xi = xi_dx * 2 * math.pi / n
    out = []
    for prec in (GP_FP32, GP_FP64):
        plan = Plan(field_params(n, 0.001, xi_over_dx=xi_dx, precision=prec))
        out.append(plan.init_rvr(0, plan.empty(), 11, mode=0, count=count, p0=r0 * xi, p1=r1 * xi))
    d = (out[0].to(torch.complex128) - out[1])
    assert float(torch.maximum(d.real.abs().max(), d.imag.abs().max())) <= 1.2e-7
