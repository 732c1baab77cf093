"""The ring field of a float32 plan is the float64 plan's field rounded, bit for bit.

The twofold float32 kernel bounds its error at every point and leaves the points where the rounding is open to
float64, so no tolerance is needed.
"""
import math

import pytest
import torch

from paper_2003_03590_gb300 import GP_FP32, GP_FP64, Plan, field_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 12, 24, 32, 48, 64, 96, 128, 192, 256])
@pytest.mark.parametrize("count,r0,r1,xi_dx", [(0, 1.0, 2.0, 1.5), (1, 0.0, 0.0, 1.5), (5, 4.0, 12.0, 2.0), (40, 4.0, 12.0, 1.5),
                                               (400, 4.0, 12.0, 1.5), (7, 1.0, 60.0, 0.05), (5, 2.0, 3.0, 40.0),
                                               (3, -8.0, 8.0, 1.5), (3, 1e7, 2e7, 1.5), (4096, 2.0, 6.0, 0.3)])
def test_float32_field_is_the_float64_one_rounded(n, count, r0, r1, xi_dx):
    if count == 4096 and n > 96:
        pytest.skip("the same kernels over more points")
    xi = xi_dx * 2 * math.pi / n
    out = []
    for prec in (GP_FP32, GP_FP64):
        plan = Plan(field_params(n, 0.001, xi_over_dx=xi_dx, precision=prec))
        out.append(plan.init_rvr(0, plan.empty(), 11 + n, mode=0, count=count, p0=r0 * xi, p1=r1 * xi))
    a, b = torch.view_as_real(out[0]), torch.view_as_real(out[1].to(torch.complex64))
    assert torch.equal(a, b), int((a != b).sum())
