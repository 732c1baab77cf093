"""The float32 diagnostics and structure functions (derivatives axis by axis) against the float64 ones.

Tolerance: the 2e-5 of the float32 diagnostics parity tests (a gradient's float32 rounding, about 1e-7
of the field, is amplified by up to N/2 relative to the smallest scales of these fields).
"""
import numpy as np
import pytest
import torch

from inputs import random_psi, smooth_psi
from paper_2003_03590_gb300 import GP_FP32, GP_FP64, Plan, field_params
from tests._util import to_gpu

pytestmark = pytest.mark.gpu
TOL = 2e-5


@pytest.mark.parametrize("n", [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256])
@pytest.mark.parametrize("white", [True, False])
def test_float32_against_float64(n, white):
    psi = random_psi(n, n, amp_jitter=0.2) if white else smooth_psi(n, n)
    psi = (psi * np.exp(1j * 2 * np.pi * np.arange(n) / n)).astype(np.complex64)
    got, ref = [], []
    for out, prec, dt in ((got, GP_FP32, np.complex64), (ref, GP_FP64, np.complex128)):
        plan = Plan(field_params(n, 0.001, xi_over_dx=1.5, precision=prec))
        x = to_gpu(psi, dt)
        d, spec = plan.diagnostics(0, x)
        out += [d, spec, plan.structure_function(0, x, order=2)]
        assert torch.equal(x, to_gpu(psi, dt))        # the field is only read
    for k, v in ref[0].items():
        assert abs(got[0][k] - v) <= TOL * max(abs(v), 1e-3 * abs(ref[0]["E"])), k
    for k, v in ref[1].items():
        assert np.max(np.abs(got[1][k] - v)) <= 10 * TOL * max(np.max(np.abs(v)), 1e-3 * abs(ref[0]["E"])), k
    assert np.max(np.abs(got[2] - ref[2])) <= 10 * TOL * np.max(np.abs(ref[2]))


def test_nonfinite_field_is_reported():
    plan = Plan(field_params(96, 0.001, xi_over_dx=1.5, precision=GP_FP32))
    x = to_gpu(random_psi(96, 1), np.complex64)
    x[3, 4, 5] = float("nan")
    with pytest.raises(Exception) as e:
        plan.diagnostics(0, x)
    assert e.value.status == 6
