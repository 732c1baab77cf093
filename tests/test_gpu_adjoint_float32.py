"""The float32 adjoint (one z sweep per step back) against the float64 one.

Tolerance: the 2e-5 of the float32 adjoint's oracle test (a handful of steps of about 2e-7 each on lengths
up to 256, the cotangent amplified by less than 2 per step at these beta dt).
"""
import numpy as np
import pytest
import torch

from inputs import random_direction, random_psi
from paper_2003_03590_gb300 import GP_FP32, GP_FP64, GP_SPLIT_KNK, GP_SPLIT_NKN, Plan, field_params
from tests._util import rel_l2, to_gpu, to_np

pytestmark = pytest.mark.gpu


def _run(n, split, m, prec, dt, psi, lam, alias=False):
    plan = Plan(field_params(n, 0.002, xi_over_dx=1.5, precision=prec, split=split))
    x = to_gpu(psi, dt)
    y = x if alias else to_gpu(lam, dt)
    plan.adjoint_step(0, x, y, m)
    if not alias:
        assert torch.equal(x, to_gpu(psi, dt))    # the state is only read
    return to_np(y)


@pytest.mark.parametrize("n", [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256])
@pytest.mark.parametrize("split", [GP_SPLIT_NKN, GP_SPLIT_KNK])
@pytest.mark.parametrize("m", [1, 2, 4])
def test_float32_against_float64(n, split, m):
    psi = random_psi(n, n + m, amp_jitter=0.2).astype(np.complex64)
    lam = random_direction(n, n).astype(np.complex64)
    got = _run(n, split, m, GP_FP32, np.complex64, psi, lam)
    ref = _run(n, split, m, GP_FP64, np.complex128, psi, lam)
    assert rel_l2(got, ref) < 2e-5


@pytest.mark.parametrize("split", [GP_SPLIT_NKN, GP_SPLIT_KNK])
def test_cotangent_in_the_state_buffer(split):
    psi = random_psi(32, 3, amp_jitter=0.2).astype(np.complex64)
    got = _run(32, split, 3, GP_FP32, np.complex64, psi, None, alias=True)
    ref = _run(32, split, 3, GP_FP64, np.complex128, psi, psi)
    assert rel_l2(got, ref) < 2e-5
