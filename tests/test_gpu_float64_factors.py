"""Float64 kinetic steps at time steps whose factors are 1, i, -1, -i up to rounding, against numpy.

Tolerance: the 1.5e-15 of the other float64 kinetic steps (six one-dimensional transforms on either side);
the reference takes each axis' factor from the same float64 phase, so the factors differ by 3 ulp at most
(5e-16, added in quadrature below that).
"""
import math

import numpy as np
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP64, GP_SPLIT_KNK, GP_SPLIT_NKN, Plan, field_params

pytestmark = pytest.mark.gpu
TOL = 1.5e-15


@pytest.mark.parametrize("n,alpha,dt,split", [(16, 0.05, math.pi, GP_SPLIT_NKN), (16, 0.05, 2 * math.pi, GP_SPLIT_KNK),
                                              (16, 0.05, -math.pi, GP_SPLIT_NKN), (32, 0.5, 2 * math.pi / 40, GP_SPLIT_NKN),
                                              (32, 0.5, 2 * math.pi / 40, GP_SPLIT_KNK), (64, 0.5, 2 * math.pi / 10, GP_SPLIT_NKN),
                                              (128, 0.5, 2 * math.pi / 20, GP_SPLIT_NKN)])
def test_white_field_against_numpy(n, alpha, dt, split):
    r = np.random.default_rng(n)
    psi = r.standard_normal((n, n, n)) + 1j * r.standard_normal((n, n, n))
    plan = Plan(field_params(n, dt, alpha=alpha, beta=0.0, precision=GP_FP64, split=split))
    x = torch.from_numpy(psi.copy()).cuda()
    plan.step([x], 1)
    plan.sync()
    k = np.where(np.arange(n) < (n + 1) // 2, np.arange(n), np.arange(n) - n).astype(float)
    parts = [dt] if split == GP_SPLIT_NKN else [0.5 * dt, 0.5 * dt]
    f = np.fft.fftn(psi)
    for s in parts:
        e = np.exp(-1j * np.fmod(alpha * k * k * s, 2 * np.pi))
        f = f * e[:, None, None] * e[None, :, None] * e[None, None, :]
    ref = np.fft.ifftn(f)
    err = np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= TOL * (1 if split == GP_SPLIT_NKN else math.sqrt(2)), err


@pytest.mark.parametrize("alpha,beta,dt", [(1e300, 0.0, 1e10), (0.05, 1e300, 1e10), (0.05, -1e300, 1e10)])
@pytest.mark.parametrize("n,split", [(12, GP_SPLIT_NKN), (64, GP_SPLIT_KNK)])
def test_phases_beyond_the_float64_range_give_nan(alpha, beta, dt, n, split):
    """Parameters whose phase overflows: NaN, as in float64 arithmetic, in the steps and in the adjoint."""
    plan = Plan(field_params(n, dt, alpha=alpha, beta=beta, precision=GP_FP64, split=split))
    start = torch.ones(n, n, n, dtype=torch.complex128, device="cuda")
    for steps in (1, 6):
        x = start.clone()
        plan.step([x], steps)
        plan.sync()
        assert bool(torch.view_as_real(x).isnan().all())
    lam = start.clone()
    plan.adjoint_step(0, start, lam, 1)
    plan.sync()
    assert bool(torch.view_as_real(lam).isnan().any())
