"""Float64 steps against extended precision (long double: 80 bits on x86, 128 on Arm) and, at 512 and 1024
points, against torch's complex128 transforms.

Tolerances, relative L2.  A transform in fixed point loses at most 1.6e-16 (1024 points; 0.75e-16 at 512, less
below), storing float64 between the sweeps 0.5e-16 each, the products of kinetic factors 1.1e-16 each.
  One axis: two transforms, six stores, three products: sqrt(2 1.6^2 + 6 0.5^2 + 3 1.1^2) 1e-16 = 3.2e-16;
  5e-16 allows 1.6 times that.  The reference takes the kinetic factors in float64, as the scheme does: at 1024 points
  their phases (13 radians) are rounded by up to 9e-16.
  Three axes against float64 transforms of about 4e-16 each: sqrt(6 4^2 + 6 1.7^2 + 3 1.1^2) 1e-16 = 1.1e-15, the
  flow N adds 3e-16 (phases of a few hundredths, rounded in float64 by the reference): 3e-15 allows 2.5 times that.
  Up to 96 points the step is closer to extended precision than numpy's float64 is.
"""
import numpy as np
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP64, GP_SPLIT_KNK, GP_SPLIT_NKN, Plan, field_params

pytestmark = pytest.mark.gpu
ALPHA, BETA, DT = 0.05, 20.0, 1e-3
ONE_AXIS_TOL, TORCH_TOL = 5e-16, 3e-15
LENGTHS = [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 512, 1024]


def _plan(n, beta, split=GP_SPLIT_NKN):
    return Plan(field_params(n, DT, alpha=ALPHA, beta=beta, precision=GP_FP64, split=split))


def _k2(n, dtype):
    k = np.where(np.arange(n) < (n + 1) // 2, np.arange(n), np.arange(n) - n).astype(dtype)
    return k * k


def _step(psi, split, beta, real):
    """One step in numpy, every number in the precision of psi (real: its real type)."""
    n = psi.shape[0]
    e = np.exp(-1j * (real(ALPHA) * real(DT) * (1 if split == GP_SPLIT_NKN else real(0.5)) * _k2(n, real)))

    def kinetic(f):
        return np.fft.ifftn(np.fft.fftn(f) * e[:, None, None] * e[None, :, None] * e[None, None, :])

    def nonlinear(f, s):
        return f * np.exp(-1j * (real(beta) * s * (f.real * f.real + f.imag * f.imag - 1)))
    if split == GP_SPLIT_NKN:
        return nonlinear(kinetic(nonlinear(psi, real(DT) / 2)), real(DT) / 2)
    return kinetic(nonlinear(kinetic(psi), real(DT)))


def _norm(x):
    return float(np.sqrt(np.sum(x.real * x.real + x.imag * x.imag)))


@pytest.mark.parametrize("n", [64, 96])
@pytest.mark.parametrize("split", [GP_SPLIT_NKN, GP_SPLIT_KNK])
def test_closer_to_extended_precision_than_float64_is(n, split):
    if np.fft.fft(np.ones(4, np.clongdouble)).dtype != np.clongdouble:
        pytest.skip("numpy without long double transforms")
    r = np.random.default_rng(n)
    psi = (1 + 0.3 * r.standard_normal((n, n, n))) * np.exp(2j * np.pi * r.random((n, n, n)))
    x = torch.from_numpy(psi.copy()).cuda()
    plan = _plan(n, BETA, split)
    plan.step([x], 1)
    plan.sync()
    ref = _step(psi.astype(np.clongdouble), split, BETA, np.longdouble)
    ours = _norm(x.cpu().numpy() - ref) / _norm(ref)
    theirs = _norm(_step(psi, split, BETA, np.float64) - ref) / _norm(ref)
    assert ours <= theirs, (ours, theirs)


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_field_of_one_axis(n, axis):
    """The field varies along one axis only, so that the kinetic step is a one-dimensional one."""
    if np.fft.fft(np.ones(4, np.clongdouble)).dtype != np.clongdouble:
        pytest.skip("numpy without long double transforms")
    r = np.random.default_rng(3 * n + axis)
    f = (1 + 0.3 * r.standard_normal(n)) * np.exp(2j * np.pi * r.random(n))
    shape = [1, 1, 1]
    shape[2 - axis] = n
    x = torch.from_numpy(f).cuda().view(shape).expand(n, n, n).contiguous()
    plan = _plan(n, 0.0)
    plan.step([x], 1)
    plan.sync()
    e = np.exp(-1j * np.fmod(ALPHA * _k2(n, np.float64) * DT, 2 * np.pi)).astype(np.clongdouble)
    ref = np.fft.ifft(np.fft.fft(f.astype(np.clongdouble)) * e)
    at = [[0, 0], [n // 2, n // 3], [n - 1, 1]]
    for a, b in at:
        y = x.movedim(2 - axis, 0)[:, a, b].cpu().numpy()
        assert _norm(y - ref) <= ONE_AXIS_TOL * _norm(ref), (a, b, _norm(y - ref) / _norm(ref))


@pytest.mark.parametrize("n", [512, 1024])
@pytest.mark.parametrize("split,steps", [(GP_SPLIT_NKN, 1), (GP_SPLIT_NKN, 2), (GP_SPLIT_KNK, 1)])
def test_large_lengths_against_torch(n, split, steps):
    """Every operation of the float64 step at the lengths with 32 elements a thread."""
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.empty(n, n, n, dtype=torch.complex128, device="cuda")
    torch.view_as_real(x).normal_(0.0, 0.7, generator=g)
    f = x.clone()
    plan = _plan(n, BETA, split)
    plan.step([x], steps)
    plan.sync()
    del plan

    def kinetic(f, s):
        e = torch.from_numpy(np.exp(-1j * np.fmod(ALPHA * _k2(n, np.float64) * s, 2 * np.pi))).cuda()
        f = torch.fft.fftn(f)
        for shape in ((n, 1, 1), (1, n, 1), (1, 1, n)):
            f *= e.view(shape)
        return torch.fft.ifftn(f)

    def nonlinear(f, s):
        for z in range(n):                                # plane by plane: no temporaries of the field's size
            p = f[z]
            ph = BETA * s * (p.real * p.real + p.imag * p.imag - 1.0)
            f[z] = p * torch.polar(torch.ones_like(ph), -ph)
        return f
    for _ in range(steps):
        if split == GP_SPLIT_NKN:
            f = nonlinear(kinetic(nonlinear(f, 0.5 * DT), DT), 0.5 * DT)
        else:
            f = kinetic(nonlinear(kinetic(f, 0.5 * DT), DT), 0.5 * DT)
    norm = torch.linalg.vector_norm(f).item()
    f -= x
    err = torch.linalg.vector_norm(f).item() / norm
    del f, x
    torch.cuda.empty_cache()
    assert err <= TORCH_TOL * (steps if split == GP_SPLIT_NKN else 2) ** 0.5, err
