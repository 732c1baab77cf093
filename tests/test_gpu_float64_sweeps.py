"""Float64 fields: the fixed-point sweeps against numpy, over the float64 range and for special values.

The kinetic flow alone (beta = 0) is linear, so a power-of-two factor on the field must come out
unchanged, bit for bit, and numpy's FFT gives the result in float64.

Tolerance.  Relative L2 error of one K step: six one-dimensional transforms on either side.  The
sweeps lose at most 0.7e-16 each up to 256 points (the fixed-point unit) plus 0.5e-16 for storing
float64 between them, numpy about 2.3e-16 each; added in quadrature sqrt(6) 2.5e-16 = 6e-16.  1.5e-15
allows 2.5 times that.
"""
import numpy as np
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP64, GP_SPLIT_KNK, GP_SPLIT_NKN, Plan, field_params

pytestmark = pytest.mark.gpu
TOL = 1.5e-15
SIZES = [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256]


def k_step(n, psi, split=GP_SPLIT_NKN):
    plan = Plan(field_params(n, 0.01, alpha=0.05, beta=0.0, precision=GP_FP64, split=split))
    x = torch.from_numpy(psi.copy()).cuda()
    plan.step([x], 1)
    plan.sync()
    return x.cpu().numpy()


def field(n, seed):
    r = np.random.default_rng(seed)
    return (1 + 0.3 * r.standard_normal((n, n, n))) * np.exp(2j * np.pi * r.random((n, n, n)))


def reference(n, psi):
    k = np.fft.fftfreq(n, 1.0 / n)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
    return np.fft.ifftn(np.exp(-1j * np.fmod(0.05 * 0.01 * k2, 2 * np.pi)) * np.fft.fftn(psi))


@pytest.mark.parametrize("n", SIZES)
def test_kinetic_step_against_numpy(n):
    psi = field(n, n)
    ref = reference(n, psi)
    assert np.linalg.norm(k_step(n, psi) - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [8, 12, 64, 96])
@pytest.mark.parametrize("power", [-1000, -880, 1, 870, 980])
def test_power_of_two_scales_come_out_exactly(n, power):
    psi = field(n, 3)
    psi[1] *= 2.0 ** -40                      # planes of very different size
    psi[:, 2] *= 2.0 ** 30
    base = k_step(n, psi)
    f = 2.0 ** power
    got = k_step(n, psi * f)
    tiny = np.abs(base) * f < 2.0 ** -1000    # results near the subnormal range lose digits
    assert np.array_equal(got[~tiny], (base * f)[~tiny])
    assert np.all(np.abs(got[tiny] - (base * f)[tiny]) <= 2.0 ** -1040)


@pytest.mark.parametrize("n", [12, 64])
@pytest.mark.parametrize("split", [GP_SPLIT_NKN, GP_SPLIT_KNK])
def test_special_values(n, split):
    z = np.zeros((n, n, n), dtype=np.complex128)
    assert not k_step(n, z, split).any()
    for bad in (np.nan, np.inf, -np.inf):
        psi = field(n, 5)
        psi[1, 2, 3] = bad
        assert not np.isfinite(k_step(n, psi, split)).any()


@pytest.mark.parametrize("n", [16, 48])
def test_a_single_mode_keeps_its_digits(n):
    """One plane wave: every pencil of the k-space holds one value or none; the step multiplies it by its
    kinetic factor, to the accuracy of the wave itself."""
    x = 2 * np.pi * np.arange(n) / n
    psi = np.exp(1j * (2 * x[None, None, :] - 3 * x[None, :, None] + x[:, None, None]))
    want = psi * np.exp(-1j * 0.05 * 0.01 * 14)
    assert np.max(np.abs(k_step(n, psi) - want)) <= 2e-15
