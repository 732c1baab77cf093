"""The float32 imaginary-time steps (grad phi branching off the transforms of phi) against the float64 ones.

Tolerance: the 2e-5 of the float32 steps' oracle tests.  A step adds dtau v . grad phi; with
dtau max|k| |v| <= 1 its rounding stays at the field's (1e-7 per step), for white fields as well.
The criteria are differences, of 1e-2 of the field or the energy here: 1e-3.
"""
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP32, GP_FP64, Plan, field_params

pytestmark = pytest.mark.gpu
TOL = 2e-5
STEPS = 5


def _field(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    r = torch.randn(2, n, n, n, generator=g, device="cuda")
    return torch.complex(1.0 + 0.2 * r[0], 0.2 * r[1])


def _run(psi, prec, dtype, flow, renorm, mode):
    n = psi.shape[0]
    plan = Plan(field_params(n, 0.01, alpha=0.05, beta=20.0, precision=prec))
    x, dtau = psi.to(dtype).clone(), 1e-3
    if mode == "one":
        out = (plan.argle(0, x, flow, dtau, STEPS, renorm=renorm),)
    elif mode == "split":
        for m in (1, 1, 3):
            out = (plan.argle(0, x, flow, dtau, m, renorm=renorm),)
    else:
        d, c1, c2, e = plan.argle_converge(0, x, flow, dtau, STEPS, 0.0, check_every=3, renorm=renorm)
        assert d == STEPS
        out = (e, c1, c2)
    return x, out


@pytest.mark.parametrize("n", [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 512])
@pytest.mark.parametrize("flow", [0, 1, 2])
def test_float32_against_float64(n, flow):
    psi = _field(n)
    for renorm in (False, True):
        ref, ref_out = _run(psi, GP_FP64, torch.complex128, flow, renorm, "check")
        for mode in ("one", "split", "check"):
            x, out = _run(psi, GP_FP32, torch.complex64, flow, renorm, mode)
            err = (torch.linalg.vector_norm(x.to(torch.complex128) - ref) / torch.linalg.vector_norm(ref)).item()
            assert err < TOL, (mode, renorm)
            assert abs(out[0] - ref_out[0]) < TOL * abs(ref_out[0])
            if mode == "check":
                assert abs(out[1] - ref_out[1]) < 1e-3 * ref_out[1] and abs(out[2] - ref_out[2]) < 1e-3 * ref_out[2]
