"""Choices of the float32 sweep kernels, copied from plan to plan.

The kernels a plan launches are read from its profile, not from the numbers it reports.
"""
import pytest
import torch

from paper_2003_03590_gb300 import Plan, field_params
from paper_2003_03590_gb300.gpqt import OP_PLANE, profile, profile_read

pytestmark = pytest.mark.gpu
KINDS = [(2, 1), (2, 2), (2, 3), (2, 4), (2, 5), (1, 1), (1, 2), (0, 6), (1, OP_PLANE)]


def _start(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.empty(n, n, n, dtype=torch.complex64, device="cuda")
    torch.view_as_real(x).normal_(0.0, 0.7, generator=g)
    return x


def _launched(plan, x, steps=2):
    """kernel names and numbers of launches of `steps` steps"""
    profile(plan)
    plan.step([x], steps)
    plan.sync()
    rec = profile_read(plan)
    profile(plan, False)
    return {k: c for k, (c, _) in rec.items()}


@pytest.mark.parametrize("n", [32, 64, 96, 128, 192, 256, 512])
@pytest.mark.parametrize("tuned", [False, True])
def test_copied_choices_give_the_same_kernels(n, tuned):
    a, b = (Plan(field_params(n, 0.001, xi_over_dx=1.5)) for _ in range(2))
    if tuned:
        a.autotune()
    for axis, op in KINDS:
        b.set_sweep_variant(n, axis, op, a.sweep_variant(n, axis, op))
    assert _launched(a, _start(n)) == _launched(b, _start(n))
