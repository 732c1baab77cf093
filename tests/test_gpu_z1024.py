"""The z sweeps of 1024 points with 16-pencil tiles: bit for bit the one-tile-per-CTA kernel's results.

Two steps of either split launch every operation (N-forward, inverse-N-forward, inverse-N, forward,
inverse).  An 8 GB field: every SM walks several hundred tiles of both kinds of landing phase.
"""
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP32, GP_SPLIT_KNK, GP_SPLIT_NKN, Plan, field_params
from paper_2003_03590_gb300.gpqt import VARIANT_PLAIN, VARIANT_TMA

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [GP_SPLIT_NKN, GP_SPLIT_KNK])
def test_matches_plain_kernel(split):
    n = 1024
    g = torch.Generator(device="cuda").manual_seed(1)
    psi = torch.empty(n, n, n, dtype=torch.complex64, device="cuda")
    torch.view_as_real(psi).normal_(0.0, 0.7, generator=g)
    out = []
    for variant in (VARIANT_TMA, VARIANT_PLAIN):
        plan = Plan(field_params(n, 0.001, xi_over_dx=1.5, precision=GP_FP32, split=split))
        for op in range(1, 6):
            plan.set_sweep_variant(n, 2, op, variant)
        x = psi.clone()
        plan.step([x], 2)
        torch.cuda.synchronize()
        out.append(x)
        del plan
    assert torch.equal(torch.view_as_real(out[0]), torch.view_as_real(out[1]))
