"""Choices of the float32 sweep kernels: copied from plan to plan, and every kernel against the plain one.

The kernels a plan launches are read from its profile, not from the numbers it reports.
"""
import pytest
import torch

from paper_2003_03590_gb300 import GP_SPLIT_KNK, GP_SPLIT_NKN, Plan, field_params
from paper_2003_03590_gb300.gpqt import (OP_PLANE, VARIANT_DEFAULT, VARIANT_PLAIN, VARIANT_TMA_2STAGE, VARIANT_TMA_FULL,
                                         VARIANT_TMA_GROUPS, VARIANT_TMA_ONE, profile, profile_read)

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


@pytest.mark.parametrize("split", [GP_SPLIT_NKN, GP_SPLIT_KNK])
@pytest.mark.parametrize("n", [32, 48, 64, 96, 128, 192, 256, 512, 1024])
def test_every_kernel_equals_the_plain_one(n, split):
    start = _start(n)
    variants = [VARIANT_PLAIN, VARIANT_DEFAULT, VARIANT_TMA_FULL, VARIANT_TMA_ONE, VARIANT_TMA_2STAGE]
    if n >= 512:
        variants.append(VARIANT_TMA_GROUPS)
    ref = None
    for fused in (False, True):
        for v in variants:
            if fused and v == VARIANT_PLAIN:
                continue
            plan = Plan(field_params(n, 0.001, xi_over_dx=1.5, split=split))
            for axis, op in KINDS:
                if op == OP_PLANE:
                    plan.set_sweep_variant(n, axis, op, v if fused else VARIANT_PLAIN)
                elif not (v == VARIANT_TMA_2STAGE and axis == 0):
                    plan.set_sweep_variant(n, axis, op, v)
            x = start.clone()
            names = {k.split("<")[0] for k in _launched(plan, x)}
            if v == VARIANT_PLAIN:
                assert all(k.startswith("k_sweep_") for k in names), names
                ref = x
            else:
                assert torch.equal(x, ref), (v, fused)
                if v != VARIANT_DEFAULT:
                    assert ("k_tma_plane" in names) == fused
                    assert not any(k.startswith("k_sweep_strided") for k in names), (v, names)
            del plan, x
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n", [32, 96, 192, 256, 512, 1024])
def test_profile_names_the_kernels(n):
    tail = "_rc" if n >= 512 or n in (96, 192) else ""
    want = {VARIANT_PLAIN: {"x": f"k_sweep_contig{tail}<float,{n}>", "y": f"k_sweep_strided{tail}<float,{n}>",
                            "z": f"k_sweep_strided{tail}<float,{n}>"},
            VARIANT_TMA_FULL: {"x": f"k_warp_sweep<{n}>" if n >= 256 else f"k_tma_contig<{n}>",
                               "y": f"k_warp_sweep<{n}>" if n in (256, 1024) else f"k_tma_strided<{n}>",
                               "z": f"k_ztile<{n}>" if n == 1024 else f"k_warp_sweep<{n}>" if n >= 256 else f"k_tma_strided<{n}>"}}
    for v, names in want.items():
        plan = Plan(field_params(n, 0.001, xi_over_dx=1.5)).set_sweep_variant(n, 1, OP_PLANE, VARIANT_PLAIN)
        for axis, op in KINDS[:-1]:
            plan.set_sweep_variant(n, axis, op, v)
        got = {}
        for k in _launched(plan, _start(n)):
            kernel, _, axis = k.split(":")
            got.setdefault(axis, set()).add(kernel)
        assert got == {a: {k} for a, k in names.items()}
