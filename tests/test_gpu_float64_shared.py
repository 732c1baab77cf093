"""Float64 fields of one plan given the same memory: advanced one after the other, in the plan's order."""
import pytest
import torch

from paper_2003_03590_gb300 import GP_FP32, GP_FP64, GP_SPLIT_KNK, GP_SPLIT_NKN, Plan, field_params

pytestmark = pytest.mark.gpu


def _field(n, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = torch.randn(2, n, n, n, generator=g, device="cuda", dtype=torch.float64)
    return torch.complex(1.0 + 0.2 * r[0], 0.2 * r[1]).to(dtype)


@pytest.mark.parametrize("params", [[(0.004, GP_SPLIT_NKN)] * 2, [(0.004, GP_SPLIT_NKN), (0.002, GP_SPLIT_KNK)],
                                    [(0.004, GP_SPLIT_KNK)] * 3])
@pytest.mark.parametrize("steps", [1, 7])
def test_same_buffer_for_several_fields(params, steps):
    n = 24
    fp = [field_params(n, dt, xi_over_dx=1.5, precision=GP_FP64, split=s) for dt, s in params]
    single = field_params(32, 0.004, xi_over_dx=1.5, precision=GP_FP32)
    x, y = _field(n, torch.complex128, 1), _field(32, torch.complex64, 2)
    ref, yref = x.clone(), y.clone()
    plan = Plan(fp + [single])
    for _ in range(2):                          # a repeated call as well
        plan.step([x] * len(fp) + [y], steps)
        plan.sync()
        for f in fp:
            Plan(f).step([ref], steps)
        Plan(single).step([yref], steps)
        torch.cuda.synchronize()
        assert torch.equal(x, ref) and torch.equal(y, yref)


def test_partly_shared_memory():
    n = 16
    fp = field_params(n, 0.004, xi_over_dx=1.5, precision=GP_FP64)
    buf = torch.cat([_field(n, torch.complex128, k).reshape(-1) for k in (3, 4)])
    ref = buf.clone()
    half = n ** 3 // 2
    Plan([fp, fp]).step([buf[:n ** 3].view(n, n, n), buf[half:half + n ** 3].view(n, n, n)], 3)
    for o in (0, half):
        Plan(fp).step([ref[o:o + n ** 3].view(n, n, n)], 3)
    torch.cuda.synchronize()
    assert torch.equal(buf, ref)
