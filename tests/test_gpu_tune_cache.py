"""The autotuner's cache file: entries of other kernels are kept but not used, its own are reused."""
import json

import pytest
import torch

from paper_2003_03590_gb300 import Plan, field_params
from paper_2003_03590_gb300.gpqt import OP_PLANE, VARIANT_TMA_ONE

pytestmark = pytest.mark.gpu
KINDS = [(2, 1), (2, 2), (2, 3), (2, 4), (2, 5), (1, 1), (1, 2), (0, 6), (1, OP_PLANE)]
N = 32


def _plan(cache):
    return Plan(field_params(N, 0.004, xi_over_dx=1.5)).autotune(cache)


def test_entries_without_the_kernels_version_are_not_used(tmp_path):
    cache = tmp_path / "tune.json"
    gpu = torch.cuda.get_device_name()
    old = {f"{gpu}|{N}|{axis}|{op}": VARIANT_TMA_ONE for axis, op in KINDS}
    cache.write_text(json.dumps(old))
    _plan(cache)
    entries = json.loads(cache.read_text())
    assert all(entries[k] == v for k, v in old.items())
    own = [k for k in entries if k not in old]
    assert len(own) == len(KINDS) and all(k.startswith(gpu + "|v") for k in own)
    # the file's own entries are obeyed: name another kernel for every kind
    for k in own:
        entries[k] = VARIANT_TMA_ONE
    cache.write_text(json.dumps(entries))
    again = _plan(cache)
    for axis, op in KINDS:
        assert again.sweep_variant(N, axis, op) == VARIANT_TMA_ONE
