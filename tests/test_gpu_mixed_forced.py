"""The tensor-core covariance and apply where a plan would run the FP32
kernels by default: the parity checks of test_gpu_mixed.py with the tensor
cores named by the tuning, and the default's own choice."""
import numpy as np
import pytest
import torch

import test_gpu_mixed as mixed
from paper_2203_06233_gb300 import stap

from _parity import to_np

pytestmark = pytest.mark.gpu


def _forced(spec, prec):
    plan = stap.Plan(spec.dims(), precision=prec)
    choices = stap.stap_plan_get_tuning(plan.handle, 0)
    choices[5], choices[8] = 3, 2
    stap.stap_plan_set_tuning(plan.handle, 0, choices)
    return plan


@pytest.mark.parametrize("prec", mixed.PRECS, ids=mixed.PIDS)
@pytest.mark.parametrize("spec", mixed.SPECS + mixed.WIDTH_SPECS,
                         ids=mixed.IDS + [f"D{s.D}" for s in mixed.WIDTH_SPECS])
def test_tensor_core_steps_named_by_the_tuning(spec, prec, monkeypatch):
    monkeypatch.setattr(mixed, "_plan", _forced)
    mixed._check_covariance(spec, prec)
    mixed.test_mixed_apply_parity(spec, prec)


# (C, T, K, R, B, S) and which apply runs by default (1 FP32, 3 tensor cores)
@pytest.mark.parametrize("dims,app", [((4, 3, 32, 4096, 64, 16), 1), ((8, 3, 16, 2048, 64, 8), 1),
                                      ((8, 3, 16, 2048, 128, 64), 3), ((16, 4, 32, 2048, 128, 8), 3),
                                      ((32, 4, 8, 8192, 256, 64), 3)])
def test_default_apply_follows_the_shape(dims, app):
    C, T, K, R, B, S = dims
    rng = np.random.default_rng(3)
    dop = torch.from_numpy((rng.standard_normal((C, K, R)) + 1j * rng.standard_normal((C, K, R)))
                           .astype(np.complex64)).cuda()
    wts = torch.from_numpy((rng.standard_normal((K, R // B, S, C * T)) + 1j)
                           .astype(np.complex64)).cuda()
    res = {}
    for kind in (0, app):
        plan = stap.Plan((C, 4, K, R, T, B, S), precision=stap.STAP_PREC_BF16X3, steps_only=True)
        choices = stap.stap_plan_get_tuning(plan.handle, 0)
        choices[5] = kind
        stap.stap_plan_set_tuning(plan.handle, 0, choices)
        res[kind] = to_np(plan.apply(dop, wts))
        plan.close()
    assert np.array_equal(res[0], res[app])
