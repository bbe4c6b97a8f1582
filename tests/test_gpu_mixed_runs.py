"""The FP16S covariance's runs of bins: a CTA that walks consecutive bins of the
same range cells keeps the maxima of the bins that the snapshots share.  A
maximum is exact, so the results (and the apply's) equal, bit for bit, those of
small pieces of the range axis, where a CTA has one tile."""
import numpy as np
import pytest
import torch

from paper_2203_06233_gb300 import stap

from _parity import to_np

pytestmark = pytest.mark.gpu


def _plan(dims):
    plan = stap.Plan(dims, precision=stap.STAP_PREC_FP16_SCALED, steps_only=True)
    choices = stap.stap_plan_get_tuning(plan.handle, 0)
    choices[5], choices[8] = 3, 2   # tensor cores, whatever the shape
    stap.stap_plan_set_tuning(plan.handle, 0, choices)
    return plan


# split and stacked forms, several systems per tile, tiles across blocks, every
# bin in each snapshot with runs as long as the bins
@pytest.mark.parametrize("C,T,K,R,B,S", [(32, 4, 128, 1024, 128, 8), (16, 4, 128, 1280, 64, 5),
                                         (9, 5, 64, 4608, 96, 3), (4, 3, 64, 8192, 64, 4),
                                         (8, 8, 8, 16384, 128, 6), (12, 8, 8, 16384, 128, 3), (30, 3, 64, 2560, 256, 33)])
def test_runs_equal_small_pieces(C, T, K, R, B, S):
    rng = np.random.default_rng(C * K)
    dop = (rng.standard_normal((C, K, R)) + 1j * rng.standard_normal((C, K, R)))
    dop *= 2.0 ** rng.integers(-6, 7, (1, K, 1)) * 2.0 ** rng.integers(-2, 3, (C, 1, R // 64)).repeat(64, 2)
    dop = torch.from_numpy(dop.astype(np.complex64)).cuda()
    wts = torch.from_numpy((rng.standard_normal((K, R // B, S, C * T)) + 1j * rng.standard_normal((K, R // B, S, C * T)))
                           .astype(np.complex64)).cuda()
    plan = _plan((C, 4, K, R, T, B, S))
    cov, out = to_np(plan.covariance(dop)), to_np(plan.apply(dop, wts))
    assert plan.status() == (stap.STAP_OK, 0)
    plan.close()
    n = int(np.lcm(B, 128))
    plan = _plan((C, 4, K, n, T, B, S))
    for r0 in sorted({0, R // n // 2 * n, R - n}):
        part, b = dop[:, :, r0:r0 + n].contiguous(), slice(r0 // B, (r0 + n) // B)
        assert np.array_equal(to_np(plan.covariance(part)), cov[:, b])
        assert np.array_equal(to_np(plan.apply(part, wts[:, b].contiguous())), out[:, :, r0:r0 + n])
    plan.close()
