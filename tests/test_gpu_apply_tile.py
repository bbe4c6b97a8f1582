"""The tiled FP32 apply at the edges of its tiles, against 64-bit sums within
the forward-error bound of an FP32 dot product (_parity.cell_bound)."""
import numpy as np
import pytest
import torch

from paper_2203_06233_gb300 import stap

from _parity import cell_bound, gather, to_np

pytestmark = pytest.mark.gpu

# (C, T, B, NB, S): blocks around the 32-, 64- and 128-cell tiles, odd range
# extents, 1 to 64 and more steering vectors around the warps' 8, snapshot
# lengths around the chunks of 16 entries
SHAPES = [(1, 1, 1, 3, 1), (3, 1, 31, 3, 7), (5, 3, 32, 2, 8), (5, 3, 33, 3, 9), (8, 2, 64, 2, 16), (16, 1, 65, 1, 17),
          (17, 1, 100, 3, 11), (11, 3, 127, 1, 63), (8, 4, 128, 2, 64), (11, 3, 129, 3, 65), (13, 4, 250, 1, 33),
          (32, 4, 257, 2, 130), (43, 2, 96, 2, 24)]


@pytest.mark.parametrize("C,T,B,NB,S", SHAPES)
def test_tiled_apply_within_the_dot_product_bound(C, T, B, NB, S):
    K, R, D = 4, NB * B, C * T
    rng = np.random.default_rng(1000 * C + B + S)
    dop = (rng.standard_normal((C, K, R)) + 1j * rng.standard_normal((C, K, R))).astype(np.complex64)
    wts = (rng.standard_normal((K, NB, S, D)) + 1j * rng.standard_normal((K, NB, S, D))).astype(np.complex64)
    plan = stap.Plan((C, 4, K, R, T, B, S), device="cuda", steps_only=True)
    choices = stap.stap_plan_get_tuning(plan.handle, 0)
    choices[5] = 2                                   # the tiled kernel for every shape
    stap.stap_plan_set_tuning(plan.handle, 0, choices)
    out = torch.full((S, K, R), float("nan"), device="cuda")
    plan.apply(torch.from_numpy(dop).cuda(), torch.from_numpy(wts).cuda(), out)
    out = to_np(out)
    plan.close()
    x = np.repeat(wts.astype(np.complex128), B, axis=1)               # [K][R][S][D]
    y = np.einsum("krsd,krd->skr", x.conj(), gather(dop.astype(np.complex128), T))
    assert np.all(np.abs(out - np.abs(y) ** 2) <= cell_bound(dop, wts, T, B))
