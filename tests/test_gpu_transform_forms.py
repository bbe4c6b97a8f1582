"""The Doppler transform's longest lengths (K = 512 in split passes) at every tile width, and the
front end's three forms, against 64-bit sums."""
import numpy as np
import pytest
import torch

from paper_2203_06233_gb300 import stap

from _parity import EPS32, to_np

pytestmark = pytest.mark.gpu


def _randc(shape, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


@pytest.mark.parametrize("tr", [0, 8, 16, 32])
@pytest.mark.parametrize("C,P,K,R,T,staggered", [(2, 512, 512, 33, 1, False), (1, 300, 512, 7, 3, True),
                                                 (2, 1024, 1024, 40, 2, False), (1, 1000, 1024, 17, 4, True)])
def test_long_transforms(C, P, K, R, T, staggered, tr):
    """Normwise per row within the FFT error bound 2 u log2 K + 4 u."""
    if tr == 32 and K == 1024:
        pytest.skip("32 columns of 1024 bins do not fit in shared memory")
    plan = stap.Plan((C, P, K, R, T, R, 2), device="cuda", steps_only=True,
                     snapshots=stap.STAP_SNAP_PRI_STAGGERED if staggered else stap.STAP_SNAP_ADJACENT_BINS)
    choices = stap.stap_plan_get_tuning(plan.handle, 0)
    choices[0] = tr
    stap.stap_plan_set_tuning(plan.handle, 0, choices)
    cube = _randc((C, P, R), K + R)
    dop = to_np(plan.doppler(torch.from_numpy(cube).cuda()))
    plan.close()
    n = P - T + 1 if staggered else P
    for t in range(T if staggered else 1):
        h = np.zeros(P)
        h[t:t + n] = np.hanning(n)
        ref = np.fft.fft(cube.astype(np.complex128) * h[None, :, None], n=K, axis=1)
        err = np.linalg.norm(dop[t * C:(t + 1) * C] - ref, axis=(1, 2)) / np.linalg.norm(ref, axis=(1, 2))
        assert err.max() <= (2 * np.log2(K) + 4) * EPS32


# positions around the forms' thresholds and odd counts; elements around the
# blocks of 32, the split form's rounds of 256 and the 512 kept at a time
@pytest.mark.parametrize("N,P,R,C", [(1, 1, 1, 1), (31, 3, 11, 4), (33, 5, 13, 5), (257, 4, 64, 4), (513, 2, 33, 3),
                                     (40, 8, 7296, 4), (520, 4, 14593, 1), (65, 64, 3649, 2), (70, 4, 58370, 9)])
def test_front_end_forms(N, P, R, C):
    """Each sum within (32 + N / 32 + 4) u of the sum of magnitudes."""
    W = _randc((C, N), N + C).astype(np.complex128)
    x = _randc((N, P, R), N + R)
    B = max(b for b in range(1, 65) if R % b == 0)
    plan = stap.Plan((C, P, max(4, 1 << (P - 1).bit_length()), R, 1, B, 2), device="cuda", front_end=W)
    y = to_np(plan.reduce_channels(torch.from_numpy(x).cuda()))
    plan.close()
    Wc = W.astype(np.complex64).astype(np.complex128)
    ref = np.tensordot(Wc.conj(), x.astype(np.complex128), axes=(1, 0))
    mag = np.tensordot(np.abs(Wc), np.abs(x.astype(np.complex128)), axes=(1, 0))
    assert np.all(np.abs(y - ref) <= (32 + N / 32 + 4) * np.sqrt(2) * EPS32 * mag)
