"""The error-free FP32 covariance at the edges of its tiles and of its grid's
bound, against 64-bit sums: 1e-10 relative Frobenius per system (the bound of
test_gpu_parity.py), each matrix scaled by its rows' norms where these differ."""
import numpy as np
import pytest
import torch

from paper_2203_06233_gb300 import stap

from _parity import gather, to_np

pytestmark = pytest.mark.gpu


def _run(C, T, B, NB, dop, K):
    plan = stap.Plan((C, 4, K, NB * B, T, B, 2), device="cuda", steps_only=True)
    cov = to_np(plan.covariance(torch.from_numpy(dop).cuda()))
    plan.close()
    x = gather(dop.astype(np.complex128), T).reshape(K, NB, B, C * T)
    return cov, np.einsum("kbri,kbrj->kbij", x, x.conj()) / B


def _dop(C, K, R, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal((C, K, R)) + 1j * rng.standard_normal((C, K, R))).astype(np.complex64)


# odd and even blocks (cells come in pairs), one to many rounds of entries per
# CTA, blocks that need chunks of cells, one bin and many bins per CTA
@pytest.mark.parametrize("C,T,B,NB,K", [(1, 1, 1, 3, 4), (1, 2, 3, 2, 8), (2, 2, 33, 5, 16), (3, 3, 50, 2, 32),
                                        (5, 4, 64, 1, 8), (7, 3, 127, 2, 4), (12, 2, 100, 3, 16),
                                        (16, 4, 129, 1, 8), (24, 1, 96, 2, 16), (33, 3, 200, 1, 4), (32, 4, 515, 1, 4),
                                        (128, 1, 40, 2, 4)])
def test_covariance_at_tile_edges(C, T, B, NB, K):
    cov, ref = _run(C, T, B, NB, _dop(C, K, NB * B, C + B), K)
    err = np.linalg.norm(cov - ref, axis=(2, 3)) / np.linalg.norm(ref, axis=(2, 3))
    assert err.max() <= 1e-10
    assert np.array_equal(cov, cov.conj().swapaxes(2, 3))


@pytest.mark.parametrize("spread", [1e3, 1e12, 1e17])
def test_rows_of_any_magnitude_keep_their_own_precision(spread):
    """Entry (i, l) is bounded by the norms of rows i and l, whatever the other
    rows are; at 1e17 the rows' squares overflow and underflow FP32."""
    C, T, B, NB, K = 6, 1, 64, 2, 4
    scale = np.logspace(-1, 1, C) ** np.log10(spread)
    dop = (_dop(C, K, NB * B, 7) * scale[:, None, None].astype(np.float32)).astype(np.complex64)
    cov, ref = _run(C, T, B, NB, dop, K)
    ok = np.abs(scale[:, None] * scale[None, :]) < 1e37 / B     # entries that FP32 products can hold
    ok &= np.abs(scale[:, None] * scale[None, :]) > 1e-20
    d = np.sqrt(np.einsum("kbii->kbi", ref).real)
    err = np.abs(cov - ref) / (d[..., :, None] * d[..., None, :])
    assert err[..., ok].max() <= 1e-10


@pytest.mark.parametrize("size", [1e18, 1.5e18, 2e18])
@pytest.mark.parametrize("C,T,B", [(3, 1, 50), (4, 3, 64), (16, 4, 128), (32, 4, 515)])
def test_rows_at_the_end_of_fp32s_range(C, T, B, size):
    """Rows whose squares sum to just under FP32's largest number (3.2e38 for the
    largest), beside rows smaller by 1e28 and by 1e33."""
    NB, K = 2, 8
    dop = _dop(C, K, NB * B, B)
    dop = dop / np.sqrt((np.abs(dop.reshape(C, K, NB, B)) ** 2).sum(3).max()) * size * 9
    dop[1::3] *= 1e-28
    dop[2::3] *= 1e-33
    cov, ref = _run(C, T, B, NB, dop.astype(np.complex64), K)
    d = np.sqrt(np.einsum("kbii->kbi", ref).real)
    assert (np.abs(cov - ref) / (d[..., :, None] * d[..., None, :])).max() <= 1e-10
