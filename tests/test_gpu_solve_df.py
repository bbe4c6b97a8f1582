"""The double-float weight solve against 64-bit solutions.

Covariances are those of strong interference over noise (40 dB), so that the
load's bound on the condition number, D / lf + 1, is nearly reached.
Tolerance per weight vector, derived: the complex64 rounding of each
component (u = 2^-24 of the vector at most), as much again for the solve's own
error (kappa 2^-44 <= 2^-25 at kappa = 2^19, the largest bound the kernels
accept), and the sqrt(2) of a complex component: 2 sqrt(2) u, the bound that
the FP64 kernels are held to.
"""
import numpy as np
import pytest
import torch

from paper_2203_06233_gb300 import stap

from _parity import EPS32, to_np

pytestmark = pytest.mark.gpu

TOL = 2 * EPS32 * np.sqrt(2)


def _covariances(n, D, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    J = rng.standard_normal((n, D, 3)) + 1j * rng.standard_normal((n, D, 3))
    N = rng.standard_normal((n, D, 2 * D)) + 1j * rng.standard_normal((n, D, 2 * D))
    R = 1e4 * J @ J.conj().swapaxes(1, 2) + N @ N.conj().swapaxes(1, 2) / (4 * D)
    i = np.arange(D)
    R[:, i, i] = R[:, i, i].real
    return R * scale


def _reference(R, v, lf):
    D = R.shape[-1]
    tr = np.einsum("nii->n", R).real
    Rl = R + (lf / D) * tr[:, None, None] * np.eye(D)
    u = np.linalg.solve(Rl, np.broadcast_to(v.T, (len(R),) + v.T.shape))
    q = np.einsum("sd,nds->ns", v.conj(), u).real
    return np.swapaxes(u, 1, 2) / np.sqrt(q)[:, :, None]


def _solve(R, C, T, S, steer=None, **kw):
    """Weights [n][S][D] of n = 8 NB systems (K = 8 bins)."""
    n, D = R.shape[0], C * T
    K, NB = 8, R.shape[0] // 8
    plan = stap.Plan((C, 8, K, NB * 4, T, 4, S), device="cuda", **kw)
    if steer is not None:
        plan.set_steering(steer)
    w = to_np(plan.solve_weights(torch.from_numpy(R.reshape(K, NB, D, D)).cuda())).reshape(n, S, D)
    status = plan.status()
    plan.close()
    return w, status


def _check(w, ref):
    err = np.linalg.norm(w - ref, axis=-1) / np.linalg.norm(ref, axis=-1)
    print(f"largest vector error {err.max():.2e}")
    assert err.max() <= TOL


def _default_steering(C, T, S, P=8, K=8):
    s = np.arange(S)
    fs = 0.5 * np.sin(np.deg2rad(-90.0 + 180.0 * (s + 0.5) / S))
    a = np.exp(2j * np.pi * fs[:, None] * np.arange(C))
    m = np.arange(T) - T // 2
    g = (np.exp(-2j * np.pi * m[:, None] * np.arange(P) / K) * np.hanning(P)).sum(1)
    return (g[None, :, None] * a[:, None, :]).reshape(S, C * T)


# every team size and row count at its edges, one and several passes of
# right-hand sides, fewer and more steering vectors than channels, odd counts
SHAPES = [(1, 1, 1), (2, 2, 3), (8, 1, 5), (4, 2, 16), (3, 3, 4), (4, 3, 7), (13, 1, 3), (4, 4, 16), (17, 1, 18),
          (8, 3, 16), (5, 5, 2), (16, 2, 33), (11, 3, 24), (16, 3, 16), (7, 7, 8), (32, 2, 40), (13, 5, 11),
          (32, 3, 64), (97, 1, 2), (25, 4, 26), (64, 2, 65), (32, 4, 64)]


@pytest.mark.parametrize("solver,refine", [(stap.STAP_SOLVE_FP64, 1), (stap.STAP_SOLVE_FP64, 0),
                                           (stap.STAP_SOLVE_MIXED_IR, 2)], ids=["default", "unrefined", "mixed_ir"])
@pytest.mark.parametrize("C,T,S", SHAPES)
def test_weights_match_64_bit_solutions(C, T, S, solver, refine):
    D = C * T
    R = _covariances(8 * 3, D, seed=D + S)
    v = _default_steering(C, T, S)
    ref = _reference(R, v, 1e-3)
    for steer in (None, v * np.exp(1j * np.arange(D))):   # separable, and any other table
        w, status = _solve(R, C, T, S, steer, refine_steps=refine, solver=solver)
        assert status == (stap.STAP_OK, 0)
        _check(w, ref if steer is None else _reference(R, steer, 1e-3))


@pytest.mark.parametrize("C,T", [(4, 2), (3, 3), (5, 2), (4, 3)])
def test_many_small_systems_take_half_a_warp_each(C, T):
    """From 2048 systems of up to 12 rows on, an odd number of teams included."""
    R = _covariances(8 * 257, C * T, seed=C)
    for S in (3, 16):
        w, status = _solve(R, C, T, S)
        assert status == (stap.STAP_OK, 0)
        _check(w, _reference(R, _default_steering(C, T, S), 1e-3))


@pytest.mark.parametrize("scale", [2.0 ** -600, 1e-40, 3e-20, 1e30, 2.0 ** 600])
def test_any_power_of_the_input_scale_gives_the_same_weights(scale):
    """Floats span 2^+-126: the system's scale is taken out of the matrix and
    put back with the normalisation (weights go like scale^-1/2)."""
    C, T, S = 5, 3, 6
    R = _covariances(8, C * T, seed=3)
    v = _default_steering(C, T, S)
    ref = _reference(R, v, 1e-3) / np.sqrt(scale)
    w, status = _solve(R * scale, C, T, S)
    assert status == (stap.STAP_OK, 0)
    inside = np.abs(ref).max() < 1e38 and np.abs(ref).min() > 1e-30
    if inside:
        _check(w, ref)
    else:   # beyond complex64: infinities above, zeros (or subnormals) below, as any rounding gives
        assert np.all(~np.isfinite(w.real) | (np.abs(w.real) > 1e30)) if scale < 1 else np.all(np.abs(w) < 1e-30)


@pytest.mark.parametrize("refine", [0, 1])
@pytest.mark.parametrize("C,T", [(11, 3), (16, 4), (13, 5), (32, 3), (97, 1), (32, 4)])
def test_rows_of_uneven_power(C, T, refine):
    """From 33 rows on the factor's sums run on grids set by the diagonal, the
    substitutions' by the factor's entries and the solution: diagonals over
    six decades, and a row that the others do not touch."""
    D, S = C * T, 7
    R = _covariances(8, D, seed=D)
    r = 10.0 ** np.random.default_rng(D).uniform(-3, 0, D)
    R = R * r[:, None] * r[None, :]
    R[:, D // 2, :D // 2] = R[:, D // 2, D // 2 + 1:] = 0
    R[:, :D // 2, D // 2] = R[:, D // 2 + 1:, D // 2] = 0
    w, status = _solve(R, C, T, S, refine_steps=refine)
    assert status == (stap.STAP_OK, 0)
    _check(w, _reference(R, _default_steering(C, T, S), 1e-3))


def test_weak_loads_take_the_fp64_kernels():
    """Nothing bounds the condition number without a load: such plans keep the
    FP64 kernels bit for bit (solve_kind 3 names one of them)."""
    C, T, S = 8, 5, 9
    R = _covariances(8, C * T, seed=4)
    K, NB = 8, 1
    out = []
    for kind in (0, 3):
        plan = stap.Plan((C, 8, K, 4, T, 4, S), device="cuda", load_factor=1e-5)
        choices = stap.stap_plan_get_tuning(plan.handle, 0)
        choices[7] = kind
        stap.stap_plan_set_tuning(plan.handle, 0, choices)
        out.append(to_np(plan.solve_weights(torch.from_numpy(R.reshape(K, NB, C * T, C * T)).cuda())))
        plan.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("C,T", [(4, 3), (8, 3), (16, 3), (24, 3)])
def test_failed_systems_are_counted_and_zeroed(C, T):
    D, S = C * T, 5
    R = _covariances(8 * 2, D, seed=9)
    bad = {1: "indefinite", 4: "nan", 7: "inf", 10: "nan off the diagonal", 15: "zero"}
    R[1] = -R[1]
    R[4, D - 1, D - 1] = np.nan
    R[7, D - 1, 0] = np.inf
    R[10, 2, 1] = np.nan
    R[15] = 0.0
    w, status = _solve(R, C, T, S)
    assert status == (stap.STAP_ERR_NOT_POSDEF, len(bad))
    good = [i for i in range(16) if i not in bad]
    assert all(np.all(w[i] == 0) for i in bad)
    _check(w[good], _reference(R[good], _default_steering(C, T, S), 1e-3))
