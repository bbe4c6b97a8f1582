"""The weight solve where the double-float kernels could leave the 64-bit
weights: steering tables and loads of any magnitude, beams that point along the
interference (the separable combination cancels), the weakest loads they
accept, and Hermitian inputs that are not quite covariances."""
import numpy as np
import pytest
import torch

from paper_2203_06233_gb300 import stap

from test_gpu_solve_df import TOL, _check, _covariances, _default_steering, _reference, _solve

pytestmark = pytest.mark.gpu

BIG_AND_SMALL = [(4, 3), (5, 3), (16, 4), (32, 4)]


@pytest.mark.parametrize("solver", [stap.STAP_SOLVE_FP64, stap.STAP_SOLVE_MIXED_IR], ids=["default", "mixed_ir"])
@pytest.mark.parametrize("C,T", BIG_AND_SMALL)
def test_weights_do_not_depend_on_the_steering_tables_scale(C, T, solver):
    """w = u / sqrt(v^H u): every finite table gives the weights of its
    directions, to the tolerance of the unscaled one."""
    D, S = C * T, 5
    R = _covariances(8, D, seed=D)
    v = _default_steering(C, T, S) * np.exp(1j * np.arange(D))
    ref = _reference(R, v, 1e-3)
    scales = [np.full(S, s) for s in (1e-320, 1e-300, 1e-30, 1e-20, 1e20, 1e30, 1e300)]
    scales.append(np.array([1e-30, 1.0, 1e30, 1e-200, 1e200]))     # one table, many magnitudes
    for s in scales:
        t = v * 1e10 * (s * 1e-10)[:, None] if s.min() > 1e-305 else v * s[:, None]
        want = ref if s.min() > 1e-305 else _reference(R, t * 2.0 ** 1000, 1e-3)   # subnormal entries are rounded
        w, status = _solve(R, C, T, S, t, solver=solver, refine_steps=2)
        assert status == (stap.STAP_OK, 0)
        _check(w, want)


@pytest.mark.parametrize("gain", [1e-30, 1e-22, 1e22, 1e30])
def test_weights_do_not_depend_on_the_front_ends_scale(gain):
    """The separable table of a front end, v_s = g (x) W^H a_s."""
    C, T, S, N = 4, 3, 9, 12
    W = np.zeros((C, N))
    for c in range(C):
        W[c, 3 * c:3 * c + 3] = 1.0
    R = torch.from_numpy(_covariances(8, C * T, seed=1).reshape(8, 1, C * T, C * T)).cuda()
    out = []
    for g in (1.0, gain):
        plan = stap.Plan((C, 8, 8, 4, T, 4, S), front_end=W * g)
        out.append(plan.solve_weights(R).cpu().numpy().reshape(8, S, C * T))
        assert plan.status() == (stap.STAP_OK, 0)
        plan.close()
    _check(out[1], out[0])


@pytest.mark.parametrize("lf", [1e3, 1e20, 1e38, 1e42, 1e100])
@pytest.mark.parametrize("C,T", BIG_AND_SMALL)
def test_loads_of_any_strength(C, T, lf):
    """Rl is scaled by its own trace, load included; R is scaled so that the
    weights stay inside complex64."""
    D, S = C * T, 5
    R = _covariances(8, D, seed=D) / lf
    for steer in (None, _default_steering(C, T, S) * np.exp(1j * np.arange(D))):
        v = _default_steering(C, T, S) if steer is None else steer
        w, status = _solve(R, C, T, S, steer, load_factor=lf)
        assert status == (stap.STAP_OK, 0)
        _check(w, _reference(R, v, lf))


def _weakest(D):
    """The smallest load that the double-float kernels accept: D / lf + 1 = 2^19."""
    return D / (2.0 ** 19 - 1.0) * (1 + 1e-9)


@pytest.mark.parametrize("refine", [0, 1])
@pytest.mark.parametrize("C,T", BIG_AND_SMALL)
def test_the_weakest_load_on_either_side_of_the_rule(C, T, refine):
    """kappa(Rl) reaches the bound within a factor of 3 (three strong sources)."""
    D, S = C * T, C + 3
    R = _covariances(8, D, seed=D)
    for lf in (_weakest(D), _weakest(D) * 0.99):
        for steer in (None, _default_steering(C, T, S) * np.exp(1j * np.arange(D))):
            v = _default_steering(C, T, S) if steer is None else steer
            w, status = _solve(R, C, T, S, steer, refine_steps=refine, load_factor=lf)
            assert status == (stap.STAP_OK, 0)
            _check(w, _reference(R, v, lf))


def _along(v, jnr, seed):
    """Noise and one source along each of v's vectors in turn, jnr per entry."""
    n, D = v.shape
    rng = np.random.default_rng(seed)
    N = rng.standard_normal((n, D, 2 * D)) + 1j * rng.standard_normal((n, D, 2 * D))
    a = v * np.sqrt(D) / np.linalg.norm(v, axis=1, keepdims=True)
    R = jnr * a[:, :, None] * a[:, None, :].conj() + N @ N.conj().swapaxes(1, 2) / (4 * D)
    i = np.arange(D)
    R[:, i, i] = R[:, i, i].real
    return R


@pytest.mark.parametrize("refine,load", [(1, "default"), (0, "default"), (2, "default"), (1, "weakest"), (0, "weakest")])
@pytest.mark.parametrize("db", [40, 60, 80])
@pytest.mark.parametrize("C,T,S", [(4, 3, 16), (4, 2, 100), (5, 3, 11), (8, 3, 16), (16, 4, 32), (32, 3, 40),
                                   (32, 4, 64)])
def test_beams_along_the_interference(C, T, S, db, refine, load):
    """The solution of such a beam is up to kappa(Rl) times smaller than the
    separable terms that it is combined from."""
    D = C * T
    lf = 1e-3 if load == "default" else _weakest(D)
    for steer in (None, _default_steering(C, T, S) * np.exp(1j * np.arange(D))):
        v = _default_steering(C, T, S) if steer is None else steer
        R = _along(v[np.linspace(0, S - 1, 16).astype(int)], 10.0 ** (db / 10), seed=S)
        w, status = _solve(R, C, T, S, steer, refine_steps=refine, load_factor=lf)
        assert status == (stap.STAP_OK, 0)
        _check(w, _reference(R, v, lf))


def test_beams_along_the_interference_in_many_small_systems():
    """Two systems share a warp: one with such a beam, one without."""
    C, T, S = 4, 3, 16
    v = _default_steering(C, T, S)
    n = 8 * 257
    R = _covariances(n, C * T, seed=2)
    R[::3] = np.resize(_along(v, 1e6, seed=4), (n, C * T, C * T))[:len(R[::3])]
    w, status = _solve(R, C, T, S)
    assert status == (stap.STAP_OK, 0)
    _check(w, _reference(R, v, 1e-3))


def test_range_slabs_take_the_whole_cpis_kernel():
    """D = 12, 8192 systems: half a warp per system, also in slabs of 1024,
    which by themselves would take a warp each and round otherwise."""
    g = torch.Generator().manual_seed(1)
    cube = torch.randn((4, 128, 1024), dtype=torch.complex64, generator=g).cuda()
    out = []
    for slabs in (1, 3, 8):
        plan = stap.Plan((4, 128, 128, 1024, 3, 16, 8))
        choices = stap.stap_plan_get_tuning(plan.handle, 0)
        choices[6] = slabs
        stap.stap_plan_set_tuning(plan.handle, 0, choices)
        out.append(plan.run_cpi(cube).clone())
        assert plan.status() == (stap.STAP_OK, 0)
        plan.close()
    assert torch.equal(out[1], out[0]) and torch.equal(out[2], out[0])


def _long_reference(R, v, lf):
    """The weights by an unpivoted LDL^H in long double (64 or more bits)."""
    n, D = R.shape[0], R.shape[-1]
    A = R.astype(np.clongdouble)
    tr = np.einsum("nii->ni", A).real.sum(1)
    i = np.arange(D)
    A[:, i, i] = A[:, i, i].real + (np.longdouble(lf) * tr / D)[:, None]
    u = np.broadcast_to(v.T.astype(np.clongdouble), (n,) + v.T.shape).copy()
    for j in range(D):                       # [A | u] -> unit upper triangular
        row = A[:, j, j + 1:] / A[:, j, j, None]
        ur = u[:, j] / A[:, j, j, None]
        f = A[:, j + 1:, j, None]
        A[:, j + 1:, j + 1:] -= f * row[:, None, :]
        u[:, j + 1:] -= f * ur[:, None, :]
        A[:, j, j + 1:], u[:, j] = row, ur
    for j in range(D - 1, 0, -1):
        u[:, :j] -= A[:, :j, j, None] * u[:, j, None, :]
    q = np.einsum("sd,nds->ns", v.conj().astype(np.clongdouble), u).real
    return (np.swapaxes(u, 1, 2) / np.sqrt(q)[:, :, None]).astype(np.complex128)


@pytest.mark.parametrize("refine", [0, 1])
@pytest.mark.parametrize("margin", [0.5, 1e-2, 1e-4, 1e-6])
@pytest.mark.parametrize("C,T", [(4, 2), (4, 3), (5, 3), (8, 3), (16, 3), (16, 4), (32, 3), (32, 4)])
def test_matrices_that_are_not_quite_covariances(C, T, margin, refine):
    """A negative eigenvalue just above minus the load: Rl is positive definite
    with kappa = 1 / margin times what a covariance's would be.  The weights
    are as good as 64-bit arithmetic leaves them, sqrt(D) kappa 2^-53 beside the
    complex64 rounding; covariances among them are not touched."""
    D, S, n, lf = C * T, 7, 16, 1e-3
    rng = np.random.default_rng(D)
    Q, _ = np.linalg.qr(rng.standard_normal((n, D, D)) + 1j * rng.standard_normal((n, D, D)))
    ev = np.concatenate([[1e4], rng.uniform(0.5, 2.0, D - 2), [0.0]])
    lo = lf / D * ev.sum() / (1 + lf / D * (1 - margin))      # its share of the trace taken off
    ev[-1] = -(1 - margin) * lo
    odd = np.arange(n) % 3 != 1
    R = (Q * np.where(odd[:, None], ev, np.abs(ev))[:, None, :]) @ Q.conj().swapaxes(1, 2)
    R = (R + R.conj().swapaxes(1, 2)) / 2
    kappa = (1e4 + lo) / (margin * lo)
    tol = TOL + np.sqrt(D) * kappa * 2.0 ** -53
    v = _default_steering(C, T, S)
    for steer in (None, v * np.exp(1j * np.arange(D))):
        w, status = _solve(R, C, T, S, steer, load_factor=lf, refine_steps=refine)
        assert status == (stap.STAP_OK, 0)
        ref = _long_reference(R, v if steer is None else steer, lf)
        err = np.linalg.norm(w - ref, axis=-1) / np.linalg.norm(ref, axis=-1)
        print(f"indefinite {err[odd].max():.2e} (kappa {kappa:.1e}, bound {tol:.1e}), covariances {err[~odd].max():.2e}")
        assert err[odd].max() <= tol and err[~odd].max() <= TOL


@pytest.mark.parametrize("refine", [0, 1])
@pytest.mark.parametrize("C,T,S,K,NB", [(3, 2, 5, 8, 3), (4, 3, 16, 8, 3), (4, 3, 16, 64, 33), (5, 3, 40, 8, 5),
                                        (4, 4, 3, 32, 33), (8, 3, 16, 8, 3), (16, 2, 9, 8, 3), (11, 3, 24, 8, 3),
                                        (16, 4, 32, 8, 3), (24, 4, 40, 8, 2), (32, 4, 64, 8, 2)])
def test_runs_and_steps_agree(C, T, S, K, NB, refine):
    """A run's solve, of its own covariances, and the step's, of any matrix, are
    kernels of their own: the same bits, also for a beam along interference."""
    B = 2 * C * T
    g = torch.Generator().manual_seed(S)
    cube = torch.randn((C, K, NB * B), dtype=torch.complex64, generator=g)
    f = 0.5 * np.sin(np.deg2rad(-90.0 + 180.0 * (S // 2 + 0.5) / S))
    line = np.exp(2j * np.pi * (f * np.arange(C)[:, None] + 3 / K * np.arange(K)[None, :]))
    cube += 1e3 * torch.from_numpy(line.astype(np.complex64))[:, :, None] * torch.randn(
        NB * B, dtype=torch.complex64, generator=g)
    plan = stap.Plan((C, K, K, NB * B, T, B, S), refine_steps=refine)
    cube = cube.cuda()
    out = plan.run_cpi(cube).clone()
    dop = plan.doppler(cube)
    steps = plan.apply(dop, plan.solve_weights(plan.covariance(dop)))
    assert plan.status() == (stap.STAP_OK, 0)
    plan.close()
    assert torch.equal(out, steps)


@pytest.mark.parametrize("solver", [stap.STAP_SOLVE_FP64, stap.STAP_SOLVE_MIXED_IR], ids=["default", "mixed_ir"])
@pytest.mark.parametrize("n", [8, 512, 520, 1024, 1032, 2040, 2048])
@pytest.mark.parametrize("C,T,S", [(3, 2, 5), (4, 2, 33), (5, 2, 16), (5, 3, 4), (4, 4, 17), (12, 2, 9)])
def test_every_split_of_small_systems(C, T, S, n, solver):
    """Teams of half a warp, a warp and 128 threads, by the systems' count and
    the right-hand sides' (at most 4, 16, more)."""
    R = _covariances(n, C * T, seed=S)
    v = _default_steering(C, T, S)
    for steer in (None, v * np.exp(1j * np.arange(C * T))):
        w, status = _solve(R, C, T, S, steer, solver=solver, refine_steps=2)
        assert status == (stap.STAP_OK, 0)
        _check(w, _reference(R, v if steer is None else steer, 1e-3))


def test_the_tuning_cache_tells_loads_apart(tmp_path):
    """A weak load is solved in FP64, with launch choices of its own; a plan
    with the default load, tuned into the same cache, does not take them."""
    dims, cache = (4, 16, 16, 256, 3, 16, 4), str(tmp_path / "tune.json")
    cube = torch.randn((4, 16, 256), dtype=torch.complex64, device="cuda")
    keys = []
    for lf in (1e-6, 1e-3):
        plan = stap.Plan(dims, load_factor=lf)
        (key, tuning), = plan.autotune(cube, cache_path=cache).items()
        keys.append(key)
        assert (tuning[7] == 0) == (lf == 1e-3), tuning
        plan.close()
    assert keys[0] != keys[1]
