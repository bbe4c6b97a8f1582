"""The work that a user of this framework has it do, as cases to be timed.

Whole CPIs through ``Plan.run_cpi`` (one CPI or a batch of uneven ones, with
or without the front end) and the chain's steps on their own (``Plan.doppler``,
``Plan.covariance``, ``Plan.solve_weights``, ``Plan.apply``), at the shapes of
the workloads in ``paper_2203_06233_gb300/synth.py`` and at odd ones between
them.  A case is a dict of plain values:

  kind       "cpi" (the whole chain), "batch" (many CPIs in one call),
             "elements" (front end, then the chain), "contractions"
             (Doppler, covariance and apply, each on inputs of its own),
             "doppler", "solve"
  C .. S     channels, pulses, Doppler bins, range cells, temporal degrees of
             freedom, cells per training block, steering vectors
  precision  arithmetic of the contractions, solver that of the solve

Launch choices are the plan's defaults: no case runs the autotuner.
"""
import math
import random

import numpy as np
import torch

from paper_2203_06233_gb300 import stap

PRECISIONS = {"fp32": stap.STAP_PREC_FP32, "bf16x3": stap.STAP_PREC_BF16X3,
              "tf32x3": stap.STAP_PREC_TF32X3, "fp16s": stap.STAP_PREC_FP16_SCALED}
SOLVERS = {"fp64": stap.STAP_SOLVE_FP64, "mixed_ir": stap.STAP_SOLVE_MIXED_IR}
TRAININGS = {"own": stap.STAP_TRAIN_OWN_BLOCK, "neighbours": stap.STAP_TRAIN_NEIGHBOURS,
             "window": stap.STAP_TRAIN_WINDOW}
SNAPSHOTS = {"adjacent": stap.STAP_SNAP_ADJACENT_BINS, "staggered": stap.STAP_SNAP_PRI_STAGGERED}

LOAD = 1e-3          # diagonal load factor of every workload
PATCHES = 64         # clutter patches


def _case(kind, C, P, K, R, T, B, S, precision="fp32", solver="fp64", training="own",
          snapshots="adjacent", cnr_db=40.0, guard=0, half=1, elements=0, n_cpi=1, dims_seed=0):
    return dict(kind=kind, C=C, P=P, K=K, R=R, T=T, B=B, S=S, precision=precision, solver=solver,
                training=training, snapshots=snapshots, cnr_db=cnr_db, guard=guard, half=half,
                elements=elements, n_cpi=n_cpi, dims_seed=dims_seed)


def listed():
    cases = {
        # one small CPI at a time, as a low-latency loop or a first trial runs it:
        # a few thousand cells, so launches and latency count
        "small_cpi": _case("cpi", 4, 32, 32, 256, 3, 32, 4, cnr_db=30.0),
        # the standard CPI in the default arithmetic (D = 12)
        "standard_cpi": _case("cpi", 4, 128, 256, 4096, 3, 64, 16),
        # odd sizes with the options that change the data flow: PRI-staggered
        # snapshots, a sliding training window with a guard group, D = 15
        "ragged_cpi": _case("cpi", 5, 100, 128, 3000, 3, 100, 11, training="window",
                            snapshots="staggered", guard=1, half=2),
        # the D = 64 CPI in its stated arithmetic (BF16 three-piece split)
        "d64_cpi": _case("cpi", 16, 256, 256, 16384, 4, 128, 32, precision="bf16x3"),
        # the D = 128 CPI in its stated arithmetic (FP16 with per-block scales),
        # a quarter of the large workload's range cells
        "d128_cpi": _case("cpi", 32, 512, 512, 8192, 4, 256, 64, precision="fp16s"),
        # many uneven CPIs in one call, the batch workload's distribution
        "batch": _case("batch", 0, 0, 0, 0, 0, 64, 0, precision="bf16x3", n_cpi=24, dims_seed=4),
        # the paper's cube shape (1000 elements x 100 pulses) with a tenth of its
        # range cells, reduced to 4 channels by the front end, then the chain
        "paper_cube": _case("elements", 4, 100, 128, 3000, 3, 100, 16, elements=1000),
        # the Doppler transform on its own, at the large workload's pulse count
        "doppler_d128": _case("doppler", 32, 512, 512, 4096, 4, 256, 64),
        # step-by-step use, default arithmetic, D = 64: the three contractions
        "plain_steps_d64": _case("contractions", 16, 256, 256, 4096, 4, 128, 32),
        # the same on the tensor cores, D = 128
        "tensor_steps_d128": _case("contractions", 32, 512, 512, 2048, 4, 256, 64, precision="fp16s"),
        # the weight solve on its own, default solver, D = 64
        "solve_d64": _case("solve", 16, 256, 256, 4096, 4, 128, 32),
        # the weight solve with the mixed-precision refinement option, D = 128
        "solve_ir_d128": _case("solve", 32, 512, 512, 1024, 4, 256, 64, solver="mixed_ir"),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_any(rng):
    kind = rng.choice(["cpi", "cpi", "cpi", "contractions", "solve", "doppler", "batch", "elements"])
    if kind == "batch":
        return _case("batch", 0, 0, 0, 0, 0, 64, 0, precision=rng.choice(["fp32", "bf16x3"]),
                     n_cpi=rng.randint(4, 24), dims_seed=rng.randint(5, 10 ** 6))
    T = rng.choice([2, 3, 3, 4])
    C = 4 if kind == "elements" else min(_log_int(rng, 3, 40), 128 // T)
    P = _log_int(rng, 24, 512)
    K = 1 << max(5, math.ceil(math.log2(P)))
    D = C * T
    # training blocks of at least about 2 D cells, powers of two and odd sizes
    B = rng.choice([32, 50, 64, 100, 128, 200, 256])
    while B < 2 * D and B < 256:
        B = {32: 50, 50: 64, 64: 100, 100: 128, 128: 200, 200: 256}[B]
    NB = _log_int(rng, 4, 256)
    S = rng.choice([4, 8, 11, 16, 24, 32, 64])
    precision = rng.choice(["fp32", "fp32", "bf16x3", "tf32x3", "fp16s"])
    solver = rng.choice(["fp64", "fp64", "mixed_ir"])
    training = rng.choice(["own", "own", "own", "neighbours", "window"]) if kind == "cpi" else "own"
    snapshots = rng.choice(["adjacent", "adjacent", "staggered"]) if kind in ("cpi", "doppler") else "adjacent"
    guard = rng.randint(0, 1) if training == "window" else 0
    half = rng.randint(1, 4) if training == "window" else 1
    return _case(kind, C, P, K, NB * B, T, B, S, precision, solver, training, snapshots,
                 rng.choice([20.0, 30.0, 40.0]), guard, half,
                 _log_int(rng, 100, 1000) if kind == "elements" else 0)


def _state_bytes(case):
    """Device bytes of one state, about."""
    total = 0
    for C, P, K, R, T, B, S in _dims(case):
        D, NB = C * T, R // B
        rows = D if case["snapshots"] == "staggered" else C
        total += 8 * max(C, case["elements"]) * P * R + 8 * rows * K * R + 32 * K * NB * D * D + \
            8 * K * NB * S * D + 4 * S * K * R
    return total


def draw(rng):
    largest = work(next(c for c in listed() if c["name"] == "d128_cpi"))
    while True:
        case = _draw_any(rng)
        w = work(case)
        if 5 * w["flops"] <= 4 * largest["flops"] and w["bytes"] <= largest["bytes"] and \
                _state_bytes(case) <= 12 << 30:
            return case


# ------------------------------------------------------------------- shapes --

def _dims(case):
    """The CPI shapes (C, P, K, R, T, B, S) of a case."""
    if case["kind"] != "batch":
        return [tuple(case[n] for n in ("C", "P", "K", "R", "T", "B", "S"))]
    rng = random.Random(case["dims_seed"])
    out = []
    for _ in range(case["n_cpi"]):
        C, T = rng.choice((4, 8, 16)), rng.choice((2, 3, 4))
        P, R, S = rng.choice((64, 128, 256)), 64 * rng.randint(16, 256), rng.choice((8, 16))
        out.append((C, P, P, R, T, 64, S))
    return out


def _refine_steps(case):
    return 2 if case["solver"] == "mixed_ir" else 1   # what each solver needs (2: see stap.h)


def _plan(case, **kw):
    dims = _dims(case)
    return stap.Plan(dims if case["kind"] == "batch" else dims[0], load_factor=LOAD,
                     refine_steps=_refine_steps(case), precision=PRECISIONS[case["precision"]],
                     solver=SOLVERS[case["solver"]], training=TRAININGS[case["training"]],
                     snapshots=SNAPSHOTS[case["snapshots"]], train_guard=case["guard"],
                     train_half=case["half"], **kw)


# ------------------------------------------------------------------- inputs --

def _generator(seed, sub=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + sub) & 0x7FFFFFFFFFFFFFFF)
    return g


def _randc(shape, g):
    return torch.randn(shape, dtype=torch.complex64, device="cuda", generator=g)   # CN(0, 1)


def _expj(x):
    return torch.complex(torch.cos(x), torch.sin(x))


def _cube(C, P, K, R, S, cnr_db, seed, sub=0):
    """Noise, a clutter ridge of 64 patches (Doppler equal to spatial frequency)
    and four targets, as radar cubes have them: complex64 [C][P][R]."""
    g = _generator(seed, sub)
    cube = _randc((C, P, R), g)
    f = 0.5 * torch.sin(torch.deg2rad(-90.0 + 180.0 * (torch.arange(PATCHES, device="cuda",
                                                                    dtype=torch.float64) + 0.5) / PATCHES))
    alpha = _randc((PATCHES, R), g) * math.sqrt(10.0 ** (cnr_db / 10.0) / PATCHES)
    c = torch.arange(C, device="cuda", dtype=torch.float64)
    p = torch.arange(P, device="cuda", dtype=torch.float64)
    ridge = _expj(2 * math.pi * (c[:, None, None] + p[None, :, None]) * f).to(torch.complex64)
    cube.view(C * P, R).addmm_(ridge.view(C * P, PATCHES), alpha)
    rng = random.Random(seed * 7919 + sub)
    for _ in range(4):
        r0, k0, s0 = rng.randrange(R), rng.randrange(K), rng.randrange(S)
        amp = math.sqrt(10.0 ** (rng.uniform(0.0, 1.5)))
        fs = 0.5 * math.sin(math.radians(-90.0 + 180.0 * (s0 + 0.5) / S))
        cube[:, :, r0] += amp * _expj(2 * math.pi * (fs * c[:, None] + k0 / K * p[None, :])).to(torch.complex64)
    return cube


def _hann(n):
    return torch.from_numpy(np.hanning(n) if n > 1 else np.ones(1)).cuda()


def _doppler(cube, K, T, snapshots, dtype):
    """The Doppler transform by torch's FFT: [rows][K][R] in `dtype`."""
    C, P, R = cube.shape
    x = cube.to(dtype)
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    if snapshots == "adjacent":
        return torch.fft.fft(x * _hann(P).to(real)[None, :, None], n=K, dim=1).contiguous()
    n = P - T + 1                                   # pulses of a sub-window
    out = torch.empty((T, C, K, R), dtype=dtype, device=cube.device)
    for t in range(T):
        h = torch.zeros(P, dtype=real, device=cube.device)
        h[t:t + n] = _hann(n).to(real)
        out[t] = torch.fft.fft(x * h[None, :, None], n=K, dim=1)
    return out.view(T * C, K, R)


def _snapshots(dop, bins, C, T, snapshots):
    """x[k][t*C + c][r] of the bins (a list) from the Doppler rows."""
    K = dop.shape[1]
    if snapshots == "staggered":
        return dop[:, bins].transpose(0, 1)
    parts = [dop[:, [(k + t - T // 2) % K for k in bins]].transpose(0, 1) for t in range(T)]
    return torch.cat(parts, dim=1)                  # [bins][T*C][R]


def _covariance(x, B, dtype=torch.complex128):
    """[bins][NB][D][D] sample covariances of x [bins][D][R]."""
    n, D, R = x.shape
    X = x.view(n, D, R // B, B).transpose(1, 2).to(dtype)
    cov = X @ X.mH / B
    torch.diagonal(cov, dim1=-2, dim2=-1).imag.zero_()
    return cov


def _prepared_covariances(case, seed):
    """Covariances as the solve meets them: of the Doppler output of a cube."""
    C, P, K, R, T, B, S = _dims(case)[0]
    dop = _doppler(_cube(C, P, K, R, S, case["cnr_db"], seed), K, T, "adjacent", torch.complex64)
    cov = torch.empty((K, R // B, C * T, C * T), dtype=torch.complex128, device="cuda")
    for k0 in range(0, K, 16):
        bins = list(range(k0, min(K, k0 + 16)))
        cov[bins] = _covariance(_snapshots(dop, bins, C, T, "adjacent"), B)
    return cov


def _prepared_weights(case, seed):
    """Unit-norm weight vectors around the steering vectors, c64 [K][NB][S][D]."""
    C, P, K, R, T, B, S = _dims(case)[0]
    v = _steering(C, P, K, T, S, "adjacent").to(torch.complex64)
    w = _randc((K, R // B, S, C * T), _generator(seed, 77)) * 0.3 + v / v.abs().mean()
    return w / torch.linalg.vector_norm(w, dim=-1, keepdim=True)


def _front_end(case):
    """Contiguous subarrays of the element channels: W [C][N]."""
    W = np.zeros((case["C"], case["elements"]), np.complex128)
    for c, idx in enumerate(np.array_split(np.arange(case["elements"]), case["C"])):
        W[c, idx] = 1.0
    return W


def prepare(case, seed):
    kind = case["kind"]
    dims = _dims(case)
    C, P, K, R, T, B, S = dims[0]
    st = {"kind": kind}
    if kind in ("cpi", "batch"):
        st["plan"] = _plan(case)
        st["cubes"] = [_cube(d[0], d[1], d[2], d[3], d[6], case["cnr_db"], seed, i) for i, d in enumerate(dims)]
        st["outs"] = [torch.empty((d[6], d[2], d[3]), device="cuda") for d in dims]
    elif kind == "elements":
        st["plan"] = _plan(case, front_end=_front_end(case))
        st["elements"] = _cube(case["elements"], P, K, R, S, case["cnr_db"], seed)
        st["cube"] = torch.empty((C, P, R), dtype=torch.complex64, device="cuda")
        st["outs"] = [torch.empty((S, K, R), device="cuda")]
    else:
        st["plan"] = _plan(case, steps_only=True)
        sh = st["plan"].shapes()
        if kind in ("doppler", "contractions"):
            st["cube"] = _cube(C, P, K, R, S, case["cnr_db"], seed)
            st["dop"] = torch.empty(sh["dop"], dtype=torch.complex64, device="cuda")
        if kind == "contractions":
            st["dop_in"] = _doppler(st["cube"], K, T, "adjacent", torch.complex64)
            st["wts_in"] = _prepared_weights(case, seed)
            st["cov"] = torch.empty(sh["cov"], dtype=torch.complex128, device="cuda")
            st["out"] = torch.empty(sh["out"], device="cuda")
        if kind == "solve":
            st["cov_in"] = _prepared_covariances(case, seed)
            st["wts"] = torch.empty(sh["wts"], dtype=torch.complex64, device="cuda")
    return st


def run(st):
    plan, kind = st["plan"], st["kind"]
    if kind in ("cpi", "batch"):
        return plan.run_cpi(st["cubes"], st["outs"])
    if kind == "elements":
        cube = plan.reduce_channels(st["elements"], st["cube"])
        return [cube] + plan.run_cpi([cube], st["outs"])
    if kind == "doppler":
        return plan.doppler(st["cube"], st["dop"])
    if kind == "solve":
        return plan.solve_weights(st["cov_in"], st["wts"])
    return [plan.doppler(st["cube"], st["dop"]), plan.covariance(st["dop_in"], st["cov"]),
            plan.apply(st["dop_in"], st["wts_in"], st["out"])]


# --------------------------------------------------------------------- work --

def work(case):
    """Bytes: each input read once, each output written once.  Flops: 5 N log2 N
    per FFT, 8 per complex multiply-add; adjacent-bin covariances share the
    products of their bin pairs; the solve counts the C basis right-hand sides
    of the separable steering and the refinement steps that the plan asks for."""
    kind, total_b, total_f = case["kind"], 0, 0
    for C, P, K, R, T, B, S in _dims(case):
        D, NB = C * T, R // B
        st = case["snapshots"] == "staggered"
        rows = D if st else C
        refine = _refine_steps(case)
        pairs = D * (D + 1) // 2 if st else T * C * C - C * (C - 1) // 2
        fft = 5 * rows * R * K * max(1, K.bit_length() - 1)
        cov = 8 * K * R * pairs
        solve = 8 * K * NB * (D ** 3 // 6 + (1 + 2 * refine) * min(C, S) * D * D)
        app = 8 * K * R * S * D
        cube, dop, covb = 8 * C * P * R, 8 * rows * K * R, 16 * K * NB * D * D
        wts, out = 8 * K * NB * S * D, 4 * S * K * R
        if kind in ("cpi", "batch"):
            total_b += cube + out
            total_f += fft + cov + solve + app
        elif kind == "elements":
            N = case["elements"]
            total_b += 8 * N * P * R + cube + out
            total_f += 8 * N * C * P * R + fft + cov + solve + app
        elif kind == "doppler":
            total_b += cube + dop
            total_f += fft
        elif kind == "solve":
            total_b += covb // 2 + wts
            total_f += solve
        else:
            total_b += cube + dop + dop + covb + dop + wts + out
            total_f += fft + cov + app
    return {"bytes": total_b, "flops": total_f}


# -------------------------------------------------------------------- exact --

def _steering(C, P, K, T, S, snapshots, W=None):
    """Steering vectors v[s][t*C + c] in complex128."""
    theta = torch.deg2rad(-90.0 + 180.0 * (torch.arange(S, dtype=torch.float64, device="cuda") + 0.5) / S)
    fs = 0.5 * torch.sin(theta)
    if W is None:
        a = _expj(2 * math.pi * fs[:, None] * torch.arange(C, dtype=torch.float64, device="cuda"))
    else:
        Wt = torch.from_numpy(W).cuda()
        n = torch.arange(Wt.shape[1], dtype=torch.float64, device="cuda")
        a = _expj(2 * math.pi * fs[:, None] * n) @ Wt.conj().T
    if snapshots == "staggered":
        g = torch.full((T,), float(_hann(P - T + 1).sum()), dtype=torch.complex128, device="cuda")
    else:
        m = torch.arange(T, dtype=torch.float64, device="cuda") - T // 2
        p = torch.arange(P, dtype=torch.float64, device="cuda")
        g = (_expj(-2 * math.pi * m[:, None] * p / K) * _hann(P)).sum(1)
    return (g[None, :, None] * a[:, None, :]).reshape(S, T * C)


def _train(cov, case):
    if case["training"] == "own":
        return cov
    g, h = (0, 1) if case["training"] == "neighbours" else (case["guard"], case["half"])
    NB = cov.shape[1]
    out = torch.empty_like(cov)
    for j in range(NB):
        idx = [i for i in list(range(j - g - h, j - g)) + list(range(j + g + 1, j + g + h + 1)) if 0 <= i < NB]
        out[:, j] = cov[:, idx].mean(dim=1)
    return out


def _weights(cov, v):
    """Unit-noise-gain weights [..][S][D] of covariances [..][D][D]."""
    D = cov.shape[-1]
    tr = torch.diagonal(cov, dim1=-2, dim2=-1).real.sum(-1)
    Rl = cov + (LOAD / D) * tr[..., None, None] * torch.eye(D, dtype=cov.dtype, device=cov.device)
    u = torch.linalg.solve(Rl, v.T.expand(*cov.shape[:-2], -1, -1))
    q = (v.T.conj() * u).real.sum(-2, keepdim=True)
    return (u / torch.sqrt(q)).mT


def _chain(cube, d, case, W=None):
    """The whole chain in complex128: power [S][K][R]."""
    C, P, K, R, T, B, S = d
    dop = _doppler(cube, K, T, case["snapshots"], torch.complex128)
    v = _steering(C, P, K, T, S, case["snapshots"], W)
    out = torch.empty((S, K, R), dtype=torch.float64, device="cuda")
    step = max(1, min(K, (1 << 27) // (C * T * max(R, (R // B) * C * T))))
    for k0 in range(0, K, step):
        bins = list(range(k0, min(K, k0 + step)))
        x = _snapshots(dop, bins, C, T, case["snapshots"])
        w = _weights(_train(_covariance(x, B), case), v)          # [bins][NB][S][D]
        X = x.reshape(len(bins), C * T, R // B, B).transpose(1, 2)  # [bins][NB][D][B]
        y = (w.conj() @ X).abs().square()                          # [bins][NB][S][B]
        out[:, bins] = y.permute(2, 0, 1, 3).reshape(S, len(bins), R)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch" or work(case)["flops"] > 4e11:
        return None                                  # minutes in 64 bits
    C, P, K, R, T, B, S = d = _dims(case)[0]
    if kind == "solve":
        cov = _prepared_covariances(case, seed)
        v = _steering(C, P, K, T, S, "adjacent")
        return torch.cat([_weights(cov[k0:k0 + 16], v) for k0 in range(0, K, 16)])
    if kind == "elements":
        W = _front_end(case)
        x = _cube(case["elements"], P, K, R, S, case["cnr_db"], seed)
        cube = torch.zeros((C, P, R), dtype=torch.complex128, device="cuda")
        Wt = torch.from_numpy(W).cuda().conj()
        for n0 in range(0, case["elements"], 50):
            part = x[n0:n0 + 50].to(torch.complex128)
            cube += (Wt[:, n0:n0 + 50] @ part.reshape(part.shape[0], -1)).view(C, P, R)
        return [cube, _chain(cube, d, case, W)]
    cube = _cube(C, P, K, R, S, case["cnr_db"], seed)
    if kind == "cpi":
        return [_chain(cube, d, case)]
    dop = _doppler(cube, K, T, case["snapshots"], torch.complex128)
    if kind == "doppler":
        return dop
    given = _doppler(cube, K, T, "adjacent", torch.complex64)
    wts = _prepared_weights(case, seed)
    cov = torch.empty((K, R // B, C * T, C * T), dtype=torch.complex128, device="cuda")
    out = torch.empty((S, K, R), dtype=torch.float64, device="cuda")
    for k0 in range(0, K, 16):
        bins = list(range(k0, min(K, k0 + 16)))
        x = _snapshots(given, bins, C, T, "adjacent")
        cov[bins] = _covariance(x, B)
        X = x.reshape(len(bins), C * T, R // B, B).transpose(1, 2).to(torch.complex128)
        y = (wts[bins].to(torch.complex128).conj() @ X).abs().square()
        out[:, bins] = y.permute(2, 0, 1, 3).reshape(S, len(bins), R)
    return [dop, cov, out]
