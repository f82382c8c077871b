"""What a user of this framework has it do: the calls that are timed, over the sizes they are made at.

A case is a family of calls with its sizes (``listed``; ``draw`` gives more of the same ranges).  ``prepare``
makes what a program holds before the call (problem handle, inputs, buffers), ``run`` is one pass through the
public entry points, ``work`` the bytes and FP64 operations a pass cannot do without and ``exact`` the same
results by plain torch in 64 bits where that is short to write.

Families:
  burgers           gradient of the final energy with respect to the initial state, batches of members:
                    forward sweep with the trajectory stored, objective, adjoint sweep (slots = 0), or the
                    checkpointed gradient call (slots > 0)
  rb                Rayleigh-Benard gradient of the kinetic energy at T, binomial checkpointing
  rb_terms          the pieces of one Rayleigh-Benard step on their own: F, its JVP and VJP, the collocation
                    transforms and the stage solves, as a caller with its own loop uses them
  kolmogorov        4D-Var gradient of a batch of (mixed) resolutions
  closure           training gradient of the learned closure: state and parameter gradient of a batch of windows
  couette           energy-gain gradient of plane Couette flow
  couette_terms     the pieces of one Couette step on their own
  evp               shear-flow eigenvalues with sensitivities for a batch of pencils
"""
import math

import numpy as np
import torch

from paper_2506_14792_gb300 import spadj

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # one small problem in an optimiser's or a notebook's loop: dependent steps, nothing to fill the chip with
        {"name": "burgers_single", "family": "burgers", "n": 256, "batch": 1, "steps": 100, "order": 2, "slots": 0},
        # the benchmark's ensemble of 16384 members over a short horizon
        {"name": "burgers_ensemble", "family": "burgers", "n": 256, "batch": 16384, "steps": 40, "order": 2, "slots": 0},
        # fourth order, another resolution, a ragged batch, a memory-bound program's checkpoints
        {"name": "burgers_sbdf4_slots", "family": "burgers", "n": 192, "batch": 1000, "steps": 60, "order": 4, "slots": 6},
        # the smallest calls: the pieces of a step at a test-sized resolution
        {"name": "rb_terms_small", "family": "rb_terms", "nx": 64, "nz": 32},
        # the benchmark's Rayleigh-Benard gradient over a short horizon, with recomputation
        {"name": "rb_gradient", "family": "rb", "nx": 256, "nz": 64, "scheme": "rk222", "steps": 40, "slots": 8},
        # third-order scheme at an odd size
        {"name": "rb_rk443", "family": "rb", "nx": 96, "nz": 40, "scheme": "rk443", "steps": 10, "slots": 4},
        # a single flow assimilated on its own
        {"name": "kolmogorov_single", "family": "kolmogorov", "sizes": "192", "count": 1, "steps": 16, "slots": 0},
        # the benchmark's mixed-resolution batch, one observation window
        {"name": "kolmogorov_batch", "family": "kolmogorov", "sizes": "128,256,384,512", "count": 64, "steps": 8, "slots": 0},
        # one training iteration's gradient of the learned closure (benchmark sizes, a shorter window)
        {"name": "closure_windows", "family": "closure", "n": 64, "batch": 128, "steps": 8},
        # the benchmark's Couette gradient over a few steps
        {"name": "couette_gradient", "family": "couette", "nx": 128, "ny": 64, "nz": 64, "steps": 8, "slots": 0},
        # the pieces of a Couette step at a ragged size
        {"name": "couette_terms_odd", "family": "couette_terms", "nx": 48, "ny": 36, "nz": 40},
        # a neutral-curve scan's batch of eigenproblems
        {"name": "evp_scan", "family": "evp", "n": 48, "pencils": 96, "iters": 20},
    ]


# resolutions whose 3/2-dealiased transforms factor into 2s and 3s
SMOOTH = sorted(4 * 2 ** a * 3 ** b for a in range(8) for b in range(4))


def _pick(rng, lo, hi, of=SMOOTH):
    """A value of `of` near exp(uniform(log lo, log hi))."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((x for x in of if lo <= x <= hi), key=lambda x: abs(math.log(x / v)))


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    f = rng.choice(["burgers", "burgers", "rb", "rb_terms", "kolmogorov", "kolmogorov", "closure", "couette",
                    "couette_terms", "evp"])
    z = [n for n in range(16, 97, 4)]
    if f == "burgers":
        n = _pick(rng, 32, 512)
        cap = 16384 * 40 * 256 // n  # member-steps of the listed ensemble
        steps = _log_int(rng, 10, 100)
        return {"family": f, "n": n, "batch": _log_int(rng, 1, max(1, min(16384, cap // (2 * steps)))), "steps": steps,
                "order": rng.choice([1, 2, 2, 3, 4]), "slots": rng.choice([0, 0, _log_int(rng, 3, 12)])}
    if f == "rb":
        return {"family": f, "nx": _pick(rng, 32, 384), "nz": _pick(rng, 16, 72, z),
                "scheme": rng.choice(["rk222", "rk222", "rk443"]), "steps": _log_int(rng, 5, 30), "slots": rng.choice([0, 3, 6])}
    if f == "rb_terms":
        return {"family": f, "nx": _pick(rng, 32, 384), "nz": _pick(rng, 16, 72, z)}
    if f == "kolmogorov":
        sizes = sorted({_pick(rng, 32, 512) for _ in range(rng.randint(1, 4))})
        return {"family": f, "sizes": ",".join(map(str, sizes)), "count": _log_int(rng, 1, 32), "steps": _log_int(rng, 4, 12),
                "slots": rng.choice([0, 0, 2])}
    if f == "closure":
        return {"family": f, "n": rng.choice([32, 48, 64, 96]), "batch": _log_int(rng, 4, 96), "steps": rng.randint(2, 8)}
    if f == "couette":
        return {"family": f, "nx": _pick(rng, 16, 128), "ny": _pick(rng, 8, 64, [8, 12, 16, 24, 32, 36, 48, 64]),
                "nz": _pick(rng, 16, 64, z), "steps": rng.randint(3, 8), "slots": rng.choice([0, 0, 3])}
    if f == "couette_terms":
        return {"family": f, "nx": _pick(rng, 16, 128), "ny": _pick(rng, 8, 64, [8, 12, 16, 24, 32, 36, 48, 64]),
                "nz": _pick(rng, 16, 64, z)}
    return {"family": f, "n": _pick(rng, 24, 64, z), "pencils": _log_int(rng, 4, 152), "iters": rng.randint(8, 30)}


# ---- inputs ---------------------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _cnormal(shape, g):
    return torch.complex(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64),
                         torch.randn(shape, generator=g, device="cuda", dtype=torch.float64))


def _burgers_state(n, batch, g):
    """Members u0 = sum_{k <= 16} k^-2 (a_k cos kx + b_k sin kx), scaled to max |u0| = 1."""
    K = n // 2
    k = torch.arange(1, min(16, K - 1) + 1, device="cuda", dtype=torch.float64)
    c = torch.zeros((batch, K), dtype=torch.complex128, device="cuda")
    c[:, 1:len(k) + 1] = _cnormal((batch, len(k)), g) / (2.0 * k * k)
    return c / _irfft(c, 1024).abs().amax(dim=1, keepdim=True)


def _kolmogorov_state(n, g):
    """Vorticity with energy spectrum k^-3 for 1 <= |k| <= n/3 and random phases, rms velocity 1."""
    kx, ky = _kol_wavenumbers(n)
    k2 = kx * kx + ky * ky
    k = k2.sqrt()
    band = (k >= 1) & (k <= n / 3.0) & (ky != -(n // 2))
    ph = torch.rand(k.shape, generator=g, device="cuda", dtype=torch.float64) * TWO_PI
    w = torch.where(band, torch.polar(1.0 / k.clamp(min=1.0), ph), 0.0)
    w = _kol_project(w)
    e = (torch.where(kx == 0, 1.0, 2.0) * w.abs() ** 2 / k2.clamp(min=1.0)).sum()
    return w / e.sqrt()


def _plane_hermitian(s):
    """(.., ky, kx, n) coefficients of a real field: no ky = -Ny/2 row, kx = 0 plane Hermitian in ky."""
    ny = s.shape[-3]
    s[..., ny // 2, :, :] = 0.0
    neg = (-torch.arange(ny, device=s.device)) % ny
    s[..., :, 0, :] = 0.5 * (s[..., :, 0, :] + s[..., neg, 0, :].conj())
    return s


def _rb_fields(nx, nz, g, amp):
    """Velocity and temperature coefficients with decaying spectra (developed convection's shape)."""
    m = torch.arange(nx // 2, device="cuda", dtype=torch.float64)[:, None]
    n = torch.arange(nz, device="cuda", dtype=torch.float64)[None, :]
    s = amp * _cnormal((3, nx // 2, nz), g) / ((1.0 + m) * (1.0 + n) ** 2)
    s[:, 0] = s[:, 0].real + 0j
    return s


def _rb_start(nx, nz, g):
    """Temperature noise 1e-3 that vanishes at both walls (phi_n = T_{n+2} - T_n), fluid at rest."""
    a = _rb_fields(nx, nz - 2, g, 1e-3)[2]
    s = torch.zeros((3, nx // 2, nz), dtype=torch.complex128, device="cuda")
    s[2, :, 2:] += a
    s[2, :, :nz - 2] -= a
    return s


def _couette_fields(nx, ny, nz, g, amp):
    kx = torch.arange(nx // 2, device="cuda", dtype=torch.float64)[None, :, None]
    ky = torch.fft.fftfreq(ny, 1.0 / ny, device="cuda", dtype=torch.float64)[:, None, None]
    n = torch.arange(nz, device="cuda", dtype=torch.float64)[None, None, :]
    s = amp * _cnormal((3, ny, nx // 2, nz), g) / ((1.0 + kx * kx + ky * ky) * (1.0 + n) ** 2)
    return _plane_hermitian(s)


def _couette_start(nx, ny, nz, g):
    """Perturbation that vanishes at both walls (each coefficient column times T_{n+2} - T_n)."""
    a = _couette_fields(nx, ny, nz - 2, g, 1e-3)
    s = torch.zeros((3, ny, nx // 2, nz), dtype=torch.complex128, device="cuda")
    s[..., 2:] += a
    s[..., :nz - 2] -= a
    return s


def _cnn_params(n, g):
    """Initial weights N(0, 1/fan_in), zero biases, small last layer (1-32-32-32-1 channels, 3 x 3)."""
    parts = []
    ch = (1, 32, 32, 32, 1)
    for i in range(4):
        w = torch.randn(ch[i + 1] * ch[i] * 9, generator=g, device="cuda", dtype=torch.float64) / math.sqrt(9 * ch[i])
        parts += [w * (0.01 if i == 3 else 1.0), torch.zeros(ch[i + 1], device="cuda", dtype=torch.float64)]
    p = torch.cat(parts)
    assert p.numel() == n
    return p


def _sizes(case):
    res = [int(v) for v in case["sizes"].split(",")]
    return [res[i * len(res) // case["count"]] for i in range(case["count"])] if case["count"] >= len(res) else res[:case["count"]]


def _obs_steps(steps):
    every = max(1, steps // 4)
    return list(range(every, steps + 1, every))


def _inputs(case, seed):
    """The case's inputs from the seed alone."""
    g, f = _gen(seed), case["family"]
    if f == "burgers":
        return {"x0": _burgers_state(case["n"], case["batch"], g)}
    if f == "rb":
        return {"x0": _rb_start(case["nx"], case["nz"], g)}
    if f == "rb_terms":
        a = [_rb_fields(case["nx"], case["nz"], g, v) for v in (0.1, 0.1, 1.0)]
        grid = torch.randn((3 * case["nz"] // 2, 3 * case["nx"] // 2), generator=g, device="cuda", dtype=torch.float64)
        return {"x": a[0], "dx": a[1], "y": a[2], "c": a[0][0].contiguous(), "g": grid}
    if f == "kolmogorov":
        sizes = _sizes(case)
        x0 = torch.cat([_kolmogorov_state(n, g).reshape(-1) for n in sizes])
        obs = torch.stack([torch.cat([_kolmogorov_state(n, g).reshape(-1) for n in sizes]) for _ in _obs_steps(case["steps"])])
        return {"x0": x0, "obs": obs}
    if f == "closure":
        n, b = case["n"], case["batch"]
        x0 = torch.stack([_kolmogorov_state(n, g) for _ in range(b)])
        obs = torch.stack([x0 + 0.01 * torch.stack([_kolmogorov_state(n, g) for _ in range(b)]) for _ in range(case["steps"])])
        return {"x0": x0, "obs": obs}
    if f == "couette":
        return {"x0": _couette_start(case["nx"], case["ny"], case["nz"], g)}
    if f == "couette_terms":
        a = [_couette_fields(case["nx"], case["ny"], case["nz"], g, v) for v in (0.1, 0.1, 1.0)]
        grid = torch.randn((3 * case["nz"] // 2, 3 * case["ny"] // 2, 3 * case["nx"] // 2), generator=g, device="cuda",
                           dtype=torch.float64)
        return {"x": a[0], "dx": a[1], "y": a[2], "c": a[0][0].contiguous(), "g": grid}
    p, n = case["pencils"], case["n"]
    rng = np.random.default_rng(int(seed))
    alpha = 0.6 + 0.7 * (np.arange(p) + rng.random(p)) / p
    return {"pencils": [(float(a), 0.0, 8000.0) for a in alpha], "shifts": [complex(0.0, -0.25 * a) for a in alpha],
            "x": _cnormal((p, 3 * n), g), "psi": _cnormal((p, 3 * n), g)}


ORDERS = {1: spadj.SPADJ_SBDF1, 2: spadj.SPADJ_SBDF2, 3: spadj.SPADJ_SBDF3, 4: spadj.SPADJ_SBDF4}
DT = {"burgers": 1e-3, "rb": 1e-3, "rb_terms": 1e-3, "kolmogorov": 5e-4, "closure": 4e-3, "couette": 5e-3, "couette_terms": 5e-3}


def prepare(case, seed):
    f = case["family"]
    s = dict(case, **_inputs(case, seed))
    if f == "burgers":
        s["p"] = p = spadj.Problem(spadj.SPADJ_BURGERS1D, ORDERS[case["order"]], [case["n"]], [TWO_PI], [0.01], DT[f],
                                   batch=case["batch"])
        x = s["x0"]
        s["grad"], s["seed_vec"], s["xn"] = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
        s["J"] = torch.empty(case["batch"], dtype=torch.float64, device="cuda")
        if not case["slots"]:
            s["traj"] = torch.empty((case["steps"] + 1,) + tuple(x.shape), dtype=x.dtype, device="cuda")
    elif f in ("rb", "rb_terms"):
        sch = spadj.SPADJ_RK443 if case.get("scheme") == "rk443" else spadj.SPADJ_RK222
        s["p"] = spadj.Problem(spadj.SPADJ_RB2D, sch, [case["nx"], case["nz"]], [4.0], [1e6, 1.0], DT[f])
    elif f == "kolmogorov":
        sizes = _sizes(case)
        s["p"] = spadj.Problem(spadj.SPADJ_KOLMOGOROV2D, spadj.SPADJ_SBDF2, [sizes[0]], [TWO_PI], [100.0, 0.0], DT[f],
                               batch=len(sizes), batch_n=sizes)
        s["p"].set_observations(_obs_steps(case["steps"]), s.pop("obs"), 32)
    elif f == "closure":
        s["p"] = spadj.Problem(spadj.SPADJ_KOLMOGOROV2D, spadj.SPADJ_SBDF2, [case["n"]], [TWO_PI], [1000.0, 0.0], DT[f],
                               batch=case["batch"], closure=True)
        s["p"].set_observations(list(range(1, case["steps"] + 1)), s.pop("obs"), case["n"] // 2 - 1)
        s["params"] = _cnn_params(s["p"].state_len(2), _gen(int(seed) + 1))
        s["grad_p"] = torch.empty_like(s["params"])
    elif f in ("couette", "couette_terms"):
        s["p"] = spadj.Problem(spadj.SPADJ_COUETTE3D, spadj.SPADJ_SBDF2, [case["nx"], case["ny"], case["nz"]],
                               [2 * TWO_PI, TWO_PI], [1000.0, 0.0], DT[f])
    else:
        s["p"] = spadj.Problem(spadj.SPADJ_SHEAR_EVP, 0, (0, 0, case["n"]), (0.0, 0.0, 0.0), (1,), 1.0, batch=case["pencils"])
        s["xi"], s["psii"] = torch.empty_like(s["x"]), torch.empty_like(s["psi"])
        s["out"] = torch.zeros((case["pencils"], 10), dtype=torch.float64, device="cuda")
    if f in ("rb", "kolmogorov", "closure", "couette"):
        s["grad"], s["xn"] = torch.empty_like(s["x0"]), torch.empty_like(s["x0"])
    if f in ("rb_terms", "couette_terms"):
        for k in ("F", "dF", "vjp", "solve", "solve_t"):
            s[k] = torch.empty_like(s["x"])
        s["c2g"], s["g2c"] = torch.empty_like(s["g"]), torch.empty_like(s["c"])
        s["c2g_adj"], s["g2c_adj"] = torch.empty_like(s["c"]), torch.empty_like(s["g"])
    return s


def run(s):
    f, p = s["family"], s["p"]
    if f == "burgers":
        if s["slots"]:
            p.gradient(s["x0"], s["steps"], s["grad"], ckpt_slots=s["slots"], want_J=False)
            return {"grad": s["grad"]}
        p.forward(s["steps"], s["x0"], s["xn"], s["traj"])
        p.objective(s["xn"], s["J"], s["seed_vec"])
        p.adjoint(s["steps"], s["traj"], s["seed_vec"], s["grad"])
        return {"xn": s["xn"], "J": s["J"], "grad": s["grad"]}
    if f == "rb":
        p.gradient(s["x0"], s["steps"], s["grad"], ckpt_slots=s["slots"], want_J=False)
        return {"grad": s["grad"]}
    if f in ("rb_terms", "couette_terms"):
        p.eval_F(s["x"], s["F"])
        p.eval_F_jvp(s["x"], s["dx"], s["dF"])
        p.eval_F_vjp(s["x"], s["y"], s["vjp"])
        p.transform(spadj.C2G, s["c"], s["c2g"])
        p.transform(spadj.G2C, s["g"], s["g2c"])
        p.transform(spadj.C2G_ADJ, s["g"], s["c2g_adj"])
        p.transform(spadj.G2C_ADJ, s["c"], s["g2c_adj"])
        p.solve(s["x"], s["solve"])
        p.solve(s["y"], s["solve_t"], transpose=True)
        return {k: s[k] for k in ("F", "dF", "vjp", "c2g", "g2c", "c2g_adj", "g2c_adj", "solve", "solve_t")}
    if f == "kolmogorov":
        p.gradient(s["x0"], s["steps"], s["grad"], objective=spadj.SPADJ_OBJ_FOURDVAR, ckpt_slots=s["slots"], want_J=False)
        return {"grad": s["grad"]}
    if f == "closure":
        p.set_params(s["params"])
        p.gradient(s["x0"], s["steps"], s["grad"], objective=spadj.SPADJ_OBJ_FOURDVAR, grad_p=s["grad_p"], want_J=False)
        return {"grad": s["grad"], "grad_p": s["grad_p"]}
    if f == "couette":
        p.gradient(s["x0"], s["steps"], s["grad"], objective=spadj.SPADJ_OBJ_GAIN, ckpt_slots=s["slots"], want_J=False)
        return {"grad": s["grad"]}
    s["xi"].copy_(s["x"])
    s["psii"].copy_(s["psi"])
    p.eigen(s["pencils"], s["shifts"], s["iters"], s["xi"], s["psii"], s["out"])
    return {"x": s["xi"], "psi": s["psii"], "out": s["out"]}


# ---- the work of a pass -----------------------------------------------------------------------------------


def _fft(n):
    """FP64 operations of one complex FFT of length n."""
    return 5.0 * n * math.log2(n)


def _rb_F(nx, nz, fields):
    """Collocation transforms of `fields` scalar fields: x FFTs of every grid row, z as folded matrices."""
    mx, mz = 3 * nx // 2, 3 * nz // 2
    return fields * (mz * 0.5 * _fft(mx) + 4.0 * (nx // 2) * nz * mz / 2)


def _cou_F(nx, ny, nz, fields):
    mx, my, mz = 3 * nx // 2, 3 * ny // 2, 3 * nz // 2
    return fields * (mz * my * 0.5 * _fft(mx) + mz * (nx // 2) * _fft(my) + 4.0 * (nx // 2) * ny * nz * mz / 2)


def work(case):
    f = case["family"]
    if f == "burgers":
        K, M = case["n"] // 2, 3 * case["n"] // 2
        state = case["batch"] * K * 16.0
        # forward step: two real transforms; adjoint step: three
        return {"bytes": state * (2 if case["slots"] else 2 + 2 * (case["steps"] + 1)),
                "flops": case["batch"] * case["steps"] * 5.0 * (0.5 * _fft(M) + 8.0 * K)}
    if f in ("rb", "rb_terms"):
        nx, nz = case["nx"], case["nz"]
        state, solve = 3 * (nx // 2) * nz * 16.0, 2.0 * (nx // 2) * (1.5 * nz) ** 2 * 4
        if f == "rb":
            st = 4 if case["scheme"] == "rk443" else 2
            return {"bytes": 2 * state, "flops": case["steps"] * st * (_rb_F(nx, nz, 11 + 22) + 2 * solve)}
        grid = 2.25 * nx * nz * 8.0
        return {"bytes": state * 12 + 4 * (grid + state / 3), "flops": _rb_F(nx, nz, 11 + 19 + 22 + 4) + 2 * solve}
    if f in ("kolmogorov", "closure"):
        sizes = _sizes(case) if f == "kolmogorov" else [case["n"]] * case["batch"]
        state = sum(n * n // 2 for n in sizes) * 16.0
        # forward step: four inverse and one forward 2D transform; adjoint step: nine
        fl = sum(14.0 * (1.5 * n * 0.5 * _fft(3 * n // 2) + 0.5 * n * _fft(3 * n // 2)) for n in sizes)
        if f == "closure":  # 3 x 3 network 1-32-32-32-1: forward, input and weight gradients on every grid point
            fl += sum(3 * 2.0 * 2.25 * n * n * 9 * (32 + 1024 + 1024 + 32) for n in sizes)
            return {"bytes": state * (2 + case["steps"]), "flops": case["steps"] * fl}
        return {"bytes": state * (2 + len(_obs_steps(case["steps"]))), "flops": case["steps"] * fl}
    if f in ("couette", "couette_terms"):
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        state, solve = 3 * (nx // 2) * ny * nz * 16.0, (nx // 2) * ny * 8.0 * 40 * 4 * nz
        if f == "couette":
            return {"bytes": 2 * state, "flops": case["steps"] * (_cou_F(nx, ny, nz, 9 + 15) + 2 * solve)}
        grid = 3.375 * nx * ny * nz * 8.0
        return {"bytes": state * 12 + 4 * (grid + state / 3), "flops": _cou_F(nx, ny, nz, 9 + 15 + 15 + 4) + 2 * solve}
    n, P = case["n"], case["pencils"]
    return {"bytes": P * (4 * 3 * n * 16.0 + 80), "flops": P * (case["iters"] * 2 * 8.0 * 40 * 4 * n + 8.0 * 4 * n * 12 * 40)}


# ---- the same results in 64 bits by plain torch -----------------------------------------------------------


def _irfft(c, M):
    """Grid values of sum_k over the Hermitian-completed half spectrum (last axis)."""
    return torch.fft.irfft(torch.nn.functional.pad(c, (0, M // 2 + 1 - c.shape[-1])), n=M) * M


def _x_c2g(c, M):
    return _irfft(c, M)


def _x_g2c(g, K):
    return torch.fft.rfft(g)[..., :K] / g.shape[-1]


def _x_weights(K):
    w = torch.full((K,), 2.0, dtype=torch.float64, device="cuda")
    w[0] = 1.0
    return w


def _x_c2g_adj(g, K):
    c = torch.fft.rfft(g)[..., :K] * _x_weights(K)
    c[..., 0] = c[..., 0].real + 0j
    return c


def _x_g2c_adj(c, M):
    return _irfft(c / _x_weights(c.shape[-1]), M) / M


SBDF = {1: ([1.0, -1.0], [1.0]), 2: ([1.5, -2.0, 0.5], [2.0, -1.0]), 3: ([11 / 6, -3.0, 1.5, -1 / 3], [3.0, -3.0, 1.0]),
        4: ([25 / 12, -4.0, 3.0, -4 / 3, 0.25], [4.0, -6.0, 4.0, -1.0])}


def _multistep_gradient(x0, steps, dt, order, lam, F, vjp, project, cotangent):
    """Trajectory X_0..X_N of the SBDF scheme (lower orders first) for dX/dt + lam X = F(X), and the exact
    discrete gradient with dJ/dX_n = cotangent(n, X) (None where J does not depend on X_n)."""
    X, Fs = [x0], []
    for n in range(1, steps + 1):
        a, c = SBDF[min(n, order)]
        Fs.append(F(X[-1]))
        r = sum(ci * Fs[n - 1 - i] for i, ci in enumerate(c)) - sum(ai / dt * X[n - 1 - i] for i, ai in enumerate(a[1:]))
        X.append(project(r / (a[0] / dt + lam)))
    Y = {}
    for n in range(steps, -1, -1):
        r = cotangent(n, X)
        r = torch.zeros_like(x0) if r is None else r.clone()
        w = None
        for i in range(1, order + 1):
            if n + i > steps:
                break
            a, c = SBDF[min(n + i, order)]
            if i < len(a):
                r = r - a[i] / dt * Y[n + i]
                w = c[i - 1] * Y[n + i] + (0 if w is None else w)
        if w is not None:
            r = r + vjp(X[n], w)
        if n == 0:
            return X, r
        Y[n] = project(r) / (SBDF[min(n, order)][0][0] / dt + lam)
        Y.pop(n + order, None)


def _exact_burgers(case, x0):
    K, M = case["n"] // 2, 3 * case["n"] // 2
    ik = 1j * torch.arange(K, device="cuda", dtype=torch.float64)

    def project(x):
        x = x.clone()
        x[:, 0] = x[:, 0].real + 0j
        return x

    def grad_of_energy(x):
        return project(x) * TWO_PI * _x_weights(K)

    X, g = _multistep_gradient(
        x0, case["steps"], DT["burgers"], case["order"], 0.01 * ik.imag ** 2,
        lambda x: -ik * _x_g2c(0.5 * _x_c2g(x, M) ** 2, K),
        lambda x, y: _x_c2g_adj(_x_c2g(x, M) * _x_g2c_adj(ik * y, M), K),
        project, lambda n, X: grad_of_energy(X[n]) if n == case["steps"] else None)
    if case["slots"]:
        return {"grad": g}
    xn = X[-1]
    return {"xn": xn, "J": 0.5 * TWO_PI * (xn[:, 0].real ** 2 + 2.0 * (xn[:, 1:].abs() ** 2).sum(dim=1)), "grad": g}


def _kol_wavenumbers(n):
    kx = torch.arange(n // 2, device="cuda", dtype=torch.float64)[:, None]
    ky = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)[None, :]
    return kx.expand(n // 2, n), ky.expand(n // 2, n)


def _kol_project(w):
    n = w.shape[-1]
    w = w.clone()
    w[..., n // 2] = 0.0
    neg = (-torch.arange(n, device=w.device)) % n
    w[..., 0, :] = 0.5 * (w[..., 0, :] + w[..., 0, neg].conj())
    w[..., 0, 0] = w[..., 0, 0].real + 0j
    return w


def _exact_kolmogorov(case, x0, obs):
    """Members of one resolution together: [b][kx][ky]."""
    sizes, steps, at = _sizes(case), case["steps"], _obs_steps(case["steps"])
    off = np.concatenate([[0], np.cumsum([n * n // 2 for n in sizes])])
    grad = torch.empty_like(x0)
    for n in sorted(set(sizes)):
        mem = [b for b, m in enumerate(sizes) if m == n]
        take = lambda v: torch.stack([v[off[b]:off[b + 1]].view(n // 2, n) for b in mem])  # noqa: E731
        M, K = 3 * n // 2, n // 2
        kx, ky = _kol_wavenumbers(n)
        k2 = kx * kx + ky * ky
        inv = torch.where(k2 > 0, 1.0 / k2.clamp(min=1.0), 0.0)
        mult = [1j * ky * inv, -1j * kx * inv, 1j * kx, 1j * ky]
        mask = ((kx <= 32) & (ky.abs() <= 32)).to(torch.float64)
        force = torch.zeros((K, n), dtype=torch.complex128, device="cuda")
        force[0, 4] = force[0, n - 4] = -2.0

        def ypad(c):
            out = torch.zeros(c.shape[:-1] + (M,), dtype=c.dtype, device="cuda")
            out[..., :K], out[..., M - K + 1:] = c[..., :K], c[..., K + 1:]
            return out

        def ycut(c):
            out = torch.zeros(c.shape[:-1] + (n,), dtype=c.dtype, device="cuda")
            out[..., :K], out[..., K + 1:] = c[..., :K], c[..., M - K + 1:]
            return out

        def c2g(c):  # grid [b][y][x]
            return _x_c2g((torch.fft.ifft(ypad(c)) * M).transpose(-1, -2), M)

        def g2c(g):
            return ycut(torch.fft.fft(_x_g2c(g, K).transpose(-1, -2)) / M)

        def c2g_adj(g):
            return ycut(torch.fft.fft(_x_c2g_adj(g, K).transpose(-1, -2)))

        def g2c_adj(c):
            return _x_g2c_adj(torch.fft.ifft(ypad(c)).transpose(-1, -2), M)

        def F(x):
            u, v, wx, wy = (c2g(m * x) for m in mult)
            return force - g2c(u * wx + v * wy)

        def vjp(x, y):
            g = g2c_adj(y)
            u, v, wx, wy = (c2g(m * x) for m in mult)
            return sum(m.conj() * c2g_adj(-g * b) for m, b in zip(mult, (wx, wy, u, v)))

        ob = [take(o) for o in obs]
        _, gr = _multistep_gradient(take(x0), steps, DT["kolmogorov"], 2, k2 / 100.0, F, vjp, _kol_project,
                                    lambda t, X: mask * (X[t] - ob[at.index(t)]) if t in at else None)
        for i, b in enumerate(mem):
            grad[off[b]:off[b + 1]] = gr[i].reshape(-1)
    return {"grad": grad}


def _cheb(N, M, scale):
    """Matrices c2g (M x N), g2c (N x M) on the Gauss grid and the derivative in the T basis (times scale)."""
    th = math.pi * (1.0 - (np.arange(M) + 0.5) / M)
    C = np.cos(np.outer(th, np.arange(N)))
    G = (np.where(np.arange(N) == 0, 1.0, 2.0)[:, None] / M) * C.T
    D = np.zeros((N, N))
    for n in range(N):
        for k in range(n - 1, -1, -2):
            D[k, n] = scale * (n if k == 0 else 2.0 * n)
    t = lambda a: torch.from_numpy(a).to("cuda", torch.float64)  # noqa: E731
    return t(C), t(G), t(D)


def _mm(a, m):
    """a @ m for complex a and real m."""
    return torch.complex(a.real @ m, a.imag @ m)


def _terms(case, s):
    """Pieces of a step shared by Rayleigh-Benard (c: [kx][n], grid [z][x]) and Couette (c: [ky][kx][n], grid
    [z][y][x]): collocation transforms and their adjoints."""
    rb = case["family"] == "rb_terms"
    N, Kx = case["nz"], case["nx"] // 2
    Mz, Mx = 3 * N // 2, 3 * Kx
    Cz, Gz, Dz = _cheb(N, Mz, 2.0 if rb else 1.0)
    if not rb:
        Ny = case["ny"]
        My, K = 3 * Ny // 2, Ny // 2

    def ypad(m):  # [z][ky][kx] -> [z][My][kx]
        out = torch.zeros((m.shape[0], My, m.shape[2]), dtype=m.dtype, device="cuda")
        out[:, :K], out[:, My - K + 1:] = m[:, :K], m[:, K + 1:]
        return out

    def ycut(m):
        out = torch.zeros((m.shape[0], Ny, m.shape[2]), dtype=m.dtype, device="cuda")
        out[:, :K], out[:, K + 1:] = m[:, :K], m[:, My - K + 1:]
        return out

    to_z = lambda c, m: _mm(c, m).movedim(-1, 0)  # noqa: E731
    from_z = lambda m, a: _mm(m.movedim(0, -1), a)  # noqa: E731
    yi = (lambda m: m) if rb else (lambda m: torch.fft.ifft(ypad(m), dim=1) * My)
    yf = (lambda m: m) if rb else (lambda m: ycut(torch.fft.fft(m, dim=1)))
    ny = 1.0 if rb else float(My)
    c2g = lambda c: _x_c2g(yi(to_z(c, Cz.T)), Mx)  # noqa: E731
    g2c = lambda g: from_z(yf(_x_g2c(g, Kx)) / ny, Gz.T)  # noqa: E731
    c2g_adj = lambda g: from_z(yf(_x_c2g_adj(g, Kx)), Cz)  # noqa: E731
    g2c_adj = lambda c: _x_g2c_adj(yi(to_z(c, Gz)) / ny, Mx)  # noqa: E731
    dz, dza = (lambda c: _mm(c, Dz.T)), (lambda c: _mm(c, Dz))
    ia = 1j * (TWO_PI / (4.0 if rb else 2 * TWO_PI)) * torch.arange(Kx, device="cuda", dtype=torch.float64)[:, None]
    x, dx, y = s["x"], s["dx"], s["y"]
    if rb:
        fields = lambda c: [c2g(v) for v in (c[0], c[1], ia * c[0], dz(c[0]), ia * c[1], dz(c[1]), ia * c[2], dz(c[2]))]  # noqa: E731
        q, d = fields(x), fields(dx)
        adv = lambda a, b: [-(a[0] * b[i] + a[1] * b[i + 1]) for i in (2, 4, 6)]  # noqa: E731
        F = torch.stack([g2c(v) for v in adv(q, q)])
        dF = torch.stack([g2c(v + w) for v, w in zip(adv(d, q), adv(q, d))])
        h = [g2c_adj(v) for v in y]
        bar = [-sum(h[i] * q[2 + 2 * i] for i in range(3)), -sum(h[i] * q[3 + 2 * i] for i in range(3))]
        grads = [c2g_adj(-h[i] * q[j]) for i in range(3) for j in (0, 1)]
        bx = [-ia * grads[2 * i] + dza(grads[2 * i + 1]) for i in range(3)]
        vjp = torch.stack([c2g_adj(bar[0]) + bx[0], c2g_adj(bar[1]) + bx[1], bx[2]])
    else:
        ib = 1j * torch.fft.fftfreq(Ny, 1.0 / Ny, device="cuda", dtype=torch.float64)[:, None, None]
        fields = lambda c: [c2g(v) for v in (c[0], c[1], c[2], ib * c[2] - dz(c[1]), dz(c[0]) - ia * c[2], ia * c[1] - ib * c[0])]  # noqa: E731
        q, d = fields(x), fields(dx)
        cross = lambda a, b: [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]  # noqa: E731
        F = torch.stack([g2c(v) for v in cross(q[:3], q[3:])])
        dF = torch.stack([g2c(v + w) for v, w in zip(cross(d[:3], q[3:]), cross(q[:3], d[3:]))])
        h = [g2c_adj(v) for v in y]
        cu, cv, cw = (c2g_adj(v) for v in cross(q[3:], h))
        ox, oy, oz = (c2g_adj(v) for v in cross(h, q[:3]))
        vjp = torch.stack([cu + dza(oy) + ib * oz, cv - dza(ox) - ia * oz, cw - ib * ox + ia * oy])
    return {"F": F, "dF": dF, "vjp": vjp, "c2g": c2g(s["c"]), "g2c": g2c(s["g"]), "c2g_adj": c2g_adj(s["g"]),
            "g2c_adj": g2c_adj(s["c"]), "solve": None, "solve_t": None}


def exact(case, seed):
    f = case["family"]
    if f not in ("burgers", "kolmogorov", "rb_terms", "couette_terms"):
        return None
    s = _inputs(case, seed)
    if f == "burgers":
        return _exact_burgers(case, s["x0"])
    if f == "kolmogorov":
        return _exact_kolmogorov(case, s["x0"], s["obs"])
    return _terms(case, s)
