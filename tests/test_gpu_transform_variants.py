"""Variants of the transforms' kernels that only some sizes and batches reach, against the oracle at the bars of the
problems' own parity tests: rows too long for the fixed-point transforms, rows of very different amplitude in one CTA, the
Kolmogorov launch with twice the threads for few long rows, and the Burgers kernels of full batches (also under a
step-size schedule)."""
import numpy as np
import pytest

import synthetic
from oracle import burgers as obur
from oracle import imex
from oracle import rayleigh_benard as orb
from tests import test_gpu_burgers as tb
from tests import test_gpu_kolmogorov as tk
from tests.gpu_util import TOL, dev, host, rel_err
from tests.rb_util import F_T, F_T_jvp, F_T_vjp, gpu_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _z(shape):
    return torch.zeros(shape, dtype=torch.complex128, device="cuda")


@pytest.mark.parametrize("rows", [0, 1, 2])
def test_rows_beyond_the_fixed_point_range(rows):
    """1152 complex points a row: FP64 butterflies, one and two inputs per job, by rows per CTA (0: timed)."""
    from paper_2506_14792_gb300 import spadj
    Nx, Nz = 1536, 8
    o = orb.RayleighBenard(Nx, Nz, 1e6)
    p = gpu_problem(Nx, Nz)
    if rows:
        p.set_option(8, rows)
    s, d = (synthetic.random_coeffs((3, o.Kx, o.N), seed=i) for i in (1, 2))
    s[:, 0], d[:, 0] = s[:, 0].real, d[:, 0].real
    g = np.random.default_rng(3).standard_normal((o.Mz, o.Mx))
    og, oc, out = torch.zeros((o.Mz, o.Mx), dtype=torch.float64, device="cuda"), _z((o.Kx, o.N)), _z((3, o.Kx, o.N))
    p.transform(spadj.C2G, dev(s[0]), og)
    assert rel_err(host(og), o.c2g(s[0])) < 1e-13
    p.transform(spadj.G2C_ADJ, dev(s[0]), og)
    assert rel_err(host(og), o.g2c_adj(s[0])) < 1e-13
    p.transform(spadj.G2C, dev(g), oc)
    assert rel_err(host(oc), o.g2c(g)) < 1e-13
    p.transform(spadj.C2G_ADJ, dev(g), oc)
    assert rel_err(host(oc), o.c2g_adj(g)) < 1e-13
    X = o.pencils(s)
    p.eval_F(dev(s), out)
    assert rel_err(host(out), F_T(o, X)) < 1e-12
    p.eval_F_jvp(dev(s), dev(d), out)
    assert rel_err(host(out), F_T_jvp(o, X, o.pencils(d))) < 1e-12
    p.eval_F_vjp(dev(s), dev(d), out)
    assert rel_err(host(out), F_T_vjp(o, X, d)) < 1e-12
    p.close()


def test_rows_of_different_amplitude_in_one_cta():
    """30 rows (no multiple of 4) of amplitudes 1 to 1e-12 and zero: the same bits for 1, 2 and 4 rows per CTA."""
    from paper_2506_14792_gb300 import spadj
    Nx, Nz = 48, 20
    o = orb.RayleighBenard(Nx, Nz, 1e6)
    g = np.random.default_rng(4).standard_normal((o.Mz, o.Mx)) * (10.0 ** -(5 * np.arange(o.Mz) % 13))[:, None]
    g[7] = g[28] = 0.0
    got = []
    for rows in (1, 2, 4):
        p = gpu_problem(Nx, Nz)
        p.set_option(8, rows)
        oc, ob = _z((o.Kx, o.N)), _z((o.Kx, o.N))
        p.transform(spadj.G2C, dev(g), oc)
        p.transform(spadj.C2G_ADJ, dev(g), ob)
        got.append((oc, ob))
        p.close()
    assert rel_err(host(got[0][0]), o.g2c(g)) < 1e-13 and rel_err(host(got[0][1]), o.c2g_adj(g)) < 1e-13
    for a, b in got[1:]:
        assert torch.equal(a, got[0][0]) and torch.equal(b, got[0][1])


@pytest.mark.parametrize("sizes", [[192], [256, 192], [1024]])
def test_kolmogorov_few_long_rows(sizes):
    """4D-Var gradients by the launch with 256 threads per CTA (more than 128 butterflies a pass, few tiles)."""
    from paper_2506_14792_gb300 import spadj
    dt, nsteps, obs_steps, kmax = 2e-3, 4, [2, 4], 8
    X0, obs, Js, gs = tk._fourdvar_case(sizes, dt, nsteps, obs_steps, kmax, 50)
    p = tk.gpu_problem(sizes, dt=dt)
    p.set_observations(obs_steps, dev(obs), kmax)
    g = _z(sum((n // 2) * n for n in sizes))
    J = p.gradient(dev(tk.pack(X0)), nsteps, g, objective=spadj.SPADJ_OBJ_FOURDVAR)
    for i, got in enumerate(tk.unpack(host(g), sizes)):
        assert abs(J[i] - Js[i]) <= TOL * abs(Js[i])
        assert rel_err(got, gs[i]) < TOL
    p.close()


@pytest.mark.parametrize("N,order,schedule", [(256, 2, False), (256, 2, True), (256, 4, False), (512, 1, True), (512, 2, False),
                                              (512, 3, False), (96, 4, False)])
def test_burgers_full_batches(N, order, schedule):
    """700 members (more than four per SM): tangent and gradient of sampled members."""
    from paper_2506_14792_gb300 import spadj
    B, n, dt = 700, 12, 1e-3
    scheme = {1: spadj.SPADJ_SBDF1, 2: spadj.SPADJ_SBDF2, 3: spadj.SPADJ_SBDF3, 4: spadj.SPADJ_SBDF4}[order]
    p = tb._problem(N, batch=B, dt=dt, scheme=scheme)
    dts = [2e-3 if k // 3 % 2 == 0 else 7e-4 for k in range(n)] if schedule else dt
    if schedule:
        p.set_dt_schedule(dts)
    X0 = synthetic.burgers_ic(N, batch=B, seed=8)
    dX0 = tb._adm(synthetic.random_coeffs((B, N // 2), seed=9))
    dx, g = _z((B, N // 2)), _z((B, N // 2))
    p.tangent(n, dev(X0), dev(dX0), dx)
    p.gradient(dev(X0), n, g)
    o, pick = obur.Burgers(N, 0.01), [0, 333, 699]
    X = imex.multistep_forward(o, X0[pick], n, dts, order)
    assert rel_err(host(dx)[pick], imex.multistep_tangent(o, X, dX0[pick], dts, order)[-1]) < TOL
    want = imex.multistep_adjoint(o, X, lambda k: o.energy_grad(X[-1]) if k == n else None, dts, order)
    assert rel_err(host(g)[pick], want) < TOL
    p.close()
