"""The imaginary part of a real field's mean coefficient is not used by the inverse transforms, however large it is or
if it is no number: grids and steps come out as with a zero in its place, bit for bit."""
import numpy as np
import pytest

import synthetic
from oracle import kolmogorov as okol
from tests.gpu_util import dev
from tests.test_gpu_closure import N as KN
from tests.test_gpu_closure import gpu_problem as closure_problem
from tests.test_gpu_couette import gpu_problem as couette_problem
from tests.rb_util import gpu_problem as rb_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
PARTS = [1e30, -1e300, np.nan, np.inf]


def _grids(p, c, shape, part):
    from paper_2506_14792_gb300 import spadj
    out = []
    for kind in (spadj.C2G, spadj.G2C_ADJ):
        for v in (0.0, part):
            x = c.copy()
            x.imag[..., 0, :] = 0.0
            x.imag[(0,) * (x.ndim - 2) + (0,)] = v  # every z mode of the mean column
            g = torch.zeros(shape, dtype=torch.float64, device="cuda")
            p.transform(kind, dev(x), g)
            out.append(g)
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[0], out[1]) and torch.equal(out[2], out[3])


@pytest.mark.parametrize("part", PARTS)
def test_rayleigh_benard_grids(part):
    _grids(rb_problem(32, 16), synthetic.random_coeffs((16, 16), seed=1), (24, 48), part)


@pytest.mark.parametrize("part", PARTS)
def test_couette_grids(part):
    _grids(couette_problem(16, 6, 12), synthetic.random_coeffs((6, 8, 12), seed=2), (18, 9, 24), part)


@pytest.mark.parametrize("part", PARTS)
def test_burgers_steps(part):
    """Forward, tangent and (from a given trajectory) adjoint steps."""
    from paper_2506_14792_gb300 import spadj
    N, n = 48, 3
    p = spadj.Problem(spadj.SPADJ_BURGERS1D, spadj.SPADJ_SBDF2, [N], [2 * np.pi], [0.01], 1e-3, batch=2)
    x, d, y = (synthetic.random_coeffs((2, N // 2), seed=s) for s in (3, 4, 5))
    got = []
    for v in (0.0, part):
        for a in (x, d):
            a[:, 0] = a[:, 0].real + 0j
            a.imag[:, 0] = v
        out, tan, adj = (torch.zeros((2, N // 2), dtype=torch.complex128, device="cuda") for _ in range(3))
        traj = torch.zeros((n + 1, 2, N // 2), dtype=torch.complex128, device="cuda")
        p.forward(n, dev(x), out, traj)
        p.tangent(n, dev(x), dev(d), tan)
        traj[:, :, 0] = torch.complex(traj[:, :, 0].real, torch.full_like(traj[:, :, 0].real, v))
        p.adjoint(n, traj, dev(y), adj)
        got.append((out, tan, adj))
    for a, b in zip(*got):
        assert torch.isfinite(torch.view_as_real(a)).all() and torch.equal(a, b)


def test_closure_input():
    """The vorticity field that the closure's network reads (the other fields are multiplied by a zero wavenumber)."""
    x = okol.Kolmogorov(KN, 1000.0).project(synthetic.kolmogorov_ic(KN, 300)).ravel()
    p = closure_problem(1)
    p.set_params(dev(synthetic.cnn_params(5, scale_out=1.0)))
    got = []
    for v in (0.0, 1e30):
        x.imag[0] = v
        f = torch.zeros(x.size, dtype=torch.complex128, device="cuda")
        p.eval_F(dev(x), f)
        got.append(f)
    assert torch.isfinite(torch.view_as_real(got[0])).all() and torch.equal(*got)
