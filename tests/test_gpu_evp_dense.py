"""Eigenproblem iterations with the dense operator (few pencils, enough steps) against as many calls of one banded step
each: iterates, eigenvalues, residuals and sensitivities, for both flows, odd N, every count of 32-column
chunks and the mean pencil; and more pencils than SMs."""
import numpy as np
import pytest

from oracle.shear_evp import ShearEVP
from tests.gpu_util import dev, host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PRM = [(1.1, 0.7, 1234.5), (0.0, 0.0, 300.0), (0.9, 0.0, 5000.0)]
SHIFT = [0.03 - 0.31j, 0.2 + 0.1j, 0.01 - 0.25j]


def _run(N, base, prm, shift, calls):
    from paper_2506_14792_gb300 import stability
    P, H = len(prm), 3 * N
    prob = stability.shear_evp_problem(N, base, P)
    rng = np.random.default_rng(N)
    x, psi = (dev(rng.standard_normal((P, H)) + 1j * rng.standard_normal((P, H))) for _ in range(2))
    out = torch.zeros((P, 10), dtype=torch.float64, device="cuda")
    for n in calls:
        prob.eigen(prm, shift, n, x, psi, out)
    prob.close()
    return host(x), host(psi), host(out)


# steps: the rule takes the dense operator from 5 + N / 10 + 3e-4 P N^2 on
@pytest.mark.parametrize("N,base,steps", [(8, "poiseuille", 8), (9, "couette", 8), (20, "poiseuille", 12), (31, "couette", 12),
                                          (42, "poiseuille", 16), (52, "poiseuille", 20), (64, "couette", 24)])
def test_matches_single_banded_steps(N, base, steps):
    """A step's solves are off by a small multiple of cond(A) 2^-53 of the iterate; errors of several steps add up at most
    (the power iteration contracts what is not along the eigenvector).  Bar: 1000 of them a step."""
    e = ShearEVP(N, base)
    xd, pd, od = _run(N, base, PRM, SHIFT, [steps])
    xb, pb, ob = _run(N, base, PRM, SHIFT, [1] * steps)
    assert np.all(np.isfinite(od))
    for i, ((a, b, Re), s) in enumerate(zip(PRM, SHIFT)):
        M, L = e.matrices(a, b, Re)[:2]
        tol = steps * 1000 * np.linalg.cond(s * M + L) * 2.0 ** -53
        assert tol < 1e-2
        assert np.linalg.norm(xd[i] - xb[i]) <= tol and np.linalg.norm(pd[i] - pb[i]) <= tol, i
        # the Rayleigh quotient divides by psi^H x, the sensitivities by <Y, M X> (about its size)
        amp = tol / min(1.0, abs(np.vdot(pb[i], xb[i])))
        lam = ob[i, 0] + 1j * ob[i, 1]
        assert abs(od[i, 0] + 1j * od[i, 1] - lam) <= 10 * amp * abs(lam - s), i
        assert np.allclose(od[i, 8:], ob[i, 8:], rtol=0, atol=10 * amp), i


def test_more_pencils_than_sms():
    """200 pencils of N = 8 with 250 steps: the converged eigenvalues, next to those of 10 calls of 25 banded steps."""
    P = 200
    prm = [(a, 0.2, 500.0) for a in np.linspace(0.5, 1.5, P)]
    shift = [0.05 - 0.4j * a for a, _, _ in prm]
    _, _, od = _run(8, "poiseuille", prm, shift, [250])
    _, _, ob = _run(8, "poiseuille", prm, shift, [25] * 10)
    good = (ob[:, 8] < 1e-12) & (od[:, 8] < 1e-12)
    assert good.sum() >= P // 2
    assert np.allclose(od[good, :2], ob[good, :2], rtol=1e-9, atol=1e-10)
