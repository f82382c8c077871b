"""The banded factorisation and solves of the eigenproblem on the GPU (one shift-invert iteration) against dense solves with the oracle's matrices, at the smallest size, at
sizes that are and are not whole chunks of sweep steps, for both flows and for the mean pencil (its own
structure)."""
import numpy as np
import pytest

from oracle.shear_evp import ShearEVP
from tests.gpu_util import dev, host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,base", [(8, "couette"), (9, "poiseuille"), (16, "poiseuille"), (30, "couette")])
def test_one_iteration_matches_dense_solves(N, base):
    """x <- Phi x / |Phi x| and psi <- Phi^H psi / |Phi^H psi| from random vectors.  A backward stable solve is
    off by a small multiple of cond(A) 2^-53; the bar is 1000 of them against a dense solve of the same matrix
    (numpy's, itself off by some)."""
    from paper_2506_14792_gb300 import stability
    e = ShearEVP(N, base)
    prm = [(1.1, 0.7, 1234.5), (0.0, 0.0, 300.0), (0.0, 1.3, 50.0), (2.5, 0.0, 10000.0)]
    shift = [0.03 - 0.31j, 0.2 + 0.1j, -0.5 + 0.0j, 5.0 - 40.0j]
    P, H = len(prm), 3 * N
    prob = stability.shear_evp_problem(N, base, P)
    rng = np.random.default_rng(N)
    x0 = rng.standard_normal((P, H)) + 1j * rng.standard_normal((P, H))
    p0 = rng.standard_normal((P, H)) + 1j * rng.standard_normal((P, H))
    x, psi = dev(x0), dev(p0)
    out = torch.zeros((P, 10), dtype=torch.float64, device="cuda")
    prob.eigen(prm, shift, 1, x, psi, out)
    xg, pg, o = host(x), host(psi), host(out)
    assert np.all(np.isfinite(o))
    for i, ((a, b, Re), s) in enumerate(zip(prm, shift)):
        M, L = e.matrices(a, b, Re)[:2]
        A = s * M + L
        S = np.zeros((A.shape[0], H))
        for f in range(3):
            S[f * N:(f + 1) * N, f * N:(f + 1) * N] = e.SS
        y = np.linalg.solve(A, S @ x0[i])[:H]
        z = S.T @ np.linalg.solve(A.conj().T, np.concatenate([p0[i], np.zeros(A.shape[0] - H)]))
        tol = 1000 * np.linalg.cond(A) * 2.0 ** -53
        assert tol < 1e-3, (i, tol)
        for got, want in ((xg[i], y), (pg[i], z)):
            want = want / np.linalg.norm(want)
            assert np.linalg.norm(got - want) <= tol, (i, np.linalg.norm(got - want), tol)
        px = np.vdot(p0[i], x0[i])
        mu = np.vdot(p0[i], y) / px
        dmu = tol * np.linalg.norm(p0[i]) * np.linalg.norm(y) / abs(px)
        assert abs(o[i, 0] + 1j * o[i, 1] - (s - 1 / mu)) <= 2 * dmu / abs(mu) ** 2
