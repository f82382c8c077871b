"""A closed eigenproblem gives its device memory back."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_closed_problems_hold_no_memory():
    """20 problems of 64 pencils at N = 64, whose factors and operators take over 100 MB each."""
    from paper_2506_14792_gb300 import stability
    P, N = 64, 64
    prm = np.stack([np.linspace(0.5, 1.5, P), np.full(P, 0.1), np.full(P, 2000.0)], axis=1)
    x, psi = (torch.ones((P, 3 * N), dtype=torch.complex128, device="cuda") for _ in range(2))
    out = torch.zeros((P, 10), dtype=torch.float64, device="cuda")
    free = []
    for _ in range(20):
        prob = stability.shear_evp_problem(N, "poiseuille", P)
        prob.eigen(prm, np.full(P, 0.02 - 0.3j), 100, x, psi, out)
        prob.close()
        free.append(torch.cuda.mem_get_info()[0])
    assert free[-1] >= free[0] - 100e6
