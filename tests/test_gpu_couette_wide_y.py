"""Couette transforms at the wavenumber counts in y where the y transforms' buffers pass the shared memory that a kernel
gets without asking, and where they no longer fit eight columns to a CTA."""
import numpy as np
import pytest

import synthetic
from oracle import couette as oco
from tests.gpu_util import dev, host, rel_err
from tests.test_gpu_couette import RE, gpu_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# columns per CTA: 8 (49.3 KB), 4 (49.2 KB), 2 (49.2 KB), 8 at the largest length that fits (222 KB), 4 in place of 8 (197 KB)
@pytest.mark.parametrize("Nx,Ny", [(16, 128), (8, 256), (4, 512), (16, 576), (16, 1024)])
def test_transforms_and_their_adjoints(Nx, Ny):
    """The same bar as the transforms' parity test; the adjoint identity to 1e-13 of the norms' product."""
    from paper_2506_14792_gb300 import spadj
    Nz = 8
    o = oco.Couette(Nx, Ny, Nz, RE, pencils=False)
    p = gpu_problem(Nx, Ny, Nz)
    c = synthetic.random_coeffs((o.Kx, o.Ny, o.N), seed=Nx + Ny)
    g = np.random.default_rng(Ny).standard_normal((o.Mx, o.My, o.Mz))
    cg = dev(np.ascontiguousarray(c.transpose(1, 0, 2)))
    gg = dev(np.ascontiguousarray(g.transpose(2, 1, 0)))
    og = torch.zeros((o.Mz, o.My, o.Mx), dtype=torch.float64, device="cuda")
    oc = torch.zeros((o.Ny, o.Kx, o.N), dtype=torch.complex128, device="cuda")
    p.transform(spadj.C2G, cg, og)
    assert rel_err(host(og).transpose(2, 1, 0), o.c2g(c)) < 1e-13
    p.transform(spadj.C2G_ADJ, gg, oc)
    assert rel_err(host(oc).transpose(1, 0, 2), o.c2g_adj(g)) < 1e-13
    dot = torch.sum(og * gg).item()
    assert abs(dot - torch.vdot(cg.reshape(-1), oc.reshape(-1)).real.item()) <= 1e-13 * og.norm().item() * gg.norm().item()
    p.transform(spadj.G2C, gg, oc)
    assert rel_err(host(oc).transpose(1, 0, 2), o.g2c(g)) < 1e-13
    p.close()
