"""Edges of the collocation transforms on the GPU, through spadj_transform of the Burgers problem (FP64
butterflies) and its trajectories (fixed point): every member (sequence) has its own scale, tiny and huge
amplitudes keep their relative accuracy, zeros stay zeros and a non-finite member does not touch the others."""
import numpy as np
import pytest

from oracle import burgers as obur
from oracle import fourier, imex
from tests.gpu_util import dev, host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [4, 12, 16, 36, 108, 256, 512])
def test_scales_are_per_sequence(N):
    """Round trip c -> grid -> c; a round trip of FP64 transforms is exact to a few units of 2^-53 times
    log2 of the length, the bar is 20 of them."""
    from paper_2506_14792_gb300 import spadj
    amps = np.array([1.0, 1e-290, 1e280, 0.0, 1e-3, np.nan, np.inf, 1e5])
    B, K, M = len(amps), N // 2, 3 * N // 2
    p = spadj.Problem(spadj.SPADJ_BURGERS1D, spadj.SPADJ_SBDF2, [N], [2 * np.pi], [0.01], 1e-3, batch=B)
    rng = np.random.default_rng(N)
    base = rng.standard_normal((B, K)) + 1j * rng.standard_normal((B, K))
    base[:, 0] = base[:, 0].real
    c = base * np.where(np.isfinite(amps), amps, 1.0)[:, None]
    c[5, K // 2], c[6, K - 1] = np.nan, np.inf
    g = torch.zeros((B, M), dtype=torch.float64, device="cuda")
    back = torch.zeros((B, K), dtype=torch.complex128, device="cuda")
    p.transform(spadj.C2G, dev(c), g)
    gh = host(g)
    p.transform(spadj.G2C, g, back)
    bh = host(back)
    tol = 20 * 2.0 ** -53
    for b in (0, 1, 2, 4, 7):
        want = fourier.c2g(base[b:b + 1], M)[0]
        scale = np.max(np.abs(want))
        assert np.max(np.abs(gh[b] / amps[b] - want)) <= tol * scale * np.sqrt(N), b
        assert np.max(np.abs(bh[b] / amps[b] - base[b])) <= tol * np.max(np.abs(base[b])) * np.sqrt(N), b
    assert not gh[3].any() and not bh[3].any()
    assert np.isnan(gh[5]).all() and not np.isfinite(gh[6]).any()


@pytest.mark.parametrize("N", [4, 12, 16, 36, 108, 256, 512])
def test_scales_are_per_member_in_the_steps(N):
    """Two SBDF2 steps of each member against the oracle's.  The products are white spectra times white
    grids; a step's rounding is bounded by some tens of units of 2^-53 of the member's largest coefficient
    (times sqrt(N) for the largest entry of a vector), the bar is 100."""
    from paper_2506_14792_gb300 import spadj
    amps = np.array([1.0, 1e-290, 0.0, 1e-3, np.nan, np.inf, 30.0])
    B, K, dt = len(amps), N // 2, 1e-5
    p = spadj.Problem(spadj.SPADJ_BURGERS1D, spadj.SPADJ_SBDF2, [N], [2 * np.pi], [0.01], dt, batch=B)
    rng = np.random.default_rng(N)
    x0 = rng.standard_normal((B, K)) + 1j * rng.standard_normal((B, K))
    x0[:, 0] = x0[:, 0].real
    x0 *= np.where(np.isfinite(amps), amps, 1.0)[:, None]
    x0[4, K // 2], x0[5, K - 1] = np.nan, np.inf
    out = torch.zeros((B, K), dtype=torch.complex128, device="cuda")
    p.forward(2, dev(x0), out)
    got = host(out)
    fin = [b for b in range(B) if np.isfinite(amps[b])]
    want = imex.multistep_forward(obur.Burgers(N, 0.01), x0[fin], 2, dt)[-1]
    for b, w in zip(fin, want):
        assert np.max(np.abs(got[b] - w)) <= 100 * 2.0 ** -53 * np.max(np.abs(w)) * np.sqrt(N), (b, amps[b])
    assert not np.isfinite(got[4]).any() and not np.isfinite(got[5]).any()
