"""Edges of the fixed-point collocation transforms on the GPU, through spadj_transform of the Burgers
problem: every member (sequence) has its own scale, tiny and huge amplitudes keep their relative accuracy,
zeros stay zeros and a non-finite member does not touch the others."""
import numpy as np
import pytest

from oracle import fourier
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
