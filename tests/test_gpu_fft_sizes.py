"""The FFT series at the sizes where its row and column pairs can go wrong:
odd and even row counts, odd transform lengths, one-pair grids, lengths of
every radix mix; against the oracle with the bounds of tests/test_gpu_fft.py
(phi within 1e-13 of its maximum, S within hbar times that over phi)."""
import numpy as np
import pytest

from oracle import fft_series as fs
from paper_1403_1937_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 2), (2, 3), (8, 5), (13, 14), (23, 41), (38, 63),
                                   (64, 65), (122, 33), (95, 161), (300, 7)])
@pytest.mark.parametrize("terms", [0, 1, 4])
def test_sizes_vs_oracle(nx, ny, terms):
    import torch
    from paper_1403_1937_gb300 import build
    build.build()
    from paper_1403_1937_gb300 import eik
    rng = np.random.default_rng(nx * 1000 + ny)
    h = 1.0 / max(nx, ny)
    f = wl.fourier_field(rng, (nx, ny), h)
    src = wl.random_sources(rng, nx * ny, 3)
    hbar = 0.08
    S_ref, phi_ref, _, _ = fs.series(f, (nx, ny), h, hbar, src, terms)
    S, phi, _ = eik.fft_series((nx, ny), h, hbar, torch.from_numpy(f).cuda(), src, terms)
    S, phi = S.cpu().numpy(), phi.cpu().numpy()
    eta = 1e-13 * np.max(np.abs(phi_ref))
    assert np.max(np.abs(phi - phi_ref)) <= eta
    ok = phi_ref > 0
    assert np.all(np.abs(S[ok] - S_ref[ok]) <= hbar * eta / phi_ref[ok] + 1e-12)
