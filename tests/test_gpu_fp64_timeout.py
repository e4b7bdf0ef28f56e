"""Failure detection without a fault in the resident FP64 CG (csrc/eik_res64.cu):
with test_flags bit 1 one block does not arrive at the first grid-wide sum of
the handle's first launch, every block's bounded wait runs out, and the solve
reports a timeout.  The context and the handle stay usable.  Tolerance as in
the other FP64 tests: componentwise residual 1e-12, S within 1e-8 hbar."""
import time

import numpy as np
import pytest

from oracle import fd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eik():
    import torch
    from paper_1403_1937_gb300 import build
    build.build()
    from paper_1403_1937_gb300 import eik as e
    assert torch.cuda.is_available()
    return e


@pytest.mark.parametrize("dims", [(30, 20), (257, 129), (31, 33, 37)])
def test_wait_that_runs_out(eik, dims):
    import torch
    from paper_1403_1937_gb300 import _lib
    rng = np.random.default_rng(sum(dims))
    h = 1.0 / (max(dims) - 1)
    hbar = 3.0 * h
    f = rng.uniform(0.5, 2.0, size=dims[::-1])
    src = np.array([0, 17])
    opt = eik.make_options(precision="fp64", tol=1e-12, test_flags=2)
    hd = eik.eik_create(dims, h, hbar, torch.from_numpy(f).cuda(), src, None, opt)
    t = time.time()
    with pytest.raises(_lib.EikError) as ei:
        eik.eik_solve(hd)
    assert ei.value.status == _lib.EIK_ERR_TIMEOUT and "timed out" in str(ei.value)
    assert time.time() - t < 10
    with pytest.raises(_lib.EikError) as ei:
        eik.eik_grad(hd, torch.ones(f.size, dtype=torch.float64, device="cuda"))
    assert ei.value.status == _lib.EIK_ERR_STATE
    S, _, _ = eik.eik_solve(hd)
    assert eik.eik_kernel_stats(hd)["cg64_resident"][0] > 0
    eik.eik_destroy(hd)
    S_ref, _, _ = fd.solve(f, dims, h, hbar, src)
    assert np.max(np.abs(S.cpu().numpy().ravel() - S_ref)) <= 1e-8 * hbar
