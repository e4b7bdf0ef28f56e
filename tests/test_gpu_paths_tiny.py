"""Backtracking on grids so fine that squared distances lie near the ends of
the single-precision range, where the test that rules sources out has no
precision of its own left: bit for bit the stated operations
(oracle/paths.py)."""
import numpy as np
import pytest

from oracle import paths as opaths

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eik():
    import torch
    from paper_1403_1937_gb300 import build
    build.build()
    from paper_1403_1937_gb300 import eik as e
    assert torch.cuda.is_available()
    return e


@pytest.mark.parametrize("nd", [2, 3])
@pytest.mark.parametrize("eps", [1e-24, 4e-23, 1e-22, 1.5e-22, 4e-22, 2e-21, 1e-20, 1.3e-19, 1e-18,
                                 1e15, 1e17, 1.84e19, 1e20])
def test_backtrack_radii_near_the_float_range(eik, nd, eps):
    import torch
    dims = (61, 47) if nd == 2 else (19, 17, 23)
    h = eps / 2.7
    n = int(np.prod(dims))
    rng = np.random.default_rng(nd)
    src = np.sort(rng.choice(n, 40, replace=False)).astype(np.int64)
    G = rng.standard_normal((nd, n))
    starts = rng.uniform(0, 1, (6000, nd)) * np.array([(d - 1) * h for d in dims])
    P, L, st = eik.backtrack(torch.from_numpy(G).cuda(), dims, h, starts, src, 0.4 * h, 3, eps)
    P_ref, L_ref, st_ref = opaths.backtrack(G, dims, h, starts, 0.4 * h, 3, src, eps)
    assert 0.02 < np.mean(L_ref == 0) < 0.98
    np.testing.assert_array_equal(L.cpu().numpy(), L_ref)
    np.testing.assert_array_equal(st.cpu().numpy(), st_ref)
    np.testing.assert_array_equal(P.cpu().numpy(), P_ref)
