"""grad S and backtracking where their fast forms could differ from the stated
operations (oracle/paths.py), bit for bit: spacings and values over the
exponent range (divisions by two corrections), more sources than a block
keeps, starts outside the grid, radii at the ends of the range."""
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


@pytest.mark.parametrize("h", [0.1, 1.0 / 3.0, 1.0 / 2047, 1.9999999999999998, 3e-57, 7e61, 5e-310])
@pytest.mark.parametrize("dims", [(1021, 257), (300, 2), (2, 300), (31, 17, 19)])
def test_grad_S_divisions(eik, h, dims):
    import torch
    rng = np.random.default_rng(int(np.prod(dims)))
    n = int(np.prod(dims))
    S = rng.standard_normal(n) * 2.0 ** rng.integers(-30, 30, n)
    S[rng.integers(0, n, n // 20)] = 0.0
    S[rng.integers(0, n, 5)] = 1e-300
    S[rng.integers(0, n, 5)] = 5e-324
    S[rng.integers(0, n, 5)] = np.inf
    S[rng.integers(0, n, 5)] = np.nan
    with np.errstate(all="ignore"):
        ref = opaths.grad_S(S, dims, h)
    np.testing.assert_array_equal(eik.grad_S(torch.from_numpy(S).cuda(), dims, h).cpu().numpy(), ref)


@pytest.mark.parametrize("nd", [2, 3])
@pytest.mark.parametrize("nsrc,eps", [(1, 2.0), (128, 0.7), (129, 0.7), (400, 0.3), (3, 0.0),
                                      (3, 1e-200), (3, 1e200)])
def test_backtrack_sources_and_radii(eik, nd, nsrc, eps):
    import torch
    dims = (61, 47) if nd == 2 else (19, 17, 23)
    h = 1.0 / 60
    n = int(np.prod(dims))
    rng = np.random.default_rng(nsrc)
    src = np.sort(rng.choice(n, nsrc, replace=False)).astype(np.int64)
    G = rng.standard_normal((nd, n))
    hi = np.array([(d - 1) * h for d in dims])
    starts = rng.uniform(-0.5, 1.5, (70, nd)) * hi      # some outside the grid
    starts[0] = 0.0
    starts[1] = hi
    P, L, st = eik.backtrack(torch.from_numpy(G).cuda(), dims, h, starts, src, 0.4 * h, 60, eps * h)
    P_ref, L_ref, st_ref = opaths.backtrack(G, dims, h, starts, 0.4 * h, 60, src, eps * h)
    np.testing.assert_array_equal(L.cpu().numpy(), L_ref)
    np.testing.assert_array_equal(st.cpu().numpy(), st_ref)
    np.testing.assert_array_equal(P.cpu().numpy(), P_ref)
