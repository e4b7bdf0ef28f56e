"""The multigrid level-0 passes (csrc/eik_mg.cu) at the edges of their tiles
(2D: 128 columns x 8 rows; 3D: 128 columns x 16 rows x 2 .. 16 planes) and of
the chunks of four columns, against the oracle.

Bounds: S within 1e-6, the mixed path's bound in the other tests (tol 1e-9
there too).  A slip in one node of a preconditioner costs iterations rather
than accuracy, so the count is bounded as well: the V-cycle contracts every
error component that the Jacobi scaling does (a sweep of it comes first), so
it takes no more iterations than Jacobi-PCG on the same grid; on tiny grids,
where both end within a few dozen, 40 are allowed."""
import numpy as np
import pytest

from oracle import fd
from paper_1403_1937_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eik():
    import torch
    from paper_1403_1937_gb300 import build
    build.build()
    from paper_1403_1937_gb300 import eik as e
    assert torch.cuda.is_available()
    return e


GRIDS = [(2, 2), (3, 9), (127, 7), (128, 8), (129, 9), (131, 17), (256, 33), (257, 16), (385, 2),
         (2, 2, 2), (5, 17, 3), (127, 15, 17), (128, 16, 16), (129, 17, 15), (130, 18, 5),
         (257, 3, 19), (9, 33, 34)]


@pytest.mark.parametrize("boundary", ["half_cell", "drop_edge"])
@pytest.mark.parametrize("dims", GRIDS)
def test_tile_edges(eik, dims, boundary):
    import torch
    rng = np.random.default_rng(sum(dims) + 31 * len(dims))
    n = int(np.prod(dims))
    h = 1.0 / (max(dims) - 1)
    hbar = 6.0 * h
    f = rng.uniform(0.5, 1.5, size=dims[::-1])
    src = wl.random_sources(rng, n, min(3, n - 1))
    U = rng.uniform(0.0, 0.01, len(src))
    out = {}
    for precond in ("multigrid", "jacobi"):
        opt = eik.make_options(precision="mixed", tol=1e-9, boundary=boundary, precond=precond)
        hd = eik.eik_create(dims, h, hbar, torch.from_numpy(f).cuda(), src, U, opt)
        S, _, st = eik.eik_solve(hd)
        if precond == "multigrid":
            S2, _, _ = eik.eik_solve(hd)
            assert torch.equal(S, S2)
        eik.eik_destroy(hd)
        out[precond] = S.cpu().numpy().ravel(), st["inner_iters"]
    S_ref, _, _ = fd.solve(f, dims, h, hbar, src, U, boundary=0 if boundary == "half_cell" else 1)
    S, iters = out["multigrid"]
    assert np.max(np.abs(S - S_ref)) <= 1e-6
    assert iters <= max(40, out["jacobi"][1])
