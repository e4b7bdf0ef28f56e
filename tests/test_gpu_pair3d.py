"""The two-pass inner CG of 3D mixed solves (csrc/eik_pair3d.cu) at the edges of
its tiles (128 columns x 16 rows x a ragged number of planes), of the chunks of
four columns and of the cells of 16 nodes, against the oracle and the one-pass
kernel.

Bounds: S within 1e-6 of the oracle, the mixed path's bound in the other tests
at tol 1e-9, so within 2e-6 of the one-pass kernel."""
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


GRIDS = [((2, 2, 2), 2.0), ((3, 2, 40), 3.0), ((5, 17, 3), 4.0), ((127, 15, 17), 6.0),
         ((128, 16, 16), 6.0), ((129, 17, 15), 6.0), ((130, 18, 5), 1.5), ((257, 3, 19), 6.0),
         ((9, 33, 70), 2.0), ((20, 20, 49), 1.5), ((260, 2, 2), 6.0), ((2, 70, 33), 3.0)]


@pytest.mark.parametrize("boundary", ["half_cell", "drop_edge"])
@pytest.mark.parametrize("dims,hb", GRIDS)
def test_vs_oracle_and_one_pass(eik, dims, hb, boundary):
    import torch
    rng = np.random.default_rng(sum(dims) + int(10 * hb))
    n = int(np.prod(dims))
    h = 1.0 / (max(dims) - 1)
    f = rng.uniform(0.5, 1.5, size=dims[::-1])
    src = wl.random_sources(rng, n, min(3, n - 1))
    U = rng.uniform(0.0, 0.01, len(src))
    out = []
    for variant in (0, 1):
        opt = eik.make_options(precision="mixed", tol=1e-9, boundary=boundary,
                               tile_override=variant)
        hd = eik.eik_create(dims, h, hb * h, torch.from_numpy(f).cuda(), src, U, opt)
        S, _, _ = eik.eik_solve(hd)
        S2, _, _ = eik.eik_solve(hd)
        eik.eik_destroy(hd)
        assert torch.equal(S, S2)
        out.append(S.cpu().numpy().ravel())
    sys = fd.assemble(f, dims, h, hb * h, src, U, boundary=0 if boundary == "half_cell" else 1)
    assert np.max(np.abs(out[0] - fd.solve_relative(sys))) <= 1e-6
    assert np.max(np.abs(out[0] - out[1])) <= 2e-6
