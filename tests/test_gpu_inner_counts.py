"""Inner iterations of the resident 2D and the two-pass 3D CG (csrc/eik_res32.cu,
csrc/eik_pair3d.cu) beside those of the one-pass kernels: FP64 refinement
repairs a wrong row of the inner operator, or a wrong term of the recurrence,
at the price of iterations, so the count shows what S does not.

Bounds: all are the same CG in exact arithmetic.  The two-sum kernels aim the
last refinement step at tol / 8, the one-pass kernels at half of their tolerance,
so these solve to tol / 4; then all steps have the same aims, end at tests four
iterations apart, and rounding may add a step on either side: 15 % and 40
iterations more are allowed.  S within 2e-6 of each other, as in the kernels'
other tests."""
import numpy as np
import pytest

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


def both(eik, dims, hb, smooth, tols, boundary="half_cell"):
    import torch
    rng = np.random.default_rng(sum(dims) + int(10 * hb))
    h = 1.0 / (max(dims) - 1)
    f = wl.fourier_field(rng, dims, h) if smooth else rng.uniform(0.5, 1.5, size=dims[::-1])
    src = wl.random_sources(rng, int(np.prod(dims)), 3)
    out = []
    for variant, tol in enumerate(tols):
        opt = eik.make_options(precision="mixed", tol=tol, boundary=boundary,
                               tile_override=variant)
        hd = eik.eik_create(dims, h, hb * h, torch.from_numpy(f).cuda(), src, None, opt)
        S, _, st = eik.eik_solve(hd)
        launches = eik.eik_kernel_stats(hd)["mixed_cg"][0]
        eik.eik_destroy(hd)
        out.append((S.cpu().numpy().ravel(), st["inner_iters"], launches))
    return out


# one tile and many, ragged chunks and tiles, every instance's tile height
GRIDS2 = [((129, 17), 6.0), ((261, 130), 6.0), ((517, 263), 6.0), ((700, 900), 9.0),
          ((1301, 1100), 13.0), ((1700, 1600), 16.0), ((333, 281), 3.0)]
GRIDS3 = [((127, 15, 17), 6.0), ((129, 17, 15), 6.0), ((130, 18, 5), 4.0), ((257, 33, 19), 6.0),
          ((9, 33, 70), 6.0), ((70, 66, 49), 5.0)]


@pytest.mark.parametrize("boundary", ["half_cell", "drop_edge"])
@pytest.mark.parametrize("dims,hb", GRIDS2 + GRIDS3)
def test_counts_beside_the_one_pass_kernels(eik, dims, hb, boundary):
    (S, it, _), (S1, it1, _) = both(eik, dims, hb, len(dims) == 2, (1e-9, 2.5e-10),
                                    boundary)
    assert np.max(np.abs(S - S1)) <= 2e-6
    assert it <= 1.15 * it1 + 40, (it, it1)


@pytest.mark.parametrize("dims,resident", [((2048, 2048), True), ((2049, 2049), False),
                                           ((2040, 2049), False)])
def test_largest_resident_grid(eik, dims, resident):
    """256 rows x 128 columns are the largest tile, and 152 blocks run at once:
    2048 rows are the most that 2048 columns can have; beyond, the one-pass
    kernels run, a launch for every iteration."""
    (S, it, n), (S1, it1, n1) = both(eik, dims, 16.0, True,
                                      (1e-7, 2.5e-8 if resident else 1e-7))
    assert n1 >= it1 and (n >= it) != resident
    if resident:
        assert it <= 1.15 * it1 + 40 and np.max(np.abs(S - S1)) <= 2e-6
    else:
        assert it == it1 and np.array_equal(S, S1)
