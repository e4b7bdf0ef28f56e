"""Cooperative kernels of several solvers at once: handles of their own, each
driven by its own host thread on its own stream, give the bits that they give
alone."""
import threading

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


# together they ask for more blocks than the device has room for
KINDS = [("mixed", (1100, 900), 10.0), ("mixed", (1100, 900), 10.0), ("fp64", (600, 500), 6.0),
         ("mixed", (70, 66, 49), 5.0), ("fp64", (90, 80, 70), 4.0), ("mixed", (300, 260), 4.0)]


def test_solvers_side_by_side(eik):
    import torch
    jobs = []
    for k, (precision, dims, hb) in enumerate(KINDS):
        rng = np.random.default_rng(k)
        h = 1.0 / (max(dims) - 1)
        f = torch.from_numpy(rng.uniform(0.5, 1.5, size=dims[::-1])).cuda()
        src = wl.random_sources(rng, int(np.prod(dims)), 3)
        s = torch.cuda.Stream()
        opt = eik.make_options(precision=precision, tol=1e-8)
        hd = eik.eik_create(dims, h, hb * h, f, src, None, opt, stream=s)
        S, _, st = eik.eik_solve(hd)
        jobs.append((hd, S.cpu().numpy(), st["inner_iters"]))
    errors = []

    def work(hd, S_alone, iters):
        try:
            out = np.empty_like(S_alone)
            for _ in range(3):
                _, _, st = eik.eik_solve(hd, S_out=out)
                assert st["inner_iters"] == iters and np.array_equal(out, S_alone)
        except BaseException as e:   # noqa: BLE001  (reported by the test's thread)
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for hd, _, _ in jobs:
        eik.eik_destroy(hd)
    assert not errors, errors
