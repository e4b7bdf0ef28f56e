"""quotient() of csrc/eik_gridsync.cuh (the step lengths of the resident CG
kernels) against correctly rounded division, over mantissas and the whole
exponent range.

Bound: the reciprocal of b's mantissa m is y (1 + e + e^2) with y a
single-precision reciprocal and e = 1 - m y below 2^-22, so exact to 2^-66 before
its rounding; that rounding, the rounding of the product with a and the
reference's own are half a unit in the last place each, of numbers whose
units differ by a factor of two at most: 3 units.  A result below the normal
range is rounded once more (scalbn): 1 unit of the subnormals besides."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "eik_gridsync.cuh"
__global__ void k(const double *a, const double *b, double *q, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) q[i] = eik::quotient(a[i], b[i]);
}
extern "C" int probe(const double *a, const double *b, double *q, int n) {
  double *d = nullptr;
  const size_t m = sizeof(double) * n;
  if (cudaMalloc(&d, 3 * m) != cudaSuccess) return 1;
  cudaMemcpy(d, a, m, cudaMemcpyHostToDevice);
  cudaMemcpy(d + n, b, m, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * (size_t)n, n);
  const cudaError_t e = cudaMemcpy(q, d + 2 * (size_t)n, m, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def quotient(tmp_path_factory):
    from paper_1403_1937_gb300 import build
    d = tmp_path_factory.mktemp("quotient")
    src, lib = d / "probe.cu", d / "probe.so"
    src.write_text(PROBE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, f"-I{build.CSRC}", "-shared",
                    "-o", str(lib), str(src)], check=True)
    dll = ctypes.CDLL(os.fspath(lib))

    def run(a, b):
        a, b = (np.ascontiguousarray(v, dtype=np.float64) for v in (a, b))
        q = np.empty_like(a)
        ptr = [v.ctypes.data_as(ctypes.c_void_p) for v in (a, b, q)]
        assert dll.probe(*ptr, len(a)) == 0
        return q

    return run


TINY = 2.0 ** -1022


def check(q, a, b):
    with np.errstate(all="ignore"):
        ref = a / b
    big = np.isinf(ref)
    assert np.all(np.isinf(q[big]) | (q[big] >= np.finfo(float).max * (1 - 2.0 ** -51)))
    assert not np.isinf(q[ref < np.finfo(float).max * (1 - 2.0 ** -50)]).any()
    u = lambda v: v.view(np.int64)   # noqa: E731  (units in the last place, also subnormal)
    fin = ~big & ~np.isinf(q)
    d = np.abs(u(q[fin]) - u(ref[fin]))
    assert np.all(d <= np.where(ref[fin] < 4 * TINY, 4, 3)), d.max()


@pytest.mark.parametrize("ea,eb", [((-40, 40), (-40, 40)), ((-1074, 1023), (-1074, 1023)),
                                   ((-1074, -1000), (-60, 60)), ((-1074, -1015), (-1074, -1015)),
                                   ((900, 1023), (-1074, -900)), ((-1040, -900), (900, 1023)),
                                   ((1000, 1023), (1000, 1023))])
def test_against_division(quotient, ea, eb):
    rng = np.random.default_rng(abs(ea[0] + 3 * eb[0]))
    n = 1 << 18
    a = np.ldexp(rng.uniform(1, 2, n), rng.integers(*ea, n, endpoint=True))
    b = np.ldexp(rng.uniform(1, 2, n), rng.integers(*eb, n, endpoint=True))
    check(quotient(a, b), a, b)


def test_edges(quotient):
    ends = np.array([5e-324, 3 * 5e-324, TINY, TINY * (1 - 2.0 ** -52), TINY * 2, 1.0, 2 - 2.0 ** -52,
                     1 + 2.0 ** -52, 2.0 ** 1023, np.finfo(float).max, 2.0 ** -1021, 2.0 ** 1022])
    a, b = (v.ravel() for v in np.meshgrid(np.concatenate([[0.0], ends]), ends))
    check(quotient(a, b), a, b)
