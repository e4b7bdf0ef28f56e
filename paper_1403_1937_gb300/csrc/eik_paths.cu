// Gradient of S and backtracking of optimal paths (path-planning section,
// Eq. PathPlanning-backTrackOnS): a path from a target point solves
// dx/dt = -grad S / |grad S| and ends once it is within eps of a source.
//
// Discretisation (the paper gives none):
// * grad S at the nodes: (S[k+1] - S[k-1]) / (2h) inside, one-sided
//   (S[1] - S[0]) / h and (S[n-1] - S[n-2]) / h on the faces;
// * between nodes: multilinear interpolation of the nodal gradient in the
//   cell holding the point (cells clamped to the grid);
// * explicit Euler steps of fixed arc length, x <- clamp(x - step g/|g|),
//   preceded by the stop tests: distance to the nearest source < eps
//   (status 0), |g| zero or not finite (status 2); status 1 after max_steps.
// One thread per path.  The results are those of explicitly rounded operations
// (no fused multiply-add) in the order stated above, so a path is reproducible
// on any IEEE machine that evaluates the same steps.
//
// What bounds them: a path is one serial chain of FP64 operations, each about
// 90 cycles here, and its step used to hold a square root and four 64-bit
// integer divisions per source besides the interpolation (12 us a step), after
// which every thread filled its own row's tail with NaN.  Now a step tests the
// sources in single precision, with a bound on the error of that, and only
// those that may be within eps in double; divisions by the spacing are two
// correction steps on a product; blocks are one warp, so that every path has
// a scheduler of its own; and the tails are filled by a pass of their own.
// 4096 paths on 2048^2 with 16 sources: 24.9 ms before, 4.4 ms now (grad S
// 146 us, 122 us).
#include <math.h>

#include <algorithm>
#include <climits>

#include "eik_internal.cuh"

namespace {

struct Dims3 {
  int n[3];
  int ndim;
  int64_t N;
};

// A divisor b and its correctly rounded reciprocal (0: not used, b is near
// the ends of the exponent range).
struct Divisor {
  double b, rb;
};
inline Divisor divisor(double b) {
  return Divisor{b, (b > 1e-60 && b < 1e60) ? 1.0 / b : 0.0};
}

// a / b, correctly rounded.  q = a rb is within two units in the last place,
// one correction with the exact remainder makes it faithful, and a second one
// then rounds correctly (P. Markstein, Computation of elementary functions on
// the IBM RISC System/6000 processor, 1990: y the rounded reciprocal, q
// faithful, r = a - b q exact; q + r y rounds to a / b).  Five FP64 operations;
// exponents far from the middle of the range go the general way.
__device__ __forceinline__ double div_by(double a, const Divisor &d) {
  const double q0 = __dmul_rn(a, d.rb);
  const unsigned ea = ((unsigned)__double2hiint(a) >> 20) & 0x7ffu;
  const unsigned eq = ((unsigned)__double2hiint(q0) >> 20) & 0x7ffu;
  if (d.rb == 0.0 || ea - 323u > 1400u || eq - 323u > 1400u) return __ddiv_rn(a, d.b);
  const double q1 = __fma_rn(__fma_rn(-q0, d.b, a), d.rb, q0);
  return __fma_rn(__fma_rn(-q1, d.b, a), d.rb, q1);
}

// Rows (y, z) by blockIdx.y, columns by blockIdx.x: no division per node.
__global__ void k_grad_S(Dims3 d, Divisor h1, Divisor h2, const double *__restrict__ S,
                         double *__restrict__ G) {
  const int64_t st[3] = {1, d.n[0], (int64_t)d.n[0] * d.n[1]};
  const int64_t rows = (int64_t)d.n[1] * d.n[2];
  for (int64_t row = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; row < rows;
       row += (int64_t)gridDim.y * blockDim.y) {
    const int z = (d.ndim == 3) ? (int)(row / d.n[1]) : 0;
    const int y = (int)(row - (int64_t)z * d.n[1]);
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < d.n[0]; x += gridDim.x * blockDim.x) {
      const int k[3] = {x, y, z};
      const int64_t i = x + (int64_t)d.n[0] * row;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (a >= d.ndim) break;
        const bool lo = k[a] == 0, hi = k[a] == d.n[a] - 1;
        const double num = __dsub_rn(S[hi ? i : i + st[a]], S[lo ? i : i - st[a]]);
        G[a * d.N + i] = (lo || hi) ? div_by(num, h1) : div_by(num, h2);
      }
    }
  }
}

// Sources whose coordinates a block keeps in shared memory; those past them
// are read from their indices at every test.
constexpr int kSrcShared = 128;

// World coordinates y_a = k_a h of source s.
template <int ND>
__device__ __forceinline__ void source_coords(const Dims3 &d, double h, int64_t s, double *y) {
#pragma unroll
  for (int a = 0; a < ND; ++a) {
    y[a] = __dmul_rn((double)(s % d.n[a]), h);
    s /= d.n[a];
  }
}
// Squared distance, the sum of rounded squares.
template <int ND>
__device__ __forceinline__ double dist2(const double *x, const double *y) {
  double acc = 0.0;
#pragma unroll
  for (int a = 0; a < ND; ++a) {
    const double dx = __dsub_rn(x[a], y[a]);
    acc = (a == 0) ? __dmul_rn(dx, dx) : __dadd_rn(acc, __dmul_rn(dx, dx));
  }
  return acc;
}

// Whether the distance to some source, sqrt of the rounded sum of squares, is
// below eps.  The square root is monotone, so the test is on the sum itself:
// t2 is the smallest double whose rounded root is not below eps.  Single
// precision rules sources out first: with coordinates up to M every |dx| is
// known to 4 2^-24 M, and the squares to 2^-21 relative while they are normal
// numbers; lim is infinite, which rules nothing out, where t2 is too small for
// that.
template <int ND>
__device__ __forceinline__ bool near_source(const double *x, const double *ys, const float4 *yf,
                                            int nsrc, double t2, float ext, float lim) {
  const float fx = (float)x[0], fy = (float)x[1], fz = (ND == 3) ? (float)x[2] : 0.f;
  const float err =
      2.4e-7f * fmaxf(ext, fmaxf(fabsf(fx), fmaxf(fabsf(fy), fabsf(fz))));   // >= 4 2^-24 M
  bool hit = false;
#pragma unroll 4
  for (int s = 0; s < nsrc; ++s) {
    const float4 y = yf[s];
    const float ax = fmaxf(fabsf(fx - y.x) - err, 0.f), ay = fmaxf(fabsf(fy - y.y) - err, 0.f);
    float q = fmaf(ax, ax, ay * ay);
    if (ND == 3) {
      const float az = fmaxf(fabsf(fz - y.z) - err, 0.f);
      q = fmaf(az, az, q);
    }
    if (!(q > lim)) {   // (also where it is not a number)
      hit = hit || dist2<ND>(x, ys + ND * s) < t2;
    }
  }
  return hit;
}

template <int ND>
__global__ void __launch_bounds__(32)
k_backtrack(Dims3 d, Divisor h, const double *__restrict__ G, const double *__restrict__ starts,
            int64_t npaths, double step, int max_steps, const int64_t *__restrict__ src,
            int64_t nsrc, double eps, float ext, double *__restrict__ paths,
            int *__restrict__ lengths, int *__restrict__ status) {
  __shared__ double ys[kSrcShared * ND];
  __shared__ float4 yf[kSrcShared];
  const int ns = (int)min(nsrc, (int64_t)kSrcShared);
  for (int s = threadIdx.x; s < ns; s += blockDim.x) {
    double y[ND];
    source_coords<ND>(d, h.b, src[s], y);
#pragma unroll
    for (int a = 0; a < ND; ++a) ys[ND * s + a] = y[a];
    yf[s] = make_float4((float)y[0], (float)y[1], (ND == 3) ? (float)y[ND - 1] : 0.f, 0.f);
  }
  __syncwarp();   // one warp per block
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npaths) return;
  const int64_t stride_p = (int64_t)(max_steps + 1) * ND;
  double *out = paths + p * stride_p;
  // the squared distances whose root is below eps are those below t2
  double t2 = __dmul_rn(eps, eps);
  if (t2 > 1e-290 && t2 < 1e290) {
    for (int k = 0; k < 8 && __dsqrt_rn(t2) >= eps; ++k)
      t2 = __longlong_as_double(__double_as_longlong(t2) - 1);
    for (int k = 0; k < 8 && __dsqrt_rn(t2) < eps; ++k)
      t2 = __longlong_as_double(__double_as_longlong(t2) + 1);
  }
  const bool by_root = !(t2 > 1e-290 && t2 < 1e290);   // eps at the ends of the range
  // 1e-30: squares of distances near eps are then normal single-precision
  // numbers (above 1.2e-38), so that 1e-4 covers their rounding
  const float lim = (t2 > 1e-30) ? (float)t2 * 1.0001f : INFINITY;
  double x[ND], hi[ND];
#pragma unroll
  for (int a = 0; a < ND; ++a) {
    x[a] = starts[p * ND + a];
    hi[a] = __dmul_rn((double)(d.n[a] - 1), h.b);
    out[a] = x[a];
  }
  auto within = [&](double acc) { return by_root ? __dsqrt_rn(acc) < eps : acc < t2; };
  auto reached = [&]() {
    bool hit = false;
    if (!by_root) {
      hit = near_source<ND>(x, ys, yf, ns, t2, ext, lim);
    } else {
      for (int s = 0; s < ns; ++s) hit = hit || within(dist2<ND>(x, ys + ND * s));
    }
    for (int64_t s = ns; s < nsrc; ++s) {
      double y[ND];
      source_coords<ND>(d, h.b, src[s], y);
      hit = hit || within(dist2<ND>(x, y));
    }
    return hit;
  };
  const int64_t strides[3] = {1, d.n[0], (int64_t)d.n[0] * d.n[1]};
  int len = 0, stat = 1;
  for (int k = 0; k < max_steps; ++k) {
    // cell and position in it; the loads start before the distance test
    int64_t idx0 = 0;
    double t[ND];
#pragma unroll
    for (int a = 0; a < ND; ++a) {
      const double u = div_by(x[a], h);
      const double cf = fmin(fmax(floor(u), 0.0), (double)(d.n[a] - 2));
      idx0 += (int64_t)cf * strides[a];
      t[a] = __dsub_rn(u, cf);
    }
    double gv[1 << ND][ND];
#pragma unroll
    for (int corner = 0; corner < (1 << ND); ++corner) {
      int64_t idx = idx0;
#pragma unroll
      for (int a = 0; a < ND; ++a) idx += ((corner >> a) & 1) ? strides[a] : 0;
#pragma unroll
      for (int a = 0; a < ND; ++a) gv[corner][a] = __ldg(G + a * d.N + idx);
    }
    if (reached()) {
      stat = 0;
      break;
    }
    // multilinear interpolation of the nodal gradient
    double g[ND];
#pragma unroll
    for (int corner = 0; corner < (1 << ND); ++corner) {
      double w = (corner & 1) ? t[0] : __dsub_rn(1.0, t[0]);
#pragma unroll
      for (int a = 1; a < ND; ++a)
        w = __dmul_rn(w, ((corner >> a) & 1) ? t[a] : __dsub_rn(1.0, t[a]));
#pragma unroll
      for (int a = 0; a < ND; ++a) {
        const double v = __dmul_rn(w, gv[corner][a]);
        g[a] = corner ? __dadd_rn(g[a], v) : __dadd_rn(0.0, v);
      }
    }
    double gg = __dmul_rn(g[0], g[0]);
#pragma unroll
    for (int a = 1; a < ND; ++a) gg = __dadd_rn(gg, __dmul_rn(g[a], g[a]));
    const double gn = __dsqrt_rn(gg);
    if (!(gn > 0.0)) {
      stat = 2;
      break;
    }
    ++len;
#pragma unroll
    for (int a = 0; a < ND; ++a) {
      const double xn = __dsub_rn(x[a], __ddiv_rn(__dmul_rn(step, g[a]), gn));
      x[a] = fmin(fmax(xn, 0.0), hi[a]);
      out[(int64_t)len * ND + a] = x[a];
    }
  }
  if (stat == 1 && reached()) stat = 0;
  lengths[p] = len;
  status[p] = stat;
}

// NaN after every path's last point; a block takes one path at a time.
__global__ void k_path_tails(double *__restrict__ paths, const int *__restrict__ lengths,
                             int64_t npaths, int max_steps, int nd) {
  const int64_t stride_p = (int64_t)(max_steps + 1) * nd;
  for (int64_t p = blockIdx.x; p < npaths; p += gridDim.x) {
    double *out = paths + p * stride_p;
    for (int64_t k = (int64_t)(lengths[p] + 1) * nd + threadIdx.x; k < stride_p; k += blockDim.x)
      out[k] = NAN;
  }
}

bool make_dims(int ndim, const int64_t *dims, Dims3 &d) {
  if (ndim != 2 && ndim != 3) return false;
  d.ndim = ndim;
  d.N = 1;
  d.n[0] = d.n[1] = d.n[2] = 1;
  for (int a = 0; a < ndim; ++a) {
    if (dims[a] < 2 || dims[a] > (int64_t)1 << 30) return false;
    d.n[a] = (int)dims[a];
    d.N *= dims[a];
  }
  return true;
}

}  // namespace

extern "C" eik_status eik_grad_S(int ndim, const int64_t *dims, double h, const double *S,
                                 double *gradS, eik_stream_t stream) {
  Dims3 d{};
  if (!dims || !S || !gradS || !(h > 0) || !make_dims(ndim, dims, d)) return EIK_ERR_ARG;
  // 256 threads: as many columns as the row has, rows beside each other
  int bx = 1;
  while (bx < d.n[0] && bx < 256) bx *= 2;
  const int by = 256 / bx, cap = 152 * 16;
  const int gx = std::min((d.n[0] + bx - 1) / bx, cap);
  const int64_t rows = ((int64_t)d.n[1] * d.n[2] + by - 1) / by;
  const int gy = (int)std::max<int64_t>(1, std::min<int64_t>(rows, cap / gx));
  k_grad_S<<<dim3(gx, gy), dim3(bx, by), 0, stream>>>(d, divisor(h), divisor(2.0 * h), S, gradS);
  return cudaGetLastError() == cudaSuccess ? EIK_OK : EIK_ERR_CUDA;
}

extern "C" eik_status eik_backtrack(int ndim, const int64_t *dims, double h, const double *gradS,
                                    const double *starts, int64_t npaths, double step,
                                    int max_steps, const int64_t *src_idx, int64_t nsrc,
                                    double eps, double *paths, int *lengths, int *status,
                                    eik_stream_t stream) {
  Dims3 d{};
  if (!dims || !(h > 0) || !make_dims(ndim, dims, d)) return EIK_ERR_ARG;
  if (npaths < 0 || nsrc < 0 || max_steps < 0 || !(step > 0) || !(eps >= 0)) return EIK_ERR_ARG;
  if (npaths == 0) return EIK_OK;
  if (!gradS || !starts || !paths || !lengths || !status || (nsrc > 0 && !src_idx))
    return EIK_ERR_ARG;
  double ext = 0.0;
  for (int a = 0; a < ndim; ++a) ext = std::max(ext, (double)(d.n[a] - 1) * h);
  const float extf = (float)ext * 1.000001f;
  const int64_t nb = (npaths + 31) / 32;
  if (nb > INT_MAX) return EIK_ERR_ARG;
  if (ndim == 2)
    k_backtrack<2><<<(int)nb, 32, 0, stream>>>(d, divisor(h), gradS, starts, npaths, step, max_steps,
                                               src_idx, nsrc, eps, extf, paths, lengths, status);
  else
    k_backtrack<3><<<(int)nb, 32, 0, stream>>>(d, divisor(h), gradS, starts, npaths, step, max_steps,
                                               src_idx, nsrc, eps, extf, paths, lengths, status);
  k_path_tails<<<(int)std::min<int64_t>(npaths, 152 * 8), 256, 0, stream>>>(paths, lengths, npaths,
                                                                          max_steps, ndim);
  return cudaGetLastError() == cudaSuccess ? EIK_OK : EIK_ERR_CUDA;
}

// Shape-from-shading forcing (shape-from-shading section, Eq. SfS-forcingFunc):
// a Lambertian image under vertical light, P = 1/sqrt(|grad S|^2 + 1), gives
// the eikonal forcing f = sqrt(1/P^2 - 1), raised to f_min where smaller
// (flat regions would give f = 0, which eik_create rejects); P outside
// (0, 1] or not finite gives NaN (eik_create rejects it).  Explicitly
// rounded operations, as in the path kernels.
namespace {
__global__ void k_sfs_forcing(const double *__restrict__ P, int64_t n, double f_min,
                              double *__restrict__ f) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double p = P[i];
    double v = NAN;
    if (p > 0.0 && p <= 1.0) {
      const double g = __dsqrt_rn(__dsub_rn(__ddiv_rn(1.0, __dmul_rn(p, p)), 1.0));
      v = fmax(g, f_min);
    }
    f[i] = v;
  }
}
}  // namespace

extern "C" eik_status eik_sfs_forcing(const double *P, int64_t n, double f_min, double *f,
                                      eik_stream_t stream) {
  if (n < 0 || !(f_min >= 0.0) || (n > 0 && (!P || !f))) return EIK_ERR_ARG;
  if (n == 0) return EIK_OK;
  const int th = 256;
  const int nb = (int)std::min<int64_t>((n + th - 1) / th, 152 * 16);
  k_sfs_forcing<<<nb, th, 0, stream>>>(P, n, f_min, f);
  return cudaGetLastError() == cudaSuccess ? EIK_OK : EIK_ERR_CUDA;
}
