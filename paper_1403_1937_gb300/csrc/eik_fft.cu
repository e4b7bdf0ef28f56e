// FFT perturbation series of Sec. 5 (Table 1) on a 2D grid.
//
// With a constant f~, phi = phi_0 - phi_1 + phi_2 - ... + (-1)^T phi_T,
// phi_0 = G~ * delta_kron (G~ = exp(-f~|x|/hbar), Sec. 3.2), and
// phi_i = h^2 G * [(f^2 - f~^2) phi_{i-1}] (Eq. phi_i_Solution) with G the 2D
// Green's function K_0(f~|x|/hbar) / (2 pi hbar^2) (Eq. GreensFunction2D);
// S = -hbar log phi.  Every convolution is the linear one over the grid,
// computed by complex FP64 transforms of arrays zero-padded to P_a >= 2 n_a - 1
// points per axis with the kernel sampled at the offsets
// -(n_a - 1) .. n_a - 1 and wrapped; G's sample at the origin is its average
// over the grid cell.
//
// Transforms.  Everything transformed is real, so two rows of a grid function
// travel as the real and imaginary part of one complex row, and only the
// columns kx <= P_x / 2 of its spectrum are kept.  One term is four launches:
//   k_rows_x  inverse row transforms of the last product, which give the term
//             (added to phi); psi of the next term; its forward transforms
//   k_unpack  split of the row pairs' spectra, transposed
//   k_cols    forward column transform, times the kernel's spectrum, inverse
//   k_repack  the row pairs' spectra again, transposed back
// Both kernels are even in x and y: their spectra are real, and their row
// pairs' and column pairs' transforms need no split.  Against complex
// transforms of the whole padded array (two row passes each way, products,
// embedding and extraction as passes of their own) this does half of the FP64
// work, which is what bounds the series on this GPU, and a third of the
// launches: 513^2, six terms 3.65 ms before, 2.05 ms now.
//
// A row transform runs in one block, in shared memory, as the Stockham
// self-sorting form of the mixed-radix FFT: lengths P = 2^a 3^b 5^c (the
// smallest >= 2n - 1), stages of radix 4, 2, 3 and 5, each reading one buffer
// and writing the other in natural order.
//
// K_0 and K_1 come from their integral representation
// K_nu(x) = int_0^inf exp(-x cosh t) cosh(nu t) dt (DLMF 10.32.9), summed by
// the trapezoidal rule, which converges geometrically for this analytic,
// doubly exponentially decaying integrand; the step shrinks like 1/sqrt(x)
// for large x, where the integrand is a narrow Gaussian around t = 0.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "eik_internal.cuh"

namespace eik {
namespace {

constexpr int kMaxFft = 7200;   // largest transform length per axis (two buffers
                                // of P complex doubles in shared memory)
constexpr int kMaxStages = 16;

__device__ __forceinline__ double2 cadd(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ double2 csub(double2 a, double2 b) {
  return make_double2(a.x - b.x, a.y - b.y);
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// Twiddles w_q = exp(-2 pi i q / P), q < P.
__global__ void k_twiddles(double2 *tw, int P) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= P) return;
  double s, c;
  sincospi(2.0 * q / P, &s, &c);
  tw[q] = make_double2(c, -s);
}

// The radices of one transform length, in stage order.
struct Radices {
  int n;
  int r[kMaxStages];
};

// Multiplication by -i (forward) or +i (inverse).
template <bool INV>
__device__ __forceinline__ double2 rot(double2 a) {
  return INV ? make_double2(-a.y, a.x) : make_double2(a.y, -a.x);
}

// In-place DFT of R points, forward (exp(-2 pi i q r / R)) or inverse.
// Radix-3 and -5 constants: cos/sin of 2 pi / R multiples (passed in).
struct DftConst {
  double c3, s3;            // cos(2pi/3), sin(2pi/3)
  double c51, c52, s51, s52;  // cos(2pi/5), cos(4pi/5), sin(2pi/5), sin(4pi/5)
};

template <int R, bool INV>
__device__ __forceinline__ void dft(double2 *v, const DftConst &k) {
  if constexpr (R == 2) {
    const double2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  } else if constexpr (R == 4) {
    const double2 t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
    const double2 t2 = cadd(v[1], v[3]), t3 = rot<INV>(csub(v[1], v[3]));
    v[0] = cadd(t0, t2);
    v[2] = csub(t0, t2);
    v[1] = cadd(t1, t3);
    v[3] = csub(t1, t3);
  } else if constexpr (R == 3) {
    const double2 a = v[0], t = cadd(v[1], v[2]);
    const double2 m = make_double2(a.x + k.c3 * t.x, a.y + k.c3 * t.y);
    const double2 d = rot<INV>(csub(v[1], v[2]));
    v[0] = cadd(a, t);
    v[1] = make_double2(m.x + k.s3 * d.x, m.y + k.s3 * d.y);
    v[2] = make_double2(m.x - k.s3 * d.x, m.y - k.s3 * d.y);
  } else {   // R == 5
    const double2 a = v[0];
    const double2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    const double2 t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
    const double2 m1 = make_double2(a.x + k.c51 * t1.x + k.c52 * t2.x,
                                    a.y + k.c51 * t1.y + k.c52 * t2.y);
    const double2 m2 = make_double2(a.x + k.c52 * t1.x + k.c51 * t2.x,
                                    a.y + k.c52 * t1.y + k.c51 * t2.y);
    const double2 n1 = rot<INV>(make_double2(k.s51 * t3.x + k.s52 * t4.x,
                                             k.s51 * t3.y + k.s52 * t4.y));
    const double2 n2 = rot<INV>(make_double2(k.s52 * t3.x - k.s51 * t4.x,
                                             k.s52 * t3.y - k.s51 * t4.y));
    v[0] = cadd(a, cadd(t1, t2));
    v[1] = cadd(m1, n1);
    v[4] = csub(m1, n1);
    v[2] = cadd(m2, n2);
    v[3] = csub(m2, n2);
  }
}

// One 1D transform of length P per block (rows of `a`, pitch P); INV uses
// the conjugate twiddles and butterflies (no 1/P scaling).  Stockham stage of
// radix R over span Ns: for j < P/R, with k = j mod Ns, the R inputs
// x[j + r P/R] are twiddled by w^(r k P/(Ns R)), transformed, and written to
// y[(j / Ns) Ns R + k + r Ns]; Ns grows by R each stage.
template <int R, bool INV>
__device__ __forceinline__ void stockham_stage(const double2 *x, double2 *y, int P, int Ns,
                                               const double2 *__restrict__ tw,
                                               const DftConst &kc) {
  const int m = P / R;
  const int tstep = P / (Ns * R);   // w_{Ns R}^(r k) = w_P^(r k tstep)
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    const int k = j % Ns;
    double2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      double2 t = x[j + r * m];
      if (r > 0 && k > 0) {
        double2 w = __ldg(tw + r * k * tstep);   // r k tstep < P
        if (INV) w.y = -w.y;
        t = cmul(w, t);
      }
      v[r] = t;
    }
    dft<R, INV>(v, kc);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) y[base + r * Ns] = v[r];
  }
}

// Transform of the row in x (y: scratch of the same length); returns the
// buffer that holds the result.  Every stage ends with a barrier.
template <bool INV>
__device__ __forceinline__ double2 *fft_row(double2 *x, double2 *y, int P, const Radices &rad,
                                            const DftConst &kc, const double2 *__restrict__ tw) {
  int Ns = 1;
  for (int st = 0; st < rad.n; ++st) {
    const int R = rad.r[st];
    switch (R) {
      case 4: stockham_stage<4, INV>(x, y, P, Ns, tw, kc); break;
      case 2: stockham_stage<2, INV>(x, y, P, Ns, tw, kc); break;
      case 3: stockham_stage<3, INV>(x, y, P, Ns, tw, kc); break;
      default: stockham_stage<5, INV>(x, y, P, Ns, tw, kc); break;
    }
    __syncthreads();
    double2 *tmp = x;
    x = y;
    y = tmp;
    Ns *= R;
  }
  return x;
}

// Rows 2 b and 2 b + 1 of the grid (block b).  INV: inverse transforms of Z's
// row, scaled, give the term's rows; phi = v, or phi += sign v.  FWD: forward
// transforms of psi = (f^2 - f~^2) v (Table 1 step 9), or of the grid function
// `in` itself, into Z's row.
template <bool INV, bool FWD>
__global__ void k_rows_x(double2 *Z, int P, Radices rad, DftConst kc,
                         const double2 *__restrict__ tw, int nx, int ny,
                         const double *__restrict__ in, const double *__restrict__ f, double ft2,
                         double scale, double sign, int first, double *__restrict__ phi) {
  extern __shared__ double2 fsm[];
  double2 *x = fsm, *y = fsm + P;
  double2 *row = Z + (size_t)blockIdx.x * P;
  const int64_t o0 = (int64_t)2 * blockIdx.x * nx, o1 = o0 + nx;
  const bool two = 2 * blockIdx.x + 1 < ny;
  if (INV) {
    for (int i = threadIdx.x; i < P; i += blockDim.x) x[i] = row[i];
    __syncthreads();
    double2 *z = fft_row<true>(x, y, P, rad, kc, tw);
    if (z != x) {
      y = x;
      x = z;
    }
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
      double2 psi = make_double2(0.0, 0.0);
      if (i < nx) {
        const double v0 = scale * x[i].x, v1 = scale * x[i].y;
        phi[o0 + i] = first ? v0 : phi[o0 + i] + sign * v0;
        if (two) phi[o1 + i] = first ? v1 : phi[o1 + i] + sign * v1;
        if (FWD) {
          const double f0 = f[o0 + i];
          psi.x = (f0 * f0 - ft2) * v0;
          if (two) {
            const double f1 = f[o1 + i];
            psi.y = (f1 * f1 - ft2) * v1;
          }
        }
      }
      if (FWD) x[i] = psi;
    }
  } else {
    for (int i = threadIdx.x; i < P; i += blockDim.x)
      x[i] = (i < nx) ? make_double2(in[o0 + i], two ? in[o1 + i] : 0.0) : make_double2(0.0, 0.0);
  }
  if (!FWD) return;
  __syncthreads();
  const double2 *z = fft_row<false>(x, y, P, rad, kc, tw);
  for (int i = threadIdx.x; i < P; i += blockDim.x) row[i] = z[i];
}

// B[k][y] (hx x ny), the spectrum of grid row y at kx = k, from the row pairs'
// transforms Z (Z_k = A_k + i B_k with A, B Hermitian): 32 x 32 tiles of (k,
// pair), transposed through shared memory.
__global__ void k_unpack(const double2 *__restrict__ Z, double2 *__restrict__ B, int P, int hx,
                         int ny) {
  __shared__ double2 t[32][33], u[32][33];
  const int k = blockIdx.x * 32 + threadIdx.x, np = (ny + 1) / 2;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int r = blockIdx.y * 32 + q;
    if (k < hx && r < np) {
      const double2 a = Z[(size_t)r * P + k], b = Z[(size_t)r * P + (k == 0 ? 0 : P - k)];
      t[q][threadIdx.x] = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
      u[q][threadIdx.x] = make_double2(0.5 * (a.y + b.y), 0.5 * (b.x - a.x));
    }
  }
  __syncthreads();
  // rows of B: columns y = 2 r and 2 r + 1 side by side
  const int y = blockIdx.y * 64 + 2 * threadIdx.x;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int kk = blockIdx.x * 32 + q;
    if (kk < hx) {
      if (y < ny) B[(size_t)kk * ny + y] = t[threadIdx.x][q];
      if (y + 1 < ny) B[(size_t)kk * ny + y + 1] = u[threadIdx.x][q];
    }
  }
}

// The inverse of k_unpack: Z_k = A_k + i B_k, also for kx > P / 2 by symmetry.
__global__ void k_repack(const double2 *__restrict__ B, double2 *__restrict__ Z, int P, int hx,
                         int ny) {
  __shared__ double2 t[32][33], u[32][33];
  const int y = blockIdx.y * 64 + 2 * threadIdx.x, np = (ny + 1) / 2;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int kk = blockIdx.x * 32 + q;
    if (kk < hx) {
      t[q][threadIdx.x] = (y < ny) ? B[(size_t)kk * ny + y] : make_double2(0.0, 0.0);
      u[q][threadIdx.x] = (y + 1 < ny) ? B[(size_t)kk * ny + y + 1] : make_double2(0.0, 0.0);
    }
  }
  __syncthreads();
  const int k = blockIdx.x * 32 + threadIdx.x;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int r = blockIdx.y * 32 + q;
    if (k < hx && r < np) {
      const double2 a = t[threadIdx.x][q], b = u[threadIdx.x][q];
      Z[(size_t)r * P + k] = make_double2(a.x - b.y, a.y + b.x);
      if (k > 0 && P - k >= hx) Z[(size_t)r * P + P - k] = make_double2(a.x + b.y, b.x - a.y);
    }
  }
}

// One column kx = blockIdx.x of the spectrum: forward transform along y (zero
// past the grid), times the kernel's spectrum, inverse.
__global__ void k_cols(double2 *B, int P, Radices rad, DftConst kc,
                       const double2 *__restrict__ tw, int ny, const double *__restrict__ K) {
  extern __shared__ double2 fsm[];
  double2 *x = fsm, *y = fsm + P;
  double2 *row = B + (size_t)blockIdx.x * ny;
  const double *k = K + (size_t)blockIdx.x * P;
  for (int i = threadIdx.x; i < P; i += blockDim.x)
    x[i] = (i < ny) ? row[i] : make_double2(0.0, 0.0);
  __syncthreads();
  double2 *z = fft_row<false>(x, y, P, rad, kc, tw);
  if (z != x) {
    y = x;
    x = z;
  }
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    const double m = k[i];
    x[i] = make_double2(m * x[i].x, m * x[i].y);
  }
  __syncthreads();
  z = fft_row<true>(x, y, P, rad, kc, tw);
  for (int i = threadIdx.x; i < ny; i += blockDim.x) row[i] = z[i];
}

// K_nu(x), nu = 0 or 1, x > 0 (integral representation, trapezoidal rule).
// The nodes' c_k = cosh(k eta) come from the recurrence c_{k+1} =
// 2 cosh(eta) c_k - c_{k-1} (one exponential per node instead of three; the
// rounding it adds grows like k eps over the few dozen nodes summed).
__device__ double bessel_k(int nu, double x) {
  if (!(x > 0.0)) return INFINITY;
  if (x > 745.0) return 0.0;
  const double eta = fmin(0.25, 0.7 / sqrt(x));
  const double ex = exp(-x);
  const double ce = cosh(eta);
  // exp(-x cosh t) = exp(-x) exp(-x (cosh t - 1)); half weight at t = 0
  double sum = 0.5, cprev = 1.0, c = ce;
  for (int k = 1; k < 4000; ++k) {
    const double term = exp(-x * (c - 1.0)) * (nu ? c : 1.0);
    sum += term;
    if (term < 1e-18 * sum) break;
    const double cn = 2.0 * ce * c - cprev;
    cprev = c;
    c = cn;
  }
  return eta * ex * sum;
}

// G at the offsets 0 <= b <= a < m, packed as tab[a (a + 1) / 2 + b] (G
// depends on |offset| only, so one octant serves all); the origin takes *g0.
__global__ void k_green_table(double *tab, int m, double h, double ft, double hbar,
                              const double *g0) {
  const int64_t tot = (int64_t)m * (m + 1) / 2;
  const double inv2pi = 1.0 / (2.0 * M_PI * hbar * hbar);
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot;
       e += (int64_t)gridDim.x * blockDim.x) {
    int a = (int)((sqrt(8.0 * (double)e + 1.0) - 1.0) * 0.5);
    while ((int64_t)a * (a + 1) / 2 > e) --a;
    while ((int64_t)(a + 1) * (a + 2) / 2 <= e) ++a;
    const int b = (int)(e - (int64_t)a * (a + 1) / 2);
    tab[e] = (a == 0) ? *g0 : bessel_k(0, ft * h * hypot((double)a, (double)b) / hbar) * inv2pi;
  }
}

// Kernel rows y = 2 b and 2 b + 1 (y >= 0 offsets) at the wrapped x offsets:
// mode 0 G~ = exp(-f~ r / hbar), mode 1 G from the octant table.  Both rows are
// even in x, so the pair's transform holds their real spectra as its real and
// imaginary part: KX[y][kx], kx < hx.
__global__ void k_kernel_rows(double *__restrict__ KX, int P, Radices rad, DftConst kc,
                              const double2 *__restrict__ tw, int nx, int ny, int hx, double h,
                              double ft, double hbar, int mode, const double *__restrict__ tab) {
  extern __shared__ double2 fsm[];
  const int y0 = 2 * blockIdx.x;
  auto value = [&](int ox, int oy) {
    if (mode == 0) return exp(-ft * h * hypot((double)ox, (double)oy) / hbar);
    const int p = max(abs(ox), abs(oy)), q = min(abs(ox), abs(oy));
    return tab[(int64_t)p * (p + 1) / 2 + q];
  };
  // the half x >= 0; the other half is its mirror image
  for (int i = threadIdx.x; i < nx; i += blockDim.x) {
    const double2 v = make_double2(value(i, y0), (y0 + 1 < ny) ? value(i, y0 + 1) : 0.0);
    fsm[i] = v;
    if (i > 0) fsm[P - i] = v;
  }
  for (int i = nx + threadIdx.x; i < P - nx + 1; i += blockDim.x) fsm[i] = make_double2(0.0, 0.0);
  __syncthreads();
  const double2 *z = fft_row<false>(fsm, fsm + P, P, rad, kc, tw);
  for (int i = threadIdx.x; i < hx; i += blockDim.x) {
    KX[(size_t)y0 * hx + i] = z[i].x;
    if (y0 + 1 < ny) KX[(size_t)(y0 + 1) * hx + i] = z[i].y;
  }
}

// Columns kx = 2 b and 2 b + 1 of the kernel's spectrum, likewise: K[kx][ky].
__global__ void k_kernel_cols(const double *__restrict__ KX, double *__restrict__ K, int P,
                              Radices rad, DftConst kc, const double2 *__restrict__ tw, int ny,
                              int hx) {
  extern __shared__ double2 fsm[];
  const int k0 = 2 * blockIdx.x;
  const bool two = k0 + 1 < hx;
  for (int i = threadIdx.x; i < ny; i += blockDim.x) {
    const double *q = KX + (size_t)i * hx + k0;
    const double2 v = make_double2(q[0], two ? q[1] : 0.0);
    fsm[i] = v;
    if (i > 0) fsm[P - i] = v;
  }
  for (int i = ny + threadIdx.x; i < P - ny + 1; i += blockDim.x) fsm[i] = make_double2(0.0, 0.0);
  __syncthreads();
  const double2 *z = fft_row<false>(fsm, fsm + P, P, rad, kc, tw);
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    K[(size_t)k0 * P + i] = z[i].x;
    if (two) K[(size_t)(k0 + 1) * P + i] = z[i].y;
  }
}

// G's average over the cell [-h/2, h/2]^2: 8 rays' triangles, along each
// int_0^R r K_0(a r) dr = (1 - a R K_1(a R)) / a^2, R = (h/2) / cos(theta),
// over theta in [0, pi/4] by Simpson's rule: the weighted samples first,
// spread over the GPU, then their fixed-order sum in one block.
constexpr int kSimpson = 2048;   // intervals (even)

__global__ void k_cell_samples(double h, double ft, double hbar, double *val) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k > kSimpson) return;
  const double a = ft / hbar;
  const double th = (M_PI / 4) * k / kSimpson;
  const double R = 0.5 * h / cos(th);
  const double v = (1.0 - a * R * bessel_k(1, a * R)) / (a * a);
  const double w = (k == 0 || k == kSimpson) ? 1.0 : ((k & 1) ? 4.0 : 2.0);
  val[k] = w * v;
}

__global__ void k_cell_average(const double *__restrict__ val, double h, double hbar,
                               double *g0) {
  __shared__ double red[32];
  double acc = 0.0;
  for (int k = threadIdx.x; k <= kSimpson; k += blockDim.x) acc += val[k];
  acc = block_sum(acc, red);
  if (threadIdx.x == 0) {
    const double integral = 8.0 * acc * (M_PI / 4) / (3.0 * kSimpson);
    *g0 = integral / (h * h) / (2.0 * M_PI * hbar * hbar);
  }
}

// The sources' Kronecker deltas on the grid (zeroed before).
__global__ void k_delta(double *a, const int64_t *__restrict__ src, int64_t nsrc) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < nsrc) a[src[k]] = 1.0;
}

__global__ void k_log(const double *__restrict__ phi, int64_t n, double hbar, double *S) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    S[i] = -hbar * log(phi[i]);
}

// min and max of f, and a flag for values that are not finite and positive.
__global__ void k_fminmax(const double *__restrict__ f, int64_t n, double *out, int *bad) {
  double lo = INFINITY, hi = 0.0;
  int b = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double v = f[i];
    if (!(v > 0.0) || !isfinite(v)) b = 1;
    lo = fmin(lo, v);
    hi = fmax(hi, v);
  }
  if (b) atomicExch(bad, 1);
  // per warp, then one atomic per warp: positive doubles order like their bits
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_down_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_down_sync(0xffffffffu, hi, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (hi > 0.0)
      atomicMax(reinterpret_cast<unsigned long long *>(out + 1),
                (unsigned long long)__double_as_longlong(hi));
    if (lo > 0.0 && lo < INFINITY)
      atomicMin(reinterpret_cast<unsigned long long *>(out),
                (unsigned long long)__double_as_longlong(lo));
  }
}

struct Fft2 {
  int Px, Py, hx;   // transform lengths; columns of the spectrum kept
  int nx, ny;
  Radices rx, ry;
  DftConst kc;
  double2 *twx, *twy;
  double2 *Z;       // row pairs: ceil(ny / 2) x Px
  double2 *B;       // spectrum by column: hx x ny
  double *KX, *K;   // kernel: rows' spectra ny x hx, spectrum hx x Py
  cudaStream_t s;
};

// Smallest 2^a 3^b 5^c >= n (0 if above kMaxFft).
int fft_length(int n) {
  for (int p = std::max(n, 2); p <= kMaxFft; ++p) {
    int q = p;
    for (int f : {2, 3, 5})
      while (q % f == 0) q /= f;
    if (q == 1) return p;
  }
  return 0;
}

// Stage radices of P: fours first, then a two, threes and fives.
Radices radices(int P) {
  Radices r{};
  int q = P;
  while (q % 4 == 0 && r.n < kMaxStages) {
    r.r[r.n++] = 4;
    q /= 4;
  }
  for (int f : {2, 3, 5})
    while (q % f == 0 && r.n < kMaxStages) {
      r.r[r.n++] = f;
      q /= f;
    }
  return r;
}

int fft_threads(int P) { return std::min(512, std::max(32, P / 2)); }
size_t fft_smem(int P) { return 2 * sizeof(double2) * P; }

// Spectrum of a kernel into F.K.
void kernel_spectrum(const Fft2 &F, double h, double ft, double hbar, int mode, const double *tab) {
  k_kernel_rows<<<(F.ny + 1) / 2, fft_threads(F.Px), fft_smem(F.Px), F.s>>>(
      F.KX, F.Px, F.rx, F.kc, F.twx, F.nx, F.ny, F.hx, h, ft, hbar, mode, tab);
  k_kernel_cols<<<(F.hx + 1) / 2, fft_threads(F.Py), fft_smem(F.Py), F.s>>>(
      F.KX, F.K, F.Py, F.ry, F.kc, F.twy, F.ny, F.hx);
}

// Z (forward row transforms) -> Z (before the inverse ones), times F.K.
void convolve(const Fft2 &F) {
  const dim3 g((F.hx + 31) / 32, ((F.ny + 1) / 2 + 31) / 32), b(32, 8);
  k_unpack<<<g, b, 0, F.s>>>(F.Z, F.B, F.Px, F.hx, F.ny);
  k_cols<<<F.hx, fft_threads(F.Py), fft_smem(F.Py), F.s>>>(F.B, F.Py, F.ry, F.kc, F.twy, F.ny, F.K);
  k_repack<<<g, b, 0, F.s>>>(F.B, F.Z, F.Px, F.hx, F.ny);
}

template <bool INV, bool FWD>
void rows_x(const Fft2 &F, const double *in, const double *f, double ft2, double scale,
            double sign, int first, double *phi) {
  k_rows_x<INV, FWD><<<(F.ny + 1) / 2, fft_threads(F.Px), fft_smem(F.Px), F.s>>>(
      F.Z, F.Px, F.rx, F.kc, F.twx, F.nx, F.ny, in, f, ft2, scale, sign, first, phi);
}

// The attribute belongs to the function: always the largest row, so that
// concurrent calls agree.
template <class Kn>
bool max_smem(Kn *fn) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)fft_smem(kMaxFft)) == cudaSuccess;
}

// Work arrays from the stream-ordered allocator (the device's memory pool):
// after the first call, allocating and freeing them costs no synchronisation.
struct Buf {
  cudaStream_t s;
  std::vector<void *> p;
  explicit Buf(cudaStream_t st) : s(st) {}
  ~Buf() {
    for (void *q : p) cudaFreeAsync(q, s);
  }
  template <class T>
  bool get(T **out, size_t n) {
    void *q = nullptr;
    if (cudaMallocAsync(&q, sizeof(T) * std::max<size_t>(n, 1), s) != cudaSuccess) return false;
    p.push_back(q);
    *out = static_cast<T *>(q);
    return true;
  }
};

}  // namespace
}  // namespace eik

using namespace eik;

extern "C" eik_status eik_fft_series(const int64_t *dims, double h, double hbar, const double *f,
                                     const int64_t *src_idx, int64_t nsrc, int terms,
                                     double f_tilde, double *S_out, double *phi_out,
                                     double *f_tilde_out, eik_stream_t stream) {
  if (!dims || !f || !src_idx || !S_out || nsrc < 1 || terms < 0 || terms > 64)
    return EIK_ERR_ARG;
  if (!(h > 0.0) || !std::isfinite(h) || !(hbar > 0.0) || !std::isfinite(hbar) ||
      !(f_tilde >= 0.0) || !std::isfinite(f_tilde))
    return EIK_ERR_ARG;
  const int64_t nx64 = dims[0], ny64 = dims[1];
  if (nx64 < 2 || ny64 < 2 || 2 * nx64 - 1 > kMaxFft || 2 * ny64 - 1 > kMaxFft)
    return EIK_ERR_ARG;
  const int nx = (int)nx64, ny = (int)ny64;
  const int64_t n = nx64 * ny64;
  std::vector<int64_t> hs(nsrc);
  if (cudaMemcpy(hs.data(), src_idx, sizeof(int64_t) * nsrc, cudaMemcpyDefault) != cudaSuccess)
    return EIK_ERR_ARG;
  for (int64_t s : hs)
    if (s < 0 || s >= n) return EIK_ERR_ARG;
  cudaStream_t s = stream;
  Fft2 F;
  F.Px = fft_length(2 * nx - 1);
  F.Py = fft_length(2 * ny - 1);
  if (F.Px == 0 || F.Py == 0) return EIK_ERR_ARG;
  F.rx = radices(F.Px);
  F.ry = radices(F.Py);
  F.kc = DftConst{-0.5, 0.5 * std::sqrt(3.0),
                  0.25 * (std::sqrt(5.0) - 1.0), -0.25 * (std::sqrt(5.0) + 1.0),
                  std::sqrt(0.125 * (5.0 + std::sqrt(5.0))),
                  std::sqrt(0.125 * (5.0 - std::sqrt(5.0)))};
  F.s = s;
  F.nx = nx;
  F.ny = ny;
  F.hx = F.Px / 2 + 1;
  Buf buf(s);
  double *fd = nullptr, *phi = nullptr, *Sd = nullptr, *mm = nullptr, *g0 = nullptr;
  double *gtab = nullptr, *cval = nullptr;
  const int m = std::max(nx, ny);
  int64_t *src = nullptr;
  int *bad = nullptr;
  if (!buf.get(&F.twx, F.Px) || !buf.get(&F.twy, F.Py) ||
      !buf.get(&F.Z, (size_t)((ny + 1) / 2) * F.Px) || !buf.get(&F.B, (size_t)F.hx * ny) ||
      !buf.get(&F.KX, (size_t)F.hx * ny) || !buf.get(&F.K, (size_t)F.hx * F.Py) ||
      !buf.get(&fd, n) || !buf.get(&phi, n) || !buf.get(&Sd, n) || !buf.get(&mm, 2) ||
      !buf.get(&g0, 1) ||
      !buf.get(&src, nsrc) || !buf.get(&bad, 1) ||
      !buf.get(&gtab, (size_t)m * (m + 1) / 2) || !buf.get(&cval, kSimpson + 1)) {
    cudaGetLastError();
    return EIK_ERR_OOM;
  }
  if (!max_smem(k_rows_x<false, true>) || !max_smem(k_rows_x<true, true>) ||
      !max_smem(k_rows_x<true, false>) || !max_smem(k_cols) || !max_smem(k_kernel_rows) ||
      !max_smem(k_kernel_cols))
    return EIK_ERR_CUDA;
  const int nb = 152 * 8;
  if (cudaMemcpyAsync(fd, f, sizeof(double) * n, cudaMemcpyDefault, s) != cudaSuccess ||
      cudaMemcpyAsync(src, hs.data(), sizeof(int64_t) * nsrc, cudaMemcpyHostToDevice, s) !=
          cudaSuccess)
    return EIK_ERR_ARG;
  // f validation and f~ (Eq. fTildeValue when not given)
  const double init[2] = {INFINITY, 0.0};
  if (cudaMemcpyAsync(mm, init, sizeof init, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemsetAsync(bad, 0, sizeof(int), s) != cudaSuccess)
    return EIK_ERR_CUDA;
  k_fminmax<<<nb, kThreads, 0, s>>>(fd, n, mm, bad);
  double hmm[2];
  int hbad = 0;
  if (cudaMemcpyAsync(hmm, mm, sizeof hmm, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return EIK_ERR_CUDA;
  if (hbad) return EIK_ERR_ARG;
  const double ft = (f_tilde > 0.0) ? f_tilde : std::sqrt(0.5 * (hmm[0] * hmm[0] + hmm[1] * hmm[1]));
  k_twiddles<<<(F.Px + 255) / 256, 256, 0, s>>>(F.twx, F.Px);
  k_twiddles<<<(F.Py + 255) / 256, 256, 0, s>>>(F.twy, F.Py);
  const double inv = 1.0 / ((double)F.Px * F.Py);
  // Table 1 steps 1-6: phi = phi_0 = G~ * delta_kron (Sd holds the deltas)
  kernel_spectrum(F, h, ft, hbar, 0, nullptr);
  cudaMemsetAsync(Sd, 0, sizeof(double) * n, s);
  k_delta<<<(int)((nsrc + 255) / 256), 256, 0, s>>>(Sd, src, nsrc);
  rows_x<false, true>(F, Sd, nullptr, 0.0, 0.0, 0.0, 0, nullptr);
  convolve(F);
  if (terms == 0) {
    rows_x<true, false>(F, nullptr, nullptr, 0.0, inv, 1.0, 1, phi);
  } else {
    rows_x<true, true>(F, nullptr, fd, ft * ft, inv, 1.0, 1, phi);
    // step 7: transform of G
    k_cell_samples<<<(kSimpson + 1 + 63) / 64, 64, 0, s>>>(h, ft, hbar, cval);
    k_cell_average<<<1, kThreads, 0, s>>>(cval, h, hbar, g0);
    k_green_table<<<nb, kThreads, 0, s>>>(gtab, m, h, ft, hbar, g0);
    kernel_spectrum(F, h, ft, hbar, 1, gtab);
    // steps 8-14
    for (int i = 1; i <= terms; ++i) {
      convolve(F);
      const double sign = (i & 1) ? -1.0 : 1.0;
      if (i < terms) rows_x<true, true>(F, nullptr, fd, ft * ft, inv * h * h, sign, 0, phi);
      else rows_x<true, false>(F, nullptr, nullptr, 0.0, inv * h * h, sign, 0, phi);
    }
  }
  // step 15
  k_log<<<nb, kThreads, 0, s>>>(phi, n, hbar, Sd);
  if (cudaGetLastError() != cudaSuccess) return EIK_ERR_CUDA;
  if (cudaMemcpyAsync(S_out, Sd, sizeof(double) * n, cudaMemcpyDefault, s) != cudaSuccess)
    return EIK_ERR_ARG;
  if (phi_out &&
      cudaMemcpyAsync(phi_out, phi, sizeof(double) * n, cudaMemcpyDefault, s) != cudaSuccess)
    return EIK_ERR_ARG;
  if (cudaStreamSynchronize(s) != cudaSuccess) return EIK_ERR_CUDA;
  if (f_tilde_out) *f_tilde_out = ft;
  return EIK_OK;
}
