// Multigrid-preconditioned inner solve of the mixed-precision path (2D, 3D).
//
// The paper names multigrid as the O(N) route for the sparse system of
// Sec. 6 (Eq. sparse-system); this file builds one that keeps the relative
// accuracy the method needs.  phi = exp(-S/hbar) spans hundreds of powers of
// two, and a componentwise tolerance asks for the far field as precisely as
// the near field, so the coarse spaces are built in relative form:
//
// * Level 0 is the Jacobi-scaled operator of the correction equation in kx
//   units, (A v)_i = v_i - sig_i sum_j omega_ij sig_j 2^(kx_i - kx_j) v_j,
//   exactly as in the Jacobi-preconditioned inner CG.
// * Coarse node C of level l + 1 aggregates a 2 x 2 (x 2) box of level-l
//   nodes.  Its basis function is, on level 0, the estimated solution shape
//   w_i = exp(kx_i ln 2 - St_i / hbar) / sig_i on the box (St_i: the cell
//   distance estimate interpolated (bi/tri)linearly between cell centres), so a
//   coarse unknown is a relative correction, constant on its box, of the
//   estimated phi.  Coarser levels take unit weights, so every coarse basis
//   function keeps that level-0 shape.
// * Every level l holds its Galerkin operator A^l = P^T A^(l-1) P (true,
//   symmetric) for vectors stored as value * 2^k, k a power-of-two exponent
//   per node: (A y)_C = a_C y_C + sum_D c_CD y_D with the row-relative
//   coefficients c_CD = A_CD 2^(k_C - k_D), one per neighbour (west, east,
//   south, north, below, above), formed in FP64.  Between an aggregate and its upstream
//   neighbour (nearer the sources) c is O(1); downstream it is tiny or 0.
//   (Storing A_CD and the factor separately would overflow FP32 on coarse
//   levels, where neighbouring exponents differ by over a hundred.)  The
//   transfers in these units: restriction g_C = sum_{i in C} P_i 2^(k_C -
//   k_i) t_i, prolongation y_i += P_i 2^(k_i - k_C) y_C, with P_i = w_i on
//   level 0 (one exponent per box there) and P_i = 2^(k_C - k_i), k_C = min
//   over the box, above; so c^(l+1)_CD = sum_{i in C, j in D} 2^(2(k_C -
//   k_i)) c_ij and a^(l+1)_C = sum_{i in C} 2^(2(k_C - k_i)) (a_i + sum_{j in
//   C} c_ij).
// * The cycle is a symmetric V-cycle down to one node: one damped-Jacobi
//   sweep (omega = 8/9) before and after each coarse correction, the single
//   node solved exactly.  Sources (sig = 0) take no part in any transfer.
//
// The outer iteration is preconditioned CG on level 0 in kx units with the
// true inner product, <u, v> = sum u_i v_i 2^(-2 kx_i) (per-thread FP32
// sums, weights relative to the smallest exponent, 0 past the FP32 range;
// FP64 across threads and blocks in a fixed order),
// one graph launch per two iterations:
//   z = M r, rho = <r, z>, beta = rho / rho_old, p = z + beta p, q = A p,
//   alpha = rho / <p, q>, d += alpha p, r -= alpha q,
// and the inner solve stops on the mixed solve's tests (scaled max norm of r
// or the componentwise test against the iterate).  Measured on a CPU model of
// this scheme (FP32 inner vectors, FP64 refinement): 56 inner iterations
// instead of 998 for Jacobi-PCG on a 513^2 workload with hbar = 10.2 h, and
// 72 / 79 with hbar = 4 h / 2 h (phi down to e^-128, no level-set bands).
#include <cuda.h>
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <climits>
#include <string>
#include <vector>

#include "eik_mg.h"

namespace eik {

namespace {

constexpr float kOmega = 8.0f / 9.0f;   // Chebyshev-optimal single step on [1/4, 2]
constexpr int kGraphIters = 2;          // even: the direction buffers alternate
// an inner solve that has not met its test after this many iterations ends
// (the refinement step then judges progress from the true residual)
constexpr int kMaxInnerIters = 1000;
// An inner solve is cut off (MixCtl.stalled = 2) where its largest residual has
// grown by kMaxGrowth, or has not fallen below its smallest value for kMaxIdle
// iterations: the FP32 recurrence has come apart, and every power of ten that
// the residual has grown by costs a refinement step to take back (measured
// without the cut-off: a 400^2 solve with hbar = 2 h whose residual had grown by
// 1e14 and 1e18 took 18 steps, or all 30, to return).  Its correction is dropped
// and the same solve, which is deterministic, runs again up to the iteration
// with the smallest residual.  Where that was not below half of the first one,
// growth may be what the solve needs (the maximum norm in kx units does not
// fall steadily in CG), and it runs again without a cut-off.
constexpr float kMaxGrowth = 1e4f;
constexpr int kMaxIdle = 200;
thread_local std::string g_msg = "no error";

enum { kW = 0, kE = 1, kS = 2, kN = 3, kB = 4, kT = 5, kDirs = 6 };

struct MgLevel {
  int nx = 0, ny = 0, nz = 1;
  float *a = nullptr;            // diagonal; a < 0 marks a node with no unknowns
  float *ia = nullptr;           // 1 / a (0 on nodes with no unknowns)
  float *c = nullptr;            // kDirs x m row-relative coefficients (W, E, S, N, B, T)
  int *k = nullptr;
  // restricted residual, its pre-smoothed correction omega g / a (written
  // beside it, so that neighbours read one array instead of two), correction
  float *g = nullptr, *yp = nullptr, *y = nullptr;
};

struct MgCtl {
  double rho;        // <r, z> of the current residual
  double alpha, beta;
  int iter, max_iter, done, status, stalled, mode, first, kmin;
  float thresh, theta;
  float r_limit;     // the inner solve is cut off where max |r| grows past this,
  int max_idle;      // or after this many iterations without a new smallest one
  float r_best;      // smallest max |r| so far and its iteration (0: the start)
  int best_iter;
  unsigned int counter[4];
};

__device__ __forceinline__ int kx_at(const CellGrid &cg, int x, int y, int z, const int *kx) {
  return kx[(x >> cg.lgB) + cg.cx * ((y >> cg.lgB) + cg.cy * (z >> cg.lgB))];
}
__device__ __forceinline__ float face(int i, int n, int boundary) {
  return (boundary == EIK_BOUNDARY_HALF_CELL && (i == 0 || i == n - 1)) ? 0.5f : 1.f;
}
// the face factor of the z axis (1 in 2D, which has no z faces)
__device__ __forceinline__ float facez(const Grid &g, int z) {
  return (g.nz > 1) ? face(z, g.nz, g.boundary) : 1.f;
}

// 2^e from its bit pattern; 0 below the normal range (such factors only
// scale terms that are negligible), e capped at 127.
__device__ __forceinline__ float p2f(int e) {
  e = min(e, 127);
  return (e < -126) ? 0.f : __int_as_float((e + 127) << 23);
}

// Grid-stride loops over the rows (y, z) of a level and its columns x: no
// 64-bit division per node.  Blocks are as wide as the row needs (grid2), so
// that short rows leave no threads idle.
#define MG_ROWS(ny_, nz_)                                                           \
  for (int rr = blockIdx.y * blockDim.y + threadIdx.y; rr < (ny_) * (nz_);          \
       rr += gridDim.y * blockDim.y)                                                \
    for (int y = rr % (ny_), z = rr / (ny_), once_ = 1; once_; once_ = 0)
#define MG_COLS(nx_) \
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < (nx_); x += gridDim.x * blockDim.x)

// Linear index of (x, y, z) on a level of pitch nx and ny rows per plane
// (DIM = 2: z is 0).
template <int DIM>
__device__ __forceinline__ int64_t lin(int x, int y, int z, int nx, int ny) {
  if constexpr (DIM == 3) return x + (int64_t)nx * (y + (int64_t)ny * z);
  else return x + (int64_t)nx * y;
}

// Coarse-level operator (A u)_t for node (x, y, z) of a level; u(j, xj, yj,
// zj) by dense index and coordinates.
template <int DIM, class V>
__device__ __forceinline__ float apply_l(const MgLevel &L, int x, int y, int z, V u) {
  const int64_t pl = (int64_t)L.nx * L.ny;
  const int64_t m = (DIM == 3) ? pl * L.nz : pl;
  const int64_t i = lin<DIM>(x, y, z, L.nx, L.ny);
  float acc = fabsf(L.a[i]) * u(i, x, y, z);
  if (x > 0) acc = fmaf(L.c[kW * m + i], u(i - 1, x - 1, y, z), acc);
  if (x + 1 < L.nx) acc = fmaf(L.c[kE * m + i], u(i + 1, x + 1, y, z), acc);
  if (y > 0) acc = fmaf(L.c[kS * m + i], u(i - L.nx, x, y - 1, z), acc);
  if (y + 1 < L.ny) acc = fmaf(L.c[kN * m + i], u(i + L.nx, x, y + 1, z), acc);
  if constexpr (DIM == 3) {
    if (z > 0) acc = fmaf(L.c[kB * m + i], u(i - pl, x, y, z - 1), acc);
    if (z + 1 < L.nz) acc = fmaf(L.c[kT * m + i], u(i + pl, x, y, z + 1), acc);
  }
  return acc;
}

// ------------------------------------------------------------- setup
// w_i = exp(kx_i ln 2 - St_i / hbar) / sig_i (0 on the sources); St_i
// interpolated linearly along each axis between the cell centres (flat
// beyond the outer ones).
__global__ void k_mg_weights(Grid g, CellGrid cg, int px, const float *__restrict__ s32,
                             const int *__restrict__ kx, const float *__restrict__ St,
                             float *__restrict__ w) {
  const float B = (float)cg.B, half = 0.5f * (B - 1.f);
  auto axis = [&](int c, int ncell, int nn, int &I0, int &I1, float &tt) {
    I0 = min(max((int)floorf(((float)c - half) / B), 0), ncell - 1);
    I1 = min(I0 + 1, ncell - 1);
    const float c0 = fminf(I0 * B + half, (float)(nn - 1));
    const float c1 = fminf(I1 * B + half, (float)(nn - 1));
    tt = (c1 > c0) ? fminf(fmaxf(((float)c - c0) / (c1 - c0), 0.f), 1.f) : 0.f;
  };
  MG_ROWS(g.ny, g.nz) MG_COLS(g.nx) {
    const int64_t i = x + (int64_t)px * rr;
    const float s = s32[i];
    if (s == 0.f) {
      w[i] = 0.f;
      continue;
    }
    int I0, I1, J0, J1, K0, K1;
    float tx, ty, tz;
    axis(x, cg.cx, g.nx, I0, I1, tx);
    axis(y, cg.cy, g.ny, J0, J1, ty);
    axis(z, cg.cz, g.nz, K0, K1, tz);
    auto Sc = [&](int I, int J, int K) { return St[I + cg.cx * (J + cg.cy * K)]; };
    const float v[8] = {Sc(I0, J0, K0), Sc(I1, J0, K0), Sc(I0, J1, K0), Sc(I1, J1, K0),
                        Sc(I0, J0, K1), Sc(I1, J0, K1), Sc(I0, J1, K1), Sc(I1, J1, K1)};
    bool fin = true;
    for (int q = 0; q < 8; ++q) fin = fin && isfinite(v[q]);
    const int ki = kx_at(cg, x, y, z, kx);
    float ex = 0.f;
    if (fin) {
      const float b0 = (1.f - ty) * ((1.f - tx) * v[0] + tx * v[1]) + ty * ((1.f - tx) * v[2] + tx * v[3]);
      const float b1 = (1.f - ty) * ((1.f - tx) * v[4] + tx * v[5]) + ty * ((1.f - tx) * v[6] + tx * v[7]);
      const float Sb = (1.f - tz) * b0 + tz * b1;
      ex = (float)((double)ki * 0.69314718055994530942 - (double)Sb / g.hbar);
      ex = fminf(fmaxf(ex, -30.f), 30.f);   // w^2 stays in the FP32 range
    }
    w[i] = expf(ex) / s;
  }
}

// Level 1 from level 0: P_i = w_i (one exponent per box: boxes lie inside
// one cell), true A_ij = -sig_i sig_j omega_ij; c_CD = 2^(k_C - k_D) sum
// w_i w_j A_ij over the edges between the two boxes.  Sums in FP64.
__global__ void k_mg_coarsen0(Grid g, CellGrid cg, int px, const float *__restrict__ s32,
                              const int *__restrict__ kx, const float *__restrict__ w, MgLevel L) {
  const int64_t m = (int64_t)L.nx * L.ny * L.nz;
  MG_ROWS(L.ny, L.nz) MG_COLS(L.nx) {
    const int64_t t = x + (int64_t)L.nx * rr;
    const int x0 = 2 * x, y0 = 2 * y, z0 = 2 * z;
    const int x1 = min(x0 + 1, g.nx - 1), y1 = min(y0 + 1, g.ny - 1), z1 = min(z0 + 1, g.nz - 1);
    auto at = [&](int a, int b, int c) { return a + (int64_t)px * (b + (int64_t)g.ny * c); };
    auto W = [&](int a, int b, int c) { return (double)w[at(a, b, c)]; };
    auto S = [&](int a, int b, int c) { return (double)s32[at(a, b, c)]; };
    // A_ij of the edges (a, b, c)-(a + 1, b, c), (a, b, c)-(a, b + 1, c), (a, b, c)-(a, b, c + 1)
    auto ax = [&](int a, int b, int c) {
      return -S(a, b, c) * S(a + 1, b, c) * (double)(face(b, g.ny, g.boundary) * facez(g, c));
    };
    auto ay = [&](int a, int b, int c) {
      return -S(a, b, c) * S(a, b + 1, c) * (double)(face(a, g.nx, g.boundary) * facez(g, c));
    };
    auto az = [&](int a, int b, int c) {
      return -S(a, b, c) * S(a, b, c + 1) *
             (double)(face(a, g.nx, g.boundary) * face(b, g.ny, g.boundary));
    };
    const int kc = kx_at(cg, x0, y0, z0, kx);
    double A = 0.0, cd[kDirs] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    bool live = false;
    for (int c = z0; c <= z1; ++c)
      for (int b = y0; b <= y1; ++b)
        for (int a = x0; a <= x1; ++a) {
          const double wi = W(a, b, c);
          if (wi != 0.0) live = true;
          A += wi * wi;
        }
    for (int c = z0; c <= z1; ++c)
      for (int b = y0; b <= y1; ++b) {
        if (x1 > x0) A += 2.0 * W(x0, b, c) * W(x1, b, c) * ax(x0, b, c);
        if (x > 0) cd[kW] += W(x0, b, c) * W(x0 - 1, b, c) * ax(x0 - 1, b, c);
        if (x + 1 < L.nx && x0 + 2 < g.nx) cd[kE] += W(x1, b, c) * W(x0 + 2, b, c) * ax(x1, b, c);
      }
    for (int c = z0; c <= z1; ++c)
      for (int a = x0; a <= x1; ++a) {
        if (y1 > y0) A += 2.0 * W(a, y0, c) * W(a, y1, c) * ay(a, y0, c);
        if (y > 0) cd[kS] += W(a, y0, c) * W(a, y0 - 1, c) * ay(a, y0 - 1, c);
        if (y + 1 < L.ny && y0 + 2 < g.ny) cd[kN] += W(a, y1, c) * W(a, y0 + 2, c) * ay(a, y1, c);
      }
    for (int b = y0; b <= y1; ++b)
      for (int a = x0; a <= x1; ++a) {
        if (z1 > z0) A += 2.0 * W(a, b, z0) * W(a, b, z1) * az(a, b, z0);
        if (z > 0) cd[kB] += W(a, b, z0) * W(a, b, z0 - 1) * az(a, b, z0 - 1);
        if (z + 1 < L.nz && z0 + 2 < g.nz) cd[kT] += W(a, b, z1) * W(a, b, z0 + 2) * az(a, b, z1);
      }
    // row-relative: times 2^(k_C - k_D), k_D the neighbouring box's cell exponent
    if (x > 0) cd[kW] *= ldexp(1.0, kc - kx_at(cg, x0 - 2, y0, z0, kx));
    if (x + 1 < L.nx && x0 + 2 < g.nx) cd[kE] *= ldexp(1.0, kc - kx_at(cg, x0 + 2, y0, z0, kx));
    if (y > 0) cd[kS] *= ldexp(1.0, kc - kx_at(cg, x0, y0 - 2, z0, kx));
    if (y + 1 < L.ny && y0 + 2 < g.ny) cd[kN] *= ldexp(1.0, kc - kx_at(cg, x0, y0 + 2, z0, kx));
    if (z > 0) cd[kB] *= ldexp(1.0, kc - kx_at(cg, x0, y0, z0 - 2, kx));
    if (z + 1 < L.nz && z0 + 2 < g.nz) cd[kT] *= ldexp(1.0, kc - kx_at(cg, x0, y0, z0 + 2, kx));
    L.a[t] = live ? (float)A : -1.f;
    L.ia[t] = live ? (float)(1.0 / A) : 0.f;
    for (int d = 0; d < kDirs; ++d) L.c[d * m + t] = live ? (float)cd[d] : 0.f;
    L.k[t] = kc;
  }
}

// Smallest exponent over the live nodes of the box (X, Y, Z) of level F;
// INT_MAX when it has none.
__device__ __forceinline__ int box_k(const MgLevel &F, int X, int Y, int Z) {
  int k = INT_MAX;
  for (int z = 2 * Z; z <= min(2 * Z + 1, F.nz - 1); ++z)
    for (int y = 2 * Y; y <= min(2 * Y + 1, F.ny - 1); ++y)
      for (int x = 2 * X; x <= min(2 * X + 1, F.nx - 1); ++x) {
        const int64_t i = x + (int64_t)F.nx * (y + (int64_t)F.ny * z);
        if (F.a[i] >= 0.f) k = min(k, F.k[i]);
      }
  return k;
}

// Level l + 1 (C) from level l (F): rows restricted with 2^(2(k_C - k_i)),
// columns prolonged with unit weight (live nodes only).
__global__ void k_mg_coarsen(MgLevel F, MgLevel C) {
  const int64_t m = (int64_t)C.nx * C.ny * C.nz;
  const int64_t mf = (int64_t)F.nx * F.ny * F.nz;
  MG_ROWS(C.ny, C.nz) MG_COLS(C.nx) {
    const int64_t t = x + (int64_t)C.nx * rr;
    const int kc = box_k(F, x, y, z);
    if (kc == INT_MAX) {
      C.a[t] = -1.f;
      C.ia[t] = 0.f;
      for (int d = 0; d < kDirs; ++d) C.c[d * m + t] = 0.f;
      C.k[t] = F.k[2 * x + (int64_t)F.nx * (2 * y + (int64_t)F.ny * 2 * z)];
      continue;
    }
    const int x0 = 2 * x, y0 = 2 * y, z0 = 2 * z;
    const int x1 = min(x0 + 1, F.nx - 1), y1 = min(y0 + 1, F.ny - 1), z1 = min(z0 + 1, F.nz - 1);
    double A = 0.0, cd[kDirs] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int c = z0; c <= z1; ++c)
      for (int b = y0; b <= y1; ++b)
        for (int a = x0; a <= x1; ++a) {
          const int64_t i = a + (int64_t)F.nx * (b + (int64_t)F.ny * c);
          if (F.a[i] < 0.f) continue;
          const double r = ldexp(1.0, 2 * (kc - F.k[i]));
          double row = (double)F.a[i];
          // neighbours inside the box join the diagonal, the others the links
          auto add = [&](bool exists, bool inside, int d) {
            if (!exists) return;
            const double cij = (double)F.c[d * mf + i];
            if (inside) row += cij;
            else cd[d] += r * cij;
          };
          add(a > 0, a - 1 >= x0, kW);
          add(a + 1 < F.nx, a + 1 <= x1, kE);
          add(b > 0, b - 1 >= y0, kS);
          add(b + 1 < F.ny, b + 1 <= y1, kN);
          add(c > 0, c - 1 >= z0, kB);
          add(c + 1 < F.nz, c + 1 <= z1, kT);
          A += r * row;
        }
    C.a[t] = (float)A;
    C.ia[t] = (float)(1.0 / A);
    C.c[kW * m + t] = (x > 0) ? (float)cd[kW] : 0.f;
    C.c[kE * m + t] = (x + 1 < C.nx) ? (float)cd[kE] : 0.f;
    C.c[kS * m + t] = (y > 0) ? (float)cd[kS] : 0.f;
    C.c[kN * m + t] = (y + 1 < C.ny) ? (float)cd[kN] : 0.f;
    C.c[kB * m + t] = (z > 0) ? (float)cd[kB] : 0.f;
    C.c[kT * m + t] = (z + 1 < C.nz) ? (float)cd[kT] : 0.f;
    C.k[t] = kc;
  }
}

// ------------------------------------------------------------- V-cycle
// Level l down (l >= 1) at coarse node (x, y, z): t = g - A yp on the box,
// restricted to level l + 1, and that level's pre-smoothed correction.
template <int DIM>
__device__ __forceinline__ void down_node(const MgLevel &F, const MgLevel &C, int x, int y, int z) {
  auto yv = [&](int64_t j, int, int, int) { return F.yp[j]; };
  const int64_t t = lin<DIM>(x, y, z, C.nx, C.ny);
  const int kc = C.k[t];
  float sum = 0.f;
  if (C.a[t] >= 0.f) {
    const int zt = (DIM == 3) ? min(2 * z + 1, F.nz - 1) : 0;
    for (int cz = 2 * z; cz <= zt; ++cz)
      for (int cy = 2 * y; cy <= min(2 * y + 1, F.ny - 1); ++cy)
        for (int cx = 2 * x; cx <= min(2 * x + 1, F.nx - 1); ++cx) {
          const int64_t i = lin<DIM>(cx, cy, cz, F.nx, F.ny);
          if (F.a[i] < 0.f) continue;
          const float ti = F.g[i] - apply_l<DIM>(F, cx, cy, cz, yv);
          sum = fmaf(p2f(2 * (kc - F.k[i])), ti, sum);
        }
  }
  C.g[t] = sum;
  C.yp[t] = kOmega * sum * C.ia[t];
}

template <int DIM>
__global__ void k_mg_down(MgLevel F, MgLevel C, const MgCtl *ctl) {
  if (ctl->done) return;
  MG_ROWS(C.ny, C.nz) MG_COLS(C.nx) down_node<DIM>(F, C, x, y, z);
}

// Level l up (l >= 1) at node (x, y, z): u = yp + y(parent);
// y = u + omega (g - A u) / a.  (Coefficients towards nodes with no unknowns
// are 0, so their parents' values do not enter.)
template <int DIM>
__device__ __forceinline__ void up_node(const MgLevel &F, const MgLevel &C, int x, int y, int z) {
  const int64_t t = lin<DIM>(x, y, z, F.nx, F.ny);
  if (F.a[t] < 0.f) {
    F.y[t] = 0.f;
    return;
  }
  auto uat = [&](int64_t j, int xj, int yj, int zj) {
    return F.yp[j] + C.y[lin<DIM>(xj >> 1, yj >> 1, zj >> 1, C.nx, C.ny)];
  };
  const float ut = uat(t, x, y, z);
  const float Au = apply_l<DIM>(F, x, y, z, uat);
  F.y[t] = fmaf(kOmega * (F.g[t] - Au), F.ia[t], ut);
}

template <int DIM>
__global__ void k_mg_up(MgLevel F, MgLevel C, const MgCtl *ctl) {
  if (ctl->done) return;
  MG_ROWS(F.ny, F.nz) MG_COLS(F.nx) up_node<DIM>(F, C, x, y, z);
}

// The small levels s .. L of the V-cycle in one block: down sweeps, the
// single-node solve, up sweeps, a block barrier between levels.
constexpr int kMaxLevels = 24;
constexpr int kTailNodes = 256;    // levels of at most this many nodes run in the tail
constexpr int kTailThreads = 1024;
struct MgTail {
  MgLevel lv[kMaxLevels];
  int s, L;
};
template <int DIM>
__global__ void __launch_bounds__(kTailThreads) k_mg_tail(MgTail T, const MgCtl *ctl) {
  if (ctl->done) return;
  for (int l = T.s; l < T.L; ++l) {
    const MgLevel &F = T.lv[l], &C = T.lv[l + 1];
    const int m = C.nx * C.ny * C.nz;
    for (int t = threadIdx.x; t < m; t += blockDim.x)
      down_node<DIM>(F, C, t % C.nx, (t / C.nx) % C.ny, t / (C.nx * C.ny));
    __syncthreads();
  }
  {
    const MgLevel &B = T.lv[T.L];
    const int m = B.nx * B.ny * B.nz;
    for (int t = threadIdx.x; t < m; t += blockDim.x) B.y[t] = B.g[t] * B.ia[t];
    __syncthreads();
  }
  for (int l = T.L - 1; l >= T.s; --l) {
    const MgLevel &F = T.lv[l], &C = T.lv[l + 1];
    const int m = F.nx * F.ny * F.nz;
    for (int t = threadIdx.x; t < m; t += blockDim.x)
      up_node<DIM>(F, C, t % F.nx, (t / F.nx) % F.ny, t / (F.nx * F.ny));
    __syncthreads();
  }
}

// ------------------------------------------------ level-0 passes (tiled)
// The three level-0 passes of an iteration share one shape: form a vector v
// from one to three arrays, apply the operator A to it, and combine.  Each
// node's u = sigma v is formed once and its neighbours' come from registers
// (z in 3D, y in 2D), a shuffle (x) and shared memory (y in 3D); gathering
// them per node, as these passes did before, formed every u five or seven
// times from up to four loads each and left them bound by load latency
// (256^3: 1.19 ms an iteration for the three, 0.23 ms now; 2048^2: 163 us, 83 us).
//   down (kDown): v = r;                g1 = sum over the box of w (r - omega (r - A' v)),
//   up   (kUp):   v = omega r + w y1,   z = v + omega (r - A v), <r, z>,
//   dir  (kDir):  v = z + beta p_old,   p = v, q = A v, <p, q>.
// Tiles are 128 columns (four per lane) x 8 rows per warp in 2D, x 16 rows x
// up to 16 planes per block in 3D: with cells of at least 16 nodes a tile
// lies in one cell row and layer, so a lane has one cell exponent, and the
// factors 2^(k_i - k_j) differ from 1 at the tile's rim only.
enum { kDown = 0, kUp = 1, kDir = 2 };

struct Mg0 {
  Grid g;
  CellGrid cg;
  int px;
  const float *s32;
  const int *kx;
  const float *w, *r, *z, *p_old;
  float *out, *out2;    // up: z; dir: p_new, q; down: the level-1 residual
  const float *y1;      // level-1 correction
  int nx1, ny1;         // level-1 extents
  const float *ia1;     // level-1 inverse diagonal (down: out2 = yp)
};

__device__ __forceinline__ float4 ld4g(const float *p) {
  return __ldg(reinterpret_cast<const float4 *>(p));
}
__device__ __forceinline__ float f4(const float4 &v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}

// One row of a tile at pitched offset o: sigma, v and the arrays that the
// output needs later (a: r in kDown and kUp, w: in kDown).  y1x/y1y: the parents'
// corrections of the lane's two column pairs.
struct Row0 {
  float4 s, v, a, w;
};
template <int MODE>
__device__ __forceinline__ Row0 row0_load(const Mg0 &A, int64_t o, bool in, float y1x, float y1y,
                                          float beta, bool first) {
  Row0 R;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  R.s = R.v = R.a = R.w = zero;
  if (!in) return R;
  R.s = ld4g(A.s32 + o);
  if (MODE == kDown) {
    R.a = R.v = ld4g(A.r + o);
    R.w = ld4g(A.w + o);
  } else if (MODE == kUp) {
    R.a = ld4g(A.r + o);
    const float4 w = ld4g(A.w + o);
    R.v = make_float4(fmaf(w.x, y1x, kOmega * R.a.x), fmaf(w.y, y1x, kOmega * R.a.y),
                      fmaf(w.z, y1y, kOmega * R.a.z), fmaf(w.w, y1y, kOmega * R.a.w));
  } else {
    R.v = ld4g(A.z + o);
    if (!first) {
      const float4 p = ld4g(A.p_old + o);
      R.v = make_float4(fmaf(beta, p.x, R.v.x), fmaf(beta, p.y, R.v.y), fmaf(beta, p.z, R.v.z),
                        fmaf(beta, p.w, R.v.w));
    }
  }
  return R;
}
// u = sigma v of one node beside the tile (column x0 - 1 or x0 + 128).
template <int MODE>
__device__ __forceinline__ float rim0(const Mg0 &A, int64_t o, bool in, float y1, float beta,
                                      bool first) {
  if (!in) return 0.f;
  const float s = __ldg(A.s32 + o);
  if (MODE == kDown) return s * __ldg(A.r + o);
  if (MODE == kUp) return s * fmaf(__ldg(A.w + o), y1, kOmega * __ldg(A.r + o));
  return s * (first ? __ldg(A.z + o) : fmaf(beta, __ldg(A.p_old + o), __ldg(A.z + o)));
}
__device__ __forceinline__ float4 mul4f(const float4 &a, const float4 &b) {
  return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
}

// Output of one row: off[i] = sigma_i sum of the neighbours' u.  Returns the
// lane's dot terms (times the weight wd) of kUp and kDir; kDown adds w t to
// the box sums c0, c1.
template <int MODE>
__device__ __forceinline__ float row0_out(const Mg0 &A, int64_t o, const Row0 &R,
                                          const float (&off)[4], float wd, float &c0, float &c1) {
  if (MODE == kDown) {
    float t[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float ri = f4(R.a, i);
      t[i] = f4(R.w, i) * (ri - kOmega * (ri - off[i]));
    }
    c0 += t[0] + t[1];
    c1 += t[2] + t[3];
    return 0.f;
  }
  float dot = 0.f, x[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float vi = f4(R.v, i), ri = f4(R.a, i);
    const bool live = f4(R.s, i) != 0.f;
    if (MODE == kUp) {
      x[i] = live ? fmaf(kOmega, ri - (vi - off[i]), vi) : 0.f;
      dot = fmaf(ri * x[i], wd, dot);
    } else {
      x[i] = live ? vi - off[i] : 0.f;
      dot = fmaf(vi * x[i], wd, dot);
    }
  }
  if (MODE == kUp) {
    *reinterpret_cast<float4 *>(A.out + o) = make_float4(x[0], x[1], x[2], x[3]);
  } else {
    *reinterpret_cast<float4 *>(A.out + o) = R.v;
    *reinterpret_cast<float4 *>(A.out2 + o) = make_float4(x[0], x[1], x[2], x[3]);
  }
  return dot;
}

// kDown: the level-1 residual and pre-smoothed correction of a lane's two
// boxes in level-1 row `row`.
__device__ __forceinline__ void coarse_out(const Mg0 &A, int64_t row, int X, float c0, float c1) {
  if (X < A.nx1) {
    A.out[row + X] = c0;
    A.out2[row + X] = kOmega * c0 * __ldg(A.ia1 + row + X);
  }
  if (X + 1 < A.nx1) {
    A.out[row + X + 1] = c1;
    A.out2[row + X + 1] = kOmega * c1 * __ldg(A.ia1 + row + X + 1);
  }
}

// What a lane keeps for all its rows: x-face weights, cell factors.
struct Lane0 {
  float hx[4], fL, fR, wd;
  int kc, kcol;
};
__device__ __forceinline__ Lane0 lane0(const Mg0 &A, int xl, int y, int z, int kmin) {
  Lane0 L;
  const int mask = A.cg.B - 1, lg = A.cg.lgB;
  const bool half = A.g.boundary == EIK_BOUNDARY_HALF_CELL;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    L.hx[i] = (half && (xl + i == 0 || xl + i == A.g.nx - 1)) ? 0.5f : 1.f;
  const int row = A.cg.cx * ((y >> lg) + A.cg.cy * (z >> lg));
  const int xc = min(xl, A.g.nx - 1);
  L.kcol = xc >> lg;
  L.kc = __ldg(A.kx + row + L.kcol);
  L.fL = (xc > 0 && (xc & mask) == 0) ? p2f(L.kc - __ldg(A.kx + row + L.kcol - 1)) : 1.f;
  L.fR = (xl + 4 < A.g.nx && ((xl + 4) & mask) == 0)
             ? p2f(L.kc - __ldg(A.kx + row + L.kcol + 1)) : 1.f;
  L.wd = p2f(2 * (kmin - L.kc));
  return L;
}

// End of a pass with a dot product: <r, z> (kUp) or <p, q> (kDir).
template <int MODE>
__device__ void dot0_end(float dot, MgCtl *ctl, double *part) {
  __shared__ double sh[32];
  __shared__ int flag;
  const double bs = block_sum((double)dot, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = bs;
  if (!last_block(&ctl->counter[MODE == kUp ? 0 : 1], &flag)) return;
  const double tot = sum_partials(part, gridDim.x, sh);
  if (threadIdx.x != 0) return;
  if (MODE == kUp) {
    ctl->beta = ctl->first ? 0.0 : tot / ctl->rho;
    ctl->rho = tot;
    ctl->counter[0] = 0u;
    if (!(tot > 0.0) || !isfinite(tot)) {   // z = M r lost positivity: stop here
      ctl->stalled = 1;
      ctl->done = 1;
    }
  } else {
    ctl->counter[1] = 0u;
    ctl->first = 0;
    if (!(tot > 0.0) || !isfinite(tot)) {
      ctl->alpha = 0.0;
      ctl->stalled = 1;
      ctl->done = 1;
    } else {
      ctl->alpha = ctl->rho / tot;
    }
  }
}

constexpr int kRows2 = 8;       // 2D: rows per warp tile
// 2D: every warp marches its tiles of 128 x kRows2 downwards.
template <int MODE>
__global__ void __launch_bounds__(kThreads)
k_mg0_2d(const Mg0 A, int tiles_x, int ntiles, MgCtl *ctl, double *part) {
  if (ctl->done) return;
  const int kmin = ctl->kmin, lane = threadIdx.x & 31;
  const float beta = (float)ctl->beta;
  const bool first = ctl->first != 0;
  const int mask = A.cg.B - 1, lg = A.cg.lgB;
  const bool half = A.g.boundary == EIK_BOUNDARY_HALF_CELL;
  const int nw = gridDim.x * (blockDim.x >> 5);
  float dot = 0.f;
  for (int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < ntiles; t += nw) {
    const int ty = t / tiles_x, x0 = (t - ty * tiles_x) * 128, y0 = ty * kRows2;
    const int xl = x0 + 4 * lane;
    const bool act = xl < A.px;
    const Lane0 L = lane0(A, xl, y0, 0, kmin);
    const int nrow = min(kRows2, A.g.ny - y0);
    // the node left (lane 0) or right (lane 31) of the tile
    const int xr = (lane == 0) ? x0 - 1 : x0 + 128;
    const bool rim = (lane == 0 && x0 > 0) || (lane == 31 && x0 + 128 < A.g.nx);
    const int X = xl >> 1;
    auto parents = [&](int y, float &a, float &b, float &c) {
      a = b = c = 0.f;
      if (MODE != kUp || y < 0 || y >= A.g.ny) return;
      const float *q = A.y1 + (int64_t)(y >> 1) * A.nx1;
      if (X < A.nx1) a = __ldg(q + X);
      if (X + 1 < A.nx1) b = __ldg(q + X + 1);
      if (rim) c = __ldg(q + (xr >> 1));
    };
    auto load = [&](int y, Row0 &R, float &ur) {
      float a, b, c;
      parents(y, a, b, c);
      const bool in = y >= 0 && y < A.g.ny;
      R = row0_load<MODE>(A, (int64_t)y * A.px + xl, in && act, a, b, beta, first);
      ur = rim0<MODE>(A, (int64_t)y * A.px + xr, in && rim, c, beta, first);
    };
    Row0 C, N;
    float urc, urn;
    load(y0 - 1, C, urc);
    float4 um = mul4f(C.s, C.v);
    load(y0, C, urc);
    float4 uc = mul4f(C.s, C.v);
    float c0 = 0.f, c1 = 0.f;
#pragma unroll 2
    for (int j = 0; j < nrow; ++j) {
      const int y = y0 + j;
      load(y + 1, N, urn);
      const float4 un = mul4f(N.s, N.v);
      float fU = 1.f, fD = 1.f;
      if ((y & mask) == 0 && y > 0)
        fU = p2f(L.kc - __ldg(A.kx + A.cg.cx * ((y >> lg) - 1) + L.kcol));
      if (((y + 1) & mask) == 0 && y + 1 < A.g.ny)
        fD = p2f(L.kc - __ldg(A.kx + A.cg.cx * ((y >> lg) + 1) + L.kcol));
      const float hy = (half && (y == 0 || y == A.g.ny - 1)) ? 0.5f : 1.f;
      float uL = __shfl_up_sync(0xffffffffu, uc.w, 1);
      float uR = __shfl_down_sync(0xffffffffu, uc.x, 1);
      if (lane == 0) uL = urc;
      if (lane == 31) uR = urc;
      const float xs[4] = {fmaf(uL, L.fL, uc.y), uc.x + uc.z, uc.y + uc.w, fmaf(uR, L.fR, uc.z)};
      float off[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        off[i] = f4(C.s, i) * fmaf(hy, xs[i], L.hx[i] * fmaf(f4(um, i), fU, f4(un, i) * fD));
      if (act) dot += row0_out<MODE>(A, (int64_t)y * A.px + xl, C, off, L.wd, c0, c1);
      if (MODE == kDown && ((j & 1) || j == nrow - 1)) {
        coarse_out(A, (int64_t)(y >> 1) * A.nx1, X, c0, c1);
        c0 = c1 = 0.f;
      }
      um = uc;
      uc = un;
      C = N;
      urc = urn;
    }
  }
  if (MODE != kDown) dot0_end<MODE>(dot, ctl, part);
}

constexpr int kRows3 = 16;                  // 3D: rows per block tile
constexpr int kThreads3 = 32 * (kRows3 / 2);
constexpr int kStages3 = 3;                 // planes of input in flight or in use
constexpr int kPlane3 = (kRows3 + 2) * 32;  // float4 of one array and plane
constexpr size_t kSmem3 = sizeof(float4) * kPlane3 * (3 * kStages3 + 3);

// 16 bytes of global memory into shared memory, zeros where !in.
__device__ __forceinline__ void copy16(float4 *dst, const float *src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(in ? 16 : 0)
               : "memory");
}

// 3D: a block marches its tile of 128 x kRows3 columns through zc planes
// (even).  Warp w owns rows y0 + 2 w and the next; the first and the last warp
// also supply u of the rows y0 - 1 and y0 + 16 (a ninth warp for them would cost
// every thread 32 registers).  Every thread copies its own four columns of the
// three input arrays into shared memory kStages3 - 1 planes ahead and reads
// them back itself, so the copies need no barrier and no registers (the loads
// of one plane ahead, in registers, left a block waiting for memory at every
// plane: 0.42 ms for the three passes on 256^3, 0.23 ms this way).  Three planes of u are shared (the one being written, the one in
// use, and the one that slower warps may still read), so a plane takes one
// barrier.
template <int MODE>
__global__ void __launch_bounds__(kThreads3, 2)
k_mg0_3d(const Mg0 A, int tiles_x, int tiles_y, int zc, int ntiles, MgCtl *ctl, double *part) {
  extern __shared__ float4 sm3[];
  float4 *us = sm3 + 3 * kStages3 * kPlane3;   // [3][kRows3 + 2][32]
  if (ctl->done) return;
  const int kmin = ctl->kmin, lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const float beta = (float)ctl->beta;
  const bool first = ctl->first != 0;
  const int mask = A.cg.B - 1, lg = A.cg.lgB;
  const bool half = A.g.boundary == EIK_BOUNDARY_HALF_CELL;
  const bool edge = wi == 0 || wi == kRows3 / 2 - 1;   // supplies a halo row
  // the input arrays: sigma, and r, w (down, up) or z, p_old (dir)
  const float *in1 = (MODE == kDir) ? A.z : A.r;
  const float *in2 = (MODE == kDir) ? A.p_old : A.w;
  // the warp's two rows in shared memory
  const int pr[2] = {(1 + 2 * wi) * 32 + lane, (2 + 2 * wi) * 32 + lane};
  const int ph = (wi == 0 ? 0 : kRows3 + 1) * 32 + lane;
  float dot = 0.f;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int tz = t / (tiles_x * tiles_y), rem = t - tz * tiles_x * tiles_y;
    const int ty = rem / tiles_x, x0 = (rem - ty * tiles_x) * 128;
    const int y0 = ty * kRows3, z0 = tz * zc;
    const int nz = min(zc, A.g.nz - z0);
    const int xl = x0 + 4 * lane;
    const bool act = xl < A.px;
    const int xr = (lane == 0) ? x0 - 1 : x0 + 128;
    const bool rim = ((lane == 0 && x0 > 0) || (lane == 31 && x0 + 128 < A.g.nx));
    const int X = xl >> 1;
    const int yr[2] = {y0 + 2 * wi, y0 + 2 * wi + 1};
    const bool yin[2] = {yr[0] < A.g.ny, yr[1] < A.g.ny};
    const int yh = (wi == 0) ? y0 - 1 : y0 + kRows3;
    const bool hin = edge && yh >= 0 && yh < A.g.ny;
    const Lane0 L = lane0(A, xl, min(yr[0], A.g.ny - 1), z0, kmin);
    const int layer = A.cg.cx * A.cg.cy;
    const int crow = L.kcol + A.cg.cx * (min(yr[0], A.g.ny - 1) >> lg) + layer * (z0 >> lg);
    float fU = 1.f, fD = 1.f;
    if (yr[0] > 0 && yr[0] < A.g.ny && (yr[0] & mask) == 0)
      fU = p2f(L.kc - __ldg(A.kx + crow - A.cg.cx));
    if (yr[1] + 1 < A.g.ny && ((yr[1] + 1) & mask) == 0)
      fD = p2f(L.kc - __ldg(A.kx + crow + A.cg.cx));
    float hy[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) hy[e] = (half && (yr[e] == 0 || yr[e] == A.g.ny - 1)) ? 0.5f : 1.f;
    // plane q of the march is z0 - 1 + q, q = 0 .. nz + 1
    auto issue = [&](int q) {
      const int z = z0 - 1 + q;
      float4 *dst = sm3 + (q % kStages3) * 3 * kPlane3;
      const bool inz = q < nz + 2 && z >= 0 && z < A.g.nz && act;
      auto row = [&](int y, bool iny, int at) {
        const bool in = inz && iny;
        const int64_t o = in ? (int64_t)A.px * (y + (int64_t)A.g.ny * z) + xl : 0;
        copy16(dst + at, A.s32 + o, in);
        copy16(dst + kPlane3 + at, in1 + o, in);
        copy16(dst + 2 * kPlane3 + at, in2 + o, in);
      };
#pragma unroll
      for (int e = 0; e < 2; ++e) row(yr[e], yin[e], pr[e]);
      if (edge) row(yh, hin, ph);
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // what a plane needs beside them: the rim node's values, the parents'
    // corrections (loaded a plane ahead)
    struct Side {
      float s[2], a[2], b[2], y0, y1, yc, yh0, yh1;   // (both rows have the same parents)
    };
    auto side = [&](int q) {
      Side S;
      const int z = z0 - 1 + q;
      const bool inz = q < nz + 2 && z >= 0 && z < A.g.nz;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        S.s[e] = S.a[e] = S.b[e] = 0.f;
        if (inz && yin[e] && rim) {
          const int64_t o = (int64_t)A.px * (yr[e] + (int64_t)A.g.ny * z) + xr;
          S.s[e] = __ldg(A.s32 + o);
          S.a[e] = __ldg(in1 + o);
          if (MODE != kDown) S.b[e] = __ldg(in2 + o);
        }
      }
      S.y0 = S.y1 = S.yc = S.yh0 = S.yh1 = 0.f;
      if (MODE == kUp && inz) {
        const float *y = A.y1 + (int64_t)A.nx1 * A.ny1 * (z >> 1);
        if (yin[0]) {
          const float *q1 = y + (int64_t)A.nx1 * (yr[0] >> 1);
          if (X < A.nx1) S.y0 = __ldg(q1 + X);
          if (X + 1 < A.nx1) S.y1 = __ldg(q1 + X + 1);
          if (rim) S.yc = __ldg(q1 + (xr >> 1));
        }
        if (hin) {
          const float *q1 = y + (int64_t)A.nx1 * (yh >> 1);
          if (X < A.nx1) S.yh0 = __ldg(q1 + X);
          if (X + 1 < A.nx1) S.yh1 = __ldg(q1 + X + 1);
        }
      }
      return S;
    };
    // sigma, v (and r, w) of the row at `at` of plane q from its inputs
    auto row_of = [&](int q, int at, float y0, float y1) {
      const float4 *src = sm3 + (q % kStages3) * 3 * kPlane3;
      Row0 R;
      R.s = src[at];
      const float4 a = src[kPlane3 + at], b = src[2 * kPlane3 + at];
      R.a = R.v = a;
      if (MODE == kDown)
        R.w = b;
      else if (MODE == kUp)
        R.v = make_float4(fmaf(b.x, y0, kOmega * a.x), fmaf(b.y, y0, kOmega * a.y),
                          fmaf(b.z, y1, kOmega * a.z), fmaf(b.w, y1, kOmega * a.w));
      else if (!first)
        R.v = make_float4(fmaf(beta, b.x, a.x), fmaf(beta, b.y, a.y), fmaf(beta, b.z, a.z),
                          fmaf(beta, b.w, a.w));
      return R;
    };
    // the two rows of plane q, u of their rim node, and (planes with a place in
    // us) u of the halo row
    auto form = [&](int q, const Side &S, Row0 (&R)[2], float (&ur)[2], float4 *u) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        R[e] = row_of(q, pr[e], S.y0, S.y1);
        if (MODE == kDown) ur[e] = S.s[e] * S.a[e];
        else if (MODE == kUp) ur[e] = S.s[e] * fmaf(S.b[e], S.yc, kOmega * S.a[e]);
        else ur[e] = S.s[e] * (first ? S.a[e] : fmaf(beta, S.b[e], S.a[e]));
      }
      if (edge && u) {
        const Row0 H = row_of(q, ph, S.yh0, S.yh1);
        u[ph] = mul4f(H.s, H.v);
      }
    };
    auto landed = [] {   // the oldest plane in flight
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages3 - 1) : "memory");
    };
    Row0 C[2], N[2];
    float urc[2], urn[2];
    float4 um[2], uc[2];
#pragma unroll
    for (int q = 0; q < kStages3; ++q) issue(q);
    Side S = side(0), Sn = side(1);
    landed();
    form(0, S, C, urc, nullptr);
    issue(kStages3);
#pragma unroll
    for (int e = 0; e < 2; ++e) um[e] = mul4f(C[e].s, C[e].v);
    S = Sn;
    Sn = side(2);
    landed();
    __syncthreads();   // the previous tile's planes of u are no longer read
    form(1, S, C, urc, us);
    issue(kStages3 + 1);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      uc[e] = mul4f(C[e].s, C[e].v);
      us[pr[e]] = uc[e];
    }
    float c0 = 0.f, c1 = 0.f;
    int cur = 0;
    for (int j = 0; j < nz; ++j) {
      const int z = z0 + j;
      S = Sn;
      Sn = side(j + 3);
      const int nxt = (cur == 2) ? 0 : cur + 1;
      landed();
      form(j + 2, S, N, urn, us + nxt * kPlane3);
      issue(j + 2 + kStages3);
      float4 un[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        un[e] = mul4f(N[e].s, N[e].v);
        us[nxt * kPlane3 + pr[e]] = un[e];
      }
      __syncthreads();
      {
        float fP = 1.f, fN = 1.f;
        if ((z & mask) == 0 && z > 0) fP = p2f(L.kc - __ldg(A.kx + crow - layer));
        if (((z + 1) & mask) == 0 && z + 1 < A.g.nz) fN = p2f(L.kc - __ldg(A.kx + crow + layer));
        const float hz = (half && (z == 0 || z == A.g.nz - 1)) ? 0.5f : 1.f;
        const float4 yu = us[cur * kPlane3 + pr[0] - 32], yd = us[cur * kPlane3 + pr[1] + 32];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float uL = __shfl_up_sync(0xffffffffu, uc[e].w, 1);
          float uR = __shfl_down_sync(0xffffffffu, uc[e].x, 1);
          if (lane == 0) uL = urc[e];
          if (lane == 31) uR = urc[e];
          const float4 up = (e == 0) ? yu : uc[0], dn = (e == 0) ? uc[1] : yd;
          const float gu = (e == 0) ? fU : 1.f, gd = (e == 0) ? 1.f : fD;
          const float xs[4] = {fmaf(uL, L.fL, uc[e].y), uc[e].x + uc[e].z, uc[e].y + uc[e].w,
                               fmaf(uR, L.fR, uc[e].z)};
          const float wx = hy[e] * hz;
          float off[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float ys = fmaf(f4(up, i), gu, f4(dn, i) * gd);
            const float zs = fmaf(f4(um[e], i), fP, f4(un[e], i) * fN);
            off[i] = f4(C[e].s, i) * fmaf(wx, xs[i], L.hx[i] * fmaf(hz, ys, hy[e] * zs));
          }
          if (act && yin[e]) {
            const int64_t o = (int64_t)A.px * (yr[e] + (int64_t)A.g.ny * z) + xl;
            dot += row0_out<MODE>(A, o, C[e], off, L.wd, c0, c1);
          }
        }
        if (MODE == kDown && ((j & 1) || j == nz - 1)) {
          if (yin[0])
            coarse_out(A, (int64_t)A.nx1 * ((yr[0] >> 1) + (int64_t)A.ny1 * (z >> 1)), X, c0, c1);
          c0 = c1 = 0.f;
        }
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        um[e] = uc[e];
        uc[e] = un[e];
        C[e] = N[e];
        urc[e] = urn[e];
      }
      cur = nxt;
    }
    // (copies past the last plane are zero fills of unused stages; they have
    // to land before the next tile issues into them)
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  if (MODE != kDown) dot0_end<MODE>(dot, ctl, part);
}

// Largest of the threads' values, in all threads of warp 0.
__device__ __forceinline__ unsigned block_max_bits(unsigned v, unsigned *sh) {
  v = __reduce_max_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0u;
    v = __reduce_max_sync(0xffffffffu, v);
  }
  return v;
}

// d += alpha p, r -= alpha q, and the stopping tests; n4 float4 groups of the
// pitched arrays (their padding columns are zero and stay so).
__global__ void __launch_bounds__(kThreads)
k_mg_step(int64_t n4, const float4 *__restrict__ p, const float4 *__restrict__ q,
          const float4 *__restrict__ xref, float4 *__restrict__ d, float4 *__restrict__ r,
          MgCtl *ctl, double *part) {
  __shared__ unsigned sh[32];
  __shared__ int flag;
  if (ctl->done) return;
  const float alpha = (float)ctl->alpha;
  const int mode = ctl->mode;
  const float theta = ctl->theta;
  float rmax = 0.f, viol = 0.f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float4 pi = p[i], qi = q[i];
    float4 di = d[i], ri = r[i];
    di = make_float4(fmaf(alpha, pi.x, di.x), fmaf(alpha, pi.y, di.y), fmaf(alpha, pi.z, di.z),
                     fmaf(alpha, pi.w, di.w));
    ri = make_float4(fmaf(-alpha, qi.x, ri.x), fmaf(-alpha, qi.y, ri.y), fmaf(-alpha, qi.z, ri.z),
                     fmaf(-alpha, qi.w, ri.w));
    d[i] = di;
    r[i] = ri;
    rmax = fmaxf(rmax, fmaxf(fmaxf(fabsf(ri.x), fabsf(ri.y)), fmaxf(fabsf(ri.z), fabsf(ri.w))));
    if (mode == 1) {
      const float4 xi = __ldg(xref + i);
      if (fabsf(ri.x) > theta * fabsf(xi.x + di.x) || fabsf(ri.y) > theta * fabsf(xi.y + di.y) ||
          fabsf(ri.z) > theta * fabsf(xi.z + di.z) || fabsf(ri.w) > theta * fabsf(xi.w + di.w))
        viol = 1.f;
    }
  }
  // (maxima of non-negative floats are maxima of their bits: the integer
  // reductions keep this off the FP64 pipe)
  const unsigned b1 = block_max_bits(__float_as_uint(rmax), sh);
  const unsigned b2 = (unsigned)__syncthreads_or(viol != 0.f);
  unsigned *ip = reinterpret_cast<unsigned *>(part);
  if (threadIdx.x == 0) {
    ip[2 * blockIdx.x] = b1;
    ip[2 * blockIdx.x + 1] = b2;
  }
  if (!last_block(&ctl->counter[2], &flag)) return;
  unsigned m1 = 0, m2 = 0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
    const uint2 v = __ldcg(reinterpret_cast<const uint2 *>(ip) + b);
    m1 = max(m1, v.x);
    m2 |= v.y;
  }
  const float rm = __uint_as_float(block_max_bits(m1, sh));
  const int vi = __syncthreads_or(m2 != 0u);
  if (threadIdx.x == 0) {
    ctl->counter[2] = 0u;
    ctl->iter += 1;
    const bool conv = (mode == 0) ? (rm <= ctl->thresh) : (vi == 0);
    if (rm < ctl->r_best) {
      ctl->r_best = rm;
      ctl->best_iter = ctl->iter;
    }
    if (!isfinite(rm)) {
      ctl->status = EIK_ERR_BREAKDOWN;
      ctl->done = 1;
    } else if (conv) {
      ctl->done = 1;
    } else if (rm > ctl->r_limit || ctl->iter - ctl->best_iter >= ctl->max_idle) {
      ctl->stalled = 2;
      ctl->done = 1;
    } else if (ctl->iter >= ctl->max_iter) {
      ctl->done = 1;
    }
  }
}

}  // namespace

// ====================================================================== host
struct MgState {
  Grid g;
  CellGrid cg;
  int px = 0, cap = 0;
  std::vector<MgLevel> lv;   // lv[0]: level-0 sizes only
  float *w = nullptr, *z = nullptr, *p[2] = {nullptr, nullptr}, *q = nullptr;
  MgCtl *ctl = nullptr, *h_ctl = nullptr;
  double *part = nullptr;
  cudaGraphExec_t graph = nullptr;
  MgFine bound{};            // arrays the graph was captured with
  int64_t launches = 0;
  bool profile = false;
  cudaEvent_t ev[2] = {nullptr, nullptr};
  int64_t timed_iters = 0;
  double ms = 0.0;
};

const char *mg_last_error() { return g_msg.c_str(); }
int mg_levels(const MgState *mg) { return mg ? (int)mg->lv.size() : 0; }
int64_t mg_launches(const MgState *mg) { return mg ? mg->launches : 0; }
void mg_set_profiling(MgState *mg, bool on) {
  if (mg) mg->profile = on;
}
void mg_time(const MgState *mg, int64_t *iters, double *ms) {
  *iters = mg ? mg->timed_iters : 0;
  *ms = mg ? mg->ms : 0.0;
}
void mg_reset(MgState *mg) {
  if (!mg) return;
  mg->launches = 0;
  mg->timed_iters = 0;
  mg->ms = 0.0;
}

#define GCK(call)                                                       \
  do {                                                                  \
    cudaError_t e_ = (call);                                            \
    if (e_ != cudaSuccess) {                                            \
      g_msg = std::string(#call) + ": " + cudaGetErrorString(e_);       \
      return EIK_ERR_CUDA;                                              \
    }                                                                   \
  } while (0)

void mg_destroy(MgState *mg) {
  if (!mg) return;
  if (mg->graph) cudaGraphExecDestroy(mg->graph);
  for (auto &e : mg->ev)
    if (e) cudaEventDestroy(e);
  for (size_t l = 1; l < mg->lv.size(); ++l) {
    MgLevel &L = mg->lv[l];
    void *arr[] = {L.a, L.ia, L.c, L.k, L.g, L.yp, L.y};
    for (void *p : arr)
      if (p) cudaFree(p);
  }
  void *arr[] = {mg->w, mg->z, mg->p[0], mg->p[1], mg->q, mg->ctl, mg->part};
  for (void *p : arr)
    if (p) cudaFree(p);
  if (mg->h_ctl) cudaFreeHost(mg->h_ctl);
  delete mg;
}

eik_status mg_create(MgState **out, const Grid &g, const CellGrid &cg, int px, int num_sms,
                     cudaStream_t s) {
  *out = nullptr;
  MgState *mg = new MgState();
  mg->g = g;
  mg->cg = cg;
  mg->px = px;
  mg->cap = num_sms * 8;
  MgLevel L0;
  L0.nx = g.nx;
  L0.ny = g.ny;
  L0.nz = g.nz;
  mg->lv.push_back(L0);
  bool ok = true;
  int nx = g.nx, ny = g.ny, nz = g.nz;
  while (ok && (nx > 1 || ny > 1 || nz > 1) && (int)mg->lv.size() < kMaxLevels) {
    nx = (nx + 1) / 2;
    ny = (ny + 1) / 2;
    nz = (nz + 1) / 2;
    MgLevel L;
    L.nx = nx;
    L.ny = ny;
    L.nz = nz;
    const size_t m = (size_t)nx * ny * nz;
    ok = cudaMalloc(&L.a, 4 * m) == cudaSuccess && cudaMalloc(&L.ia, 4 * m) == cudaSuccess &&
         cudaMalloc(&L.c, 4 * kDirs * m) == cudaSuccess &&
         cudaMalloc(&L.k, 4 * m) == cudaSuccess && cudaMalloc(&L.g, 4 * m) == cudaSuccess &&
         cudaMalloc(&L.yp, 4 * m) == cudaSuccess && cudaMalloc(&L.y, 4 * m) == cudaSuccess;
    mg->lv.push_back(L);
  }
  const size_t np = (size_t)g.ny * g.nz * px;
  ok = ok && cudaMalloc(&mg->w, 4 * np) == cudaSuccess && cudaMalloc(&mg->z, 4 * np) == cudaSuccess &&
       cudaMalloc(&mg->p[0], 4 * np) == cudaSuccess && cudaMalloc(&mg->p[1], 4 * np) == cudaSuccess &&
       cudaMalloc(&mg->q, 4 * np) == cudaSuccess &&
       cudaMalloc(&mg->ctl, sizeof(MgCtl)) == cudaSuccess &&
       cudaMalloc(&mg->part, 2 * sizeof(double) * mg->cap) == cudaSuccess &&
       cudaMallocHost(&mg->h_ctl, sizeof(MgCtl)) == cudaSuccess;
  if (ok) {
    // padding columns of the pitched arrays are read by no kernel; keep them finite
    float *arr[] = {mg->w, mg->z, mg->p[0], mg->p[1], mg->q};
    for (float *a : arr) ok = ok && cudaMemsetAsync(a, 0, 4 * np, s) == cudaSuccess;
    ok = ok && cudaMemsetAsync(mg->ctl, 0, sizeof(MgCtl), s) == cudaSuccess &&
         cudaStreamSynchronize(s) == cudaSuccess;
  }
  if (!ok) {
    cudaGetLastError();
    mg_destroy(mg);
    g_msg = "multigrid: device allocation failed";
    return EIK_ERR_OOM;
  }
  if (g.ndim == 3 &&
      (cudaFuncSetAttribute(k_mg0_3d<kDown>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                            (int)kSmem3) != cudaSuccess ||
       cudaFuncSetAttribute(k_mg0_3d<kUp>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                            (int)kSmem3) != cudaSuccess ||
       cudaFuncSetAttribute(k_mg0_3d<kDir>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                            (int)kSmem3) != cudaSuccess)) {
    cudaGetLastError();
    mg_destroy(mg);
    g_msg = "multigrid: cannot reserve shared memory";
    return EIK_ERR_CUDA;
  }
  *out = mg;
  return EIK_OK;
}

// Row-strided launch shape of a level: blocks of kThreads threads, as many
// columns as the row has up to kThreads (a power of two), rows beside each
// other; at most cap blocks.
struct Shape {
  dim3 grid, block;
};
static Shape shape_of(const MgState *mg, const MgLevel &L) {
  int bx = 1;
  while (bx < L.nx && bx < kThreads) bx *= 2;
  const int by = kThreads / bx;
  const int gx = std::max(1, std::min((L.nx + bx - 1) / bx, mg->cap));
  const int64_t rows = ((int64_t)L.ny * L.nz + by - 1) / by;
  const int gy = (int)std::max<int64_t>(1, std::min<int64_t>(rows, mg->cap / gx));
  return Shape{dim3((unsigned)gx, (unsigned)gy, 1), dim3((unsigned)bx, (unsigned)by, 1)};
}

eik_status mg_setup(MgState *mg, const MgFine &f, int kmin, cudaStream_t s) {
  const Grid &g = mg->g;
  const Shape s0 = shape_of(mg, mg->lv[0]);
  k_mg_weights<<<s0.grid, s0.block, 0, s>>>(g, mg->cg, mg->px, f.s32, f.kx, f.St, mg->w);
  MgLevel &L1 = mg->lv[1];
  const Shape s1 = shape_of(mg, L1);
  k_mg_coarsen0<<<s1.grid, s1.block, 0, s>>>(g, mg->cg, mg->px, f.s32, f.kx, mg->w, L1);
  mg->launches += 2;
  for (size_t l = 1; l + 1 < mg->lv.size(); ++l) {
    MgLevel &C = mg->lv[l + 1];
    const Shape sh = shape_of(mg, C);
    k_mg_coarsen<<<sh.grid, sh.block, 0, s>>>(mg->lv[l], C);
    mg->launches++;
  }
  GCK(cudaGetLastError());
  mg->h_ctl->kmin = kmin;
  return EIK_OK;
}

// One PCG iteration (direction buffers: read p[set], write p[1 - set]).
// First level handled by the tail kernel: the first of at most kTailNodes
// nodes, level 1 at the earliest.
static int tail_start(const MgState *mg) {
  int l = 1;
  while (l < (int)mg->lv.size() - 1 &&
         (int64_t)mg->lv[l].nx * mg->lv[l].ny * mg->lv[l].nz > kTailNodes)
    ++l;
  return l;
}

// One level-0 pass.
template <int MODE>
static void launch0(MgState *mg, const MgFine &f, int set, cudaStream_t s) {
  const Grid &g = mg->g;
  Mg0 a{};
  a.g = g;
  a.cg = mg->cg;
  a.px = mg->px;
  a.s32 = f.s32;
  a.kx = f.kx;
  a.w = mg->w;
  a.r = f.r;
  a.z = mg->z;
  a.p_old = mg->p[set];
  a.out = (MODE == kDown) ? mg->lv[1].g : (MODE == kUp) ? mg->z : mg->p[1 - set];
  a.out2 = (MODE == kDown) ? mg->lv[1].yp : mg->q;
  a.ia1 = mg->lv[1].ia;
  a.y1 = mg->lv[1].y;
  a.nx1 = mg->lv[1].nx;
  a.ny1 = mg->lv[1].ny;
  const int tx = (g.nx + 127) / 128;
  if (g.ndim == 2) {
    const int64_t nt = (int64_t)tx * ((g.ny + kRows2 - 1) / kRows2);
    const int64_t nb = (nt + kThreads / 32 - 1) / (kThreads / 32);
    k_mg0_2d<MODE><<<(int)std::min<int64_t>(nb, mg->cap), kThreads, 0, s>>>(a, tx, (int)nt,
                                                                            mg->ctl, mg->part);
  } else {
    // planes per tile: as many as leave two blocks per SM (each tile reads
    // two planes beside its own); divisors of the cell edge
    const int ty = (g.ny + kRows3 - 1) / kRows3;
    int zc = 16;
    while (zc > 2 && (int64_t)tx * ty * ((g.nz + zc - 1) / zc) < mg->cap / 4) zc /= 2;
    const int64_t nt = (int64_t)tx * ty * ((g.nz + zc - 1) / zc);
    k_mg0_3d<MODE><<<(int)std::min<int64_t>(nt, mg->cap), kThreads3, kSmem3, s>>>(
        a, tx, ty, zc, (int)nt, mg->ctl, mg->part);
  }
}

template <int DIM>
static void launch_iter_d(MgState *mg, const MgFine &f, int set, cudaStream_t s) {
  const Grid &g = mg->g;
  const int L = (int)mg->lv.size() - 1;   // coarsest level index
  launch0<kDown>(mg, f, set, s);
  // levels 1 .. ts - 1 one launch each way; ts .. L in the single-block tail
  const int ts = tail_start(mg);
  for (int l = 1; l < ts; ++l) {
    const Shape sh = shape_of(mg, mg->lv[l + 1]);
    k_mg_down<DIM><<<sh.grid, sh.block, 0, s>>>(mg->lv[l], mg->lv[l + 1], mg->ctl);
  }
  MgTail T{};
  for (int l = ts; l <= L; ++l) T.lv[l] = mg->lv[l];
  T.s = ts;
  T.L = L;
  k_mg_tail<DIM><<<1, kTailThreads, 0, s>>>(T, mg->ctl);
  for (int l = ts - 1; l >= 1; --l) {
    const Shape sh = shape_of(mg, mg->lv[l]);
    k_mg_up<DIM><<<sh.grid, sh.block, 0, s>>>(mg->lv[l], mg->lv[l + 1], mg->ctl);
  }
  launch0<kUp>(mg, f, set, s);
  launch0<kDir>(mg, f, set, s);
  const int64_t n4 = (int64_t)(mg->px / 4) * g.ny * g.nz;
  const int nb = (int)std::max<int64_t>(1, std::min<int64_t>((n4 + kThreads - 1) / kThreads, mg->cap));
  auto v4 = [](const float *p) { return reinterpret_cast<const float4 *>(p); };
  k_mg_step<<<nb, kThreads, 0, s>>>(n4, v4(mg->p[1 - set]), v4(mg->q), v4(f.xref),
                                    reinterpret_cast<float4 *>(f.d),
                                    reinterpret_cast<float4 *>(f.r), mg->ctl, mg->part);
}

// One PCG iteration with the kernels specialised to the grid's dimension.
static void launch_iter(MgState *mg, const MgFine &f, int set, cudaStream_t s) {
  if (mg->g.ndim == 3)
    launch_iter_d<3>(mg, f, set, s);
  else
    launch_iter_d<2>(mg, f, set, s);
}

static int launches_per_iter(const MgState *mg) { return 2 * (tail_start(mg) - 1) + 5; }

eik_status mg_inner(MgState *mg, const MgFine &f, MixCtl *h_st, int *again, cudaStream_t s) {
  if (mg->graph && (f.r != mg->bound.r || f.d != mg->bound.d || f.xref != mg->bound.xref ||
                    f.s32 != mg->bound.s32 || f.kx != mg->bound.kx)) {
    cudaGraphExecDestroy(mg->graph);
    mg->graph = nullptr;
  }
  if (!mg->graph) {
    cudaGraph_t graph;
    GCK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    for (int it = 0; it < kGraphIters; ++it) launch_iter(mg, f, it & 1, s);
    GCK(cudaStreamEndCapture(s, &graph));
    GCK(cudaGraphInstantiate(&mg->graph, graph, 0));
    GCK(cudaGraphDestroy(graph));
    mg->bound = f;
  }
  MgCtl c{};
  c.kmin = mg->h_ctl->kmin;
  const bool guard = *again == kMgFirst;
  c.max_iter = std::max(1, std::min(h_st->max_iter, *again > 0 ? *again : kMaxInnerIters));
  c.mode = h_st->mode;
  c.thresh = h_st->thresh;
  c.theta = h_st->theta;
  c.r_best = (float)h_st->r_inf;
  c.r_limit = guard ? kMaxGrowth * c.r_best : INFINITY;
  c.max_idle = guard ? kMaxIdle : INT_MAX;
  c.first = 1;
  *mg->h_ctl = c;
  GCK(cudaMemcpyAsync(mg->ctl, mg->h_ctl, sizeof(MgCtl), cudaMemcpyHostToDevice, s));
  if (mg->profile && !mg->ev[0])
    for (auto &e : mg->ev) GCK(cudaEventCreate(&e));
  int before = 0;
  for (;;) {
    if (mg->profile) GCK(cudaEventRecord(mg->ev[0], s));
    GCK(cudaGraphLaunch(mg->graph, s));
    if (mg->profile) GCK(cudaEventRecord(mg->ev[1], s));
    GCK(cudaMemcpyAsync(mg->h_ctl, mg->ctl, sizeof(MgCtl), cudaMemcpyDeviceToHost, s));
    GCK(cudaStreamSynchronize(s));
    // every kernel of the graph launches (those past the end return at once)
    mg->launches += (int64_t)kGraphIters * launches_per_iter(mg);
    const int done_iters = mg->h_ctl->iter - before;
    before = mg->h_ctl->iter;
    if (mg->profile && done_iters == kGraphIters) {
      float t = 0.f;
      GCK(cudaEventElapsedTime(&t, mg->ev[0], mg->ev[1]));
      mg->ms += t;
      mg->timed_iters += done_iters;
    }
    if (mg->h_ctl->done) break;
  }
  h_st->iter = mg->h_ctl->iter;
  h_st->status = mg->h_ctl->status;
  h_st->stalled = mg->h_ctl->stalled;
  h_st->done = 1;
  *again = kMgFirst;
  if (h_st->stalled == 2)
    *again = (mg->h_ctl->r_best <= 0.5f * c.r_best) ? mg->h_ctl->best_iter : kMgNoCutoff;
  return EIK_OK;
}

}  // namespace eik
