// Two-pass FP32 inner CG of the 3D mixed solve (operator, units and frames as
// in eik_cg32.h), the two-reduction Jacobi-PCG:
//   dir:  p = r + beta p, q = A p, <p, q>              20 B per node
//   step: d += alpha p, r -= alpha q, <r, r>, <r, q>   24 B per node
//
// What bounds it: HBM.  The one-pass kernel (k_cg3d) moves 28 B per node, but
// forms p, A p, r and A r with two-node halos, a barrier and 2.5 us per plane
// of its 16-row blocks: 228 us on 256^3, a third of the copy bandwidth.  Here
// the stencil is applied once, with a one-node halo, and the other pass is a
// plain stream.  The step pass walks the rows backwards, so that it starts on
// the p, q and r that dir has just left in L2, and dir starts on the r that step
// has.
// Measured per iteration (one-pass kernel, this one): 256^3 228 us, 145 us (5.1
// TB/s of the 44 B per node, 0.75 of the copy bandwidth); 192^3 140 us, 80 us;
// 96^3 47 us, 36 us; 24^3 45 us, 25 us (two launches, their tails and the
// latency of a tile's planes).  It was the faster one at each of twelve grids
// from 24^3 to 256^3, thin and ragged ones among them, so it serves every 3D
// grid; k_cg3d remains for explicitly chosen variants and where the device
// refuses this kernel's memory.
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <climits>

#include "eik_pair3d.h"

namespace eik {

// Recurrence between the two passes: <r,r> = gm 2^gs with gm in [0.5, 1), frame
// F that r and p are in once multiplied by `scale` (dir does so for p, step for
// r), <p, A p> and 2 beta <p, A p_old> of the next direction (units of 2^gs).
struct PairCtl {
  double gm, beta, ps, conj2;
  int gs, F, fd, check;
  float alpha, alphaF, scale, thetaF;
  unsigned pexp;          // exponent bits of the largest |p|
  unsigned counter[2];
};

namespace {

constexpr int kRows = 16;                  // rows per block tile
constexpr int kDirThreads = 32 * (kRows / 2);
constexpr int kStages = 3;                 // planes of input in flight or in use
constexpr int kPlane = (kRows + 2) * 32;   // float4 of one array and plane
constexpr size_t kDirSmem = sizeof(float4) * kPlane * (3 * kStages + 3);
constexpr int kDirPerSm = 2;
constexpr int kStepPerSm = 6;
constexpr int kRescale = 8;                // r and p move to a new frame past 2^+-8

struct PairArgs {
  Grid g;
  CellGrid cg;
  int px;
  const int *kx;
  const float *s32, *xref;
  const float *p_old;
  float *r, *p, *q, *d;
  MixCtl *st;
  PairCtl *c;
  double *part;
};

__device__ __forceinline__ float p2f(int n) {
  n = min(max(n, -126), 127);
  return __int_as_float((n + 127) << 23);
}
__device__ __forceinline__ float at4(const float4 &v, int i) {
  return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
}
__device__ __forceinline__ float4 mul4(const float4 &a, const float4 &b) {
  return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
}
__device__ __forceinline__ float max4(float m, const float4 &v) {
  return fmaxf(fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
}
// 16 bytes of global memory into shared memory, zeros where !in.
__device__ __forceinline__ void copy16(float4 *dst, const float *src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(in ? 16 : 0)
               : "memory");
}
// Largest of the threads' values (bits of non-negative floats), in warp 0.
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
__device__ __forceinline__ void finish(MixCtl *st, int status, bool stalled) {
  if (stalled) st->stalled = 1;
  st->status = status;
  st->done = 1;
}

// The block of a level-0 pass of the multigrid cycle (k_mg0_3d): tiles of 128
// x kRows columns march through zc planes, warp w owns rows y0 + 2 w and the
// next, the first and the last warp also supply u of the rows beside the tile,
// and every thread copies its own columns to shared memory kStages - 1 planes
// ahead.  Cells have at least 16 nodes an edge, so a tile lies in one cell row;
// it may cross layers, where the lane's factors are looked up again.
__global__ void __launch_bounds__(kDirThreads, kDirPerSm)
k_pair_dir(const PairArgs A, int tiles_x, int tiles_y, int zc, int ntiles) {
  extern __shared__ float4 sm3[];
  __shared__ double shd[32];
  __shared__ unsigned shu[32];
  __shared__ int flag;
  MixCtl *st = A.st;
  PairCtl *c = A.c;
  if (st->done) return;
  float4 *us = sm3 + 3 * kStages * kPlane;   // u of three planes [3][kRows + 2][32]
  const bool start = st->iter == 0;
  const int dF0 = st->dF, F0 = st->F + dF0;
  const float scale = start ? p2f(-dF0) : c->scale;
  const float beta = start ? 0.f : (float)c->beta * scale;
  const int fd = start ? st->gam_s - 2 * F0 : c->fd;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int mask = A.cg.B - 1, lg = A.cg.lgB, layer = A.cg.cx * A.cg.cy;
  const bool half = A.g.boundary == EIK_BOUNDARY_HALF_CELL;
  const int nx = A.g.nx, ny = A.g.ny;
  const bool edge = wi == 0 || wi == kRows / 2 - 1;   // supplies a halo row
  const int pr[2] = {(1 + 2 * wi) * 32 + lane, (2 + 2 * wi) * 32 + lane};
  const int ph = (wi == 0 ? 0 : kRows + 1) * 32 + lane;
  float dot = 0.f, pmax = 0.f;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int tz = t / (tiles_x * tiles_y), rem = t - tz * tiles_x * tiles_y;
    const int ty = rem / tiles_x, x0 = (rem - ty * tiles_x) * 128;
    const int y0 = ty * kRows, z0 = tz * zc;
    const int nz = min(zc, A.g.nz - z0);
    const int xl = x0 + 4 * lane;
    const bool act = xl < A.px;
    // the node left (lane 0) or right (lane 31) of the tile
    const int xr = (lane == 0) ? x0 - 1 : x0 + 128;
    const bool rim = (lane == 0 && x0 > 0) || (lane == 31 && x0 + 128 < nx);
    const int yr[2] = {y0 + 2 * wi, y0 + 2 * wi + 1};
    const bool yin[2] = {yr[0] < ny, yr[1] < ny};
    const int yh = (wi == 0) ? y0 - 1 : y0 + kRows;
    const bool hin = edge && yh >= 0 && yh < ny;
    float hx[4], hy[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) hx[i] = (half && (xl + i == 0 || xl + i == nx - 1)) ? 0.5f : 1.f;
#pragma unroll
    for (int e = 0; e < 2; ++e) hy[e] = (half && (yr[e] == 0 || yr[e] == ny - 1)) ? 0.5f : 1.f;
    // factors of the lane's cell in the layer of plane z
    const int kcol = min(xl, nx - 1) >> lg;
    const int krow = A.cg.cx * (min(yr[0], ny - 1) >> lg);
    int kc = 0, crow = 0;
    float fL = 1.f, fR = 1.f, fU = 1.f, fD = 1.f, W = 0.f;
    auto cell = [&](int z) {
      crow = kcol + krow + layer * (z >> lg);
      kc = __ldg(A.kx + crow);
      fL = (xl > 0 && xl < nx && (xl & mask) == 0) ? p2f(kc - __ldg(A.kx + crow - 1)) : 1.f;
      fR = (xl + 4 < nx && ((xl + 4) & mask) == 0) ? p2f(kc - __ldg(A.kx + crow + 1)) : 1.f;
      fU = (yr[0] > 0 && yin[0] && (yr[0] & mask) == 0)
               ? p2f(kc - __ldg(A.kx + crow - A.cg.cx)) : 1.f;
      fD = (yr[1] + 1 < ny && ((yr[1] + 1) & mask) == 0)
               ? p2f(kc - __ldg(A.kx + crow + A.cg.cx)) : 1.f;
      W = p2f(-2 * kc - fd);
    };
    cell(z0);
    // plane k of the march is z0 - 1 + k, k = 0 .. nz + 1
    auto issue = [&](int k) {
      const int z = z0 - 1 + k;
      float4 *dst = sm3 + (k % kStages) * 3 * kPlane;
      const bool inz = k < nz + 2 && z >= 0 && z < A.g.nz && act;
      auto row = [&](int y, bool iny, int at) {
        const bool in = inz && iny;
        const int64_t o = in ? (int64_t)A.px * (y + (int64_t)ny * z) + xl : 0;
        copy16(dst + at, A.s32 + o, in);
        copy16(dst + kPlane + at, A.r + o, in);
        copy16(dst + 2 * kPlane + at, A.p_old + o, in);
      };
#pragma unroll
      for (int e = 0; e < 2; ++e) row(yr[e], yin[e], pr[e]);
      if (edge) row(yh, hin, ph);
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // u of the rim nodes of the warp's rows in plane k (loaded a plane ahead)
    struct Side {
      float s[2], r[2], p[2];
    };
    auto side = [&](int k) {
      Side S;
      const int z = z0 - 1 + k;
      const bool inz = k < nz + 2 && z >= 0 && z < A.g.nz;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        S.s[e] = S.r[e] = S.p[e] = 0.f;
        if (inz && yin[e] && rim) {
          const int64_t o = (int64_t)A.px * (yr[e] + (int64_t)ny * z) + xr;
          S.s[e] = __ldg(A.s32 + o);
          S.r[e] = __ldg(A.r + o);
          S.p[e] = __ldg(A.p_old + o);
        }
      }
      return S;
    };
    // sigma and p of the row at `at` of plane k
    auto row_of = [&](int k, int at, float4 &s, float4 &p) {
      const float4 *src = sm3 + (k % kStages) * 3 * kPlane;
      s = src[at];
      const float4 a = src[kPlane + at], b = src[2 * kPlane + at];
      p = make_float4(fmaf(beta, b.x, scale * a.x), fmaf(beta, b.y, scale * a.y),
                      fmaf(beta, b.z, scale * a.z), fmaf(beta, b.w, scale * a.w));
    };
    auto form = [&](int k, const Side &S, float4 (&s)[2], float4 (&p)[2], float (&ur)[2],
                    float4 *u) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        row_of(k, pr[e], s[e], p[e]);
        ur[e] = S.s[e] * fmaf(beta, S.p[e], scale * S.r[e]);
      }
      if (edge && u) {
        float4 hs, hp;
        row_of(k, ph, hs, hp);
        u[ph] = mul4(hs, hp);
      }
    };
    auto landed = [] {   // the oldest plane in flight
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1) : "memory");
    };
    float4 sc[2], pc[2], sn[2], pn[2], um[2], uc[2];
    float urc[2], urn[2];
#pragma unroll
    for (int k = 0; k < kStages; ++k) issue(k);
    Side S = side(0), Sn = side(1);
    landed();
    form(0, S, sc, pc, urc, nullptr);
    issue(kStages);
#pragma unroll
    for (int e = 0; e < 2; ++e) um[e] = mul4(sc[e], pc[e]);
    S = Sn;
    Sn = side(2);
    landed();
    __syncthreads();   // the previous tile's planes of u are no longer read
    form(1, S, sc, pc, urc, us);
    issue(kStages + 1);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      uc[e] = mul4(sc[e], pc[e]);
      us[pr[e]] = uc[e];
    }
    int cur = 0;
    for (int j = 0; j < nz; ++j) {
      const int z = z0 + j;
      S = Sn;
      Sn = side(j + 3);
      const int nxt = (cur == 2) ? 0 : cur + 1;
      landed();
      form(j + 2, S, sn, pn, urn, us + nxt * kPlane);
      issue(j + 2 + kStages);
      float4 un[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        un[e] = mul4(sn[e], pn[e]);
        us[nxt * kPlane + pr[e]] = un[e];
      }
      __syncthreads();
      if (j > 0 && (z & mask) == 0) cell(z);
      float fP = 1.f, fN = 1.f;
      if ((z & mask) == 0 && z > 0) fP = p2f(kc - __ldg(A.kx + crow - layer));
      if (((z + 1) & mask) == 0 && z + 1 < A.g.nz) fN = p2f(kc - __ldg(A.kx + crow + layer));
      const float hz = (half && (z == 0 || z == A.g.nz - 1)) ? 0.5f : 1.f;
      const float4 yu = us[cur * kPlane + pr[0] - 32], yd = us[cur * kPlane + pr[1] + 32];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float uL = __shfl_up_sync(0xffffffffu, uc[e].w, 1);
        float uR = __shfl_down_sync(0xffffffffu, uc[e].x, 1);
        if (lane == 0) uL = urc[e];
        if (lane == 31) uR = urc[e];
        const float4 up = (e == 0) ? yu : uc[0], dn = (e == 0) ? uc[1] : yd;
        const float gu = (e == 0) ? fU : 1.f, gd = (e == 0) ? 1.f : fD;
        const float xs[4] = {fmaf(uL, fL, uc[e].y), uc[e].x + uc[e].z, uc[e].y + uc[e].w,
                             fmaf(uR, fR, uc[e].z)};
        const float wx = hy[e] * hz;
        float x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float ys = fmaf(at4(up, i), gu, at4(dn, i) * gd);
          const float zs = fmaf(at4(um[e], i), fP, at4(un[e], i) * fN);
          const float si = at4(sc[e], i), pi = at4(pc[e], i);
          x[i] = fmaf(-si, fmaf(wx, xs[i], hx[i] * fmaf(hz, ys, hy[e] * zs)), pi);
        }
        if (act && yin[e]) {
          const int64_t o = (int64_t)A.px * (yr[e] + (int64_t)ny * z) + xl;
          // (weights first: W spans the range that the squares would leave)
          dot = fmaf(pc[e].x * W, x[0], fmaf(pc[e].y * W, x[1],
                fmaf(pc[e].z * W, x[2], fmaf(pc[e].w * W, x[3], dot))));
          pmax = max4(pmax, pc[e]);
          *reinterpret_cast<float4 *>(A.p + o) = pc[e];
          *reinterpret_cast<float4 *>(A.q + o) = make_float4(x[0], x[1], x[2], x[3]);
        }
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        um[e] = uc[e];
        uc[e] = un[e];
        sc[e] = sn[e];
        pc[e] = pn[e];
        urc[e] = urn[e];
      }
      cur = nxt;
    }
    // (copies past the last plane are zero fills of unused stages; they have
    // to land before the next tile issues into them)
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  const double bs = block_sum((double)dot, shd);
  const unsigned bm = block_max_bits(__float_as_uint(pmax), shu);
  unsigned *mx = reinterpret_cast<unsigned *>(A.part + gridDim.x);
  if (threadIdx.x == 0) {
    A.part[blockIdx.x] = bs;
    mx[blockIdx.x] = bm;
  }
  if (!last_block(&c->counter[0], &flag)) return;
  const double ps = sum_partials(A.part, gridDim.x, shd);
  unsigned m = 0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) m = max(m, __ldcg(mx + b));
  m = block_max_bits(m, shu);
  if (threadIdx.x != 0) return;
  c->counter[0] = 0u;
  c->pexp = m >> 23;
  if (start) {
    c->gm = st->gam_m;
    c->gs = st->gam_s;
    c->F = F0;
    c->fd = fd;
    c->scale = scale;
    c->conj2 = 0.0;
    c->check = 0;
    c->thetaF = ldexpf(st->theta, -F0);
  }
  // units of 2^(2 F + fd) = 2^gs: alpha = gm / (<p, A p> - 2 beta <p, A p_old>).
  // Without the correction FP32 rounding lets the directions lose conjugacy
  // unnoticed; once the difference is not positive the inner solve ends, its
  // correction so far is kept, and the refinement restarts from the true
  // residual (the resident 2D kernel does the same)
  const double gm = c->gm, den = ps - c->conj2;
  const bool pos = ps > 0.0 && den > 0.0 && isfinite(den);
  const float al = pos ? (float)(gm / den) : 0.f;
  c->ps = ps;
  c->alpha = al;
  c->alphaF = ldexpf(al, c->F);
  if (gm == 0.0) finish(st, EIK_OK, false);
  else if (!isfinite(ps)) finish(st, EIK_ERR_BREAKDOWN, false);
  else if (!(pos && isfinite(al)))
    finish(st, start ? EIK_ERR_BREAKDOWN : EIK_OK, !start);
}

// Blocks of step_x x step_y threads: float4 columns by rows, last rows first.
__global__ void __launch_bounds__(kThreads, kStepPerSm)
k_pair_step(const PairArgs A, int bx, int by) {
  __shared__ double shd[32];
  __shared__ unsigned shu[32];
  __shared__ int flag;
  MixCtl *st = A.st;
  PairCtl *c = A.c;
  if (st->done) return;
  const float alpha = c->alpha, alphaF = c->alphaF, thetaF = c->thetaF, scale = c->scale;
  const int fd = c->fd, lg = A.cg.lgB;
  const bool check = c->check != 0;
  const int n4 = A.px / 4, ny = A.g.ny, nrow = ny * A.g.nz;
  const int tx = threadIdx.x % bx, ty = threadIdx.x / bx;
  float gam = 0.f, rs = 0.f, rmax = 0.f;
  int bad = 0;
  for (int k = blockIdx.x * by + ty; k < nrow; k += gridDim.x * by) {
    const int row = nrow - 1 - k, z = row / ny, y = row - z * ny;
    const int *kr = A.kx + A.cg.cx * ((y >> lg) + A.cg.cy * (z >> lg));
    for (int i = tx; i < n4; i += bx) {
      const int64_t o = (int64_t)A.px * row + 4 * i;
      const float4 p = *reinterpret_cast<const float4 *>(A.p + o);
      const float4 q = *reinterpret_cast<const float4 *>(A.q + o);
      float4 d = *reinterpret_cast<const float4 *>(A.d + o);
      float4 r = *reinterpret_cast<const float4 *>(A.r + o);
      d = make_float4(fmaf(alphaF, p.x, d.x), fmaf(alphaF, p.y, d.y), fmaf(alphaF, p.z, d.z),
                      fmaf(alphaF, p.w, d.w));
      r = make_float4(fmaf(-alpha, q.x, scale * r.x), fmaf(-alpha, q.y, scale * r.y),
                      fmaf(-alpha, q.z, scale * r.z), fmaf(-alpha, q.w, scale * r.w));
      *reinterpret_cast<float4 *>(A.d + o) = d;
      *reinterpret_cast<float4 *>(A.r + o) = r;
      const float W = p2f(-2 * __ldg(kr + ((4 * i) >> lg)) - fd);
      rmax = max4(rmax, r);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float t = at4(r, e) * W;
        gam = fmaf(t, at4(r, e), gam);
        rs = fmaf(t, at4(q, e), rs);
      }
      if (check) {
        const float4 x = __ldg(reinterpret_cast<const float4 *>(A.xref + o));
        if (fabsf(r.x) > thetaF * fabsf(x.x + d.x) || fabsf(r.y) > thetaF * fabsf(x.y + d.y) ||
            fabsf(r.z) > thetaF * fabsf(x.z + d.z) || fabsf(r.w) > thetaF * fabsf(x.w + d.w))
          bad = 1;
      }
    }
  }
  const double b0 = block_sum((double)gam, shd), b1 = block_sum((double)rs, shd);
  const unsigned bm = block_max_bits(__float_as_uint(rmax), shu);
  const int any = __syncthreads_or(bad);
  double *part = A.part;
  uint2 *mx = reinterpret_cast<uint2 *>(part + 2 * gridDim.x);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = b0;
    part[gridDim.x + blockIdx.x] = b1;
    mx[blockIdx.x] = make_uint2(bm, any ? 1u : 0u);
  }
  if (!last_block(&c->counter[1], &flag)) return;
  const double G = sum_partials(part, gridDim.x, shd);
  const double rst = sum_partials(part + gridDim.x, gridDim.x, shd);
  unsigned m = 0, fl = 0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) {
    const uint2 v = __ldcg(mx + b);
    m = max(m, v.x);
    fl |= v.y;
  }
  m = block_max_bits(m, shu);
  const int viol = __syncthreads_or(fl != 0u);
  if (threadIdx.x != 0) return;
  c->counter[1] = 0u;
  const int iter = ++st->iter;
  ++st->total_iter;
  const float R = __uint_as_float(m);
  int F = c->F;
  const unsigned pexp = c->pexp;
  if (!isfinite(G) || !isfinite(R) || pexp == 255u) {
    finish(st, EIK_ERR_BREAKDOWN, false);
  } else if (G == 0.0 || (st->mode == 0 ? ldexpf(R, F) <= st->thresh : (check && !viol))) {
    finish(st, EIK_OK, false);
  } else if (iter >= st->max_iter) {
    finish(st, EIK_ERR_NOT_CONVERGED, false);
  } else {
    // <r,r> = G 2^gs as mantissa and exponent; the next direction's beta and
    // 2 beta <p, A p_old> = 2 beta (<r_new, A p> + beta <p, A p>)
    int eg;
    const double gn = frexp(G, &eg);
    const double bm = gn / c->gm, be = scalbn(bm, eg);
    c->conj2 = 2.0 * bm * fma(be, c->ps, rst);
    c->beta = be;
    c->gm = gn;
    c->gs += eg;
    // the frame follows the largest stored value
    const int e = max((int)(m >> 23), (int)pexp) - 127;
    const int dF = (e >= kRescale || e <= -kRescale) ? e : 0;
    F += dF;
    c->F = F;
    c->scale = p2f(-dF);
    c->fd = c->gs - 2 * F;
    c->thetaF = ldexpf(st->theta, -F);
    c->check = st->mode != 0 && (iter & 3) == 3;
  }
  st->F = F;
  st->alpha = c->alpha;
  st->beta = c->beta;
}

}  // namespace

void pair3_plan(Pair3Plan *pl, const Grid &g, const CellGrid &cg, int num_sms, cudaStream_t s) {
  *pl = Pair3Plan{};
  if (g.ndim != 3 || (int64_t)g.ny * g.nz > INT_MAX / 2) return;
  pl->tiles_x = (g.nx + 127) / 128;
  pl->tiles_y = (g.ny + kRows - 1) / kRows;
  // planes per tile: the fewest rounds over the resident blocks, each plane of
  // a round and its two halo planes counted
  const int64_t slots = (int64_t)num_sms * kDirPerSm, col = (int64_t)pl->tiles_x * pl->tiles_y;
  int64_t best = INT64_MAX;
  for (int zc = 1; zc <= g.nz; ++zc) {
    const int64_t nt = col * ((g.nz + zc - 1) / zc);
    const int64_t cost = (nt + slots - 1) / slots * (zc + 2);
    if (nt <= INT_MAX / 2 && cost < best) {
      best = cost;
      pl->zc = zc;
      pl->ntiles = (int)nt;
    }
  }
  if (best == INT64_MAX) return;
  pl->nblk_dir = (int)std::min<int64_t>(pl->ntiles, slots);
  const int n4 = (g.nx + 3) / 4;
  int bx = 1;
  while (bx < n4 && bx < kThreads) bx *= 2;
  pl->step_x = bx;
  pl->step_y = kThreads / bx;
  const int64_t rows = ((int64_t)g.ny * g.nz + pl->step_y - 1) / pl->step_y;
  pl->nblk_step = (int)std::min<int64_t>(rows, (int64_t)num_sms * kStepPerSm);
  if (cudaFuncSetAttribute(k_pair_dir, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kDirSmem) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  const size_t bytes = sizeof(double) * 3 * (size_t)std::max(pl->nblk_dir, pl->nblk_step);
  if (cudaMalloc((void **)&pl->ctl, sizeof(PairCtl)) != cudaSuccess ||
      cudaMalloc((void **)&pl->part, bytes) != cudaSuccess ||
      cudaMemsetAsync(pl->ctl, 0, sizeof(PairCtl), s) != cudaSuccess) {
    cudaGetLastError();
    return;   // freed by pair3_destroy
  }
  pl->ok = true;
}

void pair3_destroy(Pair3Plan *pl) {
  if (pl->ctl) cudaFree(pl->ctl);
  if (pl->part) cudaFree(pl->part);
  *pl = Pair3Plan{};
}

void pair3_iter(const Pair3Plan &pl, const Grid &g, const CellGrid &cg, const Cg32Buffers &b,
                int set, cudaStream_t s) {
  PairArgs a{};
  a.g = g;
  a.cg = cg;
  a.px = b.px;
  a.kx = b.kx;
  a.s32 = b.s32;
  a.xref = b.xref;
  a.p_old = b.p[set];
  a.r = b.r[0];
  a.p = b.p[1 - set];
  a.q = b.r[1];
  a.d = b.d;
  a.st = b.st;
  a.c = pl.ctl;
  a.part = pl.part;
  k_pair_dir<<<pl.nblk_dir, kDirThreads, kDirSmem, s>>>(a, pl.tiles_x, pl.tiles_y, pl.zc,
                                                        pl.ntiles);
  k_pair_step<<<pl.nblk_step, kThreads, 0, s>>>(a, pl.step_x, pl.step_y);
}

}  // namespace eik
