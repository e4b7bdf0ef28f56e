// Resident FP64 CG for grids whose CG vectors fit on chip: one cooperative
// kernel runs up to kRes64Iters iterations of the two-reduction Jacobi-PCG of
// eik_cg64.cu.
//
// What bounds it: the two-pass form moves 88 B per node and iteration through
// L2 and pays two launches, each with its own tail (block sums, a ticket, and
// a last block that adds the partials), 22 us together on a 129^2 grid whose
// arithmetic takes 0.3 us.  Here r, p (and x) live in registers, sigma and
// u = sigma p in shared memory, and only the faces of a block's brick go
// through L2; the face values go as tagged messages and the two grid-wide
// sums per iteration through one counter (eik_gridsync.cuh).  What is left is the FP64 pipe (two lanes per
// clock and SM on this GPU: 10 instructions per node in 2D, 12 in 3D) and two
// message round trips.  Measured per iteration (two-pass form, this one):
// 129^2 22 us, 10 us; 733 x 517 37 us, 14 us; 120 x 97 x 85 63 us, 35 us.
// Larger grids, which do not fit, keep the two passes.
//
// Split: bricks of nearly equal size, at most one block per SM, kMinNodes
// nodes per block until half of the SMs have one, 2 kMinNodes beyond.  More
// blocks shorten an iteration further (129^2: 16 blocks 8 us, 65 blocks 7 us),
// but cooperative grids run side by side only where they fit, and a batch
// solves up to 16 instances at a time; with these sizes both gain.  512
// threads hold up to 16 nodes each; sums are added in a fixed order, so a
// solve is deterministic, and the split depends on the grid alone, so a batch
// repeats the bits of single solves.
#include <math.h>

#include <algorithm>

#include "eik_gridsync.cuh"
#include "eik_res64.h"

namespace eik {

namespace {

constexpr int kT = 512;             // threads per block
constexpr int kMinNodes = 1024;     // nodes per block, at least (see above)
constexpr int kRes64Iters = 256;    // iterations per launch, at most
constexpr int kCheckEvery = 4;      // iterations between componentwise tests
constexpr size_t kMaxSmem = 222 * 1024;   // beside ~4 KB of static shared memory

// node: local coordinates in the brick and flags
constexpr unsigned kFx = 1u << 27, kFy = 1u << 28, kFz = 1u << 29, kBnd = 1u << 30;
constexpr unsigned kFaces = kFx | kFy | kFz;

// outcomes of an iteration besides 0 (go on): kStop + eik_status, or a wait
// that ran out
constexpr int kStop = 16, kLate = 1;

struct Res64Args {
  Grid g;
  int cx, cy, cz, bx, by, bz, halo;
  const double *sig, *w;
  double *x, *r, *p;
  CgState *st;
  unsigned long long *msg, *inbox;
  unsigned epoch;
  int max_it;
  int withhold;   // test hook: block 0 does not arrive in the first exchange
};

// Shared-memory layout (doubles first).
struct Layout {
  size_t u, sg, q, hp, hr, hi, total;
};
inline __host__ __device__ Layout layout(int bx, int by, int bz, int dim, int halo, bool qs) {
  Layout L;
  const size_t V = (size_t)bx * by * bz;
  const size_t H = (size_t)(bx + 2) * (by + 2) * (dim == 3 ? bz + 2 : 1);
  L.u = 0;
  L.sg = L.u + 8 * H;
  L.q = L.sg + 8 * V;
  L.hp = L.q + (qs ? 8 * V : 0);
  L.hr = L.hp + 8 * (size_t)halo;
  L.hi = L.hr + 8 * (size_t)halo;
  L.total = L.hi + 4 * (size_t)halo;
  return L;
}

// Nodes of the three kinds of brick faces, and tagged-value slots of a
// block's inbox: its halo nodes' r, face by face (-x, +x, -y, +y, -z, +z).
inline __host__ __device__ int inbox_slots(int bx, int by, int bz, int dim) {
  return 2 * (by * bz + bx * bz + (dim == 3 ? bx * by : 0));
}

__device__ __forceinline__ bool finite64(double v) {   // without the FP64 pipe
  return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}

// The same value, of which the compiler knows nothing: positions are computed
// again in every phase instead of being kept in registers through all of them.
__device__ __forceinline__ unsigned opaque(unsigned m) {
  asm volatile("" : "+r"(m));
  return m;
}

// v 2^-e without the FP64 pipe (0 below the normal range).
__device__ __forceinline__ double scale_down(double v, int e) {
  const int hi = __double2hiint(v);
  const bool ok = (hi & 0x7ff00000) > (e << 20);
  return __hiloint2double(ok ? hi - (e << 20) : 0, ok ? __double2loint(v) : 0);
}

// Sum over the block in a fixed order, valid in all lanes of warp 0; the
// return value of __syncthreads_or(flag) goes to *any.  One FP64 addition
// keeps a quarter of the SM's FP64 lanes busy for 64 cycles, so a shuffle tree
// in every warp would take 1,280 of them; here four warps (one per quarter)
// add four values per lane, and warp 0 the rest.  Warps 4 and up go on.
__device__ __forceinline__ double block_sum_w0(double v, double *red, int flag, int *any) {
  red[threadIdx.x] = v;
  *any = __syncthreads_or(flag);
  double s = 0.0;
  if (threadIdx.x < 128) {
    const double a = (red[threadIdx.x] + red[threadIdx.x + 128]) +
                     (red[threadIdx.x + 256] + red[threadIdx.x + 384]);
    red[threadIdx.x] = a;   // read by nobody else
    bar_first(1, 128);
    if (threadIdx.x < 32) {
      s = (a + red[threadIdx.x + 32]) + (red[threadIdx.x + 64] + red[threadIdx.x + 96]);
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
  }
  return s;
}

// K nodes per thread.  QS: q = A p is parked in shared memory and x stays in
// global memory (16 nodes per thread leave no registers for them).
template <int DIM, int K, bool QS>
__global__ void __launch_bounds__(kT, 1) k_cg64_res(const Res64Args A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[kT];
  __shared__ double sh_val;
  __shared__ int sh_stop;   // 0 go on, else an outcome
  if (A.st->done) return;
  const Grid &g = A.g;
  const int nblk = A.cx * A.cy * A.cz;
  const Layout L = layout(A.bx, A.by, A.bz, DIM, A.halo, QS);
  double *u = reinterpret_cast<double *>(smem_raw + L.u);
  double *sg = reinterpret_cast<double *>(smem_raw + L.sg);
  double *qs = reinterpret_cast<double *>(smem_raw + L.q);
  double *hp = reinterpret_cast<double *>(smem_raw + L.hp);
  double *hr = reinterpret_cast<double *>(smem_raw + L.hr);
  int *hi = reinterpret_cast<int *>(smem_raw + L.hi);
  const int tid = threadIdx.x;
  // the block's brick
  const int b = blockIdx.x;
  const int ix = b % A.cx, iy = (b / A.cx) % A.cy, iz = b / (A.cx * A.cy);
  const int x0 = (int)((int64_t)ix * g.nx / A.cx), x1 = (int)((int64_t)(ix + 1) * g.nx / A.cx);
  const int y0 = (int)((int64_t)iy * g.ny / A.cy), y1 = (int)((int64_t)(iy + 1) * g.ny / A.cy);
  const int z0 = (int)((int64_t)iz * g.nz / A.cz), z1 = (int)((int64_t)(iz + 1) * g.nz / A.cz);
  const int bx = x1 - x0, by = y1 - y0, bz = z1 - z0;
  const int V = bx * by * bz;
  const int HX = bx + 2, PL = HX * (by + 2);
  const int HN = (DIM == 3) ? PL * (bz + 2) : PL;
  const int g0 = x0 + g.nx * (y0 + g.ny * z0);
  const bool half = g.boundary == EIK_BOUNDARY_HALF_CELL;
  auto spos = [&](int lx, int ly, int lz) {
    return lx + 1 + HX * (ly + 1) + (DIM == 3 ? PL * (lz + 1) : 0);
  };
  auto gidx = [&](unsigned m) {
    return g0 + (int)(m & 1023u) + g.nx * ((int)((m >> 10) & 1023u) + g.ny * (int)((m >> 20) & 127u));
  };

  for (int s = tid; s < HN; s += kT) u[s] = 0.0;
  // halo nodes: the faces of the brick that have a neighbour.  A node's r
  // comes from the neighbour through this block's inbox; bricks are cut along
  // whole planes, so both sides number a face alike.
  const int mx = A.by * A.bz, my = A.bx * A.bz, mz = A.bx * A.by;
  const int slots = inbox_slots(A.bx, A.by, A.bz, DIM);
  const int f0 = (x0 > 0) ? by * bz : 0, f1 = (x1 < g.nx) ? by * bz : 0;
  const int f2 = (y0 > 0) ? bx * bz : 0, f3 = (y1 < g.ny) ? bx * bz : 0;
  const int f4 = (DIM == 3 && z0 > 0) ? bx * by : 0, f5 = (DIM == 3 && z1 < g.nz) ? bx * by : 0;
  const int nh = f0 + f1 + f2 + f3 + f4 + f5;
  // face and number within it of halo node h, and its inbox slot
  auto halo_at = [&](int h, int &lx, int &ly, int &lz) {
    int e = h;
    if (e < f0 + f1) {
      const bool hi_side = e >= f0;
      if (hi_side) e -= f0;
      lx = hi_side ? bx : -1;
      ly = e % by;
      lz = e / by;
      return (hi_side ? mx : 0) + e;
    }
    e -= f0 + f1;
    if (e < f2 + f3) {
      const bool hi_side = e >= f2;
      if (hi_side) e -= f2;
      ly = hi_side ? by : -1;
      lx = e % bx;
      lz = e / bx;
      return 2 * mx + (hi_side ? my : 0) + e;
    }
    e -= f2 + f3;
    const bool hi_side = e >= f4;
    if (hi_side) e -= f4;
    lz = hi_side ? bz : -1;
    lx = e % bx;
    ly = e / bx;
    return 2 * (mx + my) + (hi_side ? mz : 0) + e;
  };
  for (int h = tid; h < nh; h += kT) {
    int lx, ly, lz;
    const int sl = halo_at(h, lx, ly, lz);
    const int gi = g0 + lx + g.nx * (ly + g.ny * lz);
    hi[h] = spos(lx, ly, lz) | (sl << 16);
    hp[h] = A.p[gi];
    hr[h] = A.r[gi];
  }
  // sigma of the thread's first halo node stays in a register (thin bricks
  // have no more); further ones are read again from L1
  double hs0 = 0.0;
  auto halo_sigma = [&](int h) {
    int lx, ly, lz;
    halo_at(h, lx, ly, lz);
    return __ldg(A.sig + (g0 + lx + g.nx * (ly + g.ny * lz)));
  };
  if (tid < nh) hs0 = halo_sigma(tid);
  unsigned meta[K];
  double r[K], p[K], x[QS ? 1 : K], q[QS ? 1 : K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int l = tid + k * kT;
    r[k] = p[k] = 0.0;
    meta[k] = 0u;
    if (!QS) x[QS ? 0 : k] = q[QS ? 0 : k] = 0.0;
    if (l < V) {
      const int lx = l % bx, ly = (l / bx) % by, lz = l / (bx * by);
      const int gx = x0 + lx, gy = y0 + ly, gz = z0 + lz;
      unsigned m = (unsigned)lx | ((unsigned)ly << 10) | ((unsigned)lz << 20);
      if (half && (gx == 0 || gx == g.nx - 1)) m |= kFx;
      if (half && (gy == 0 || gy == g.ny - 1)) m |= kFy;
      if (DIM == 3 && half && (gz == 0 || gz == g.nz - 1)) m |= kFz;
      if (lx == 0 || lx == bx - 1 || ly == 0 || ly == by - 1 ||
          (DIM == 3 && (lz == 0 || lz == bz - 1)))
        m |= kBnd;
      meta[k] = m;
      const int gi = gidx(m);
      sg[l] = A.sig[gi];
      r[k] = A.r[gi];
      p[k] = A.p[gi];
      if (!QS) x[QS ? 0 : k] = A.x[gi];
    }
  }
  double beta = A.st->beta, rho = A.st->rho;
  const double tol = A.st->tol, nw = A.st->tol * A.st->tol * A.st->bnorm2;
  const bool cw = A.st->stop_norm == EIK_STOP_COMPONENTWISE;
  const int max_iter = A.st->max_iter;
  int iter = A.st->iter, stop = 0, late = 0;
  unsigned tag = A.epoch, arrivals = 0;
  __syncthreads();

  for (int it = 0; it < A.max_it; ++it) {
    // ---- p = r + beta p and u = sigma p on the brick and its halo
    for (int h = tid; h < nh; h += kT) {
      const double ph = fma(beta, hp[h], hr[h]);
      hp[h] = ph;
      u[hi[h] & 0xffff] = (h == tid ? hs0 : halo_sigma(h)) * ph;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int l = tid + k * kT;
      if (l < V) {
        const unsigned m = opaque(meta[k]);
        p[k] = fma(beta, p[k], r[k]);
        u[spos(m & 1023u, (m >> 10) & 1023u, (m >> 20) & 127u)] = sg[l] * p[k];
      }
    }
    __syncthreads();
    // ---- q = A p and <p, q>
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int l = tid + k * kT;
      if (l < V) {
        const unsigned m = opaque(meta[k]);
        const double *c = u + spos(m & 1023u, (m >> 10) & 1023u, (m >> 20) & 127u);
        double sx = c[-1] + c[1], sy = c[-HX] + c[HX], sz = 0.0;
        if (DIM == 3) sz = c[-PL] + c[PL];
        if (m & kFaces) {
          // edge weights: a factor 1/2 per face axis other than the edge's
          // (on the integer pipe: a brick with face nodes must not be slower
          // than the others)
          const int ex = (m >> 27) & 1, ey = (m >> 28) & 1, ez = (m >> 29) & 1;
          sx = scale_down(sx, ey + ez);
          sy = scale_down(sy, ex + ez);
          if (DIM == 3) sz = scale_down(sz, ex + ey);
        }
        double nb = sx + sy;
        if (DIM == 3) nb += sz;
        const double qv = fma(-sg[l], nb, p[k]);
        acc = fma(p[k], qv, acc);
        if (QS) qs[l] = qv;
        else q[QS ? 0 : k] = qv;
      }
    }
    int any;
    double s = block_sum_w0(acc, red, late, &any);
    ++tag;
    if (tid < 32) {
      // (a block whose halo never came does not arrive, so every block stops)
      if (tid == 0 && !any && !(A.withhold && it == 0 && b == 0)) {
        sync_put(A.msg, tag, 0, b, s);
        sync_arrive(A.msg);
      }
      arrivals += nblk;
      const bool ok = !any && sync_wait(A.msg, arrivals);
      double v[kSyncBlocks / 32];
      sync_get(A.msg, tag, 0, nblk, v);
      const double pq = sync_sum(v);
      if (tid == 0) {
        const bool pos = pq > 0.0 && finite64(pq);
        sh_val = pos ? quotient(rho, pq) : 0.0;
        sh_stop = !ok ? kLate : pos ? 0 : (rho == 0.0) ? kStop + EIK_OK : kStop + EIK_ERR_BREAKDOWN;
      }
    }
    __syncthreads();
    stop = sh_stop;   // the same in every block
    if (stop != 0) break;
    const double alpha = sh_val;
    // ---- x += alpha p, r -= alpha q, <r, r>, the componentwise test
    const bool check = cw && ((iter + 1) % kCheckEvery) == 0;
    const unsigned rtag = tag + 1;
    int bad = 0;
    acc = 0.0;
    // x += alpha p (and, in checking iterations, the test)
    auto update_x = [&]() {
      constexpr int kChunk = QS ? 4 : K;
#pragma unroll
      for (int k0 = 0; k0 < K; k0 += kChunk) {
        double xg[QS ? kChunk : 1];
        if (QS) {   // loads of a chunk before its arithmetic
#pragma unroll
          for (int j = 0; j < kChunk; ++j)
            if (tid + (k0 + j) * kT < V) xg[QS ? j : 0] = __ldcg(A.x + gidx(opaque(meta[k0 + j])));
        }
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          const int k = k0 + j;
          if (tid + k * kT < V) {
            double xn;
            if (QS) {
              xn = fma(alpha, p[k], xg[QS ? j : 0]);
              __stcg(A.x + gidx(opaque(meta[k])), xn);
            } else {
              xn = x[QS ? 0 : k] = fma(alpha, p[k], x[QS ? 0 : k]);
            }
            if (check) {
              // as in the two-pass form: |w r| <= tol (adjoint) or |r| <= tol |x|
              if (A.w) bad |= !(fabs(__ldg(A.w + gidx(opaque(meta[k]))) * r[k]) <= tol);
              else bad |= !(fabs(r[k]) <= tol * fabs(xn));
            }
          }
        }
      }
    };
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int l = tid + k * kT;
      if (l < V) {
        const unsigned m = opaque(meta[k]);
        const double rn = fma(-alpha, QS ? qs[l] : q[QS ? 0 : k], r[k]);
        r[k] = rn;
        acc = fma(rn, rn, acc);
        if (m & kBnd) {   // to the inboxes of the blocks this node is a halo of
          const int lx = m & 1023u, ly = (m >> 10) & 1023u, lz = (m >> 20) & 127u;
          auto send = [&](int nb, int slot) {
            tagged_put(A.inbox + 2 * ((size_t)nb * slots + slot), rtag, rn);
          };
          if (lx == 0 && f0) send(b - 1, mx + ly + by * lz);
          if (lx == bx - 1 && f1) send(b + 1, ly + by * lz);
          if (ly == 0 && f2) send(b - A.cx, 2 * mx + my + lx + bx * lz);
          if (ly == by - 1 && f3) send(b + A.cx, 2 * mx + lx + bx * lz);
          if (DIM == 3) {
            if (lz == 0 && f4) send(b - A.cx * A.cy, 2 * (mx + my) + mz + lx + bx * ly);
            if (lz == bz - 1 && f5) send(b + A.cx * A.cy, 2 * (mx + my) + lx + bx * ly);
          }
        }
      }
    }
    ++tag;
    ++iter;
    // x first where the test needs it, else while the messages travel (one
    // copy of its code)
#pragma unroll 1
    for (int half_step = 0; half_step < 2; ++half_step) {
      if ((half_step == 0) == check) update_x();
      if (half_step == 0) {
        s = block_sum_w0(acc, red, bad, &any);
        if (tid == 0) {
          if (check) sync_put(A.msg, tag, 1, b, any ? 1.0 : 0.0);
          sync_put(A.msg, tag, 0, b, s);
          sync_arrive(A.msg);
        }
      }
    }
    // meanwhile the neighbours' new r, and 1 / rho
    late = 0;
    for (int h = tid; h < nh; h += kT)
      late |= !tagged_wait(A.inbox + 2 * ((size_t)b * slots + (hi[h] >> 16)), tag, hr + h);
    if (tid < 32) {
      const double inv_rho = (rho != 0.0) ? 1.0 / rho : 0.0;
      arrivals += nblk;
      const bool ok = sync_wait(A.msg, arrivals);
      double v[kSyncBlocks / 32];
      bool fl = false;
      if (check) {
        sync_get(A.msg, tag, 1, nblk, v);
#pragma unroll
        for (int j = 0; j < kSyncBlocks / 32; ++j) fl = fl || __double2hiint(v[j]) != 0;
      }
      fl = __any_sync(0xffffffffu, fl);
      sync_get(A.msg, tag, 0, nblk, v);
      const double rr = sync_sum(v);
      if (tid == 0) {
        // (below about 5.6e-309 rho has no finite reciprocal; a solve whose phi
        // spans more than 1e150 passes through there before rho reaches 0 and
        // the loop ends for a restart from the true residual)
        sh_val = finite64(inv_rho) ? rr * inv_rho : rr / rho;
        const bool conv = cw ? (check && !fl) : rr <= nw;
        sh_stop = !ok ? kLate
                  : !finite64(rr) ? kStop + EIK_ERR_BREAKDOWN
                  : conv ? kStop + EIK_OK
                  : iter >= max_iter ? kStop + EIK_ERR_NOT_CONVERGED : 0;
        rho = rr;
      }
    }
    __syncthreads();
    stop = sh_stop;
    beta = sh_val;
    if (stop != 0) break;
  }

#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (tid + k * kT < V) {
      const int gi = gidx(opaque(meta[k]));
      if (!QS) A.x[gi] = x[QS ? 0 : k];
      A.r[gi] = r[k];
      A.p[gi] = p[k];
    }
  }
  if (tid == 0) {
    if (stop == kLate) {   // any block that sees a timeout reports it
      atomicExch(&A.st->status, (int)EIK_ERR_TIMEOUT);
      atomicExch(&A.st->done, 1);
    } else if (b == 0) {
      A.st->rho = rho;
      A.st->beta = beta;
      A.st->iter = iter;
      if (stop != 0) {
        atomicCAS(&A.st->status, (int)EIK_OK, stop - kStop);
        atomicExch(&A.st->done, 1);
      }
    }
  }
}

using Kern = void (*)(Res64Args);

// Nodes per thread the kernel is compiled for (one row per dimension).
Kern kernel_for(int dim, int K) {
  switch (K) {
    case 1: return dim == 2 ? k_cg64_res<2, 1, false> : k_cg64_res<3, 1, false>;
    case 2: return dim == 2 ? k_cg64_res<2, 2, false> : k_cg64_res<3, 2, false>;
    case 4: return dim == 2 ? k_cg64_res<2, 4, false> : k_cg64_res<3, 4, false>;
    case 8: return dim == 2 ? k_cg64_res<2, 8, false> : k_cg64_res<3, 8, false>;
    default: return dim == 2 ? k_cg64_res<2, 16, true> : k_cg64_res<3, 16, true>;
  }
}

}  // namespace

void res64_plan(Res64Plan *pl, const Grid &g, int num_sms) {
  *pl = Res64Plan{};
  int coop = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
    return;
  const int sms = std::min(num_sms, kSyncBlocks);
  if (g.n > (int64_t)sms * kT * 16) return;
  const int cap = (int)std::max<int64_t>(
      1, std::min<int64_t>(
             sms, std::max(std::min<int64_t>(sms / 2, g.n / kMinNodes), g.n / (2 * kMinNodes))));
  // the split with the least FP64 work per iteration in its largest brick:
  // about 10 instructions per node, 2 per halo node
  double best = 1e300;
  for (int cz = 1; cz <= std::min(cap, g.nz); ++cz)
    for (int cy = 1; cy * cz <= cap && cy <= g.ny; ++cy) {
      const int cx = std::min(cap / (cy * cz), g.nx);
      const int bx = (g.nx + cx - 1) / cx, by = (g.ny + cy - 1) / cy, bz = (g.nz + cz - 1) / cz;
      const int64_t V = (int64_t)bx * by * bz;
      if (V > kT * 16 || bx > 1023 || by > 1023 || bz > 127) continue;
      const int halo = (cx > 1 ? 2 * by * bz : 0) + (cy > 1 ? 2 * bx * bz : 0) +
                       (cz > 1 ? 2 * bx * by : 0);
      const bool qs = V > kT * 8;
      const Layout L = layout(bx, by, bz, g.ndim, halo, qs);
      // (a halo node's position and inbox slot share a word)
      if (L.total > kMaxSmem || (int64_t)(bx + 2) * (by + 2) * (bz + 2) > 65535 ||
          inbox_slots(bx, by, bz, g.ndim) > 32767)
        continue;
      const double cost = 10.0 * V + 2.0 * halo;
      if (cost < best) {
        best = cost;
        pl->cx = cx;
        pl->cy = cy;
        pl->cz = cz;
        pl->bx = bx;
        pl->by = by;
        pl->bz = bz;
        pl->halo = halo;
        pl->smem = L.total;
        int K = 1;
        while ((int64_t)K * kT < V) K *= 2;
        pl->per_thread = K;
      }
    }
  if (best == 1e300) return;
  pl->nblk = pl->cx * pl->cy * pl->cz;
  pl->inbox_words = (size_t)2 * pl->nblk * inbox_slots(pl->bx, pl->by, pl->bz, g.ndim);
  const Kern fn = kernel_for(g.ndim, pl->per_thread);
  int per = 0;
  // (the attribute belongs to the function, not to one solver: always the
  // largest size, so that concurrent solvers agree)
  if (cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kMaxSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, (const void *)fn, kT, pl->smem) !=
          cudaSuccess ||
      per < 1 || per * sms < pl->nblk) {
    cudaGetLastError();
    return;
  }
  pl->ok = true;
}

cudaError_t launch_res64(Res64Plan *pl, const Grid &g, const double *sig, double *x, double *r,
                         double *p, const double *cw_weight, CgState *st,
                         unsigned long long *msg, unsigned long long *inbox, bool withhold,
                         cudaStream_t s) {
  Res64Args a{};
  a.withhold = withhold ? 1 : 0;
  a.g = g;
  a.cx = pl->cx;
  a.cy = pl->cy;
  a.cz = pl->cz;
  a.bx = pl->bx;
  a.by = pl->by;
  a.bz = pl->bz;
  a.halo = pl->halo;
  a.sig = sig;
  a.w = cw_weight;
  a.x = x;
  a.r = r;
  a.p = p;
  a.st = st;
  a.msg = msg;
  a.inbox = inbox;
  a.epoch = pl->epoch;
  a.max_it = kRes64Iters;
  pl->epoch += 2u * kRes64Iters;
  const cudaError_t e = cudaMemsetAsync(msg, 0, sizeof(unsigned), s);   // the arrivals
  if (e != cudaSuccess) return e;
  void *args[] = {&a};
  return cudaLaunchCooperativeKernel((const void *)kernel_for(g.ndim, pl->per_thread),
                                     dim3(pl->nblk), dim3(kT), args, pl->smem, s);
}

}  // namespace eik
