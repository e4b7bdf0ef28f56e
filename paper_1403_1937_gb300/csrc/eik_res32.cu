// Resident FP32 inner CG of the 2D mixed solve (operator, units and frames as
// in eik_cg32.h): one cooperative kernel runs up to kRes32Iters iterations of
// the two-reduction Jacobi-PCG
//   p = r + beta p, s = A p, alpha = <r,r> / <p,s>, d += alpha p, r -= alpha s.
//
// What bounds it: the one-pass kernel (k_cg2d) moves 28 B per node and
// iteration through L2 and HBM, computes every row's p, s and r_new with a
// two-node halo, and pays a launch and its tail per iteration: 41 us on
// 2048^2, 23 us on 512^2.  Here r stays in
// registers, p and sigma in shared memory (220 KB of it on 2048^2, where d is
// the one array left in L2; smaller tiles keep d in registers too), and the
// halo of a tile and the two grid-wide sums per iteration travel as tagged
// messages (eik_gridsync.cuh).  Two sums per iteration instead of one, but no
// redundant halo arithmetic and no second stencil on r.  s = A p is computed
// once for <p,s> and again for r, since holding it would take another quarter
// of the registers.
// Measured per iteration of a solve (one-pass kernel, this one): 300 x 260
// 25.9 us, 10.5 us; 512^2 25.6 us, 8.6 us; 611 x 733 25.7 us, 10.1 us; 1500^2
// 33.0 us, 18.4 us; 2048^2 46.1 us, 34.4 us.  128 registers a thread are not
// enough beside r: tiles of up to 32 rows spill nothing, of 64 rows 72 B, of 128
// 268 B, of 256 592 B a thread (bytes stored), which bounds the largest grids.
// <r_new, A p>, <p, A p> and beta take FP64 like <r, r>, as in the one-pass
// kernels; adding <r_new, A p> in a second warp keeps that off the chain that
// the block waits for (in the same warp: 0.3 us an iteration).
//
// Split: tiles of up to 128 columns (a lane owns four of them) and 256 rows
// (222 KB of p and sigma), at most one block per SM: with 152 SMs 2048 x 2048 is
// the largest square, and larger grids take the one-pass kernels.  There are
// no more blocks than keep kMinNodes nodes each: the two sums take about 4 us
// whatever the tile, so smaller ones do not pay, and the SMs left free run
// other solves.  Sums are FP32 per warp, FP64 across warps and blocks in a fixed
// order: deterministic, and the split depends on the grid alone.
#include <math.h>

#include <algorithm>

#include "eik_gridsync.cuh"
#include "eik_res32.h"

namespace eik {

namespace {

constexpr int kMinNodes = 4096;     // nodes per block, at least
constexpr int kRes32Iters = 256;    // iterations per launch, at most
constexpr size_t kMaxSmem = 222 * 1024;   // beside ~3 KB of static shared memory
constexpr int kTab = 256;           // cell exponents of a tile and its rim
constexpr int kRescale = 8;         // r and p move to a new frame past 2^+-8

struct Res32Args {
  int nx, ny, px, boundary;
  CellGrid cg;
  const int *kx;
  int tx, ty, pw, ht;
  const float *s32, *xref;
  float *r, *p, *d;
  MixCtl *st;
  unsigned long long *msg, *inbox;
  unsigned epoch;
  int max_it;
};

// Recurrence scalars of the current iteration, set by one thread.
struct Scalars {
  float alpha, alphaF, beta, scale, thetaF;
  int fd, check, stop;
};
// The recurrence itself, kept by thread 0: <r,r> = gm 2^gs with gm in
// [0.5, 1), frame F (and the step dF to it that r and p still lack), beta and its
// mantissa, <p, A p>, <r_new, A p> and 2 beta <p, A p_old> of the next direction
// (units of 2^gs).
struct Recurrence {
  double gm, inv_gm, beta, bm, ps, rst, conj2;
  int gs, F, dF, iter;
  float alpha;
};
// outcomes besides 0 (go on): kStop + eik_status, kStall (positivity lost), a
// wait that ran out
constexpr int kStop = 16, kLate = 1, kStall = 2;

__device__ __forceinline__ float p2f(int n) {
  n = min(max(n, -126), 127);
  return __int_as_float((n + 127) << 23);
}
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 mul4(const float4 &a, const float4 &b) {
  return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
}
__device__ __forceinline__ bool finite64(double v) {
  return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}
__device__ __forceinline__ bool finite32(float v) {
  return (__float_as_int(v) & 0x7f800000) != 0x7f800000;
}

// One 32-bit value with its 32-bit tag in a word.
__device__ __forceinline__ unsigned long long tagged32(unsigned tag, float v) {
  return ((unsigned long long)tag << 32) | (unsigned)__float_as_int(v);
}
__device__ __forceinline__ void put32(unsigned long long *slot, unsigned tag, float v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(slot), "l"(tagged32(tag, v)) : "memory");
}
__device__ __forceinline__ bool wait32(const unsigned long long *slot, unsigned tag, float *v) {
  unsigned long long t0 = 0;
  for (unsigned spins = 1;; ++spins) {
    unsigned long long w;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(slot) : "memory");
    *v = __int_as_float((int)(unsigned)w);
    if ((unsigned)(w >> 32) == tag) return true;
    if ((spins & 255u) == 0u) {
      const unsigned long long t = sync_now();
      if (t0 == 0) t0 = t;
      else if (t - t0 > kSyncWaitNs) return false;
    }
  }
}

// T threads, ROWS rows per warp at most; DREG: d in registers.
template <int kT, int ROWS, bool DREG>
__global__ void __launch_bounds__(kT, 1) k_cg2d_res(const Res32Args A) {
  constexpr int kWarps = kT / 32, kHalo = 1024 / kT;   // halo nodes per thread
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float wsum[kWarps], wsum2[kWarps];   // FP32 per warp
  __shared__ unsigned wmax[kWarps];
  __shared__ int ktab[kTab];
  __shared__ Scalars sc;
  __shared__ Recurrence rec;
  MixCtl *st = A.st;
  if (st->done) return;
  const int tid = threadIdx.x, lane = tid & 31, wi = tid >> 5;
  const int b = blockIdx.x, nblk = A.tx * A.ty;
  const int bx = b % A.tx, by = b / A.tx;
  const int n4 = (A.nx + 3) / 4;
  const int xs = 4 * (int)((int64_t)bx * n4 / A.tx), xe = 4 * (int)((int64_t)(bx + 1) * n4 / A.tx);
  const int ys = (int)((int64_t)by * A.ny / A.ty), ye = (int)((int64_t)(by + 1) * A.ny / A.ty);
  const int w = xe - xs, h = ye - ys, pw = A.pw;
  // rows -1 and ht of sigma hold 1 and those of p the neighbours' u, so that
  // u = sigma p without a case for the rim
  float *P = reinterpret_cast<float *>(smem_raw) + pw;      // [-1 .. ht][pw]
  float *SG = P + (size_t)(A.ht + 2) * pw;                  // [-1 .. ht][pw]
  float *ul = SG + (size_t)(A.ht + 1) * pw;                 // u of the columns left and right
  float *ur = ul + A.ht;
  const CellGrid cg = A.cg;
  const int mask = cg.B - 1, lg = cg.lgB;
  const bool half = A.boundary == EIK_BOUNDARY_HALF_CELL;

  // cell exponents of the tile and its rim
  const int cc0 = max(xs - 1, 0) >> lg, cc1 = min(xe, A.nx - 1) >> lg;
  const int cr0 = max(ys - 1, 0) >> lg, cr1 = min(ye, A.ny - 1) >> lg;
  const int ncol = cc1 - cc0 + 1;
  for (int e = tid; e < ncol * (cr1 - cr0 + 1); e += kT)
    ktab[e] = A.kx[(cr0 + e / ncol) * cg.cx + cc0 + e % ncol];
  for (int e = tid; e < pw; e += kT) {
    P[e - pw] = P[h * pw + e] = 0.f;
    SG[e - pw] = SG[h * pw + e] = 1.f;
  }
  for (int e = tid; e < 2 * A.ht; e += kT) ul[e] = 0.f;

  // the lane's four columns
  const int xl = xs + 4 * lane;
  const bool act = xl < xe;
  const int c = act ? 4 * lane : 0;             // column in the tile
  const bool lastl = act && xl + 4 >= xe;
  unsigned xface = 0;                           // columns on an x face
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (half && (xl + i == 0 || xl + i == A.nx - 1)) xface |= 1u << i;
  const int xq = act ? xl : xs;
  const int kcol = (xq >> lg) - cc0;
  const int kcl = (max(xq - 1, 0) >> lg) - cc0, kcr = (min(xq + 4, A.nx - 1) >> lg) - cc0;
  const bool ccr = kcr > kcol;                  // (a chunk past the grid has none)
  // the warp's rows [j0, j0 + nr) of the tile
  const int j0 = h * wi / kWarps, nr = h * (wi + 1) / kWarps - j0;

  // halo nodes: row above, row below, column left, column right; thread t
  // holds p and sigma of nodes t and t + kT
  const int slots = 2 * (pw + A.ht);
  const int nt = (ys > 0) ? w : 0, nb = (ye < A.ny) ? w : 0;
  const int nl = (xs > 0) ? h : 0, nrt = (xe < 4 * n4) ? h : 0;
  const int nh = nt + nb + nl + nrt;
  // position of halo node q: its inbox slot, its u in shared memory, and its
  // global index
  auto halo_at = [&](int q, int64_t &gi, int &u) {
    if (q < nt) {
      gi = (int64_t)(ys - 1) * A.px + xs + q;
      u = q - pw;
      return q;
    }
    q -= nt;
    if (q < nb) {
      gi = (int64_t)ye * A.px + xs + q;
      u = h * pw + q;
      return pw + q;
    }
    q -= nb;
    if (q < nl) {
      gi = (int64_t)(ys + q) * A.px + xs - 1;
      u = (int)(ul - P) + q;
      return 2 * pw + q;
    }
    q -= nl;
    gi = (int64_t)(ys + q) * A.px + xe;
    u = (int)(ur - P) + q;
    return 2 * pw + A.ht + q;
  };
  float hp[kHalo], hs[kHalo], hr[kHalo];
  int hslot[kHalo];
  int hu[kHalo];
#pragma unroll
  for (int e = 0; e < kHalo; ++e) {
    const int q = tid + e * kT;
    hp[e] = hs[e] = hr[e] = 0.f;
    hslot[e] = -1;
    hu[e] = 0;
    if (q < nh) {
      int64_t gi;
      hslot[e] = halo_at(q, gi, hu[e]);
      hs[e] = A.s32[gi];
      hp[e] = A.p[gi];
      hr[e] = A.r[gi];
    }
  }
  float r[ROWS][4];
  float d[DREG ? ROWS : 1][4];
#pragma unroll
  for (int j = 0; j < ROWS; ++j) {
    r[j][0] = r[j][1] = r[j][2] = r[j][3] = 0.f;
    if (DREG) d[DREG ? j : 0][0] = d[DREG ? j : 0][1] = d[DREG ? j : 0][2] = d[DREG ? j : 0][3] = 0.f;
    if (j < nr && act) {
      const int64_t gi = (int64_t)(ys + j0 + j) * A.px + xl;
      const float4 r4 = ld4(A.r + gi);
      r[j][0] = r4.x; r[j][1] = r4.y; r[j][2] = r4.z; r[j][3] = r4.w;
      if (DREG) {
        const float4 d4 = ld4(A.d + gi);
        d[DREG ? j : 0][0] = d4.x; d[DREG ? j : 0][1] = d4.y;
        d[DREG ? j : 0][2] = d4.z; d[DREG ? j : 0][3] = d4.w;
      }
      const int o = (j0 + j) * pw + c;
      *reinterpret_cast<float4 *>(P + o) = ld4(A.p + gi);
      *reinterpret_cast<float4 *>(SG + o) = ld4(A.s32 + gi);
    }
  }
  // 2 beta <p, A p_old> from one launch of an inner solve to the next, beside
  // the arrivals
  double *carry = reinterpret_cast<double *>(A.msg + 1);
  const bool withhold = st->withhold != 0 && st->iter == 0 && b == 0;
  if (tid == 0) {
    rec.gm = st->gam_m;
    rec.gs = st->gam_s;
    rec.F = st->F + st->dF;
    rec.iter = st->iter;
    rec.dF = 0;
    rec.beta = st->beta;
    rec.alpha = 0.f;
    rec.bm = rec.ps = rec.rst = 0.0;
    rec.conj2 = (rec.iter == 0) ? 0.0 : *carry;
    sc.beta = (float)rec.beta;
    sc.scale = p2f(-st->dF);
    sc.fd = rec.gs - 2 * rec.F;
    sc.thetaF = ldexpf(st->theta, -rec.F);
    sc.check = st->mode != 0 && (rec.iter & 3) == 3;
    sc.stop = 0;
  }
  unsigned tag = A.epoch, arrivals = 0;
  int stop = 0, late = 0;
  __syncthreads();

  // factors of the current row: left and right neighbour columns, rows above
  // and below (2^(kx_i - kx_j), 1 inside a cell), the y face, the dots' weight.
  // They change at the rows marked in `special` only.
  float fL = 1.f, fR = 1.f, fU = 1.f, fD = 1.f, hy = 1.f, W = 0.f;
  unsigned special = 1u;
  for (int jj = 1; jj < nr; ++jj) {
    const int y = ys + j0 + jj;
    auto rim = [&](int v) {
      return (v & mask) == 0 || ((v + 1) & mask) == 0 || v == 0 || v == A.ny - 1;
    };
    if (rim(y) || rim(y - 1)) special |= 1u << jj;
  }
  auto row_factors = [&](int y, int fd) {
    const int *t = ktab + ((y >> lg) - cr0) * ncol;
    const int kc = t[kcol];
    fL = p2f(kc - t[kcl]);
    fR = ccr ? p2f(kc - t[kcr]) : 1.f;
    fU = ((y & mask) == 0 && y > 0) ? p2f(kc - t[kcol - ncol]) : 1.f;
    fD = (((y + 1) & mask) == 0 && y + 1 < A.ny) ? p2f(kc - t[kcol + ncol]) : 1.f;
    hy = (half && (y == 0 || y == A.ny - 1)) ? 0.5f : 1.f;
    W = p2f(-2 * kc - fd);
  };
  // (A p)_i of the lane's nodes of row j, given u of rows j - 1 .. j + 1
  auto apply = [&](int j, const float4 &um, const float4 &uc, const float4 &un, const float4 &p4,
                   const float4 &s4, float (&s)[4]) {
    float uL = __shfl_up_sync(0xffffffffu, uc.w, 1);
    float uR = __shfl_down_sync(0xffffffffu, uc.x, 1);
    if (lane == 0) uL = ul[j];
    if (lastl) uR = ur[j];
    const float xv[4] = {fmaf(uL, fL, uc.y), uc.x + uc.z, uc.y + uc.w, fmaf(uR, fR, uc.z)};
    const float uu[4] = {um.x, um.y, um.z, um.w}, ud[4] = {un.x, un.y, un.z, un.w};
    const float pv[4] = {p4.x, p4.y, p4.z, p4.w}, sv[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float yv = fmaf(uu[i], fU, ud[i] * fD);
      if (xface & (1u << i)) yv *= 0.5f;
      s[i] = fmaf(-sv[i], fmaf(hy, xv[i], yv), pv[i]);
    }
  };
  // sums over the block of two per-thread FP32 values, FP64 across warps in a
  // fixed order: in the lower (v) and the upper (v2) half of warp 0, so that
  // the second takes no instructions of its own; and the largest of a
  // non-negative value's bits
  static_assert(kWarps == 16, "a half warp adds the warps' values");
  auto block_sum = [&](float v, float v2, unsigned mx, int flag, int *any, unsigned *mo,
                       double *s2) {
    for (int o = 16; o > 0; o >>= 1) {
      v += __shfl_xor_sync(0xffffffffu, v, o);
      v2 += __shfl_xor_sync(0xffffffffu, v2, o);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) {
      wsum[wi] = v;
      wsum2[wi] = v2;
      wmax[wi] = mx;
    }
    *any = __syncthreads_or(flag);
    double s = 0.0;
    if (wi == 0) {
      s = (double)(lane < kWarps ? wsum[lane] : wsum2[lane - kWarps]);
      for (int o = kWarps / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (s2) *s2 = __shfl_sync(0xffffffffu, s, kWarps);
      *mo = __reduce_max_sync(0xffffffffu, lane < kWarps ? wmax[lane] : 0u);
    }
    return s;
  };
  for (int it = 0; it < A.max_it; ++it) {
    // ---- p = r + beta p (both first moved to the current frame)
    const float beta = sc.beta, scale = sc.scale;
    const int fd = sc.fd;
    float pmax = 0.f;
#pragma unroll
    for (int e = 0; e < kHalo; ++e) {
      if (hslot[e] >= 0) {
        hp[e] = fmaf(beta, hp[e] * scale, hr[e] * scale);
        P[hu[e]] = hs[e] * hp[e];
      }
    }
#pragma unroll
    for (int j = 0; j < ROWS; ++j) {
      if (j < nr && act) {
        float4 *pp = reinterpret_cast<float4 *>(P + (j0 + j) * pw + c);
        float4 p4 = *pp;
        if (scale != 1.f) {
#pragma unroll
          for (int i = 0; i < 4; ++i) r[j][i] *= scale;
          p4 = make_float4(p4.x * scale, p4.y * scale, p4.z * scale, p4.w * scale);
        }
        p4 = make_float4(fmaf(beta, p4.x, r[j][0]), fmaf(beta, p4.y, r[j][1]),
                         fmaf(beta, p4.z, r[j][2]), fmaf(beta, p4.w, r[j][3]));
        *pp = p4;
        pmax = fmaxf(fmaxf(pmax, fmaxf(fabsf(p4.x), fabsf(p4.y))),
                     fmaxf(fabsf(p4.z), fabsf(p4.w)));
      }
    }
    __syncthreads();
    // ---- <p, A p>
    float pap = 0.f;
    const float *Pr = P + j0 * pw + c, *Sr = SG + j0 * pw + c;
    {
      float4 um = mul4(ld4(Sr - pw), ld4(Pr - pw));
      float4 pc = ld4(Pr), sg = ld4(Sr), uc = mul4(sg, pc);
      constexpr int kUnroll = ROWS < 16 ? 2 : 4;   // (fewest spills)
#pragma unroll kUnroll
      for (int jj = 0; jj < nr; ++jj) {
        const float4 pn = ld4(Pr + (jj + 1) * pw), sn = ld4(Sr + (jj + 1) * pw);
        const float4 un = mul4(sn, pn);
        if ((special >> jj) & 1u) row_factors(ys + j0 + jj, fd);
        float s[4];
        apply(j0 + jj, um, uc, un, pc, sg, s);
        // (weights first: W spans the range that the squares would leave)
        if (act)
          pap = fmaf(pc.x * W, s[0], fmaf(pc.y * W, s[1],
                fmaf(pc.z * W, s[2], fmaf(pc.w * W, s[3], pap))));
        um = uc;
        uc = un;
        pc = pn;
        sg = sn;
      }
    }
    int any;
    unsigned mo = 0;
    double rs_b = 0.0;
    double sum = block_sum(pap, 0.f, (unsigned)__float_as_int(pmax), late, &any, &mo, nullptr);
    ++tag;
    unsigned pm = mo;
    if (wi == 0) {
      // (a block whose halo never came does not arrive, so every block stops)
      if (tid == 0 && !any && !(withhold && it == 0)) {
        sync_put(A.msg, tag, 0, b, sum);
        sync_arrive(A.msg);
      }
      // (while the sums travel) <p, A p_old> = <r_new, A p> + beta <p, A p>
      if (tid == 0 && it > 0) rec.conj2 = 2.0 * rec.bm * fma(rec.beta, rec.ps, rec.rst);
      arrivals += nblk;
      const bool ok = !any && sync_wait(A.msg, arrivals);
      double v[kSyncBlocks / 32];
      sync_get(A.msg, tag, 0, nblk, v);
      const double ps = sync_sum(v);
      if (tid == 0) {
        // units of 2^(2 F + fd) = 2^gs: alpha = gm / ps.  The FP32 recurrence
        // has lost the directions' conjugacy once <p, A p> is not above
        // 2 beta <p, A p_old> (then <r, A r> < beta^2 <p_old, A p_old>, which
        // CG excludes); the inner solve ends there, its correction so far is
        // kept, and the refinement restarts from the true residual
        rec.ps = ps;
        // alpha's denominator is <p, A p> less that term: <p, A p> as CG's
        // orthogonality gives it, as in the one-pass kernels (textbook
        // <p, A p> itself let a 512^2 solve without sweeps grow its residual
        // to 1e22 before it stalled)
        const double den = ps - rec.conj2;
        const bool pos = ps > 0.0 && den > 0.0 && finite64(den);
        const double al = pos ? quotient(rec.gm, den) : 0.0;
        const float alf = (float)al;
        rec.alpha = sc.alpha = alf;
        sc.alphaF = ldexpf(alf, rec.F);
        sc.stop = !ok ? kLate
                  : rec.gm == 0.0 ? kStop + EIK_OK
                  : !finite64(ps) ? kStop + EIK_ERR_BREAKDOWN
                  : (pos && finite32(alf)) ? 0
                  : rec.iter == 0 ? kStop + EIK_ERR_BREAKDOWN : kStall;
      }
    }
    __syncthreads();
    stop = sc.stop;
    if (stop != 0) break;
    // ---- r -= alpha s, <r, r>; rows and columns that neighbours need go out
    const float alpha = sc.alpha, alphaF = sc.alphaF, thetaF = sc.thetaF;
    const bool check = sc.check != 0;
    float gam = 0.f, rmax = 0.f, rs = 0.f;
    int bad = 0;
    ++tag;
    {
      float4 um = mul4(ld4(Sr - pw), ld4(Pr - pw));
      float4 pc = ld4(Pr), sg = ld4(Sr), uc = mul4(sg, pc);
#pragma unroll
      for (int jj = 0; jj < ROWS; ++jj) {
        if (jj < nr) {
          const int j = j0 + jj;
          const float4 pn = ld4(Pr + (jj + 1) * pw), sn = ld4(Sr + (jj + 1) * pw);
          const float4 un = mul4(sn, pn);
          if ((special >> jj) & 1u) row_factors(ys + j, fd);
          float s[4];
          apply(j, um, uc, un, pc, sg, s);
          if (act) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              r[jj][i] = fmaf(-alpha, s[i], r[jj][i]);
              rmax = fmaxf(rmax, fabsf(r[jj][i]));
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float t = r[jj][i] * W;
              gam = fmaf(t, r[jj][i], gam);
              rs = fmaf(t, s[i], rs);
            }
            if (j == 0 && nt) {
              unsigned long long *o = A.inbox + (size_t)(b - A.tx) * slots + pw + c;
#pragma unroll
              for (int i = 0; i < 4; ++i) put32(o + i, tag, r[jj][i]);
            }
            if (j == h - 1 && nb) {
              unsigned long long *o = A.inbox + (size_t)(b + A.tx) * slots + c;
#pragma unroll
              for (int i = 0; i < 4; ++i) put32(o + i, tag, r[jj][i]);
            }
            if (lane == 0 && nl)
              put32(A.inbox + (size_t)(b - 1) * slots + 2 * pw + A.ht + j, tag, r[jj][0]);
            if (lastl && nrt) put32(A.inbox + (size_t)(b + 1) * slots + 2 * pw + j, tag, r[jj][3]);
          }
          um = uc;
          uc = un;
          pc = pn;
          sg = sn;
          // (no loads of later rows above this point: they would fill the
          // registers that r needs)
          asm volatile("" ::: "memory");
        }
      }
    }
    // d += alpha p 2^F: before the sums where the test needs it, else while
    // the messages travel (one copy of its code)
#pragma unroll 1
    for (int step = 0; step < 2; ++step) {
      if ((step == 0) == check) {
        constexpr int kChunk = ROWS < 8 ? ROWS : ROWS < 16 ? 4 : 2;   // loads of a chunk before its stores
#pragma unroll
        for (int k0 = 0; k0 < ROWS; k0 += kChunk) {
          float4 dv[kChunk], xv[kChunk];
#pragma unroll
          for (int k = 0; k < kChunk; ++k) {
            const int jj = k0 + k;
            if (DREG) {
              const int e = DREG ? jj : 0;
              dv[k] = make_float4(d[e][0], d[e][1], d[e][2], d[e][3]);
            }
            if (jj < nr && act) {
              const int64_t gi = (int64_t)(ys + j0 + jj) * A.px + xl;
              if (!DREG) dv[k] = __ldcg(reinterpret_cast<const float4 *>(A.d + gi));
              if (check) xv[k] = __ldg(reinterpret_cast<const float4 *>(A.xref + gi));
            }
          }
#pragma unroll
          for (int k = 0; k < kChunk; ++k) {
            const int jj = k0 + k;
            if (jj < nr && act) {
              const float4 p4 = ld4(Pr + jj * pw);
              const float4 d4 = make_float4(fmaf(alphaF, p4.x, dv[k].x), fmaf(alphaF, p4.y, dv[k].y),
                                            fmaf(alphaF, p4.z, dv[k].z), fmaf(alphaF, p4.w, dv[k].w));
              if (DREG) {
                const int e = DREG ? jj : 0;
                d[e][0] = d4.x; d[e][1] = d4.y; d[e][2] = d4.z; d[e][3] = d4.w;
              } else {
                const int64_t gi = (int64_t)(ys + j0 + jj) * A.px + xl;
                __stcg(reinterpret_cast<float4 *>(A.d + gi), d4);
              }
              if (check &&
                  (fabsf(r[jj][0]) > thetaF * fabsf(xv[k].x + d4.x) ||
                   fabsf(r[jj][1]) > thetaF * fabsf(xv[k].y + d4.y) ||
                   fabsf(r[jj][2]) > thetaF * fabsf(xv[k].z + d4.z) ||
                   fabsf(r[jj][3]) > thetaF * fabsf(xv[k].w + d4.w)))
                bad = 1;
            }
          }
        }
      }
      if (step == 0) {
        sum = block_sum(gam, rs, (unsigned)__float_as_int(rmax), bad, &any, &mo, &rs_b);
        if (tid == 0) {
          // besides <r, r>: <r_new, A p>; and largest |r|, the exponent of the
          // largest |p|, the test's flag in one word
          sync_put(A.msg, tag, 1, b,
                   __hiloint2double((int)mo, (int)((pm >> 23) << 1 | (any ? 1u : 0u))));
          sync_put(A.msg, tag, 2, b, rs_b);
          sync_put(A.msg, tag, 0, b, sum);
          sync_arrive(A.msg);
        }
      }
    }
    // meanwhile the neighbours' new r
    late = 0;
#pragma unroll
    for (int e = 0; e < kHalo; ++e)
      if (hslot[e] >= 0)
        late |= !wait32(A.inbox + (size_t)b * slots + hslot[e], tag, &hr[e]);
    if (wi == 0) {
      if (tid == 0) rec.inv_gm = 1.0 / rec.gm;
      arrivals += nblk;
      const bool ok = sync_wait(A.msg, arrivals);
      asm volatile("bar.arrive 2, 64;" ::: "memory");   // warp 1 goes on
      double v[kSyncBlocks / 32];
      sync_get(A.msg, tag, 1, nblk, v);
      unsigned rm = 0, pmx = 0, fl = 0;
#pragma unroll
      for (int j = 0; j < kSyncBlocks / 32; ++j) {
        const unsigned lo = (unsigned)__double2loint(v[j]);
        rm = max(rm, (unsigned)__double2hiint(v[j]));
        pmx = max(pmx, (lo >> 1) & 0xffu);
        fl |= lo & 1u;
      }
      sync_get(A.msg, tag, 0, nblk, v);
      const double G = sync_sum(v);
      rm = __reduce_max_sync(0xffffffffu, rm);
      pmx = __reduce_max_sync(0xffffffffu, pmx);
      fl = __reduce_or_sync(0xffffffffu, fl);
      if (tid == 0) {
        const int iter = ++rec.iter, mode = st->mode;
        const float R = __int_as_float((int)rm);
        int F = rec.F, out = 0;
        if (!ok) out = kLate;
        else if (!finite64(G) || !finite32(R) || pmx == 255u) out = kStop + EIK_ERR_BREAKDOWN;
        else if (G == 0.0 || (mode == 0 ? ldexpf(R, F) <= st->thresh : (check && fl == 0)))
          out = kStop + EIK_OK;
        else if (iter >= st->max_iter) out = kStop + EIK_ERR_NOT_CONVERGED;
        // <r,r> = G 2^gs: mantissa and exponent; the next direction's beta
        // (G == 0 or subnormal: the solve ends or stalls)
        const int eb = ((__double2hiint(G) >> 20) & 0x7ff) - 1022;
        const int eg = eb > -1022 ? eb : 0;
        const double gn = eb > -1022 ? __hiloint2double((__double2hiint(G) & 0x800fffff) | 0x3fe00000,
                                                        __double2loint(G)) : G;
        const double bm = gn * rec.inv_gm;   // beta = bm 2^eg
        const int hb = __double2hiint(bm), xb = (hb >> 20) + eg;
        const double be = (hb >> 20) > 0 && xb > 0 && xb < 2047
                              ? __hiloint2double(hb + (eg << 20), __double2loint(bm))
                              : scalbn(bm, eg);
        rec.bm = bm;   // (beta in the new units)
        rec.beta = be;
        rec.gm = gn;
        rec.gs += eg;
        // the frame follows the largest stored value
        const int e = max(__float_as_int(R) >> 23, (int)pmx) - 127;
        rec.dF = (e >= kRescale || e <= -kRescale) ? e : 0;
        if (it + 1 < A.max_it && out == 0) {
          F += rec.dF;
          sc.scale = p2f(-rec.dF);
          rec.F = F;
          rec.dF = 0;
        }
        sc.beta = (float)be;
        sc.fd = rec.gs - 2 * F;
        sc.thetaF = ldexpf(st->theta, -F);
        sc.check = mode != 0 && (iter & 3) == 3;
        sc.stop = out;
      }
    }
    // <r_new, A p> beside it, on an FP64 pipe of its own; needed in the next
    // exchange only
    if (wi == 1) {
      asm volatile("bar.sync 2, 64;" ::: "memory");
      double v[kSyncBlocks / 32];
      sync_get(A.msg, tag, 2, nblk, v);
      const double rst = sync_sum(v);
      if (lane == 0) rec.rst = rst;
    }
    __syncthreads();
    stop = sc.stop;
    if (stop != 0) break;
  }

#pragma unroll
  for (int j = 0; j < ROWS; ++j) {
    if (j < nr && act) {
      const int64_t gi = (int64_t)(ys + j0 + j) * A.px + xl;
      if (DREG)
        *reinterpret_cast<float4 *>(A.d + gi) =
            make_float4(d[DREG ? j : 0][0], d[DREG ? j : 0][1], d[DREG ? j : 0][2],
                        d[DREG ? j : 0][3]);
      if (stop == 0) {   // the next launch goes on from here
        *reinterpret_cast<float4 *>(A.r + gi) = make_float4(r[j][0], r[j][1], r[j][2], r[j][3]);
        *reinterpret_cast<float4 *>(A.p + gi) = ld4(P + (j0 + j) * pw + c);
      }
    }
  }
  if (tid == 0) {
    if (stop == kLate) {   // any block that sees a timeout reports it
      atomicExch(&st->status, (int)EIK_ERR_TIMEOUT);
      atomicExch(&st->done, 1);
    } else if (b == 0) {
      st->gam_m = rec.gm;
      st->gam_s = rec.gs;
      st->alpha = rec.alpha;
      st->beta = rec.beta;
      st->F = rec.F;
      st->dF = rec.dF;
      st->fd = rec.gs - 2 * rec.F;
      st->total_iter += rec.iter - st->iter;
      st->iter = rec.iter;
      *carry = 2.0 * rec.bm * fma(rec.beta, rec.ps, rec.rst);
      if (stop != 0) {
        if (stop == kStall) st->stalled = 1;
        atomicCAS(&st->status, (int)EIK_OK, stop == kStall ? (int)EIK_OK : stop - kStop);
        atomicExch(&st->done, 1);
      }
    }
  }
}

using Kern = void (*)(Res32Args);

// Instances by tile height (rows per warp of 16 warps).  Taller tiles leave no
// registers for d.
struct Instance {
  Kern fn;
  int threads, max_ht;
};
const Instance kInstances[] = {{k_cg2d_res<512, 2, true>, 512, 32},
                               {k_cg2d_res<512, 4, true>, 512, 64},
                               {k_cg2d_res<512, 8, false>, 512, 128},
                               {k_cg2d_res<512, 16, false>, 512, 256}};
constexpr int kNumInstances = 4, kMaxHt = 256;

int instance_for(int ht) {
  int k = 0;
  while (k + 1 < kNumInstances && kInstances[k].max_ht < ht) ++k;
  return k;
}

size_t smem_of(int pw, int ht) { return sizeof(float) * (2 * (size_t)pw * (ht + 2) + 2 * ht); }

}  // namespace

void res32_plan(Res32Plan *pl, const Grid &g, const CellGrid &cg, int num_sms, cudaStream_t s) {
  *pl = Res32Plan{};
  if (g.ndim != 2) return;
  int coop = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
    return;
  const int sms = std::min(num_sms, kSyncBlocks);
  const int n4 = (g.nx + 3) / 4;
  const int64_t padded = (int64_t)n4 * 4 * g.ny;
  if (padded > (int64_t)sms * kMaxSmem / 8) return;
  // the fewest rows per warp (about 560 cycles each, beside 8,000 for the two
  // sums), then the fewest blocks
  const int cap = (int)std::max<int64_t>(1, std::min<int64_t>(sms, padded / kMinNodes));
  int best = 1 << 30, best_blk = 0;
  for (int pass = 0; pass < 2 && best == 1 << 30; ++pass) {
    const int lim = pass == 0 ? cap : sms;   // past cap only where the tiles need it
    for (int tx = 1; tx <= std::min(lim, n4); ++tx) {
      const int pw = 4 * ((n4 + tx - 1) / tx);
      if (pw > 128) continue;
      for (int ty = 1; tx * ty <= lim && ty <= g.ny; ++ty) {
        const int ht = (g.ny + ty - 1) / ty;
        if (ht > kMaxHt || smem_of(pw, ht) > kMaxSmem || 2 * (pw + ht) > 1024) continue;
        const int ncol = pw / cg.B + 3, nrow = ht / cg.B + 3;
        if (ncol * nrow > kTab) continue;
        const int rows = (ht + 15) / 16;
        if (rows < best || (rows == best && tx * ty < best_blk)) {
          best = rows;
          best_blk = tx * ty;
          pl->tx = tx;
          pl->ty = ty;
          pl->pw = pw;
          pl->ht = ht;
        }
      }
    }
  }
  if (best == 1 << 30) return;
  pl->nblk = best_blk;
  pl->instance = instance_for(pl->ht);
  pl->smem = smem_of(pl->pw, pl->ht);
  const Kern fn = kInstances[pl->instance].fn;
  int per = 0;
  // (the attribute belongs to the function, not to one solver: always the
  // largest size, so that concurrent solvers agree)
  if (cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kMaxSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &per, (const void *)fn, kInstances[pl->instance].threads, pl->smem) !=
          cudaSuccess ||
      per < 1 || per * sms < pl->nblk) {
    cudaGetLastError();
    return;
  }
  pl->inbox_words = (size_t)pl->nblk * 2 * (pl->pw + pl->ht);
  const size_t bytes = kSyncBytes + sizeof(unsigned long long) * pl->inbox_words;
  if (cudaMalloc((void **)&pl->msg, bytes) != cudaSuccess) {
    cudaGetLastError();
    pl->msg = nullptr;
    return;
  }
  if (cudaMemsetAsync(pl->msg, 0, bytes, s) != cudaSuccess) {
    cudaGetLastError();
    return;   // the buffer is freed by res32_destroy
  }
  pl->ok = true;
}

void res32_destroy(Res32Plan *pl) {
  if (pl->msg) cudaFree(pl->msg);
  pl->msg = nullptr;
  pl->ok = false;
}

cudaError_t launch_res32(Res32Plan *pl, const Grid &g, const CellGrid &cg, const Cg32Buffers &b,
                         cudaStream_t s) {
  Res32Args a{};
  a.nx = g.nx;
  a.ny = g.ny;
  a.px = b.px;
  a.boundary = g.boundary;
  a.cg = cg;
  a.kx = b.kx;
  a.tx = pl->tx;
  a.ty = pl->ty;
  a.pw = pl->pw;
  a.ht = pl->ht;
  a.s32 = b.s32;
  a.xref = b.xref;
  a.r = b.r[0];
  a.p = b.p[0];
  a.d = b.d;
  a.st = b.st;
  a.msg = pl->msg;
  a.inbox = pl->msg + kSyncBytes / sizeof(unsigned long long);
  a.epoch = pl->epoch;
  a.max_it = kRes32Iters;
  pl->epoch += 2u * kRes32Iters;
  const cudaError_t e = cudaMemsetAsync(pl->msg, 0, sizeof(unsigned), s);   // the arrivals
  if (e != cudaSuccess) return e;
  void *args[] = {&a};
  const Instance &in = kInstances[pl->instance];
  return cudaLaunchCooperativeKernel((const void *)in.fn, dim3(pl->nblk), dim3(in.threads), args,
                                     pl->smem, s);
}

}  // namespace eik
