// vdp_multigrid.cu -- geometric multigrid V-cycle that preconditions CG for the variable-
// coefficient operator A of div((1/rho) grad .) (Sec. 3.4) on any grid whose coarsening reaches
// at most 512 cells (all sizes even down to it), where the FFT passes of the spectral
// preconditioner need lengths built from 2 and 3.
//
// The cycle (cell-centred, periodic, FP32, unscaled variables):
//   levels      halve every direction while all sizes are even and the level has > 64 cells;
//   coarse A    face coefficient = 1/2 x the sum of the four fine low faces under the coarse low
//               face (the 2h rediscretisation of the face flux, 8 x the 2h operator for constant
//               rho: the restricted equations are sums over 8 children);
//   P, R        cell-centred linear interpolation (3/4 parent, 1/4 its neighbour on the fine
//               cell's side, per axis) and its transpose;
//   smoothing   one weighted Jacobi sweep (weight 0.8) before the coarse correction, from zero,
//               and one after it;
//   coarsest    the dense pseudo-inverse of -A (built in double precision by one cluster).
// Same smoother before and after, R = P^T and a symmetric coarse solve make the cycle a fixed
// symmetric positive (semi-)definite operator M ~ (-A)^-1, as CG needs.  Used on the solve's
// scaled residual rt = D^-1/2 r: z = W M W rt with W = D^1/2 (the weight omega), like the
// spectral preconditioner.
//
// Per level and cycle four launches: pre-smoothing + residual (down), restriction, prolongation
// + pre-smoothed iterate, post-smoothing (up); the levels of up to 4096 cells and the coarsest take
// one launch of one block.  The level
// sweeps are z-marching column kernels (one-wave work-item plan); the z-neighbours are carried in
// registers.  All launches return at once unless the solve is in its preconditioner phase.
#include <cuda_runtime.h>

#include <cstdint>

#include "vdp_device.cuh"
#include "vdp_march.cuh"
#include "vdp_multigrid.h"

namespace vdp {

namespace {

constexpr int kMgThreads = kMarchTx * kMarchTy;  // 1-D blocks of 256 (tile 32 x 8)
// Levels that one block takes (k_mg_tail): up to 4096 cells.  CG solves, mixed, to 1e-9, with no such
// levels / up to 1024 / 4096 / 8192 / 32768 cells, ms: 32^3 0.83 / 0.74 / 0.75 / 0.75 / 0.75, 40^3 1.00
// / 0.92 / 0.92 / 1.03 / 1.03, 96^3 1.54 / 1.44 / 1.38 / 1.38 / 1.67, 128^3 2.21 / 2.12 / 2.14 / 2.14 /
// 2.99, 160^3 3.43 / 3.35 / 3.35 / 3.51 / 3.51, 256 x 128 x 128 5.72 / 5.44 / 5.44 / 5.70 / 5.70.
constexpr int kMgTailThreads = 1024, kMgTailLevels = 6, kMgTailCells = 4096;

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(double v) { return narrow(v); }
__device__ __forceinline__ void from_f(float v, float* out) { *out = v; }
__device__ __forceinline__ void from_f(float v, double* out) { *out = widen(v); }

__device__ __forceinline__ bool mg_active(const InstState* st) {  // one load per block
  if (st == nullptr) return true;
  return __syncthreads_or(threadIdx.x == 0 && __ldcg(&st->phase) == PH_SPEC) != 0;
}

struct Nbr {
  long long dxm, dxp, dym, dyp;
};

__device__ __forceinline__ Nbr neighbours(int x, int y, int nx, int ny) {
  Nbr d;
  d.dxm = x == 0 ? (long long)(nx - 1) : -1;
  d.dxp = x == nx - 1 ? -(long long)(nx - 1) : 1;
  d.dym = y == 0 ? (long long)(ny - 1) * nx : -(long long)nx;
  d.dyp = y == ny - 1 ? -(long long)(ny - 1) * nx : (long long)nx;
  return d;
}

#define MG_MARCH_BEGIN(lv)                                                                      \
  const int nx = (lv).nx, ny = (lv).ny, nz = (lv).nz;                                          \
  const long long plane = (long long)nx * ny;                                                  \
  for (int it = blockIdx.x; it < m.items; it += gridDim.x) {                                   \
    int x, y, z0, z1;                                                                          \
    if (!march_item(m, it, threadIdx.x & 31, threadIdx.x >> 5, nx, ny, nz, x, y, z0, z1))      \
      continue;                                                                                \
    const Nbr d = neighbours(x, y, nx, ny);                                                    \
    long long c = x + (long long)nx * y + plane * z0;

// Every smoothed level works in scaled variables (y = W x, W = D^1/2 = omega): the scaled operator
// At = W^-1 (-A) W^-1 = I - offdiag(bt) has a unit diagonal, so a Jacobi sweep is y += w (rt - At y)
// and no diagonal is read.  lv.bx, by, bz hold bt in FP32; level 0 takes W from the solve, the
// coarser levels keep their own (om, oinv = 1 / om).  Restriction and prolongation act on the
// unscaled quantities.

// Down: y1 = w rt (from zero), scaled residual rt - At y1 = (1 - w) rt + w sum bt rt_nb, stored
// unscaled (times omega) in t for the restriction.
template <class T>
__global__ void __launch_bounds__(kMgThreads, 4)
    k_mg_down0(MgLevel lv, MarchPlan m, const T* __restrict__ rt, const float* __restrict__ om,
               const InstState* st) {
  if (!mg_active(st)) return;
  const float w = kMgOmega;
  MG_MARCH_BEGIN(lv)
  float r_m = to_f(__ldg(rt + (z0 == 0 ? c + plane * (nz - 1) : c - plane)));
  float r_c = to_f(__ldg(rt + c));
  float bz_c = __ldg(lv.bz + c);
  for (int z = z0; z < z1; ++z) {
    const long long czp = z == nz - 1 ? c - plane * (nz - 1) : c + plane;
    const float r_p = to_f(__ldg(rt + czp));
    const float bz_p = __ldg(lv.bz + czp);
    float s = __ldg(lv.bx + c) * to_f(__ldg(rt + c + d.dxm));
    s = fmaf(__ldg(lv.bx + c + d.dxp), to_f(__ldg(rt + c + d.dxp)), s);
    s = fmaf(__ldg(lv.by + c), to_f(__ldg(rt + c + d.dym)), s);
    s = fmaf(__ldg(lv.by + c + d.dyp), to_f(__ldg(rt + c + d.dyp)), s);
    s = fmaf(bz_c, r_m, s);
    s = fmaf(bz_p, r_p, s);
    lv.t[c] = __ldg(om + c) * fmaf(1.f - w, r_c, w * s);
    r_m = r_c;
    r_c = r_p;
    bz_c = bz_p;
    c += plane;
  }
  }
}

// Up: y3 = y2 + w (rt - At y2) = (1 - w) y2 + w (rt + sum bt y2_nb), y2 = t.  Level 0 (COARSE
// false) stores y3 as the solve's scaled z and, with a state, <rt, z>, and completes the sweep; a
// coarser level stores its unscaled result x = oinv y3 for the next finer prolongation.
template <class T, class TOUT, bool COARSE>
__global__ void __launch_bounds__(kMgThreads, 4)
    k_mg_up(MgLevel lv, MarchPlan m, const T* __restrict__ rt, TOUT* __restrict__ out,
            InstState* st, const InstDesc* I) {
  if (!mg_active(st)) return;
  const float w = kMgOmega;
  const float* __restrict__ t = lv.t;
  float acc = 0.f;
  MG_MARCH_BEGIN(lv)
  float v_m = __ldg(t + (z0 == 0 ? c + plane * (nz - 1) : c - plane));
  float v_c = __ldg(t + c);
  float bz_c = __ldg(lv.bz + c);
  for (int z = z0; z < z1; ++z) {
    const long long czp = z == nz - 1 ? c - plane * (nz - 1) : c + plane;
    const float v_p = __ldg(t + czp);
    const float bz_p = __ldg(lv.bz + czp);
    float s = to_f(__ldg(rt + c));
    const float r_c = s;
    s = fmaf(__ldg(lv.bx + c), __ldg(t + c + d.dxm), s);
    s = fmaf(__ldg(lv.bx + c + d.dxp), __ldg(t + c + d.dxp), s);
    s = fmaf(__ldg(lv.by + c), __ldg(t + c + d.dym), s);
    s = fmaf(__ldg(lv.by + c + d.dyp), __ldg(t + c + d.dyp), s);
    s = fmaf(bz_c, v_m, s);
    s = fmaf(bz_p, v_p, s);
    const float y3 = fmaf(1.f - w, v_c, w * s);
    if constexpr (COARSE) {
      lv.x[c] = __ldg(lv.oinv + c) * y3;
    } else {
      from_f(y3, out + c);
      acc = fmaf(r_c, y3, acc);
    }
    v_m = v_c;
    v_c = v_p;
    bz_c = bz_p;
    c += plane;
  }
  }
  if constexpr (!COARSE) {
    if (st) {
      const float part[1] = {acc};
      store_partials<1, float>(part, I->part, gridDim.x, blockIdx.x);
      finish_sweep(*I, st, PH_SPEC, gridDim.x);
    }
  }
}

// Prolongation.  A thread has the two fine columns 2I, 2I + 1 of a fine row y and marches the coarse
// planes K of a chunk: the bilinear xy interpolations of plane K at the two columns, L(K), are
// computed once and carried (fine plane 2K takes 3/4 L(K) + 1/4 L(K-1), plane 2K + 1 3/4 L(K) + 1/4
// L(K+1)), so four fine cells cost two 8-byte loads each of rt and omega and six coarse values,
// and all of a step's loads are issued together (one column and one cell per step before: the whole
// cycle at 160^3 157 -> 136 us with this and the coarsest level below).  With the pre-smoothed iterate:
// t = w rt + omega P xc   (scaled: y1 + W P xc; xc is the coarse level's unscaled result)
__global__ void __launch_bounds__(kMgThreads, 4)
    k_mg_prolong(MgLevel lv, MgLevel cv, MarchPlan m, const float* __restrict__ rt,
                 const float* __restrict__ om, int wall_x, const InstState* st) {
  if (!mg_active(st)) return;
  const int nx = lv.nx, ny = lv.ny, cx = cv.nx, cy = cv.ny, cz = cv.nz;
  const long long plane = (long long)nx * ny, cplane = (long long)cx * cy;
  const float* __restrict__ xc = cv.x;
  for (int it = blockIdx.x; it < m.items; it += gridDim.x) {
    int I, y, K0, K1;
    if (!march_item(m, it, threadIdx.x & 31, threadIdx.x >> 5, cx, ny, cz, I, y, K0, K1)) continue;
    const int J0 = y >> 1;
    // neighbours of the parent on the fine cells' sides; at the duct's x ends the parent itself
    const int Im = I == 0 ? (wall_x ? I : cx - 1) : I - 1;
    const int Ip = I + 1 == cx ? (wall_x ? I : 0) : I + 1;
    const int J1 = (y & 1) ? (J0 + 1 == cy ? 0 : J0 + 1) : (J0 == 0 ? cy - 1 : J0 - 1);
    const long long r0 = (long long)cx * J0, r1 = (long long)cx * J1;
    auto L = [&](int K) {
      const float* p0 = xc + cplane * K + r0;
      const float* p1 = xc + cplane * K + r1;
      const float c0 = __ldg(p0 + I), l0 = __ldg(p0 + Im), h0 = __ldg(p0 + Ip);
      const float c1 = __ldg(p1 + I), l1 = __ldg(p1 + Im), h1 = __ldg(p1 + Ip);
      const float al = fmaf(0.75f, c0, 0.25f * l0), bl = fmaf(0.75f, c1, 0.25f * l1);
      const float ah = fmaf(0.75f, c0, 0.25f * h0), bh = fmaf(0.75f, c1, 0.25f * h1);
      return make_float2(fmaf(0.75f, al, 0.25f * bl), fmaf(0.75f, ah, 0.25f * bh));
    };
    long long c = 2 * I + (long long)nx * y + plane * (2 * K0);
    float2 Lm = L(K0 == 0 ? cz - 1 : K0 - 1), Lc = L(K0);
    for (int K = K0; K < K1; ++K, c += 2 * plane) {
      const float2 Lp = L(K + 1 == cz ? 0 : K + 1);
      const float2 ra = __ldg(reinterpret_cast<const float2*>(rt + c));
      const float2 rb = __ldg(reinterpret_cast<const float2*>(rt + c + plane));
      const float2 wa = __ldg(reinterpret_cast<const float2*>(om + c));
      const float2 wb = __ldg(reinterpret_cast<const float2*>(om + c + plane));
      float2 ta, tb;
      ta.x = fmaf(kMgOmega, ra.x, wa.x * fmaf(0.75f, Lc.x, 0.25f * Lm.x));
      ta.y = fmaf(kMgOmega, ra.y, wa.y * fmaf(0.75f, Lc.y, 0.25f * Lm.y));
      tb.x = fmaf(kMgOmega, rb.x, wb.x * fmaf(0.75f, Lc.x, 0.25f * Lp.x));
      tb.y = fmaf(kMgOmega, rb.y, wb.y * fmaf(0.75f, Lc.y, 0.25f * Lp.y));
      *reinterpret_cast<float2*>(lv.t + c) = ta;
      *reinterpret_cast<float2*>(lv.t + c + plane) = tb;
      Lm = Lc;
      Lc = Lp;
    }
  }
}

// Restriction r_coarse = P^T t, marching the coarse column (I, J) along K: a warp covers 32
// consecutive I of one coarse row, each lane loads its two fine cells (2I, 2I + 1) of a fine row
// as one float2 and takes 2I - 1 and 2I + 2 from its neighbour lanes (edge lanes load them), so a
// fine row costs one 8-byte load per coarse cell.  The xy sums of fine planes 2K - 1 and 2K are
// carried from the previous K.
// The coarse right side is stored scaled (times oinv) unless the coarse level is the coarsest
// (solved unscaled by the pseudo-inverse; oinv null).
__global__ void __launch_bounds__(kMgThreads, 4)
    k_mg_restrict(MgLevel fv, MgLevel cv, MarchPlan m, const float* __restrict__ oinv,
                  int wall_x, const InstState* st) {
  if (!mg_active(st)) return;
  const int nx = fv.nx, ny = fv.ny, nz = fv.nz;
  const int cx = cv.nx, cy = cv.ny, cz = cv.nz;
  const long long fplane = (long long)nx * ny, cplane = (long long)cx * cy;
  const float* __restrict__ t = fv.t;
  const int lane = threadIdx.x & 31;
  for (int it = blockIdx.x; it < m.items; it += gridDim.x) {
    int I, J, K0, K1;
    const bool on = march_item(m, it, lane, threadIdx.x >> 5, cx, cy, cz, I, J, K0, K1);
    // the whole warp takes part in the shuffles; a warp never straddles two coarse rows
    const int Jc = J < cy ? J : cy - 1;
    const int Ic = on ? I : 0;
    int yj[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) yj[b] = (2 * Jc - 1 + b + ny) % ny;
    const bool lload = lane == 0 || !on || Ic == 0;                 // 2I - 1 not in lane - 1
    const bool rload = lane == 31 || Ic == cx - 1;                  // 2I + 2 not in lane + 1
    const int xl = 2 * Ic == 0 ? nx - 1 : 2 * Ic - 1;
    const int xr = 2 * Ic + 2 == nx ? 0 : 2 * Ic + 2;
    // xy sum of fine plane k (weights 1/4, 3/4, 3/4, 1/4 per axis)
    auto plane_sum = [&](int k) {
      const float* pk = t + fplane * k;
      float sum = 0.f;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const float* row = pk + (long long)nx * yj[b];
        float2 v = make_float2(0.f, 0.f);
        if (on) v = __ldg(reinterpret_cast<const float2*>(row + 2 * Ic));
        float left = __shfl_up_sync(0xffffffffu, v.y, 1);
        float right = __shfl_down_sync(0xffffffffu, v.x, 1);
        if (on && lload) left = __ldg(row + xl);
        if (on && rload) right = __ldg(row + xr);
        // the duct's x ends: the end child took the quarter the far side would have given
        if (wall_x && Ic == 0) left = v.x;
        if (wall_x && Ic == cx - 1) right = v.y;
        const float rs = fmaf(0.25f, left + right, 0.75f * (v.x + v.y));
        const float wb = (b == 0 || b == 3) ? 0.25f : 0.75f;
        sum = fmaf(wb, rs, sum);
      }
      return sum;
    };
    int kk = 2 * K0 - 1;
    float s_a = plane_sum(kk < 0 ? kk + nz : kk);   // fine plane 2K - 1
    float s_b = plane_sum(2 * K0);                  // fine plane 2K
    for (int K = K0; K < K1; ++K) {
      const float s_c = plane_sum(2 * K + 1);
      const float s_d = plane_sum(2 * K + 2 == nz ? 0 : 2 * K + 2);
      if (on) {
        const long long C = I + (long long)cx * J + cplane * K;
        const float v = fmaf(0.25f, s_a + s_d, 0.75f * (s_b + s_c));
        cv.r[C] = oinv ? __ldg(oinv + C) * v : v;
      }
      s_a = s_c;
      s_b = s_d;
    }
  }
}

// Coarsest level: x = pinv r, a warp per four rows (one block with a thread per row and all its
// products in sequence took 13 us for 125 cells).
constexpr int kCoarseRows = 4 * (kMgThreads / 32);  // rows of a block

// Rows i0 .. i0 + 3 of x = pinv r by one warp.
__device__ __forceinline__ void coarse_rows(const MgLevel& lv, const float* __restrict__ pinv, int n,
                                            int i0, int lane) {
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  for (int j = lane; j < n; j += 32) {
    const float r = lv.r[j];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i0 + q < n) s[q] = fmaf(__ldg(pinv + (long long)(i0 + q) * n + j), r, s[q]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float v = warp_sum(s[q]);
    if (lane == 0 && i0 + q < n) lv.x[i0 + q] = v;
  }
}

__global__ void __launch_bounds__(kMgThreads)
    k_mg_coarse(MgLevel lv, const float* __restrict__ pinv, int n, const InstState* st) {
  if (!mg_active(st)) return;
  coarse_rows(lv, pinv, n, blockIdx.x * kCoarseRows + (threadIdx.x >> 5) * 4, threadIdx.x & 31);
}

// The coarse levels of a cycle in one block: down, restriction, ..., coarsest, ..., prolongation and up
// of every level from h.lev[0] on, separated by block barriers.  A level of a few thousand cells is a
// microsecond or two of work for one block (trips to L2), and a launch of its own per step took three to
// four.  Same operations per cell, in the same order, as the kernels above; fields that
// this kernel writes are read by plain loads.
struct MgTail {
  MgLevel lev[kMgTailLevels];
  int nlev;  // the last one is the coarsest
  const float* pinv;
  int ncoarse, wall_x;
};

__global__ void __launch_bounds__(kMgTailThreads) k_mg_tail(const __grid_constant__ MgTail h,
                                                            const InstState* st) {
  if (!mg_active(st)) return;
  const float w = kMgOmega;
  const int tid = threadIdx.x, lane = tid & 31;
  // the sum of the six neighbours' bt v around cell c, added to s
  auto neighbour_sum = [&](const MgLevel& lv, const float* v, int c, float s, bool up) {
    const int nx = lv.nx, ny = lv.ny, nz = lv.nz, plane = nx * ny;
    const int z = c / plane, y = (c - z * plane) / nx, x = c - z * plane - y * nx;
    const int xm = x == 0 ? c + nx - 1 : c - 1, xp = x == nx - 1 ? c - (nx - 1) : c + 1;
    const int ym = y == 0 ? c + (ny - 1) * nx : c - nx, yp = y == ny - 1 ? c - (ny - 1) * nx : c + nx;
    const int zm = z == 0 ? c + (nz - 1) * plane : c - plane, zp = z == nz - 1 ? c - (nz - 1) * plane : c + plane;
    s = up ? fmaf(__ldg(lv.bx + c), v[xm], s) : __ldg(lv.bx + c) * v[xm];
    s = fmaf(__ldg(lv.bx + xp), v[xp], s);
    s = fmaf(__ldg(lv.by + c), v[ym], s);
    s = fmaf(__ldg(lv.by + yp), v[yp], s);
    s = fmaf(__ldg(lv.bz + c), v[zm], s);
    return fmaf(__ldg(lv.bz + zp), v[zp], s);
  };
  for (int l = 0; l < h.nlev - 1; ++l) {
    const MgLevel &f = h.lev[l], &cv = h.lev[l + 1];
    for (int c = tid; c < (int)f.n; c += kMgTailThreads) {
      const float r = f.r[c];
      f.t[c] = __ldg(f.om + c) * fmaf(1.f - w, r, w * neighbour_sum(f, f.r, c, 0.f, false));
    }
    __syncthreads();
    const int nx = f.nx, ny = f.ny, nz = f.nz, cx = cv.nx, cy = cv.ny;
    for (int C = tid; C < (int)cv.n; C += kMgTailThreads) {
      const int K = C / (cx * cy), J = (C - K * cx * cy) / cx, I = C - K * cx * cy - J * cx;
      const int xl = I == 0 ? nx - 1 : 2 * I - 1, xr = 2 * I + 2 == nx ? 0 : 2 * I + 2;
      float s[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {  // fine planes 2K - 1 .. 2K + 2
        const int k = 2 * K - 1 + a, kk = k < 0 ? k + nz : k == nz ? 0 : k;
        float sum = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int j = 2 * J - 1 + b, jj = j < 0 ? j + ny : j == ny ? 0 : j;
          const float* row = f.t + (kk * ny + jj) * nx;
          const float2 v = *reinterpret_cast<const float2*>(row + 2 * I);
          const float left = h.wall_x && I == 0 ? v.x : row[xl];
          const float right = h.wall_x && I == cx - 1 ? v.y : row[xr];
          const float rs = fmaf(0.25f, left + right, 0.75f * (v.x + v.y));
          sum = fmaf(b == 0 || b == 3 ? 0.25f : 0.75f, rs, sum);
        }
        s[a] = sum;
      }
      const float v = fmaf(0.25f, s[0] + s[3], 0.75f * (s[1] + s[2]));
      cv.r[C] = l + 1 < h.nlev - 1 ? __ldg(cv.oinv + C) * v : v;
    }
    __syncthreads();
  }
  const MgLevel& last = h.lev[h.nlev - 1];
  for (int i0 = (tid >> 5) * 4; i0 < h.ncoarse; i0 += kMgTailThreads / 32 * 4)
    coarse_rows(last, h.pinv, h.ncoarse, i0, lane);
  __syncthreads();
  for (int l = h.nlev - 2; l >= 0; --l) {
    const MgLevel &f = h.lev[l], &cv = h.lev[l + 1];
    const int nx = f.nx, ny = f.ny, cx = cv.nx, cy = cv.ny, cz = cv.nz;
    for (int q = tid; q < (int)(f.n / 2); q += kMgTailThreads) {  // two cells of a row
      const int z = q / (cx * ny), y = (q - z * cx * ny) / cx, I = q - z * cx * ny - y * cx;
      const int K = z >> 1, Kn = z & 1 ? (K + 1 == cz ? 0 : K + 1) : (K == 0 ? cz - 1 : K - 1);
      const int J0 = y >> 1;
      const int Im = I == 0 ? (h.wall_x ? I : cx - 1) : I - 1, Ip = I + 1 == cx ? (h.wall_x ? I : 0) : I + 1;
      const int J1 = (y & 1) ? (J0 + 1 == cy ? 0 : J0 + 1) : (J0 == 0 ? cy - 1 : J0 - 1);
      auto L = [&](int k) {
        const float *p0 = cv.x + (k * cy + J0) * cx, *p1 = cv.x + (k * cy + J1) * cx;
        const float al = fmaf(0.75f, p0[I], 0.25f * p0[Im]), bl = fmaf(0.75f, p1[I], 0.25f * p1[Im]);
        const float ah = fmaf(0.75f, p0[I], 0.25f * p0[Ip]), bh = fmaf(0.75f, p1[I], 0.25f * p1[Ip]);
        return make_float2(fmaf(0.75f, al, 0.25f * bl), fmaf(0.75f, ah, 0.25f * bh));
      };
      const float2 Lc = L(K), Ln = L(Kn);
      const int c = (z * ny + y) * nx + 2 * I;
      const float2 r = *reinterpret_cast<const float2*>(f.r + c);
      const float2 om = __ldg(reinterpret_cast<const float2*>(f.om + c));
      *reinterpret_cast<float2*>(f.t + c) =
          make_float2(fmaf(w, r.x, om.x * fmaf(0.75f, Lc.x, 0.25f * Ln.x)),
                      fmaf(w, r.y, om.y * fmaf(0.75f, Lc.y, 0.25f * Ln.y)));
    }
    __syncthreads();
    for (int c = tid; c < (int)f.n; c += kMgTailThreads)
      f.x[c] = __ldg(f.oinv + c) * fmaf(1.f - w, f.t[c], w * neighbour_sum(f, f.t, c, f.r[c], true));
    __syncthreads();
  }
}

// First level of the tail, or 0: none.
int tail_level(const MgHier& h) {
  int l = h.nlev - 1;
  while (l > 1 && h.nlev - l < kMgTailLevels && h.lev[l - 1].n <= kMgTailCells) --l;
  return l < h.nlev - 1 ? l : 0;
}

// ---- set-up -------------------------------------------------------------------------------------

// level 0 from the FP64 face coefficients: the scaled coefficients bt = b sinv sinv_nb in FP32
__global__ void k_mg_level0(const double* __restrict__ bx, const double* __restrict__ by,
                            const double* __restrict__ bz, const double* __restrict__ sinv,
                            MgLevel lv) {
  const int nx = lv.nx, ny = lv.ny, nz = lv.nz;
  const long long plane = (long long)nx * ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < lv.n;
       c += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(c % nx), y = (int)((c / nx) % ny), z = (int)(c / plane);
    const long long xm = c - x + (x == 0 ? nx - 1 : x - 1);
    const long long ym = c + (long long)((y == 0 ? ny - 1 : y - 1) - y) * nx;
    const long long zm = c + (long long)((z == 0 ? nz - 1 : z - 1) - z) * plane;
    const double s = sinv[c];
    lv.bx[c] = (float)(bx[c] * s * sinv[xm]);
    lv.by[c] = (float)(by[c] * s * sinv[ym]);
    lv.bz[c] = (float)(bz[c] * s * sinv[zm]);
  }
}

// coarse faces: 1/2 x the sum of the four fine low faces under each coarse low face
template <class TB>
__global__ void k_mg_coarsen(const TB* __restrict__ fbx, const TB* __restrict__ fby,
                             const TB* __restrict__ fbz, int fnx, int fny, MgLevel cv) {
  for (long long C = blockIdx.x * (long long)blockDim.x + threadIdx.x; C < cv.n;
       C += (long long)gridDim.x * blockDim.x) {
    const int I = (int)(C % cv.nx), J = (int)((C / cv.nx) % cv.ny);
    const int K = (int)(C / ((long long)cv.nx * cv.ny));
    auto f = [&](int i, int j, int k) { return (long long)i + (long long)fnx * (j + (long long)fny * k); };
    const int i0 = 2 * I, j0 = 2 * J, k0 = 2 * K;
    const double sx = (double)fbx[f(i0, j0, k0)] + (double)fbx[f(i0, j0 + 1, k0)] +
                      (double)fbx[f(i0, j0, k0 + 1)] + (double)fbx[f(i0, j0 + 1, k0 + 1)];
    const double sy = (double)fby[f(i0, j0, k0)] + (double)fby[f(i0 + 1, j0, k0)] +
                      (double)fby[f(i0, j0, k0 + 1)] + (double)fby[f(i0 + 1, j0, k0 + 1)];
    const double sz = (double)fbz[f(i0, j0, k0)] + (double)fbz[f(i0 + 1, j0, k0)] +
                      (double)fbz[f(i0, j0 + 1, k0)] + (double)fbz[f(i0 + 1, j0 + 1, k0)];
    cv.bx[C] = (float)(0.5 * sx);
    cv.by[C] = (float)(0.5 * sy);
    cv.bz[C] = (float)(0.5 * sz);
  }
}

// W = D^1/2 and 1 / W of an (unscaled) coarse level
__global__ void k_mg_weights(MgLevel lv) {
  const int nx = lv.nx, ny = lv.ny, nz = lv.nz;
  const long long plane = (long long)nx * ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < lv.n;
       c += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(c % nx), y = (int)((c / nx) % ny), z = (int)(c / plane);
    const long long xp = c - x + (x == nx - 1 ? 0 : x + 1);
    const long long yp = c + (long long)((y == ny - 1 ? 0 : y + 1) - y) * nx;
    const long long zp = c + (long long)((z == nz - 1 ? 0 : z + 1) - z) * plane;
    const double D = (double)lv.bx[c] + lv.bx[xp] + lv.by[c] + lv.by[yp] + lv.bz[c] + lv.bz[zp];
    const double w = sqrt(D);
    lv.om[c] = (float)w;
    lv.oinv[c] = (float)(1.0 / w);
  }
}

// scale a coarse level's faces in place: bt = b oinv oinv_nb (after the next level was coarsened
// from the unscaled faces)
__global__ void k_mg_scale_faces(MgLevel lv) {
  const int nx = lv.nx, ny = lv.ny, nz = lv.nz;
  const long long plane = (long long)nx * ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < lv.n;
       c += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(c % nx), y = (int)((c / nx) % ny), z = (int)(c / plane);
    const long long xm = c - x + (x == 0 ? nx - 1 : x - 1);
    const long long ym = c + (long long)((y == 0 ? ny - 1 : y - 1) - y) * nx;
    const long long zm = c + (long long)((z == 0 ? nz - 1 : z - 1) - z) * plane;
    const float s = lv.oinv[c];
    lv.bx[c] = lv.bx[c] * s * lv.oinv[xm];
    lv.by[c] = lv.by[c] * s * lv.oinv[ym];
    lv.bz[c] = lv.bz[c] * s * lv.oinv[zm];
  }
}

// Pseudo-inverse of the singular SPD matrix -A of the coarsest level (n x n, null space: constants)
// in double: (-A)^+ = (-A + a J/n)^-1 - J / (a n), J the all-ones matrix, a > 0 (the mean diagonal).
//
// One cluster of 16 blocks inverts -A + a J/n in place by Gauss-Jordan elimination (positive
// definite: no pivoting).  The rows are dealt round robin (at most 32 x 512 doubles a block, 131 KB
// of shared memory); step k's owner publishes the scaled pivot row in its shared memory, the
// cluster barrier follows, and every block reads it from there.  The owner of the next pivot row
// updates that row first and publishes it before the others, so a step costs one barrier, one
// remote read and the longest of them.  It replaces a Cholesky inverse on the host (with copies
// both ways and two synchronisations): 160^3 (125 cells) 1.6 -> 0.2 ms of a density's set-up.
constexpr int kPinvBlocks = 16, kPinvThreads = 256;
constexpr int kPinvRows = (kMgMaxCoarsest + kPinvBlocks - 1) / kPinvBlocks;

__device__ __forceinline__ unsigned remote_smem(const void* p, unsigned block) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(block));
  return r;
}
__device__ __forceinline__ double load_remote(unsigned addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(kPinvThreads) k_mg_pinv(MgLevel lv, int n, float* __restrict__ pinv, int* bad) {
  extern __shared__ double rows[];  // this block's rows: rank, rank + 16, ...
  __shared__ double pivot[2][kMgMaxCoarsest];  // published pivot rows (even and odd steps)
  __shared__ double prow[kMgMaxCoarsest];
  __shared__ double total[kPinvThreads];
  const int rank = blockIdx.x, t = threadIdx.x;
  const int nr = (n - rank + kPinvBlocks - 1) / kPinvBlocks;  // (may be 0)
  const int nx = lv.nx, ny = lv.ny, nz = lv.nz;
  // neighbours and face coefficients of cell c: low and high x, y, z
  auto cell = [&](int c, int (&nb)[6], double (&w)[6]) {
    const int i = c % nx, j = c / nx % ny, k = c / (nx * ny);
    nb[0] = c - i + (i == 0 ? nx - 1 : i - 1);
    nb[1] = c - i + (i == nx - 1 ? 0 : i + 1);
    nb[2] = c + ((j == 0 ? ny - 1 : j - 1) - j) * nx;
    nb[3] = c + ((j == ny - 1 ? 0 : j + 1) - j) * nx;
    nb[4] = c + ((k == 0 ? nz - 1 : k - 1) - k) * nx * ny;
    nb[5] = c + ((k == nz - 1 ? 0 : k + 1) - k) * nx * ny;
    w[0] = lv.bx[c];
    w[1] = lv.bx[nb[1]];
    w[2] = lv.by[c];
    w[3] = lv.by[nb[3]];
    w[4] = lv.bz[c];
    w[5] = lv.bz[nb[5]];
  };
  double d = 0.0;  // sum of the diagonal (a face from a cell to itself cancels)
  for (int c = t; c < n; c += kPinvThreads) {
    int nb[6];
    double w[6];
    cell(c, nb, w);
    for (int q = 0; q < 6; ++q)
      if (nb[q] != c) d += w[q];
  }
  total[t] = d;
  __syncthreads();
  for (int s = kPinvThreads / 2; s > 0; s /= 2) {
    if (t < s) total[t] += total[t + s];
    __syncthreads();
  }
  const double a = total[0] > 0.0 ? total[0] / n : 1.0;
  for (int r = 0; r < nr; ++r)
    for (int j = t; j < n; j += kPinvThreads) rows[r * n + j] = a / n;
  __syncthreads();
  for (int r = t; r < nr; r += kPinvThreads) {
    const int c = rank + kPinvBlocks * r;
    int nb[6];
    double w[6];
    cell(c, nb, w);
    for (int q = 0; q < 6; ++q)
      if (nb[q] != c) {
        rows[r * n + c] += w[q];
        rows[r * n + nb[q]] -= w[q];
      }
  }
  __syncthreads();
  // the owner of row k scales and publishes it; every thread of that block calls it
  auto publish = [&](int k) {
    double* row = rows + k / kPinvBlocks * n;
    const double d = row[k], inv = quotient(1.0, d);
    if (t == 0 && !(d > 0.0 && isfinite(d))) *bad = 1;
    __syncthreads();
    for (int j = t; j < n; j += kPinvThreads) {
      const double v = j == k ? inv : row[j] * inv;
      row[j] = v;
      pivot[k & 1][j] = v;
    }
  };
  auto eliminate = [&](int r, int k) {  // row r of this block with pivot row k (in prow)
    double* row = rows + r * n;
    const double f = row[k];
    __syncthreads();
    for (int j = t; j < n; j += kPinvThreads) row[j] = j == k ? -f * prow[j] : fma(-f, prow[j], row[j]);
  };
  if (rank == 0) publish(0);
  cluster_arrive();
  for (int k = 0; k < n; ++k) {
    cluster_wait();  // row k is published; everyone has read row k - 1
    const unsigned src = remote_smem(pivot[k & 1], k % kPinvBlocks);
    for (int j = t; j < n; j += kPinvThreads) prow[j] = load_remote(src + 8u * j);
    __syncthreads();
    const int next = k + 1;
    const bool mine = next < n && next % kPinvBlocks == rank;
    if (mine) {
      eliminate(next / kPinvBlocks, k);
      __syncthreads();
      publish(next);
    }
    cluster_arrive();
    // the other rows: a warp each, so that no barrier separates them
    for (int r = t / 32; r < nr; r += kPinvThreads / 32) {
      const int i = rank + kPinvBlocks * r;
      if (i == k || (mine && i == next)) continue;
      double* row = rows + r * n;
      const double f = row[k];
      __syncwarp();
      for (int j = t & 31; j < n; j += 32) row[j] = j == k ? -f * prow[j] : fma(-f, prow[j], row[j]);
    }
    __syncthreads();  // prow is reused
  }
  cluster_wait();  // no block leaves while its pivot rows may still be read
  for (int r = 0; r < nr; ++r)
    for (int j = t; j < n; j += kPinvThreads)
      pinv[(long long)(rank + kPinvBlocks * r) * n + j] = (float)(rows[r * n + j] - 1.0 / (a * n));
}

cudaError_t launch_pinv(const MgLevel& lv, int n, float* pinv, int* bad, cudaStream_t s) {
  const size_t smem = sizeof(double) * (size_t)((n + kPinvBlocks - 1) / kPinvBlocks) * n;
  // (per call: the limits belong to the current device's copy of the kernel)
  cudaError_t e = cudaFuncSetAttribute(k_mg_pinv, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mg_pinv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(double) * kPinvRows * kMgMaxCoarsest));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kPinvBlocks);
  cfg.blockDim = dim3(kPinvThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kPinvBlocks;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mg_pinv, lv, n, pinv, bad);
}

// out = in rounded to FP32 (the FP64 solve's scaled residual, read by the level-0 sweeps)
__global__ void k_mg_narrow(const double* __restrict__ in, long long n, float* __restrict__ out,
                            const InstState* st) {
  if (!mg_active(st)) return;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x)
    out[c] = narrow(in[c]);
}

// out = in * sinv (between the unscaled and the scaled variables of level 0)
__global__ void k_mg_scale(const double* __restrict__ in, const double* __restrict__ sinv,
                           long long n, double* __restrict__ out) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x)
    out[c] = in[c] * sinv[c];
}

int flat_grid(long long n) {
  long long b = (n + kMgThreads - 1) / kMgThreads;
  if (b > 152 * 8) b = 152 * 8;
  return (int)(b < 1 ? 1 : b);
}

template <class K>
int cached_resident(K kernel, int* cache) {
  if (*cache <= 0) *cache = resident_blocks(kernel);
  return *cache;
}

}  // namespace

int mg_level_dims(int nx, int ny, int nz, int (*dims)[3]) {
  int n = 0;
  int x = nx, y = ny, z = nz;
  for (;;) {
    dims[n][0] = x;
    dims[n][1] = y;
    dims[n][2] = z;
    ++n;
    if (x % 2 || y % 2 || z % 2 || (long long)x * y * z <= kMgMinCoarsen || n == kMgMaxLevels) break;
    x /= 2;
    y /= 2;
    z /= 2;
  }
  // at least one coarser level (a grid of at most 64 cells is not a multigrid problem)
  return n >= 2 && (long long)x * y * z <= kMgMaxCoarsest ? n : 0;
}

size_t mg_bytes(int nx, int ny, int nz) {
  int d[kMgMaxLevels][3];
  const int L = mg_level_dims(nx, ny, nz, d);
  if (!L) return 0;
  size_t cells = 0;
  for (int l = 0; l < L; ++l) cells += (size_t)(l == 0 ? 5 : 8) * d[l][0] * d[l][1] * d[l][2];
  const size_t nc = (size_t)d[L - 1][0] * d[L - 1][1] * d[L - 1][2];
  return sizeof(float) * (cells + nc * nc) + 64 * (size_t)(8 * L + 1);
}

cudaError_t mg_alloc(MgHier* h, int nx, int ny, int nz, int wall_x) {
  int d[kMgMaxLevels][3];
  const int L = mg_level_dims(nx, ny, nz, d);
  if (!L) return cudaErrorInvalidValue;
  const size_t bytes = mg_bytes(nx, ny, nz);
  void* mem = nullptr;
  cudaError_t e = cudaMalloc(&mem, bytes);
  if (e != cudaSuccess) return e;
  char* p = static_cast<char*>(mem);
  auto take = [&](size_t count) {
    float* q = reinterpret_cast<float*>(p);
    p += ((sizeof(float) * count + 63) / 64) * 64;  // 64-byte aligned arrays
    return q;
  };
  MgHier hh;
  hh.nlev = L;
  hh.wall_x = wall_x;
  for (int l = 0; l < L; ++l) {
    MgLevel& v = hh.lev[l];
    v.nx = d[l][0];
    v.ny = d[l][1];
    v.nz = d[l][2];
    v.n = (long long)v.nx * v.ny * v.nz;
    v.bx = take(v.n);
    v.by = take(v.n);
    v.bz = take(v.n);
    v.om = l ? take(v.n) : nullptr;  // level 0 uses the solve's W
    v.oinv = l ? take(v.n) : nullptr;
    v.t = take(v.n);
    v.r = take(v.n);  // level 0: the FP32 copy of an FP64 right side
    v.x = l ? take(v.n) : nullptr;
  }
  hh.ncoarse = (int)hh.lev[L - 1].n;
  hh.pinv = take((size_t)hh.ncoarse * hh.ncoarse);
  hh.bad = reinterpret_cast<int*>(take(1));
  hh.mem = mem;
  hh.bytes = bytes;
  *h = hh;
  return cudaSuccess;
}

void mg_free(MgHier* h) {
  if (h->mem) cudaFree(h->mem);
  *h = MgHier();
}

cudaError_t mg_setup(MgHier* h, const double* bx, const double* by, const double* bz,
                     const double* sinv, cudaStream_t s) {
  if (!h->mem) return cudaErrorInvalidValue;
  const MgLevel& l0 = h->lev[0];
  k_mg_level0<<<flat_grid(l0.n), kMgThreads, 0, s>>>(bx, by, bz, sinv, l0);
  for (int l = 1; l < h->nlev; ++l) {
    const MgLevel& f = h->lev[l - 1];
    const MgLevel& c = h->lev[l];
    if (l == 1)  // from the FP64 coefficients
      k_mg_coarsen<double><<<flat_grid(c.n), kMgThreads, 0, s>>>(bx, by, bz, f.nx, f.ny, c);
    else
      k_mg_coarsen<float><<<flat_grid(c.n), kMgThreads, 0, s>>>(f.bx, f.by, f.bz, f.nx, f.ny, c);
    if (l >= 2)  // level l - 1 has been coarsened from: scale it now (the coarsest stays unscaled)
      k_mg_scale_faces<<<flat_grid(f.n), kMgThreads, 0, s>>>(f);
    if (l < h->nlev - 1) k_mg_weights<<<flat_grid(c.n), kMgThreads, 0, s>>>(c);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const cudaError_t e2 = cudaMemsetAsync(h->bad, 0, sizeof(int), s);
  if (e2 != cudaSuccess) return e2;
  return launch_pinv(h->lev[h->nlev - 1], h->ncoarse, h->pinv, h->bad, s);
}

int mg_launches(const MgHier& h, int prec) {
  const int tail = tail_level(h);
  return 4 * (tail ? tail : h.nlev - 1) + 1 + (prec == PREC_FP64);
}

// One V-cycle; T is the type of the solve's rt and z.  An FP64 rt is rounded to FP32 once (into
// level 0's r), so the level-0 sweeps read FP32 only.
template <class T>
static cudaError_t vcycle(const MgHier& h, const MgArgs& a, cudaStream_t s) {
  static int r_down = 0, r_up0 = 0, r_up = 0, r_pro = 0, r_res = 0;
  const int L = h.nlev;
  if (L < 2 || !a.omega) return cudaErrorInvalidValue;
  const float* in;
  if constexpr (sizeof(T) == 8) {
    k_mg_narrow<<<flat_grid(h.lev[0].n), kMgThreads, 0, s>>>(static_cast<const double*>(a.in),
                                                             h.lev[0].n, h.lev[0].r, a.st);
    in = h.lev[0].r;
  } else {
    in = static_cast<const float*>(a.in);
  }
  T* out = static_cast<T*>(a.out);
  auto rhs = [&](int l) { return l == 0 ? in : static_cast<const float*>(h.lev[l].r); };
  auto wgt = [&](int l) { return l == 0 ? a.omega : static_cast<const float*>(h.lev[l].om); };
  const int tail = tail_level(h), top = tail ? tail : L - 1;  // levels 0 .. top - 1 by launches of their own
  for (int l = 0; l < top; ++l) {
    const MgLevel& v = h.lev[l];
    const MgLevel& cv = h.lev[l + 1];
    const MarchPlan m = march_plan(v.nx, v.ny, v.nz, cached_resident(k_mg_down0<float>, &r_down));
    k_mg_down0<float><<<m.blocks, kMgThreads, 0, s>>>(v, m, rhs(l), wgt(l), a.st);
    const MarchPlan mr = march_plan(cv.nx, cv.ny, cv.nz, cached_resident(k_mg_restrict, &r_res));
    k_mg_restrict<<<mr.blocks, kMgThreads, 0, s>>>(v, cv, mr, l + 1 < L - 1 ? cv.oinv : nullptr,
                                                   h.wall_x, a.st);
  }
  if (tail) {
    MgTail t = {};
    for (int l = tail; l < L; ++l) t.lev[l - tail] = h.lev[l];
    t.nlev = L - tail;
    t.pinv = h.pinv;
    t.ncoarse = h.ncoarse;
    t.wall_x = h.wall_x;
    k_mg_tail<<<1, kMgTailThreads, 0, s>>>(t, a.st);
  } else {
    k_mg_coarse<<<(h.ncoarse + kCoarseRows - 1) / kCoarseRows, kMgThreads, 0, s>>>(h.lev[L - 1], h.pinv,
                                                                                   h.ncoarse, a.st);
  }
  for (int l = top - 1; l >= 0; --l) {
    const MgLevel& v = h.lev[l];
    const MgLevel& cv = h.lev[l + 1];
    const MarchPlan mp = march_plan(cv.nx, v.ny, cv.nz, cached_resident(k_mg_prolong, &r_pro));
    k_mg_prolong<<<mp.blocks, kMgThreads, 0, s>>>(v, h.lev[l + 1], mp, rhs(l), wgt(l),
                                                         h.wall_x, a.st);
    if (l == 0) {
      const MarchPlan m = march_plan(v.nx, v.ny, v.nz, cached_resident(k_mg_up<float, T, false>, &r_up0));
      k_mg_up<float, T, false><<<m.blocks, kMgThreads, 0, s>>>(v, m, in, out, a.st, a.I);
    } else {
      const MarchPlan m = march_plan(v.nx, v.ny, v.nz, cached_resident(k_mg_up<float, float, true>, &r_up));
      k_mg_up<float, float, true><<<m.blocks, kMgThreads, 0, s>>>(v, m, rhs(l), nullptr, a.st, a.I);
    }
  }
  return cudaGetLastError();
}

cudaError_t launch_mg_scale(const double* in, const double* sinv, long long n, double* out,
                            cudaStream_t s) {
  k_mg_scale<<<flat_grid(n), kMgThreads, 0, s>>>(in, sinv, n, out);
  return cudaGetLastError();
}

cudaError_t launch_mg_vcycle(const MgHier& h, int prec, const MgArgs& a, cudaStream_t s) {
  if (!h.mem) return cudaErrorInvalidValue;
  return prec == PREC_FP64 ? vcycle<double>(h, a, s) : vcycle<float>(h, a, s);
}

}  // namespace vdp
