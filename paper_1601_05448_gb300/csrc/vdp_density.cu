// vdp_density.cu -- the density form of the inner iteration, used with the constant-coefficient
// inverse (the paper's fixed-point iteration and spectrally preconditioned CG).
//
// The Jacobi-scaled form of vdp_kernels.cu exists for preconditioners that need a unit diagonal.
// The spectral inverse does not: in unscaled variables its passes need no weights, and the
// operator's three face coefficients per cell are functions of one field, the density, so a sweep
// that reads rho (4 bytes, the neighbours' values from L1 / L2) computes them.  With
//     rho' = rho / 2^e0 (FP32; e0 the exponent of the first cell),  kappa = 2^e0 hx^2,
//     A' = kappa A:  face values 2 / (rho'_l + rho'_r) x (hx / h_d)^2,
// an inner solve of (-A') X = r gives the correction p -= kappa X, whatever the units of rho and
// of the box.  Per cell and iteration of the FP32 fixed-point solve this moves
//     X+  g 4            (weights and rt: 8)        X-  z 4            (z and weight: 8)
//     sweep  z, rho', g, X read, g, X written: 24   (z, three coefficients, rt, x: 32)
// besides the half spectrum: 32 bytes instead of 48.  Fixed point: g = rho' r is the stored
// residual (the right side of the paper's L_h dp = rho r), so X+ reads one field.
//
// The sweep is bound by HBM on grids beyond L2: 4.25 reciprocals (approximation instruction and a
// Newton step, relative error of the FP32 rounding) and about 50 FP32 operations per cell take a
// third of the time its 24 bytes take.  The march is that of sweep_stencil_direct: a thread owns
// 16 bytes of one row, three planes of z and two of rho' in registers, x neighbours by shuffle.
#include "vdp_device.cuh"
#include "vdp_internal.cuh"
#include "vdp_launch.h"

namespace vdp {

namespace {

constexpr int kV = 4;  // cells per thread

__device__ __forceinline__ void ld4(const float* p, float (&o)[kV]) {
  const float4 t = __ldg(reinterpret_cast<const float4*>(p));
  o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
}
__device__ __forceinline__ void ld4rw(const float* p, float (&o)[kV]) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
}
__device__ __forceinline__ void st4(float* p, const float (&v)[kV]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// c / (a + b): the approximate reciprocal and one Newton step.  Symmetric in a and b, so the two
// cells of a face compute the same value.
__device__ __forceinline__ float face(float c, float a, float b) {
  const float s = a + b, y = rcp_approx(s);
  return c * fmaf(y, fmaf(-s, y, 1.f), y);
}

// KIND 0: the fixed-point iteration, z = damping (-L')^-1 g: X += z, g -= rho' (-A') z and the sum
// of r^2 / D' (the norm of the scaled residual, which steers the inner stop).
// KIND 1, 2: CG, d = z + beta d_old (1: first iteration, d = z), q = (-A') d and the sum of d q.
template <int KIND>
__device__ __forceinline__ void sweep_density(const InstDesc& I, const InstState* st, int unit,
                                              float& part) {
  constexpr bool kFixed = KIND == 0, kOld = KIND == 2;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int tpr = nx / kV;
  const int tile = unit % I.uy, chunk = unit / I.uy;
  const int row = threadIdx.x / tpr;
  const int x0 = (threadIdx.x - row * tpr) * kV;
  const int yr = tile * I.ty + row;
  const bool active = row < I.ty && yr < ny;
  const int y = active ? yr : ny - 1;  // idle threads follow a valid row (shuffles need them)
  const int z0 = (int)((long long)chunk * nz / I.zc), z1 = (int)((long long)(chunk + 1) * nz / I.zc);
  const int lane = threadIdx.x & 31;
  const bool row_start = x0 == 0, row_end = x0 + kV == nx;
  const bool left_load = lane == 0 || row_start, right_load = lane == 31 || row_end;
  const bool wall_l = I.duct && row_start, wall_r = I.duct && row_end;
  const float cx = 2.f, cy = I.cy, cz = I.cz;
  const float beta = (float)st->beta;
  const bool first = st->inner_iters == 0;
  const float* rho = I.rho32;
  const float* src = static_cast<const float*>(I.za);
  const float* dold = static_cast<const float*>(st->parity ? I.d1 : I.d0);
  float* dnew = static_cast<float*>(st->parity ? I.d0 : I.d1);
  float* q = static_cast<float*>(I.q);
  float* g = static_cast<float*>(I.r);
  float* X = static_cast<float*>(I.x);
  const long long plane = (long long)nx * ny;
  const long long dym = y == 0 ? (long long)(ny - 1) * nx : -(long long)nx;
  const long long dyp = y == ny - 1 ? -(long long)(ny - 1) * nx : (long long)nx;
  const int dxl = row_start ? nx - 1 : -1, dxr = row_end ? -x0 : kV;
  const long long cell0 = (long long)y * nx + x0;
  auto zoff = [&](int z) -> long long {
    return (long long)(z < 0 ? z + nz : (z >= nz ? z - nz : z)) * plane + cell0;
  };
  auto field = [&](long long o, float (&d)[kV]) {  // the marched field
    ld4(src + o, d);
    if (kOld) {
      float b[kV];
      ld4(dold + o, b);
#pragma unroll
      for (int k = 0; k < kV; ++k) d[k] = fmaf(beta, b[k], d[k]);
    }
  };
  auto field1 = [&](long long o) -> float {
    return kOld ? fmaf(beta, __ldg(dold + o), __ldg(src + o)) : __ldg(src + o);
  };
  float um[kV], uc[kV], rc[kV], bzl[kV], sum[kV];
#pragma unroll
  for (int k = 0; k < kV; ++k) sum[k] = 0.f;
  if (z0 < z1) {
    float rm[kV];
    field(zoff(z0 - 1), um);
    field(zoff(z0), uc);
    ld4(rho + zoff(z0 - 1), rm);
    ld4(rho + zoff(z0), rc);
#pragma unroll
    for (int k = 0; k < kV; ++k) bzl[k] = face(cz, rm[k], rc[k]);
  }
  for (int z = z0; z < z1; ++z) {
    const long long o = zoff(z), op = zoff(z + 1);
    float up[kV], rp[kV], ua[kV], ub[kV], ra[kV], rb[kV], gv[kV], xv[kV];
    field(op, up);
    ld4(rho + op, rp);
    field(o + dym, ua);
    field(o + dyp, ub);
    ld4(rho + o + dym, ra);
    ld4(rho + o + dyp, rb);
    if (kFixed) {
      ld4rw(g + o, gv);  // rewritten by this thread only
      if (first) {
#pragma unroll
        for (int k = 0; k < kV; ++k) xv[k] = 0.f;
      } else {
        ld4rw(X + o, xv);
      }
    }
    float ul = __shfl_up_sync(0xffffffffu, uc[kV - 1], 1), ur = __shfl_down_sync(0xffffffffu, uc[0], 1);
    float rl = __shfl_up_sync(0xffffffffu, rc[kV - 1], 1), rr = __shfl_down_sync(0xffffffffu, rc[0], 1);
    if (left_load) {
      ul = field1(o + dxl);
      rl = __ldg(rho + o + dxl);
    }
    if (right_load) {
      ur = field1(o + dxr);
      rr = __ldg(rho + o + dxr);
    }
    float bl = wall_l ? 0.f : face(cx, rl, rc[0]);
    float au[kV];
#pragma unroll
    for (int k = 0; k < kV; ++k) {
      const bool end = k == kV - 1;
      const float u = uc[k];
      const float br = end && wall_r ? 0.f : face(cx, rc[k], end ? rr : rc[k + 1]);
      const float ba = face(cy, ra[k], rc[k]), bb = face(cy, rc[k], rb[k]);
      const float bz = face(cz, rc[k], rp[k]);
      float a = bl * (u - (k == 0 ? ul : uc[k - 1]));  // differences: a constant field gives 0
      a = fmaf(br, u - (end ? ur : uc[k + 1]), a);
      a = fmaf(ba, u - ua[k], a);
      a = fmaf(bb, u - ub[k], a);
      a = fmaf(bzl[k], u - um[k], a);
      a = fmaf(bz, u - up[k], a);
      if (kFixed) {
        const float D = ((bl + br) + (ba + bb)) + (bzl[k] + bz);
        gv[k] = fmaf(-rc[k], a, gv[k]);
        xv[k] += u;
        const float r = gv[k] * rcp_approx(rc[k]);
        sum[k] = fmaf(r * rcp_approx(D), r, sum[k]);
      } else {
        au[k] = a;
        sum[k] = fmaf(u, a, sum[k]);
      }
      bl = br;
      bzl[k] = bz;
    }
    if (active) {
      if (kFixed) {
        st4(g + o, gv);
        st4(X + o, xv);
      } else {
        st4(dnew + o, uc);
        st4(q + o, au);
      }
    }
#pragma unroll
    for (int k = 0; k < kV; ++k) {
      um[k] = uc[k];
      uc[k] = up[k];
      rc[k] = rp[k];
    }
  }
  part = active ? (sum[0] + sum[1]) + (sum[2] + sum[3]) : 0.f;
}

}  // namespace

// STENCIL phase of the instances in the density form: FIXED the fixed-point iteration, else CG.
template <bool FIXED>
__global__ void __launch_bounds__(kDirectThreads, 3)
    k_density(const InstDesc* __restrict__ insts, const UnitRef* __restrict__ units) {
  const UnitRef ur = units[blockIdx.x];
  const InstDesc& I = insts[ur.inst];
  InstState* st = I.st;
  if (__ldcg(&st->phase) != PH_STENCIL || I.form == 0 || (I.pc == PC_FIXED) != FIXED) return;
  const InstState sn = snapshot(st);
  float part[1] = {0.f};
  if constexpr (FIXED) {
    sweep_density<0>(I, &sn, ur.unit, part[0]);
  } else {
    if (sn.inner_iters > 0)
      sweep_density<2>(I, &sn, ur.unit, part[0]);
    else
      sweep_density<1>(I, &sn, ur.unit, part[0]);
  }
  store_partials<1, float>(part, I.part, I.nunits, ur.unit);
  finish_sweep(I, st, PH_STENCIL, I.nunits);
}

cudaError_t launch_density(int kind, const InstDesc* desc, const UnitRef* units, int nunits,
                           int threads, cudaStream_t s) {
  if (kind == kSweepDensityFixed)
    k_density<true><<<nunits, threads, 0, s>>>(desc, units);
  else
    k_density<false><<<nunits, threads, 0, s>>>(desc, units);
  return cudaGetLastError();
}

}  // namespace vdp
