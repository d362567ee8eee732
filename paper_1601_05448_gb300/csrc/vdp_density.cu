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
// The march is that of sweep_stencil_direct: a thread owns 16 bytes of one row and walks a z chunk,
// x neighbours come by shuffle, the rows above and below and the plane above by loads.  Written
// with plain loads the sweep waited for memory (ncu at 256^3: 8.2 of 13 stall cycles per issue on
// long-scoreboard, 47 % of the DRAM rate): each thread therefore fetches its operands of the next
// plane by cp.async into slots of shared memory that only it reads, so no barrier is needed, no
// registers are held while they fly, and the arithmetic of one plane covers the latency of the
// next.  Sums, products and Newton steps of the four cells run as paired FP32 instructions, and
// the fluxes through the x faces and the upper z face are computed once for both cells.
#include "vdp_device.cuh"
#include "vdp_internal.cuh"
#include "vdp_launch.h"

namespace vdp {

namespace {

constexpr int kV = 4;       // cells per thread
constexpr int kStages = 2;  // planes of operands in flight or in use

using f2 = unsigned long long;  // two FP32 values

__device__ __forceinline__ f2 pk(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 up2(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// c / (a + b) of a face: the approximate reciprocal and one Newton step (nc = -c; the reciprocal of
// the negated sum leaves the residual 1 - s y as one FMA).  Symmetric in a and b, so the two cells
// of a face compute the same value, and each lane of the paired form the scalar form's.
__device__ __forceinline__ float face(float nc, float a, float b) {
  const float s = a + b, y = rcp_approx(-s);
  const float w = nc * y;
  return fmaf(w, fmaf(s, y, 1.f), w);
}
__device__ __forceinline__ f2 face2(f2 nc, f2 a, f2 b) {
  const f2 s = add2(a, b);
  const float2 v = up2(s);
  const f2 y = pk(rcp_approx(-v.x), rcp_approx(-v.y));
  const f2 w = mul2(nc, y);
  return fma2(w, fma2(s, y, pk(1.f, 1.f)), w);
}

__device__ __forceinline__ void fetch16(void* smem, const float* g) {  // through L1
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(smem)),
               "l"(g)
               : "memory");
}
__device__ __forceinline__ void fetch16_once(void* smem, const float* g) {  // L2 only
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(smem)),
               "l"(g)
               : "memory");
}
__device__ __forceinline__ void fetch_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// this thread's own copies: all but the newest group have landed
__device__ __forceinline__ void fetch_wait_previous() {
  asm volatile("cp.async.wait_group 1;" ::: "memory");
}

// Operand streams of a plane z (16 bytes per thread each): z+1 and the rows above and below of the
// marched field and of the density, then what the kind needs besides.
enum Stream { S_UP, S_UA, S_UB, S_RP, S_RA, S_RB, S_0, S_1, S_2 };
template <int KIND> struct Streams { static constexpr int kCount = KIND == 0 ? 8 : (KIND == 1 ? 6 : 9); };

// KIND 0: the fixed-point iteration, z = damping (-L')^-1 g: X += z, g -= rho' (-A') z and the sum
// of r^2 / D' (the norm of the scaled residual, which steers the inner stop).
// KIND 1, 2: CG, d = z + beta d_old (1: first iteration, d = z), q = (-A') d and the sum of d q.
template <int KIND>
__device__ __forceinline__ void sweep_density(const InstDesc& I, const InstState* st, int unit,
                                              float& part, ulonglong2* slots) {
  constexpr bool kFixed = KIND == 0, kOld = KIND == 2;
  constexpr int NS = Streams<KIND>::kCount;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int tpr = nx / kV;
  const int tile = unit % I.uy, chunk = unit / I.uy;
  const int row = threadIdx.x / tpr;
  const int x0 = (threadIdx.x - row * tpr) * kV;
  const int yr = tile * I.ty + row;
  const bool active = row < I.ty && yr < ny;
  const int y = active ? yr : ny - 1;  // idle threads follow a valid row (shuffles need them)
  const int z0 = (int)((long long)chunk * nz / I.zc), z1 = (int)((long long)(chunk + 1) * nz / I.zc);
  part = 0.f;
  if (z0 >= z1) return;
  const int lane = threadIdx.x & 31;
  const bool row_start = x0 == 0, row_end = x0 + kV == nx;
  const bool left_load = lane == 0 || row_start, right_load = lane == 31 || row_end;
  const bool wall_l = I.duct && row_start, wall_r = I.duct && row_end;
  const f2 ny2 = pk(-I.cy, -I.cy), nz2 = pk(-I.cz, -I.cz);
  const float beta = (float)st->beta;
  const f2 beta2 = pk(beta, beta);
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
  const long long dz_last = plane * (nz - 1);  // from plane nz - 1 back to plane 0
  // stream k of stage b of this thread
  auto slot = [&](int b, int k) { return slots + (b * NS + k) * blockDim.x + threadIdx.x; };
  auto fetch = [&](int b, int z, long long o) {  // the operands of plane z (cells at o)
    const long long op = z == nz - 1 ? o - dz_last : o + plane;
    fetch16(slot(b, S_UP), src + op);
    fetch16(slot(b, S_UA), src + o + dym);
    fetch16(slot(b, S_UB), src + o + dyp);
    fetch16(slot(b, S_RP), rho + op);
    fetch16(slot(b, S_RA), rho + o + dym);
    fetch16(slot(b, S_RB), rho + o + dyp);
    if (kFixed) {  // rewritten by this thread only, after this plane's copies have landed
      fetch16_once(slot(b, S_0), g + o);
      if (!first) fetch16_once(slot(b, S_1), X + o);
    }
    if (kOld) {
      fetch16(slot(b, S_0), dold + op);
      fetch16(slot(b, S_1), dold + o + dym);
      fetch16(slot(b, S_2), dold + o + dyp);
    }
  };
  auto ldg2 = [](const float* p, f2& a, f2& b) {
    const ulonglong2 t = __ldg(reinterpret_cast<const ulonglong2*>(p));
    a = t.x;
    b = t.y;
  };
  auto field1 = [&](long long o) -> float {
    return kOld ? fmaf(beta, __ldg(dold + o), __ldg(src + o)) : __ldg(src + o);
  };
  long long o = (long long)z0 * plane + cell0;
  fetch(0, z0, o);
  fetch_commit();
  // the field and the density of planes z0 - 1 and z0; the flux through the face between them
  f2 u[2], r[2], bzl[2], fz[2];
  {
    const long long om = z0 == 0 ? o + dz_last : o - plane;
    f2 um[2], rm[2];
    ldg2(src + om, um[0], um[1]);
    ldg2(src + o, u[0], u[1]);
    ldg2(rho + om, rm[0], rm[1]);
    ldg2(rho + o, r[0], r[1]);
    if (kOld) {
      f2 dm[2], dc[2];
      ldg2(dold + om, dm[0], dm[1]);
      ldg2(dold + o, dc[0], dc[1]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        um[h] = fma2(beta2, dm[h], um[h]);
        u[h] = fma2(beta2, dc[h], u[h]);
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      bzl[h] = face2(nz2, rm[h], r[h]);
      fz[h] = mul2(bzl[h], sub2(u[h], um[h]));
    }
  }
  f2 sum[2] = {0ull, 0ull};
  int b = 0;
  for (int z = z0; z < z1; ++z) {
    if (z + 1 < z1) fetch(b ^ 1, z + 1, o + plane);
    fetch_commit();
    // x neighbours: adjacent lanes, or a load at row ends and warp ends
    const float2 u01 = up2(u[0]), u23 = up2(u[1]), r01 = up2(r[0]), r23 = up2(r[1]);
    float ul = __shfl_up_sync(0xffffffffu, u23.y, 1), ur = __shfl_down_sync(0xffffffffu, u01.x, 1);
    float rl = __shfl_up_sync(0xffffffffu, r23.y, 1), rr = __shfl_down_sync(0xffffffffu, r01.x, 1);
    if (left_load) {
      ul = field1(o + dxl);
      rl = __ldg(rho + o + dxl);
    }
    if (right_load) {
      ur = field1(o + dxr);
      rr = __ldg(rho + o + dxr);
    }
    // faces and fluxes b (u_k - u_{k-1}) through the five x faces of the four cells
    const float b0 = wall_l ? 0.f : face(-2.f, rl, r01.x), b1 = face(-2.f, r01.x, r01.y);
    const float b2 = face(-2.f, r01.y, r23.x), b3 = face(-2.f, r23.x, r23.y);
    const float b4 = wall_r ? 0.f : face(-2.f, r23.y, rr);
    const float f0 = b0 * (u01.x - ul), f1 = b1 * (u01.y - u01.x), fm = b2 * (u23.x - u01.y);
    const float f3 = b3 * (u23.y - u23.x), f4 = b4 * (ur - u23.y);
    f2 a[2] = {pk(f1 - f0, fm - f1), pk(f3 - fm, f4 - f3)};  // A' u, accumulated
    f2 D[2] = {pk(b0 + b1, b1 + b2), pk(b2 + b3, b3 + b4)};
    fetch_wait_previous();
    ulonglong2 t = *slot(b, S_UP);
    f2 un[2] = {t.x, t.y};
    if (kOld) {
      t = *slot(b, S_0);
      un[0] = fma2(beta2, t.x, un[0]);
      un[1] = fma2(beta2, t.y, un[1]);
    }
    t = *slot(b, S_RP);
    const f2 rn[2] = {t.x, t.y};
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // upper z face: its flux is the next plane's lower one
      const f2 bz = face2(nz2, r[h], rn[h]);
      const f2 f = mul2(bz, sub2(un[h], u[h]));
      a[h] = add2(a[h], sub2(f, fz[h]));
      fz[h] = f;
      if (kFixed) D[h] = add2(D[h], add2(bzl[h], bz));
      bzl[h] = bz;
    }
#pragma unroll
    for (int side = 0; side < 2; ++side) {  // the rows above and below
      t = *slot(b, side ? S_UB : S_UA);
      f2 v[2] = {t.x, t.y};
      if (kOld) {
        t = *slot(b, side ? S_2 : S_1);
        v[0] = fma2(beta2, t.x, v[0]);
        v[1] = fma2(beta2, t.y, v[1]);
      }
      t = *slot(b, side ? S_RB : S_RA);
      const f2 rv[2] = {t.x, t.y};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const f2 by = face2(ny2, rv[h], r[h]);
        a[h] = fma2(by, sub2(v[h], u[h]), a[h]);
        if (kFixed) D[h] = add2(D[h], by);
      }
    }
    if constexpr (kFixed) {
      t = *slot(b, S_0);
      f2 gv[2] = {t.x, t.y}, xv[2] = {u[0], u[1]};
      if (!first) {
        t = *slot(b, S_1);
        xv[0] = add2(t.x, u[0]);
        xv[1] = add2(t.y, u[1]);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        gv[h] = fma2(r[h], a[h], gv[h]);
        const float2 d = up2(D[h]), rv = up2(r[h]);
        const f2 w = mul2(gv[h], pk(rcp_approx(rv.x), rcp_approx(rv.y)));
        sum[h] = fma2(mul2(w, w), pk(rcp_approx(d.x), rcp_approx(d.y)), sum[h]);
      }
      if (active) {
        *reinterpret_cast<ulonglong2*>(g + o) = make_ulonglong2(gv[0], gv[1]);
        *reinterpret_cast<ulonglong2*>(X + o) = make_ulonglong2(xv[0], xv[1]);
      }
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        a[h] = sub2(0ull, a[h]);
        sum[h] = fma2(u[h], a[h], sum[h]);
      }
      if (active) {
        *reinterpret_cast<ulonglong2*>(dnew + o) = make_ulonglong2(u[0], u[1]);
        *reinterpret_cast<ulonglong2*>(q + o) = make_ulonglong2(a[0], a[1]);
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      u[h] = un[h];
      r[h] = rn[h];
    }
    o += plane;
    b ^= 1;
  }
  const float2 s = up2(add2(sum[0], sum[1]));
  part = active ? s.x + s.y : 0.f;
}

size_t density_smem(bool fixed, int threads) {
  const int streams = fixed ? Streams<0>::kCount : Streams<2>::kCount;
  return sizeof(ulonglong2) * (size_t)kStages * streams * threads;
}

}  // namespace

// STENCIL phase of the instances in the density form: FIXED the fixed-point iteration, else CG.
template <bool FIXED>
// Two blocks per SM: with three the slots leave so little L1 that every neighbour row comes from L2
// (512^3: 715 us against 550, 256^3: 113 against 94; plain loads at three blocks: 595 and 103).
__global__ void __launch_bounds__(kDirectThreads, 2)
    k_density(const InstDesc* __restrict__ insts, const UnitRef* __restrict__ units) {
  extern __shared__ __align__(16) ulonglong2 slots[];
  const UnitRef ur = units[blockIdx.x];
  const InstDesc& I = insts[ur.inst];
  InstState* st = I.st;
  const InstState& sn = block_state(st);
  if (sn.phase != PH_STENCIL || I.form == 0 || (I.pc == PC_FIXED) != FIXED) return;
  float part[1] = {0.f};
  if constexpr (FIXED) {
    sweep_density<0>(I, &sn, ur.unit, part[0], slots);
  } else {
    if (sn.inner_iters > 0)
      sweep_density<2>(I, &sn, ur.unit, part[0], slots);
    else
      sweep_density<1>(I, &sn, ur.unit, part[0], slots);
  }
  store_partials<1, float>(part, I.part, I.nunits, ur.unit);
  finish_sweep(I, st, PH_STENCIL, I.nunits);
}

cudaError_t prepare_density() {
  const cudaError_t e = cudaFuncSetAttribute(k_density<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)density_smem(true, kDirectThreads));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_density<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)density_smem(false, kDirectThreads));
}

cudaError_t launch_density(int kind, const InstDesc* desc, const UnitRef* units, int nunits,
                           int threads, cudaStream_t s) {
  if (kind == kSweepDensityFixed)
    k_density<true><<<nunits, threads, density_smem(true, threads), s>>>(desc, units);
  else
    k_density<false><<<nunits, threads, density_smem(false, threads), s>>>(desc, units);
  return cudaGetLastError();
}

}  // namespace vdp
