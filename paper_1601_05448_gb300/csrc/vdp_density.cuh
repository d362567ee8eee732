// vdp_density.cuh -- the density form of the FP64 inner iteration, used with the constant-coefficient
// inverse (the paper's fixed-point iteration and spectrally preconditioned CG).
//
// The Jacobi-scaled form of vdp_kernels.cu exists for preconditioners that need a unit diagonal.
// The spectral inverse does not: in unscaled variables its passes need no weights, and the
// operator's three face coefficients per cell are functions of one field, the density, so a sweep
// that reads rho (its neighbours' values from L1 / L2) computes them.  With
//     rho' = rho / 2^e0 (e0 the exponent of the first cell),  s = 2^(2 m), m the exponent of hx,
//     A' = kappa A, kappa = 2^e0 s:  face values (2 s / h_d^2) / (rho'_l + rho'_r),
// an inner solve of (-A') X = r gives the correction p -= kappa X, whatever the units of rho and
// of the box; kappa is a power of two, so the scaling rounds nothing.
//
// FP32 inner solves keep the scaled form.  The rounding of the FP32 product is part of what decides
// where a mixed solve stops (the FP64 residual after an inner solve, and the targets drawn from
// it): with the coefficients computed in FP32 the fixed-point iteration took another number of
// iterations on 7 of 60 inputs of 256^3, on 1 of 40 of 192^3 and 1 of 5 of 512^3, and its pressures
// moved by up to 1.2e-9.
//
// z comes out of the FP32 transforms, so it is an FP32 field in this solve too; r, X, d and q are
// FP64.  The product A' z in FP64 instructions bounds the sweep by the FP64 pipe (8 instructions
// per cell at 2 per clock and SM: 282 us at 256^3, where its bytes take 118).  Here coefficients
// and product are pairs of FP32 numbers (unevaluated sums hi + lo, about 47 bits): rho' as such a
// pair, the quotient by a Newton step and a corrected remainder, the differences of z exact, the
// products by FMA with their rounding errors, the six terms summed with the errors carried along.
// Only the update of the FP64 fields is FP64: three instructions per cell (fixed point), four
// (CG).  The sweep also leaves rho' r in FP32 for the X+ pass, which read r and rho' and narrowed
// the product itself: four bytes more here, eight fewer there, and X+ runs its FP32 form (256^3:
// 75 -> 35 us).  The 47 bits act on differences of z across a face, not on z D as in the scaled form, and
// the refinement's FP64 residual is evaluated from p with the FP64 coefficients as before: over 242
// spectral and 242 fixed-point inputs of 32^3 to 256^3 no pressure was further from the one in 64 bits
// than with the FP64 product.
//
// The march is that of sweep_stencil_direct: a thread owns 16 bytes of one row and walks a z chunk,
// x neighbours come by shuffle, the rows above and below and the plane above by loads.  Each thread
// fetches its operands of the next plane by cp.async into slots of shared memory that only it
// reads, so no barrier is needed, no registers are held while they fly, and the arithmetic of one
// plane covers the latency of the next.  The x neighbours at row and warp ends come the same way
// (loaded at their use, they cost every plane a trip to L2).  Sums, products and Newton steps of the
// four cells run as paired FP32 instructions, and the fluxes through the x faces and the upper z face
// are computed once for both cells.  The fused sweep takes 206 us at 256^3 and 64 on the 256 x 128 x
// 128 duct (95 in the scaled form), CG's 41 at 128^3 (64): bound by instruction issue and latency at
// three blocks of 128 threads per SM (two 270, four 289 us).
#pragma once

#include "vdp_device.cuh"
#include "vdp_internal.cuh"
#include "vdp_sweeps.cuh"

namespace vdp {

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
__device__ __forceinline__ void fetch4(void* smem, const float* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(smem)),
               "l"(g)
               : "memory");
}
__device__ __forceinline__ void fetch_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// this thread's own copies: all but the newest group have landed
__device__ __forceinline__ void fetch_wait_previous() {
  asm volatile("cp.async.wait_group 1;" ::: "memory");
}

// An unevaluated sum h + l
struct df {
  f2 h, l;
};

// h + l = a + b exactly
__device__ __forceinline__ df two_sum(f2 a, f2 b) {
  df r;
  r.h = add2(a, b);
  const f2 t = sub2(r.h, a);
  r.l = add2(sub2(a, sub2(r.h, t)), sub2(b, t));
  return r;
}
__device__ __forceinline__ df two_diff(f2 a, f2 b) {
  df r;
  r.h = sub2(a, b);
  const f2 t = sub2(r.h, a);
  r.l = sub2(sub2(a, sub2(r.h, t)), add2(b, t));
  return r;
}

// A face coefficient c / (a + b), c = ch + cl = -(nch + ncl): h and the negatives of both parts (the
// paired instructions have no negated operands, and the products below want them).
struct dface {
  f2 h, nh, nl;
};
struct consts {
  f2 ch, nch, cl;
};
__device__ __forceinline__ dface face_df(const consts& c, df a, df b) {
  df s = two_sum(a.h, b.h);
  s.l = add2(s.l, add2(a.l, b.l));
  const float2 v = up2(s.h);
  f2 y = pk(rcp_approx(-v.x), rcp_approx(-v.y));  // -1 / s
  y = fma2(y, fma2(s.h, y, pk(1.f, 1.f)), y);
  dface q;
  q.h = mul2(c.nch, y);
  q.nh = mul2(c.ch, y);
  const f2 t = add2(fma2(q.nh, s.l, fma2(q.nh, s.h, c.ch)), c.cl);  // c - q s
  q.nl = mul2(t, y);
  return q;
}

// The flux b d through a face from the exact difference d, as h - nl
struct dflux {
  f2 h, nl;
};
__device__ __forceinline__ dflux flux_df(const dface& b, df d) {
  dflux f;
  f.h = mul2(b.h, d.h);
  f.nl = fma2(b.nl, d.h, fma2(b.nh, d.l, fma2(b.nh, d.h, f.h)));  // f.h - b d
  return f;
}

// acc += f, acc -= f
__device__ __forceinline__ void accumulate_plus(df& acc, const dflux& f) {
  const df s = two_sum(acc.h, f.h);
  acc.h = s.h;
  acc.l = add2(acc.l, sub2(s.l, f.nl));
}
__device__ __forceinline__ void accumulate_minus(df& acc, const dflux& f) {
  const df s = two_diff(acc.h, f.h);
  acc.h = s.h;
  acc.l = add2(acc.l, add2(s.l, f.nl));
}

// Operands of a plane z (16 bytes per thread each): z + 1 and the rows above and below of z and of both
// parts of the density, then the two FP64 fields.
enum Stream64 { T_UP, T_UA, T_UB, T_HP, T_HA, T_HB, T_LP, T_LA, T_LB, T_P0, T_P1, T_Q0, T_Q1, kStreams64 };

// NC: z is not written while the kernel runs (read-only loads).
// thread: this thread's place in the unit (a block may hold two units).
// FIXED: X += z, r -= (-A') z and the sum of r^2 / D' (FP32, steers the inner stop).
// CG: d = z + beta d_old, q = (-A') z + beta q_old, and the sum of d q.
template <bool FIXED, bool NC = true>
__device__ __forceinline__ void sweep_density64(const InstDesc& I, const InstState& st, int unit,
                                                double& part, ulonglong2* slots,
                                                int thread = threadIdx.x) {
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int tpr = nx / kV;
  const int tile = unit % I.uy, chunk = unit / I.uy;
  const int row = thread / tpr;
  const int x0 = (thread - row * tpr) * kV;
  const int yr = tile * I.ty + row;
  const bool active = row < I.ty && yr < ny;
  const int y = active ? yr : ny - 1;
  const int z0 = (int)((long long)chunk * nz / I.zc), z1 = (int)((long long)(chunk + 1) * nz / I.zc);
  part = 0.0;
  if (z0 >= z1 || !__any_sync(0xffffffffu, active)) return;  // (no block barrier below)
  const int lane = threadIdx.x & 31;
  const bool row_start = x0 == 0, row_end = x0 + kV == nx;
  const bool left_load = lane == 0 || row_start, right_load = lane == 31 || row_end;
  const bool wall_l = I.duct && row_start, wall_r = I.duct && row_end;
  consts cf[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    cf[d].ch = pk(I.ch[d], I.ch[d]);
    cf[d].nch = pk(-I.ch[d], -I.ch[d]);
    cf[d].cl = pk(I.cl[d], I.cl[d]);
  }
  const double beta = st.beta;
  const int rexp = st.rexp;
  const bool first = st.inner_iters == 0;  // no X (fixed point), no history (CG) yet
  const float* rhi = I.rho32;
  const float* rlo = I.rho_lo;
  const float* src = static_cast<const float*>(I.za);
  // p, q: the two FP64 fields read and written (fixed point r, X; CG d, q)
  const double* pin = static_cast<const double*>(FIXED ? I.r : (st.parity ? I.d1 : I.d0));
  double* pout = static_cast<double*>(FIXED ? I.r : (st.parity ? I.d0 : I.d1));
  double* q = static_cast<double*>(FIXED ? I.x : I.q);
  const long long plane = (long long)nx * ny;
  const long long dym = y == 0 ? (long long)(ny - 1) * nx : -(long long)nx;
  const long long dyp = y == ny - 1 ? -(long long)(ny - 1) * nx : (long long)nx;
  const int dxl = row_start ? nx - 1 : -1, dxr = row_end ? -x0 : kV;
  const long long cell0 = (long long)y * nx + x0;
  const long long dz_last = plane * (nz - 1);
  auto slot = [&](int b, int k) { return slots + (b * kStreams64 + k) * blockDim.x + threadIdx.x; };
  // x neighbours beyond the warp or the row: value k (z, rho' high and low), side 0 left, 1 right
  float* edges = reinterpret_cast<float*>(slots + kStages * kStreams64 * blockDim.x);
  auto edge = [&](int b, int k, int side) {
    return edges + ((b * 3 + k) * 2 + side) * blockDim.x + threadIdx.x;
  };
  auto fetch = [&](int b, int z, long long o) {
    if (left_load) {
      fetch4(edge(b, 0, 0), src + o + dxl);
      fetch4(edge(b, 1, 0), rhi + o + dxl);
      fetch4(edge(b, 2, 0), rlo + o + dxl);
    }
    if (right_load) {
      fetch4(edge(b, 0, 1), src + o + dxr);
      fetch4(edge(b, 1, 1), rhi + o + dxr);
      fetch4(edge(b, 2, 1), rlo + o + dxr);
    }
    const long long op = z == nz - 1 ? o - dz_last : o + plane;
    fetch16(slot(b, T_UP), src + op);
    fetch16(slot(b, T_UA), src + o + dym);
    fetch16(slot(b, T_UB), src + o + dyp);
    fetch16(slot(b, T_HP), rhi + op);
    fetch16(slot(b, T_HA), rhi + o + dym);
    fetch16(slot(b, T_HB), rhi + o + dyp);
    fetch16(slot(b, T_LP), rlo + op);
    fetch16(slot(b, T_LA), rlo + o + dym);
    fetch16(slot(b, T_LB), rlo + o + dyp);
    if (FIXED || !first) {
      fetch16_once(slot(b, T_P0), reinterpret_cast<const float*>(pin + o));
      fetch16_once(slot(b, T_P1), reinterpret_cast<const float*>(pin + o + 2));
    }
    if (!first) {
      fetch16_once(slot(b, T_Q0), reinterpret_cast<const float*>(q + o));
      fetch16_once(slot(b, T_Q1), reinterpret_cast<const float*>(q + o + 2));
    }
  };
  auto ldg2 = [](const float* p, f2& a, f2& b) {
    const ulonglong2* v = reinterpret_cast<const ulonglong2*>(p);
    const ulonglong2 t = NC ? __ldg(v) : *v;
    a = t.x;
    b = t.y;
  };
  long long o = (long long)z0 * plane + cell0;
  fetch(0, z0, o);
  fetch_commit();
  f2 u[2];
  df r[2];
  f2 bzl[2];    // lower z face: its coefficient (leading part) and flux b (z - z below)
  dflux fz[2];
  {
    const long long om = z0 == 0 ? o + dz_last : o - plane;
    f2 um[2];
    df rm[2];
    ldg2(src + om, um[0], um[1]);
    ldg2(src + o, u[0], u[1]);
    ldg2(rhi + om, rm[0].h, rm[1].h);
    ldg2(rlo + om, rm[0].l, rm[1].l);
    ldg2(rhi + o, r[0].h, r[1].h);
    ldg2(rlo + o, r[0].l, r[1].l);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const dface b = face_df(cf[2], rm[h], r[h]);
      bzl[h] = b.h;
      fz[h] = flux_df(b, two_diff(u[h], um[h]));
    }
  }
  double sum = 0.0;
  float sumf = 0.f;
  int b = 0;
  for (int z = z0; z < z1; ++z) {
    if (z + 1 < z1) fetch(b ^ 1, z + 1, o + plane);
    fetch_commit();
    fetch_wait_previous();
    df acc[2];
    f2 D[2];
    {  // x: faces 0 .. 4 of the four cells, as pairs (0, 1), (2, 3) and 4
      const float2 u01 = up2(u[0]), u23 = up2(u[1]);
      const float2 h01 = up2(r[0].h), h23 = up2(r[1].h), l01 = up2(r[0].l), l23 = up2(r[1].l);
      float ul = __shfl_up_sync(0xffffffffu, u23.y, 1), ur = __shfl_down_sync(0xffffffffu, u01.x, 1);
      float hl = __shfl_up_sync(0xffffffffu, h23.y, 1), hr = __shfl_down_sync(0xffffffffu, h01.x, 1);
      float ll = __shfl_up_sync(0xffffffffu, l23.y, 1), lr = __shfl_down_sync(0xffffffffu, l01.x, 1);
      if (left_load) {
        ul = *edge(b, 0, 0);
        hl = *edge(b, 1, 0);
        ll = *edge(b, 2, 0);
      }
      if (right_load) {
        ur = *edge(b, 0, 1);
        hr = *edge(b, 1, 1);
        lr = *edge(b, 2, 1);
      }
      dface b01 = face_df(cf[0], df{pk(hl, h01.x), pk(ll, l01.x)}, r[0]);
      const dface b23 = face_df(cf[0], df{pk(h01.y, h23.x), pk(l01.y, l23.x)}, r[1]);
      dface b44 = face_df(cf[0], df{pk(h23.y, h23.y), pk(l23.y, l23.y)}, df{pk(hr, hr), pk(lr, lr)});
      if (wall_l) {
        b01.h = pk(0.f, up2(b01.h).y);
        b01.nh = pk(0.f, up2(b01.nh).y);
        b01.nl = pk(0.f, up2(b01.nl).y);
      }
      if (wall_r) b44.h = b44.nh = b44.nl = 0ull;
      // fluxes b (u_k - u_{k-1}); A' z = sum of (upper flux - lower flux)
      const dflux f01 = flux_df(b01, two_diff(u[0], pk(ul, u01.x)));
      const dflux f23 = flux_df(b23, two_diff(u[1], pk(u01.y, u23.x)));
      const dflux f44 = flux_df(b44, two_diff(pk(ur, ur), pk(u23.y, u23.y)));
      const float2 fh01 = up2(f01.h), fh23 = up2(f23.h), fl01 = up2(f01.nl), fl23 = up2(f23.nl);
      acc[0] = df{pk(fh01.y, fh23.x), sub2(0ull, pk(fl01.y, fl23.x))};
      acc[1] = df{pk(fh23.y, up2(f44.h).x), sub2(0ull, pk(fl23.y, up2(f44.nl).x))};
      accumulate_minus(acc[0], f01);
      accumulate_minus(acc[1], f23);
      if (FIXED) {
        const float2 bh01 = up2(b01.h), bh23 = up2(b23.h);
        D[0] = add2(b01.h, pk(bh01.y, bh23.x));
        D[1] = add2(b23.h, pk(bh23.y, up2(b44.h).x));
      }
    }
    ulonglong2 t = *slot(b, T_UP);
    const f2 un[2] = {t.x, t.y};
    t = *slot(b, T_HP);
    const ulonglong2 t2 = *slot(b, T_LP);
    const df rn[2] = {{t.x, t2.x}, {t.y, t2.y}};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const dface bz = face_df(cf[2], r[h], rn[h]);
      const dflux f = flux_df(bz, two_diff(un[h], u[h]));
      accumulate_plus(acc[h], f);
      accumulate_minus(acc[h], fz[h]);
      fz[h] = f;
      if (FIXED) D[h] = add2(D[h], add2(bzl[h], bz.h));
      bzl[h] = bz.h;
    }
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      t = *slot(b, side ? T_UB : T_UA);
      const f2 v[2] = {t.x, t.y};
      t = *slot(b, side ? T_HB : T_HA);
      const ulonglong2 tl = *slot(b, side ? T_LB : T_LA);
      const df rv[2] = {{t.x, tl.x}, {t.y, tl.y}};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const dface by = face_df(cf[1], rv[h], r[h]);
        accumulate_plus(acc[h], flux_df(by, two_diff(v[h], u[h])));
        if (FIXED) D[h] = add2(D[h], by.h);
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 ah = up2(acc[h].h), al = up2(acc[h].l), uu = up2(u[h]);
      const double2 pv = *reinterpret_cast<const double2*>(slot(b, h ? T_P1 : T_P0));
      const double2 qv = *reinterpret_cast<const double2*>(slot(b, h ? T_Q1 : T_Q0));
      double2 po, qo;
      if constexpr (FIXED) {
        po.x = (pv.x + widen_scaled(ah.x, -rexp)) + widen_scaled(al.x, -rexp);
        po.y = (pv.y + widen_scaled(ah.y, -rexp)) + widen_scaled(al.y, -rexp);
        qo.x = widen_scaled(uu.x, -rexp);
        qo.y = widen_scaled(uu.y, -rexp);
        if (!first) {
          qo.x += qv.x;
          qo.y += qv.y;
        }
        const float2 d = up2(D[h]), rho = up2(r[h].h);
        const float rx = narrow_pow2(po.x, rexp), ry = narrow_pow2(po.y, rexp);
        if (active) *reinterpret_cast<float2*>(I.g32 + o + 2 * h) = make_float2(rho.x * rx, rho.y * ry);
        sumf = fmaf(rx * rcp_approx(d.x), rx, sumf);
        sumf = fmaf(ry * rcp_approx(d.y), ry, sumf);
      } else {
        po.x = widen_scaled(uu.x, -rexp);
        po.y = widen_scaled(uu.y, -rexp);
        qo.x = -(widen_scaled(ah.x, -rexp) + widen_scaled(al.x, -rexp));
        qo.y = -(widen_scaled(ah.y, -rexp) + widen_scaled(al.y, -rexp));
        if (!first) {
          po.x = fma(beta, pv.x, po.x);
          po.y = fma(beta, pv.y, po.y);
          qo.x = fma(beta, qv.x, qo.x);
          qo.y = fma(beta, qv.y, qo.y);
        }
        sum = fma(po.x, qo.x, sum);
        sum = fma(po.y, qo.y, sum);
      }
      if (active) {
        *reinterpret_cast<double2*>(pout + o + 2 * h) = po;
        *reinterpret_cast<double2*>(q + o + 2 * h) = qo;
      }
      u[h] = un[h];
      r[h] = rn[h];
    }
    o += plane;
    b ^= 1;
  }
  part = active ? (FIXED ? (double)sumf : sum) : 0.0;
}

constexpr int kDensity64Threads = kDirectThreads / 2;  // four cells per thread, the FP64 layout has two

inline size_t density64_smem(int threads) {  // operand slots and x edges
  return (sizeof(ulonglong2) * kStreams64 + 6 * sizeof(float)) * (size_t)kStages * threads;
}

}  // namespace vdp
