// vdp_sweeps.cuh -- device code of the sweeps that several kernels run (vdp_kernels.cu: one sweep per
// launch; vdp_resident.cu: a whole solve per launch): element-wise sweeps, the direct stencil march
// and the FP64 residual march.  Internal to libvdp.
#pragma once

#include "vdp_device.cuh"
#include "vdp_internal.cuh"

namespace vdp {

// ---- small helpers ----------------------------------------------------------------------------

// Vector width per thread: 16-byte accesses of the inner type.
template <class T> struct VecW;
template <> struct VecW<float> { static constexpr int V = 4; };
template <> struct VecW<double> { static constexpr int V = 2; };

// two neighbouring cells, the first at an even index
__device__ __forceinline__ void store2(float* p, float a, float b) {
  *reinterpret_cast<float2*>(p) = make_float2(a, b);
}
__device__ __forceinline__ void store2(double* p, double a, double b) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
}

template <class T, int V> struct VecIO;
template <> struct VecIO<float, 4> {
  static __device__ __forceinline__ void ld(const float* p, float (&o)[4]) {
    float4 t = *reinterpret_cast<const float4*>(p);
    o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
  }
  static __device__ __forceinline__ void st(float* p, const float (&o)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
  }
};
template <> struct VecIO<double, 2> {
  static __device__ __forceinline__ void ld(const double* p, double (&o)[2]) {
    double2 t = *reinterpret_cast<const double2*>(p);
    o[0] = t.x; o[1] = t.y;
  }
  static __device__ __forceinline__ void st(double* p, const double (&o)[2]) {
    *reinterpret_cast<double2*>(p) = make_double2(o[0], o[1]);
  }
};

// the same, through the read-only (non-coherent) load path: only for data no thread of the
// running kernel writes
template <class T, int V> struct LdgIO;
template <> struct LdgIO<float, 4> {
  static __device__ __forceinline__ void ld(const float* p, float (&o)[4]) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
  }
};
template <> struct LdgIO<double, 2> {
  static __device__ __forceinline__ void ld(const double* p, double (&o)[2]) {
    const double2 t = __ldg(reinterpret_cast<const double2*>(p));
    o[0] = t.x; o[1] = t.y;
  }
};
// read-only loads where the data are constant for the whole kernel (NC), plain ones otherwise
template <bool NC, class T, int V> struct RoIO {
  static __device__ __forceinline__ void ld(const T* p, T (&o)[V]) {
    if constexpr (NC)
      LdgIO<T, V>::ld(p, o);
    else
      VecIO<T, V>::ld(p, o);
  }
};
template <bool NC, class T> __device__ __forceinline__ T ro1(const T* p) { return NC ? __ldg(p) : *p; }
// V coefficients of storage type BT into arithmetic type T
template <class BT, class T, int V> struct CoefIO;
template <> struct CoefIO<float, float, 4> {
  static __device__ __forceinline__ void ld(const float* p, float (&o)[4]) {
    VecIO<float, 4>::ld(p, o);
  }
  static __device__ __forceinline__ void ldg(const float* p, float (&o)[4]) {
    LdgIO<float, 4>::ld(p, o);
  }
};
template <> struct CoefIO<double, double, 2> {
  static __device__ __forceinline__ void ld(const double* p, double (&o)[2]) {
    VecIO<double, 2>::ld(p, o);
  }
  static __device__ __forceinline__ void ldg(const double* p, double (&o)[2]) {
    LdgIO<double, 2>::ld(p, o);
  }
};
template <> struct CoefIO<__nv_bfloat16, float, 4> {
  static __device__ __forceinline__ void ld(const __nv_bfloat16* p, float (&o)[4]) {
    uint2 u = *reinterpret_cast<const uint2*>(p);
    __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162*>(&u.x);
    __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162*>(&u.y);
    float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
    o[0] = fa.x; o[1] = fa.y; o[2] = fb.x; o[3] = fb.y;
  }
  static __device__ __forceinline__ void ldg(const __nv_bfloat16* p, float (&o)[4]) {
    uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    o[0] = __uint_as_float(u.x << 16); o[1] = __uint_as_float(u.x & 0xffff0000u);
    o[2] = __uint_as_float(u.y << 16); o[3] = __uint_as_float(u.y & 0xffff0000u);
  }
};

__device__ __forceinline__ float ldg1(const float* p) { return __ldg(p); }
__device__ __forceinline__ double ldg1(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ldg1(const __nv_bfloat16* p) {
  const unsigned short u = __ldg(reinterpret_cast<const unsigned short*>(p));
  return __uint_as_float((unsigned)u << 16);
}

__device__ __forceinline__ float ld1(const float* p) { return *p; }
__device__ __forceinline__ double ld1(const double* p) { return *p; }
__device__ __forceinline__ float ld1(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// ---- flat (element-wise) sweeps ------------------------------------------------------------------
// Run by k_flat, a kernel without dynamic shared memory (full occupancy).  Flat unit u of
// nunits_f covers the contiguous cells [flat_begin(u), flat_begin(u + 1)), multiples of 8, so
// every access is a 16-byte vector; each thread keeps four vectors in flight and several
// independent partial sums.

__device__ __forceinline__ long long flat_begin(const InstDesc& I, int u) {
  return ((long long)u * (I.ncell / 8) / I.nunits_f) * 8;
}

// Vectors per thread kept in flight by the FP64 flat sweeps below: all loads of a round are issued
// before the first use (one vector per thread per round left these sweeps latency bound).
constexpr int kFlatU = 4;

__device__ __forceinline__ double widen_t(float v, int p) { return widen_scaled(v, p); }
__device__ __forceinline__ double widen_t(double v, int) { return v; }

// <f>, ||f||^2; p := 0 unless p is the caller's initial guess.
static __device__ void sweep_meanf(const InstDesc& I, long long c0, long long c1, double& sum) {
  // <f> in FP64, one addition per cell.  p is not cleared here: from p = 0 the first residual
  // does not read it, the first correction writes it without reading it, and the gauge writes
  // zeros if no correction ever came.
  double s[2] = {0.0, 0.0};
  const long long step = 2LL * blockDim.x;
  for (long long cb = c0 + 2 * threadIdx.x; cb < c1; cb += kFlatU * step) {
    double2 fv[kFlatU];
#pragma unroll
    for (int u = 0; u < kFlatU; ++u) {
      const long long c = cb + u * step;
      fv[u] = c < c1 ? __ldg(reinterpret_cast<const double2*>(I.rhs + c)) : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int u = 0; u < kFlatU; ++u) {
      s[0] += fv[u].x;
      s[1] += fv[u].y;
    }
  }
  sum = s[0] + s[1];
}

// p -= D^-1/2 x (x in the inner type, FP32 with the factor 2^texp; DENS, the density form: p -=
// kappa x); sums the new p (the final gauge needs its mean).  fresh: p is still the zero start (never
// written), so it is not read.
template <class T, bool DENS = false>
__device__ void sweep_correct(const InstDesc& I, long long c0, long long c1, bool fresh,
                              int texp, double& psum) {
  const T* x = static_cast<const T*>(I.x);
  const double kappa = DENS ? I.dsc[0] : 0.0;
  double s = 0.0;
  const long long step = 2LL * blockDim.x;
  constexpr int U = kFlatU / 2;  // four operands per vector: half the vectors in flight
  for (long long cb = c0 + 2 * threadIdx.x; cb < c1; cb += U * step) {
    double2 sv[U], pv[U];
    T xa[U], xb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long c = cb + u * step;
      if (c < c1) {
        sv[u] = DENS ? make_double2(kappa, kappa) : __ldg(reinterpret_cast<const double2*>(I.sinv + c));
        pv[u] = fresh ? make_double2(0.0, 0.0) : *reinterpret_cast<const double2*>(I.p + c);
        xa[u] = x[c];
        xb[u] = x[c + 1];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long c = cb + u * step;
      if (c < c1) {
        double2 p = pv[u];
        p.x = fma(-sv[u].x, widen_t(xa[u], -texp), p.x);
        p.y = fma(-sv[u].y, widen_t(xb[u], -texp), p.y);
        *reinterpret_cast<double2*>(I.p + c) = p;
        s += p.x + p.y;
      }
    }
  }
  psum = s;
}

// p -= <p>   (or p = 0 when the right-hand side was constant)
static __device__ void sweep_final(const InstDesc& I, const InstState* st, long long c0, long long c1) {
  const double mp = st->sum_p / (double)I.ncell;
  const bool zero = st->zero_sol != 0 || st->p_set == 0;  // no iterate: the answer is p = 0
  const long long step = 2LL * blockDim.x;
  for (long long cb = c0 + 2 * threadIdx.x; cb < c1; cb += kFlatU * step) {
    double2 pv[kFlatU];
#pragma unroll
    for (int u = 0; u < kFlatU; ++u) {
      const long long c = cb + u * step;
      if (c < c1) pv[u] = *reinterpret_cast<const double2*>(I.p + c);
    }
#pragma unroll
    for (int u = 0; u < kFlatU; ++u) {
      const long long c = cb + u * step;
      if (c < c1)
        *reinterpret_cast<double2*>(I.p + c) =
            zero ? make_double2(0.0, 0.0) : make_double2(pv[u].x - mp, pv[u].y - mp);
    }
  }
}

// x += alpha d (x = alpha d on the first inner iteration); rt -= alpha q; <rt, rt>
template <class T>
__device__ void sweep_update(const InstDesc& I, const InstState* st, long long c0, long long c1,
                             T& part) {
  constexpr int V = VecW<T>::V;
  constexpr int U = 2;  // vectors per thread per round
  const T alpha = (T)st->alpha;
  const bool first = st->inner_iters == 0;
  // written by the last stencil sweep (the fixed-point iteration's direction is z itself)
  const T* d = static_cast<const T*>(I.pc == PC_FIXED ? I.za : (st->parity ? I.d0 : I.d1));
  const T* q = static_cast<const T*>(I.q);
  T* x = static_cast<T*>(I.x);
  T* rt = static_cast<T*>(I.r);
  T s[U];
#pragma unroll
  for (int u = 0; u < U; ++u) s[u] = 0;
  const long long step = (long long)V * blockDim.x;
  for (long long cb = c0 + (long long)V * threadIdx.x; cb < c1; cb += U * step) {
    T dv[U][V], qv[U][V], xv[U][V], rv[U][V];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long c = cb + u * step;
      if (c < c1) {
        VecIO<T, V>::ld(d + c, dv[u]);
        VecIO<T, V>::ld(q + c, qv[u]);
        VecIO<T, V>::ld(rt + c, rv[u]);
        if (!first) VecIO<T, V>::ld(x + c, xv[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long c = cb + u * step;
      if (c >= c1) continue;
#pragma unroll
      for (int k = 0; k < V; ++k) {
        xv[u][k] = fma(alpha, dv[u][k], first ? (T)0 : xv[u][k]);
        rv[u][k] = fma(-alpha, qv[u][k], rv[u][k]);
        s[u] = fma(rv[u][k], rv[u][k], s[u]);
      }
      VecIO<T, V>::st(x + c, xv[u]);
      VecIO<T, V>::st(rt + c, rv[u]);
      if constexpr (sizeof(T) == 8)
        if (I.g32) *reinterpret_cast<float2*>(I.g32 + c) = make_float2(narrow_pow2(rv[u][0], st->rexp), narrow_pow2(rv[u][1], st->rexp));
    }
  }
  T tot = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) tot += s[u];
  part = tot;
}

// BF16 coefficients carry a per-cell diagonal correction (see k_diag_correction).
template <class BT> struct CoefTraits { static constexpr bool kDiag = false; };
template <> struct CoefTraits<__nv_bfloat16> { static constexpr bool kDiag = true; };

// ---- the stencil sweep, direct form: register z march, no shared memory, no block barrier --------
// Each thread owns V consecutive cells of one row of the unit's row tile (tile = blockDim * V / nx
// rows) and marches them through the unit's z chunk, keeping d of planes z-1, z, z+1 in registers.
// Per plane it loads, as 16-byte vectors, rt and d_old of its own row at z+1 and of the rows above
// and below at z (forming d there: the neighbouring threads' rows, so these loads hit L1/L2), and
// the coefficients of its cells; x neighbours come from the adjacent lanes by warp shuffle (row
// ends, which wrap, are loaded).  Nothing waits on another warp, so many warps per SM keep many
// independent loads in flight.  Measured on the 256^3 FP32 sweep this runs at about 90 % of the
// HBM copy bandwidth, against about 50 % for the TMA-staged variant above, whose per-plane block
// barrier serialises the copy latency with the arithmetic.
//
// CHEB = true: one sweep j of the Chebyshev polynomial preconditioner instead (same march, the
// marched field is the Chebyshev iterate z_j, z_1 = rt / theta formed on the fly):
//   d_j = rho_j rho_{j-1} d_{j-1} + (2 rho_j / delta) (rt - At z_j),  z_{j+1} = z_j + d_j,
// with rho_0 = 1 / sigma, rho_j = 1 / (2 sigma - rho_{j-1}), sigma = theta / delta, d_0 = z_1;
// the last sweep also sums <rt, z>.
template <class T> struct IsF64 { static constexpr bool value = false; };
template <> struct IsF64<double> { static constexpr bool value = true; };

// NC: the marched field and its history are not written while the kernel runs (read-only loads);
// false in a kernel that runs several sweeps.
// VAR selects the variant at compile time (a predicated-off FMA still costs FP64-pipe slots):
//   0  first iteration of an inner CG solve (no search-direction history), or a Chebyshev sweep
//   1  CG with history (d = z + beta d_old)
//   2  the paper's fixed-point iteration (no history, no <d, q>, d not stored)
template <class T, class BT, bool CHEB, int VAR, bool NC = true>
__device__ void sweep_stencil_direct(const InstDesc& I, const InstState* st, int unit, T& part) {
  constexpr int V = VecW<T>::V;
  constexpr bool kDiag = CoefTraits<BT>::kDiag;
  // FP64 sweeps are bound by the FP64 pipe, not by HBM: there the stencil is applied to the
  // preconditioned residual z itself, and q = At d follows from q = At z + beta q_old, with
  // d = z + beta d_old formed for the thread's own cells only (9 FP64 operations per cell
  // instead of also forming d for the rows above and below and the row ends).  FP32 sweeps are
  // HBM bound and keep forming d, which reads one vector (q_old) less.
  constexpr bool QREC = !CHEB && IsF64<T>::value;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int tpr = nx / V;  // threads per row
  const int tile = unit % I.uy, chunk = unit / I.uy;
  const int row = threadIdx.x / tpr;
  const int x0 = (threadIdx.x - row * tpr) * V;
  const int yr = tile * I.ty + row;
  const bool active = row < I.ty && yr < ny;
  const int y = active ? yr : ny - 1;  // idle threads follow a valid row (shuffles need them)
  const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
  const int z0 = (int)((long long)chunk * nz / I.zc), z1 = (int)((long long)(chunk + 1) * nz / I.zc);
  part = 0;
  if (!__any_sync(0xffffffffu, active)) return;  // a warp without cells (no block barrier below)
  const int lane = threadIdx.x & 31;
  const bool row_start = x0 == 0, row_end = x0 + V == nx;
  const int xl = row_start ? nx - 1 : x0 - 1, xr = row_end ? 0 : x0 + V;
  // STENCIL: marched field d = src + beta d_old, src = rt (Jacobi) or the final Chebyshev z
  // CHEB:    marched field z_j = src * scale, src = rt / z buffer, scale = 1 / theta or 1
  const int cj = CHEB ? st->cheb_j : 0;
  const bool last = CHEB && cj == I.cheb_k - 1;
  T beta = (T)st->beta, scale = 1, c1 = 0, c2 = 0;
  // the paper's fixed-point iteration has no search-direction history (beta = 0) and needs
  // neither d nor q: the sweep applies the update itself on the thread's own cells,
  // x += z and rt -= At z, and sums <rt, rt> (one pass instead of a stencil and an update sweep)
  constexpr bool fixed = VAR == 2;
  const bool first_inner = st->inner_iters == 0;
  T* xv = static_cast<T*>(I.x);
  T* rw = static_cast<T*>(I.r);
  constexpr bool use_old = VAR == 1 && !CHEB;
  constexpr bool form = use_old && !QREC;  // form d = src + beta d_old for every marched value
  const T* rt = static_cast<const T*>(I.r);
  const T* src = I.pc != PC_JACOBI ? static_cast<const T*>(I.za) : rt;
  // the fixed-point iteration's z comes from the FP32 spectral passes and is stored as FP32
  // (exactly representable: widening it loses nothing)
  const float* srcf = static_cast<const float*>(I.za);
  const T* dold = static_cast<const T*>(st->parity ? I.d1 : I.d0);
  T* dnew = static_cast<T*>(st->parity ? I.d0 : I.d1);
  T* q = static_cast<T*>(I.q);
  T* zout = nullptr;
  T* dch = static_cast<T*>(I.dch);
  if (CHEB) {
    // sweep j reads z_j from buffer (k - j) % 2 and writes z_{j+1} to (k - 1 - j) % 2, so the
    // last sweep (j = k - 1) leaves z in za
    const int k = I.cheb_k;
    src = cj == 1 ? rt : static_cast<const T*>(((k - cj) & 1) ? I.zb : I.za);
    zout = static_cast<T*>(((k - 1 - cj) & 1) ? I.zb : I.za);
    scale = cj == 1 ? (T)(1.0 / I.cheb_theta) : (T)1;
    const double sigma = I.cheb_theta / I.cheb_delta;
    double rp = 1.0 / sigma, r = rp;
    for (int i = 1; i <= cj; ++i) {
      rp = r;
      r = 1.0 / (2.0 * sigma - rp);
    }
    c1 = (T)(r * rp);                  // rho_j rho_{j-1}
    c2 = (T)(2.0 * r / I.cheb_delta);  // 2 rho_j / delta
    beta = 0;
  }
  const BT* sx = static_cast<const BT*>(I.sx);
  const BT* sy = static_cast<const BT*>(I.sy);
  const BT* sz = static_cast<const BT*>(I.sz);
  const BT* sd = static_cast<const BT*>(I.sd);
  const long long plane = (long long)nx * ny;
  const long long dym = (long long)(ym - y) * nx, dyp = (long long)(yp - y) * nx;
  const int dxl = xl - x0, dxr = xr - x0;
  const long long cell0 = (long long)y * nx + x0;  // offset of the thread's cells in a plane
  auto zoff = [&](int z) -> long long {             // plane z (may be -1 or nz) + own cells
    return (long long)(z < 0 ? z + nz : (z >= nz ? z - nz : z)) * plane + cell0;
  };
  // all loads of a plane are issued together (non-coherent read-only path), then used
  auto dvec = [&](long long o, T (&d)[V]) {  // marched field, V cells at offset o
    if constexpr (fixed && IsF64<T>::value) {
#pragma unroll
      for (int k = 0; k < V; k += 2) {
        const float2* z2 = reinterpret_cast<const float2*>(srcf + o + k);
        const float2 t = NC ? __ldg(z2) : *z2;
        d[k] = widen(t.x);
        d[k + 1] = widen(t.y);
      }
    } else {
      RoIO<NC, T, V>::ld(src + o, d);
    }
    if (CHEB) {
#pragma unroll
      for (int k = 0; k < V; ++k) d[k] *= scale;
    } else if (form) {
      T b[V];
      RoIO<NC, T, V>::ld(dold + o, b);
#pragma unroll
      for (int k = 0; k < V; ++k) d[k] = fma(beta, b[k], d[k]);
    }
  };
  auto d1 = [&](long long o) -> T {
    if constexpr (fixed && IsF64<T>::value) return widen(ro1<NC>(srcf + o));
    if (CHEB) return ro1<NC>(src + o) * scale;
    return form ? fma(beta, ro1<NC>(dold + o), ro1<NC>(src + o)) : ro1<NC>(src + o);
  };

  T dm[V], dc[V], dp[V];
  if (z0 < z1) {
    dvec(zoff(z0 - 1), dm);
    dvec(zoff(z0), dc);
  }
  T sum[V];
#pragma unroll
  for (int k = 0; k < V; ++k) sum[k] = 0;
  float sumf = 0.f;  // FP64 fixed-point sweep: <rt, rt> in FP32
  for (int z = z0; z < z1; ++z) {
    const long long oc = zoff(z), op = zoff(z + 1);
    T du[V], dd[V], bx[V], by[V], byd[V], bz[V], bzp[V], bd[V];
    dvec(op, dp);
    dvec(oc + dym, du);
    dvec(oc + dyp, dd);
    CoefIO<BT, T, V>::ldg(sx + oc, bx);
    CoefIO<BT, T, V>::ldg(sy + oc, by);
    CoefIO<BT, T, V>::ldg(sy + oc + dyp, byd);
    CoefIO<BT, T, V>::ldg(sz + oc, bz);
    CoefIO<BT, T, V>::ldg(sz + op, bzp);
    if (kDiag) CoefIO<BT, T, V>::ldg(sd + oc, bd);
    T qo[V], dol[V];  // QREC: q_old and d_old of the own cells
    if (QREC && use_old) {
      VecIO<T, V>::ld(q + oc, qo);  // q is rewritten below by this thread only
      RoIO<NC, T, V>::ld(dold + oc, dol);
    }
    T ro[V], xo[V];  // fixed point: rt and x of the own cells (rewritten by this thread only)
    if (fixed) {
      VecIO<T, V>::ld(rw + oc, ro);
      if (first_inner) {
#pragma unroll
        for (int k = 0; k < V; ++k) xo[k] = 0;
      } else {
        VecIO<T, V>::ld(xv + oc, xo);
      }
    }
    const T bxr = (T)ldg1(sx + oc + dxr);
    // x neighbours of the first and last cell: adjacent lanes, or a load at row ends / warp ends
    T left = __shfl_up_sync(0xffffffffu, dc[V - 1], 1);
    T right = __shfl_down_sync(0xffffffffu, dc[0], 1);
    if (lane == 0 || row_start) left = d1(oc + dxl);
    if (lane == 31 || row_end) right = d1(oc + dxr);
    T qv[V];
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const T l = k == 0 ? left : dc[k - 1];
      const T r = k == V - 1 ? right : dc[k + 1];
      const T br = k == V - 1 ? bxr : bx[k + 1];
      T a = dc[k];
      if (kDiag) a = fma(bd[k], dc[k], a);
      a = fma(-bx[k], l, a);
      a = fma(-br, r, a);
      a = fma(-by[k], du[k], a);
      a = fma(-byd[k], dd[k], a);
      a = fma(-bz[k], dm[k], a);
      a = fma(-bzp[k], dp[k], a);
      qv[k] = a;
      if (!CHEB && !QREC && !fixed) sum[k] = fma(dc[k], a, sum[k]);
    }
    if (fixed) {
#pragma unroll
      for (int k = 0; k < V; ++k) {
        ro[k] -= qv[k];
        xo[k] += dc[k];
        if constexpr (IsF64<T>::value) {  // <rt, rt> only steers the inner stop: FP32 suffices,
          const float rf = narrow(ro[k]);   // and keeps the FP64 pipe to the update itself
          sumf = fmaf(rf, rf, sumf);
        } else {
          sum[k] = fma(ro[k], ro[k], sum[k]);
        }
      }
    }
    T dn[V];
    if (QREC && !fixed) {
#pragma unroll
      for (int k = 0; k < V; ++k) {
        dn[k] = use_old ? fma(beta, dol[k], dc[k]) : dc[k];
        qv[k] = use_old ? fma(beta, qo[k], qv[k]) : qv[k];
        if (!fixed) sum[k] = fma(dn[k], qv[k], sum[k]);
      }
    }
    if (CHEB) {
      T r[V], dprev[V], zn[V], dn[V];
      RoIO<NC, T, V>::ld(rt + oc, r);
      if (cj == 1) {
#pragma unroll
        for (int k = 0; k < V; ++k) dprev[k] = dc[k];  // d_0 = z_1
      } else {
        RoIO<NC, T, V>::ld(dch + oc, dprev);
      }
#pragma unroll
      for (int k = 0; k < V; ++k) {
        dn[k] = fma(c1, dprev[k], c2 * (r[k] - qv[k]));
        zn[k] = dc[k] + dn[k];
        if (last) sum[k] = fma(r[k], zn[k], sum[k]);
      }
      if (active) {
        VecIO<T, V>::st(zout + oc, zn);
        if (!last) VecIO<T, V>::st(dch + oc, dn);
      }
    } else if (active && fixed) {
      VecIO<T, V>::st(rw + oc, ro);
      VecIO<T, V>::st(xv + oc, xo);
    } else if (active) {
      if (QREC)
        VecIO<T, V>::st(dnew + oc, dn);
      else
        VecIO<T, V>::st(dnew + oc, dc);
      VecIO<T, V>::st(q + oc, qv);
    }
#pragma unroll
    for (int k = 0; k < V; ++k) {
      dm[k] = dc[k];
      dc[k] = dp[k];
    }
  }
  if (!active) {
#pragma unroll
    for (int k = 0; k < V; ++k) sum[k] = 0;
    sumf = 0.f;
  }
  T tot = 0;
#pragma unroll
  for (int k = 0; k < V; ++k) tot += sum[k];
  if (fixed && IsF64<T>::value) tot = (T)sumf;
  part = tot;
}

// FP64 residual sweep in the same direct form (same unit and thread geometry as the stencil
// sweep: a thread owns VR = 16 / sizeof(T) cells of one row): p of planes z-1, z, z+1 in
// registers, rows above and below loaded per plane.  r = (f - <f>) - A p with the FP64 face
// coefficients; rt = D^-1/2 r stored in the inner type; sums of r^2, rt^2, p and, on the first
// call, (f - <f>)^2.  The sweep is bound by the FP64 pipe, so the residual is formed in the
// diagonal form r = (f - <f>) + D p_c - sum of b_face p_neighbour (D stored per cell): one FMA
// per term, 8 FP64 operations per cell against 13 for the face-difference form; in the mixed
// precisions the scaling rt = D^-1/2 r is an FP32 product; the norms are summed in FP32.
// What the residual sweep hands to the inner solve in the density form (DENS, FP64): r, X+'s FP32
// input (fixed point rho' r, CG r), and the norm's terms: fixed point r^2 / D' (D' = kappa D), CG
// r^2.
struct DensityResidual {
  bool fixed;
  int ek;      // kappa = 2^ek x mk
  float mk;
  const float* rho;
  __device__ __forceinline__ DensityResidual() : fixed(false), ek(0), mk(0.f), rho(nullptr) {}
  __device__ __forceinline__ explicit DensityResidual(const InstDesc& I)
      : fixed(I.pc == PC_FIXED), rho(I.rho32) {
    const double k = I.dsc[0];
    ek = ((__double2hiint(k) >> 20) & 0x7ff) - 1023;
    mk = narrow_pow2(k, -ek);
  }
  __device__ __forceinline__ float inv_diag(double D) const {
    return rcp_approx(narrow_pow2(D, ek) * mk);
  }
};

template <class T, bool FIRST, bool DENS, bool F0 = false>
__device__ __forceinline__ void res64_march(const InstDesc& I, const InstState* st, int unit,
                                            double (&acc)[kSlots]) {
  static_assert(!DENS || IsF64<T>::value, "the density form is an FP64 one");
  constexpr int VR = VecW<T>::V;  // cells per thread (4 for FP32 inner, 2 for FP64)
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int tpr = nx / VR;
  const int tile = unit % I.uy, chunk = unit / I.uy;
  const int row = threadIdx.x / tpr;
  const int x0 = (threadIdx.x - row * tpr) * VR;
  const int yr = tile * I.ty + row;
  const bool active = row < I.ty && yr < ny;
  const int y = active ? yr : ny - 1;
  const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
  const int z0 = (int)((long long)chunk * nz / I.zc), z1 = (int)((long long)(chunk + 1) * nz / I.zc);
  if (!__any_sync(0xffffffffu, active)) return;  // a warp without cells: acc stays 0
  const int lane = threadIdx.x & 31;
  const bool row_start = x0 == 0, row_end = x0 + VR == nx;
  const int xl = row_start ? nx - 1 : x0 - 1, xr = row_end ? 0 : x0 + VR;
  const double mu = st->mu_f;
  const int rexp = st->rexp, sexp = st->texp - st->rexp;
  const double* p = I.p;
  T* rt = static_cast<T*>(I.r);
  const DensityResidual dr = DENS ? DensityResidual(I) : DensityResidual();
  auto at = [&](int z, int yy) -> long long {
    const int zz = z < 0 ? z + nz : (z >= nz ? z - nz : z);
    return ((long long)zz * ny + yy) * nx;
  };
  auto ldv = [&](const double* a, long long o, double (&v)[VR]) {
#pragma unroll
    for (int k = 0; k < VR; k += 2) {
      const double2 t = *reinterpret_cast<const double2*>(a + o + k);
      v[k] = t.x;
      v[k + 1] = t.y;
    }
  };
  double pm[VR], pc[VR], pp[VR];
  if (z0 < z1) {
    ldv(p, at(z0 - 1, y) + x0, pm);
    ldv(p, at(z0, y) + x0, pc);
  }
  double a2 = 0, a3 = 0;
  float a0 = 0.f, a1 = 0.f;  // norms steer the refinement only: summed in FP32 (cells narrowed
                             // by integer repacking), the FP64 pipe kept for the residual itself
  for (int z = z0; z < z1; ++z) {
    const long long oc = at(z, y), op = at(z + 1, y), oyp = at(z, yp), oym = at(z, ym);
    ldv(p, op + x0, pp);
    const double bxr = I.bx[oc + xr];
    double left = __shfl_up_sync(0xffffffffu, pc[VR - 1], 1);
    double right = __shfl_down_sync(0xffffffffu, pc[0], 1);
    if (lane == 0 || row_start) left = p[oc + xl];
    if (lane == 31 || row_end) right = p[oc + xr];
    // two cells at a time keeps the live registers down
#pragma unroll
    for (int h = 0; h < VR; h += 2) {
      const long long o = oc + x0 + h;
      const double2 pu = *reinterpret_cast<const double2*>(p + oym + x0 + h);
      const double2 pd = *reinterpret_cast<const double2*>(p + oyp + x0 + h);
      const double2 bx = *reinterpret_cast<const double2*>(I.bx + o);
      const double2 by = *reinterpret_cast<const double2*>(I.by + o);
      const double2 byd = *reinterpret_cast<const double2*>(I.by + oyp + x0 + h);
      const double2 bz = *reinterpret_cast<const double2*>(I.bz + o);
      const double2 bzp = *reinterpret_cast<const double2*>(I.bz + op + x0 + h);
      const double2 dg = *reinterpret_cast<const double2*>(I.dg + o);
      // F0: f - <f> as the first residual stored it (one FP64 operation fewer per cell)
      const double2 f = *reinterpret_cast<const double2*>((F0 ? I.f0 : I.rhs) + o);
      double2 si = make_double2(0.0, 0.0);
      float2 rh = make_float2(1.f, 1.f);
      if (!DENS) si = *reinterpret_cast<const double2*>(I.sinv + o);
      if (DENS && dr.fixed) rh = __ldg(reinterpret_cast<const float2*>(dr.rho + o));
      const double l0 = h == 0 ? left : pc[h - 1];
      const double r1 = h + 2 == VR ? right : pc[h + 2];
      const double br1 = h + 2 == VR ? bxr : I.bx[o + 2];
      const double c0 = pc[h], c1 = pc[h + 1];
      // r = (f - <f>) - A p with (A p)_c = sum of b_face p_neighbour - D_c p_c: the diagonal
      // term first, then one FMA per face (8 FP64 operations per cell; rounding error of order
      // eps D |p|, below 1e-12 of ||f - <f>|| on the grids here)
      double res0 = fma(dg.x, c0, F0 ? f.x : f.x - mu), res1 = fma(dg.y, c1, F0 ? f.y : f.y - mu);
      res0 = fma(-bx.x, l0, res0);
      res0 = fma(-bx.y, c1, res0);
      res1 = fma(-bx.y, c0, res1);
      res1 = fma(-br1, r1, res1);
      res0 = fma(-by.x, pu.x, res0);
      res1 = fma(-by.y, pu.y, res1);
      res0 = fma(-byd.x, pd.x, res0);
      res1 = fma(-byd.y, pd.y, res1);
      res0 = fma(-bz.x, pm[h], res0);
      res1 = fma(-bz.y, pm[h + 1], res1);
      res0 = fma(-bzp.x, pp[h], res0);
      res1 = fma(-bzp.y, pp[h + 1], res1);
      T t0, t1;
      float r0f = narrow_pow2(res0, rexp), r1f = narrow_pow2(res1, rexp), t0f, t1f;
      if constexpr (DENS) {
        t0 = res0;
        t1 = res1;
        t0f = dr.fixed ? r0f * r0f * dr.inv_diag(dg.x) : r0f * r0f;  // the norm's terms
        t1f = dr.fixed ? r1f * r1f * dr.inv_diag(dg.y) : r1f * r1f;
      } else if constexpr (IsF64<T>::value) {
        t0 = si.x * res0;
        t1 = si.y * res1;
        t0f = narrow(t0);
        t1f = narrow(t1);
      } else {  // the inner residual in FP32: D^-1/2 r from the FP32 factors (the inner solve's
                // own rounding), no FP64 multiply
        t0 = t0f = narrow_pow2(si.x, sexp) * r0f;
        t1 = t1f = narrow_pow2(si.y, sexp) * r1f;
      }
      if (active) {
        store2(rt + o, t0, t1);
        if constexpr (DENS)
          *reinterpret_cast<float2*>(I.g32 + o) = make_float2(rh.x * r0f, rh.y * r1f);
        a0 = fmaf(r0f, r0f, fmaf(r1f, r1f, a0));
        a1 = DENS ? a1 + (t0f + t1f) : fmaf(t0f, t0f, fmaf(t1f, t1f, a1));
        if (FIRST) {
          const double f0 = f.x - mu, f1 = f.y - mu;
          a2 += c0 + c1;
          a3 = fma(f0, f0, fma(f1, f1, a3));
        }
      }
    }
#pragma unroll
    for (int k = 0; k < VR; ++k) {
      pm[k] = pc[k];
      pc[k] = pp[k];
    }
  }
  acc[0] = (double)a0;
  acc[1] = (double)a1;
  if (DENS && !dr.fixed && rexp) acc[1] = ldexp(acc[1], -2 * rexp);  // CG's norms are FP64
  acc[2] = a2;
  acc[3] = a3;
}

// The first residual of a solve started from p = 0 is r = f - <f>: no stencil, no p reads.
template <class T, bool DENS>
__device__ void res64_zero_p(const InstDesc& I, const InstState* st, int unit,
                             double (&acc)[kSlots]) {
  constexpr int VR = VecW<T>::V;
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int tpr = nx / VR;
  const int tile = unit % I.uy, chunk = unit / I.uy;
  const int row = threadIdx.x / tpr;
  const int x0 = (threadIdx.x - row * tpr) * VR;
  const int yr = tile * I.ty + row;
  const int z0 = (int)((long long)chunk * nz / I.zc), z1 = (int)((long long)(chunk + 1) * nz / I.zc);
  const double mu = st->mu_f;
  const int rexp = st->rexp, sexp = st->texp - st->rexp;
  T* rt = static_cast<T*>(I.r);
  const DensityResidual dr = DENS ? DensityResidual(I) : DensityResidual();
  double a0 = 0;
  T a1 = 0;
  float a1f = 0.f;  // DENS
  // two planes' loads before the first plane's stores (which the compiler cannot move loads across):
  // 512^3 mixed 730 -> 582 us (28 bytes a cell: 6.5 TB/s), 256^3 152 -> 96, FP64 157 -> 122
  struct Cells {
    double2 f[VR / 2], w[VR / 2];  // w: D (density form), else D^-1/2
    float2 rho[VR / 2];
  };
  const bool diag = DENS && dr.fixed;
  auto load = [&](int z, Cells& c) {
    const long long o = ((long long)z * ny + yr) * nx + x0;
#pragma unroll
    for (int h = 0; h < VR; h += 2) {
      c.f[h / 2] = *reinterpret_cast<const double2*>(I.rhs + o + h);
      if (!DENS || diag) c.w[h / 2] = *reinterpret_cast<const double2*>((DENS ? I.dg : I.sinv) + o + h);
      if (diag) c.rho[h / 2] = __ldg(reinterpret_cast<const float2*>(dr.rho + o + h));
    }
  };
  auto store = [&](int z, const Cells& c) {
    const long long o = ((long long)z * ny + yr) * nx + x0;
#pragma unroll
    for (int h = 0; h < VR; h += 2) {
      const double f0 = c.f[h / 2].x - mu, f1 = c.f[h / 2].y - mu;
      if (I.f0) *reinterpret_cast<double2*>(I.f0 + o + h) = make_double2(f0, f1);
      if constexpr (DENS) {
        const float r0 = narrow_pow2(f0, rexp), r1 = narrow_pow2(f1, rexp);
        const float2 rh = diag ? c.rho[h / 2] : make_float2(1.f, 1.f);
        float2 d = make_float2(1.f, 1.f);
        if (diag) d = make_float2(dr.inv_diag(c.w[h / 2].x), dr.inv_diag(c.w[h / 2].y));
        store2(rt + o + h, f0, f1);
        *reinterpret_cast<float2*>(I.g32 + o + h) = make_float2(rh.x * r0, rh.y * r1);
        a0 = fma(f0, f0, fma(f1, f1, a0));
        a1f = fmaf(r0 * d.x, r0, fmaf(r1 * d.y, r1, a1f));
      } else if constexpr (IsF64<T>::value) {
        const double2 si = c.w[h / 2];
        const T t0 = si.x * f0, t1 = si.y * f1;
        store2(rt + o + h, t0, t1);
        a0 = fma(f0, f0, fma(f1, f1, a0));
        a1 = fma(t0, t0, fma(t1, t1, a1));
      } else {  // as the full residual of the mixed precisions: the FP32 product of the narrowed
                // factors; ||f - <f>||^2, the denominator of every relative residual of the
                // solve, stays an FP64 sum (any magnitude of f)
        const double2 si = c.w[h / 2];
        const float t0 = narrow_pow2(si.x, sexp) * narrow_pow2(f0, rexp);
        const float t1 = narrow_pow2(si.y, sexp) * narrow_pow2(f1, rexp);
        store2(rt + o + h, t0, t1);
        a0 = fma(f0, f0, fma(f1, f1, a0));
        a1 = fmaf(t0, t0, fmaf(t1, t1, a1));
      }
    }
  };
  if (row < I.ty && yr < ny) {
    Cells c[2];
    for (int z = z0; z < z1; z += 2) {
      load(z, c[0]);
      if (z + 1 < z1) load(z + 1, c[1]);
      store(z, c[0]);
      if (z + 1 < z1) store(z + 1, c[1]);
    }
  }
  acc[0] = rexp ? ldexp(a0, 2 * rexp) : a0;  // ||r||^2, in the units of the later sweeps' sums
  acc[1] = DENS ? (dr.fixed ? (double)a1f : a0) : (double)a1;  // ||rt||^2 (density form: see above)
  acc[2] = 0.0;         // sum of p
  acc[3] = a0;          // ||f - <f>||^2 (this is the first residual)
}

template <class T, bool DENS = false>
__device__ void sweep_res64_direct(const InstDesc& I, const InstState* st, int unit,
                                   double (&acc)[kSlots]) {
  if (st->first_res != 0 && !st->use_guess)
    res64_zero_p<T, DENS>(I, st, unit, acc);
  else if (st->first_res != 0)
    res64_march<T, true, DENS>(I, st, unit, acc);
  else if (I.f0 && !st->use_guess)  // f - <f> stored by the first residual
    res64_march<T, false, DENS, true>(I, st, unit, acc);
  else
    res64_march<T, false, DENS>(I, st, unit, acc);
}

}  // namespace vdp
