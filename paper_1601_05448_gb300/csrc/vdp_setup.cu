// vdp_setup.cu -- what vdp_set_density builds from rho: the FP64 face coefficients
// b_d = 2 / (rho_l + rho_r) / h_d^2 on the low faces, the diagonal D (sum of the six faces of a
// cell), the Jacobi scaling D^-1/2, the scaled inner coefficients, the weights of the scaled spectral
// passes, and the density as two FP32 numbers for the FP64 density-form sweeps (vdp_density.cu).
//
// What bounds these kernels.  The FP64 pipe of this GPU issues 2 FMA per clock and SM, 1/64 of the
// FP32 rate: an IEEE double division costs about ten such instructions and a reciprocal square
// root more, so a set-up written with `/` and `sqrt` is bound by that pipe at several times the
// HBM time (512^3: 16.3 ms against about 1 ms of traffic).  Here both start from the FP32
// approximation instruction (relative error below 2^-22, on the mantissa alone; where operands or quotient
// leave the middle of the binary64 range, the division and the root themselves run).  The root takes one third-order Newton step in FP64.  The quotient is
// refined in pairs of FP32 numbers to about 2^-44 and assembled into a double by integer
// operations; its FP64 remainder then gives the last bits: three FP64 instructions a face (the sum
// included) instead of more than ten.  512^3: 16.3 ms with both written out; now 4.0 in the density
// form (FP64 solves), 8.5 with D^-1/2, the scaled coefficients and the weights (FP32).
//
// Layout: a thread owns two neighbouring cells of a row (16-byte accesses) and marches a z chunk,
// so the plane below is in registers; the row above comes from L1 / L2.
#include <cmath>

#include "vdp_device.cuh"
#include "vdp_internal.cuh"
#include "vdp_launch.h"

namespace vdp {

namespace {

constexpr int kSetupThreads = 256;

// A face factor c split for face_quotient: 2^e (h + l), h in [1, 2).
struct FaceFactor {
  double c;
  float h, l;
  int e;  // kSlow: outside the middle of the binary64 range
};
constexpr int kSlow = 1 << 20;

// c / s, s > 0.  With s = 2^E (sh + sl): y ~ 1 / sh, th = h y, tl = (h + l - th (sh + sl)) y, so
// t = 2^(e - E) (th + tl) is c / s to about 2^-44 (the part of the sum that FP32 rounds off is added
// to the double as an integer number of its last places); then c / s = t + (c - s t) / s with y for
// 1 / s, rounded once.
__device__ __forceinline__ double face_quotient(const FaceFactor& f, double s) {
  if (f.e == kSlow || !mid_range(s)) return f.c / s;
  const unsigned lo = (unsigned)__double2loint(s);
  const int E = exponent_of(s) - 1023;
  // each factor may be far out while the quotient is itself near the ends of the range, or past them
  if ((unsigned)(f.e - E + 1000) > 2000u) return f.c / s;
  const float sh = mantissa_f(s);
  const float sl = (__uint_as_float(0x3f800000u | ((lo & 0x1fffffffu) >> 6)) - 1.f) * 0x1p-23f;
  const float y = rcp_approx(sh);
  const float th = f.h * y;
  const float rem = fmaf(-th, sl, fmaf(-th, sh, f.h)) + f.l;
  const float tl = rem * y;
  const float t1 = th + tl, t2 = tl - (t1 - th);  // the same sum, t2 at most half a place of t1
  const int et = (int)(__float_as_uint(t1) >> 23) - 127;
  int places = __float2int_rn(t2 * __uint_as_float((unsigned)(127 + 52 - et) << 23));
  // below a power of two the places are half as wide
  if (places < 0 && (__float_as_uint(t1) & 0x7fffffu) == 0) places *= 2;
  const double t = __longlong_as_double(__double_as_longlong(widen_pow2(t1, f.e - E)) + places);
  const double r = fma(-s, t, f.c);
  return fma(r, widen_pow2(y, -E), t);
}

// D^-1/2 for D > 0: seed Y0, e = 1 - D Y0^2, Y0 (1 + e/2 + 3 e^2/8).
__device__ __forceinline__ double inv_sqrt(double D) {
  if (!mid_range(D)) return 1.0 / sqrt(D);
  const int ex = exponent_of(D) - 1023, odd = ex & 1;
  const float m = __uint_as_float(__float_as_uint(mantissa_f(D)) + ((unsigned)odd << 23));
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(m));
  const double Y = widen_pow2(y, -((ex - odd) / 2));
  const double e = fma(-D * Y, Y, 1.0);
  return fma(Y * e, fma(e, 0.375, 0.5), Y);
}

// v times 2^p as FP32, rounded to nearest, by integer operations (below the FP32 range: 0).
__device__ __forceinline__ float narrow_rn_pow2(double v, int p) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const int e = (int)((hi >> 20) & 0x7ffu) - 1023 + 127 + p;
  const unsigned sign = hi & 0x80000000u;
  if (e <= 0) return __uint_as_float(sign);
  if (e >= 255) return __uint_as_float(sign | 0x7f800000u);
  return __uint_as_float(sign | ((((unsigned)e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29)) + ((lo >> 28) & 1u)));
}

// Thread geometry of the set-up kernels: pair q = two cells of a row, z chunk [z0, z1).
struct PairMarch {
  int x, y, z0, z1;
  bool on;
};

__device__ __forceinline__ PairMarch pair_march(int nx, int ny, int nz) {
  PairMarch m;
  const unsigned q = blockIdx.x * (unsigned)kSetupThreads + threadIdx.x, hx = (unsigned)nx / 2;
  m.y = (int)(q / hx);
  m.x = (int)(q - (unsigned)m.y * hx) * 2;
  m.z0 = (int)((long long)blockIdx.y * nz / gridDim.y);
  m.z1 = (int)((long long)(blockIdx.y + 1) * nz / gridDim.y);
  m.on = m.y < ny;
  return m;
}

// Whether the check of this call's density failed: nothing is built then, so that the previous
// density stays in force, and the host reads the verdict once, after the last kernel.
__device__ __forceinline__ bool rejected(const int* bad, int gen) {
  return bad && __ldcg(bad) == gen;
}

__device__ __forceinline__ double2 ld2(const double* p) {
  return __ldg(reinterpret_cast<const double2*>(p));
}

}  // namespace

// *bad = gen when an entry is <= 0, NaN or infinite: an integer test of the bits (positive and
// below the infinity pattern), which leaves the FP64 pipe alone.
__global__ void k_check_density(const double* __restrict__ rho, long long n, int gen, int* bad) {
  bool ok = true;
  const long long step = (long long)gridDim.x * blockDim.x * 2;
  auto good = [](double v) {
    const unsigned hi = (unsigned)__double2hiint(v);
    return hi < 0x7ff00000u && (hi | (unsigned)__double2loint(v)) != 0u;
  };
  if (((uintptr_t)rho & 15) == 0) {
    for (long long c = (blockIdx.x * (long long)blockDim.x + threadIdx.x) * 2; c < n; c += 2 * step) {
      const double2 u = ld2(rho + c);
      const double2 v = c + step < n ? ld2(rho + c + step) : u;
      ok = ok && good(u.x) && good(u.y) && good(v.x) && good(v.y);
    }
  } else {  // host-order arrays need no 16-byte alignment
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += step / 2)
      ok = ok && good(rho[c]);
  }
  if (!ok) *bad = gen;
}

// b_d[c] = 2 / (rho[c - e_d] + rho[c]) / h_d^2 on the low d-face of every cell; with rho32 also the
// FP32 density, scaled by the power of two of the first cell's (2^-e0), rho_lo what that
// rounds off, and dsc[0] = 2^e0 s2, the factor between the density-form operator and A
// (vdp_density.cu).  far[0] = gen when a density is more than 2^60 from the first cell's, or below the
// normal range: the density form's FP32 fields and coefficients do not hold that, the scaled form's do.
// duct: the face at the x ends (slot x = 0, shared by x = 0 and x = Lx) carries no flux.
__global__ void __launch_bounds__(kSetupThreads)
    k_faces(const double* __restrict__ rho, int nx, int ny, int nz, FaceFactor cx, FaceFactor cy, FaceFactor cz,
            int duct, double* __restrict__ bx, double* __restrict__ by, double* __restrict__ bz,
            float* __restrict__ rho32, float* __restrict__ rho_lo, double* dsc, double s2,
            const int* bad, int* far, int gen) {
  if (rejected(bad, gen)) return;
  const PairMarch m = pair_march(nx, ny, nz);
  const int e0 = exponent_of(__ldg(rho)) - 1023;
  if (dsc && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) dsc[0] = ldexp(s2, e0);
  if (!m.on) return;
  const bool wide = ((uintptr_t)rho & 15) == 0;  // 16-byte loads of the caller's array
  auto load = [&](long long o) {
    return wide ? ld2(rho + o) : make_double2(__ldg(rho + o), __ldg(rho + o + 1));
  };
  const long long plane = (long long)nx * ny;
  const long long dl = m.x == 0 ? nx - 1 : -1;
  const long long dy = m.y == 0 ? (long long)(ny - 1) * nx : -(long long)nx;
  long long c = m.x + (long long)nx * m.y + plane * m.z0;
  double2 lo = load(m.z0 == 0 ? c + plane * (nz - 1) : c - plane);
  for (int z = m.z0; z < m.z1; ++z, c += plane) {
    const double2 r = load(c), ry = load(c + dy);
    const double rl = __ldg(rho + c + dl);
    double2 vx, vy, vz;
    vx.x = face_quotient(cx, rl + r.x);
    vx.y = face_quotient(cx, r.x + r.y);
    vy.x = face_quotient(cy, ry.x + r.x);
    vy.y = face_quotient(cy, ry.y + r.y);
    vz.x = face_quotient(cz, lo.x + r.x);
    vz.y = face_quotient(cz, lo.y + r.y);
    if (duct && m.x == 0) vx.x = 0.0;
    *reinterpret_cast<double2*>(bx + c) = vx;
    *reinterpret_cast<double2*>(by + c) = vy;
    *reinterpret_cast<double2*>(bz + c) = vz;
    if (rho32) {
      const unsigned ex = (unsigned)exponent_of(r.x), ey = (unsigned)exponent_of(r.y);
      if (ex - (unsigned)(e0 + 963) > 120u || ey - (unsigned)(e0 + 963) > 120u || ex == 0u || ey == 0u) *far = gen;
      const float2 h = make_float2(narrow_rn_pow2(r.x, -e0), narrow_rn_pow2(r.y, -e0));
      *reinterpret_cast<float2*>(rho32 + c) = h;
      *reinterpret_cast<float2*>(rho_lo + c) =
          make_float2(narrow_rn_pow2(r.x - widen_pow2(h.x, e0), -e0),
                      narrow_rn_pow2(r.y - widen_pow2(h.y, e0), -e0));
    }
    lo = r;
  }
}

// D = sum of the six face coefficients of the cell; with sinv also D^-1/2
__global__ void __launch_bounds__(kSetupThreads)
    k_diag(const double* __restrict__ bx, const double* __restrict__ by,
           const double* __restrict__ bz, int nx, int ny, int nz, double* __restrict__ sinv,
           double* __restrict__ dg, const int* bad, int gen) {
  if (rejected(bad, gen)) return;
  const PairMarch m = pair_march(nx, ny, nz);
  if (!m.on) return;
  const long long plane = (long long)nx * ny;
  const long long dr = m.x + 2 == nx ? -(long long)m.x : 2;
  const long long dy = m.y == ny - 1 ? -(long long)(ny - 1) * nx : nx;
  long long c = m.x + (long long)nx * m.y + plane * m.z0;
  double2 z_lo = ld2(bz + c);
  for (int z = m.z0; z < m.z1; ++z, c += plane) {
    const double2 x = ld2(bx + c), y = ld2(by + c), yp = ld2(by + c + dy);
    const double xr = __ldg(bx + c + dr);
    const double2 z_hi = ld2(bz + (z == nz - 1 ? c - plane * (nz - 1) : c + plane));
    double2 D;
    D.x = x.x + x.y + y.x + yp.x + z_lo.x + z_hi.x;
    D.y = x.y + xr + y.y + yp.y + z_lo.y + z_hi.y;
    *reinterpret_cast<double2*>(dg + c) = D;
    if (sinv) *reinterpret_cast<double2*>(sinv + c) = make_double2(inv_sqrt(D.x), inv_sqrt(D.y));
    z_lo = z_hi;
  }
}

// D^-1/2 alone, for a context whose density was set for the density form
__global__ void k_sinv(const double* __restrict__ dg, long long n, double* __restrict__ sinv) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x)
    sinv[c] = inv_sqrt(dg[c]);
}

// Rounded to nearest: the rounding errors of the stored off-diagonals have no common sign, so
// they do not add up to a spurious diagonal shift that would swamp the operator's smallest
// eigenvalues (a directed rounding would, at BF16 precision).
template <class BT> struct CoefPair;
template <> struct CoefPair<double> {
  static __device__ __forceinline__ void st(double* p, double a, double b) {
    *reinterpret_cast<double2*>(p) = make_double2(a, b);
  }
};
template <> struct CoefPair<float> {
  static __device__ __forceinline__ void st(float* p, double a, double b) {
    *reinterpret_cast<float2*>(p) = make_float2(__double2float_rn(a), __double2float_rn(b));
  }
};
template <> struct CoefPair<__nv_bfloat16> {
  static __device__ __forceinline__ void st(__nv_bfloat16* p, double a, double b) {
    *reinterpret_cast<__nv_bfloat162*>(p) =
        __halves2bfloat162(__double2bfloat16(a), __double2bfloat16(b));
  }
};

// bt_d[c] = b_d[c] sinv[c - e_d] sinv[c]
template <class BT>
__global__ void __launch_bounds__(kSetupThreads)
    k_scaled(const double* __restrict__ bx, const double* __restrict__ by,
             const double* __restrict__ bz, const double* __restrict__ sinv, int nx, int ny, int nz,
             BT* __restrict__ sx, BT* __restrict__ sy, BT* __restrict__ sz, const int* bad, int gen) {
  if (rejected(bad, gen)) return;
  const PairMarch m = pair_march(nx, ny, nz);
  if (!m.on) return;
  const long long plane = (long long)nx * ny;
  const long long dl = m.x == 0 ? nx - 1 : -1;
  const long long dy = m.y == 0 ? (long long)(ny - 1) * nx : -(long long)nx;
  long long c = m.x + (long long)nx * m.y + plane * m.z0;
  double2 lo = ld2(sinv + (m.z0 == 0 ? c + plane * (nz - 1) : c - plane));
  for (int z = m.z0; z < m.z1; ++z, c += plane) {
    const double2 s = ld2(sinv + c), sm = ld2(sinv + c + dy);
    const double sl = __ldg(sinv + c + dl);
    const double2 x = ld2(bx + c), y = ld2(by + c), w = ld2(bz + c);
    CoefPair<BT>::st(sx + c, x.x * sl * s.x, x.y * s.x * s.y);
    CoefPair<BT>::st(sy + c, y.x * sm.x * s.x, y.y * sm.y * s.y);
    CoefPair<BT>::st(sz + c, w.x * lo.x * s.x, w.y * lo.y * s.y);
    lo = s;
  }
}

// BF16 coefficients: the rounded off-diagonals no longer sum (with the weights sqrt(D)) to the
// unit diagonal, and at BF16 precision that inconsistency is large enough to create spurious
// near-zero or negative eigenvalues.  The correction dg = sum_faces bt' s_nb / s_c - 1 (s =
// sqrt(D), bt' the stored BF16 values) restores sqrt(D) as an exact null vector of the stored
// inner operator  (1 + dg) I - offdiag(bt'), which is then congruent to a graph Laplacian with
// non-negative weights, i.e. symmetric positive semi-definite.
__global__ void k_diag_correction(const __nv_bfloat16* __restrict__ sx,
                                  const __nv_bfloat16* __restrict__ sy,
                                  const __nv_bfloat16* __restrict__ sz,
                                  const double* __restrict__ sinv, int nx, int ny, int nz,
                                  __nv_bfloat16* dg, const int* bad, int gen) {
  if (rejected(bad, gen)) return;
  const long long n = (long long)nx * ny * nz;
  const long long plane = (long long)nx * ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(c % nx);
    const int y = (int)((c / nx) % ny);
    const int z = (int)(c / plane);
    const long long cxm = c - x + (x == 0 ? nx - 1 : x - 1), cxp = c - x + (x == nx - 1 ? 0 : x + 1);
    const long long cym = c + (long long)((y == 0 ? ny - 1 : y - 1) - y) * nx;
    const long long cyp = c + (long long)((y == ny - 1 ? 0 : y + 1) - y) * nx;
    const long long czm = c + (long long)((z == 0 ? nz - 1 : z - 1) - z) * plane;
    const long long czp = c + (long long)((z == nz - 1 ? 0 : z + 1) - z) * plane;
    // s_nb / s_c = sinv_c / sinv_nb
    const double sc = sinv[c];
    double g = (double)__bfloat162float(sx[c]) * sc / sinv[cxm] +
               (double)__bfloat162float(sx[cxp]) * sc / sinv[cxp] +
               (double)__bfloat162float(sy[c]) * sc / sinv[cym] +
               (double)__bfloat162float(sy[cyp]) * sc / sinv[cyp] +
               (double)__bfloat162float(sz[c]) * sc / sinv[czm] +
               (double)__bfloat162float(sz[czp]) * sc / sinv[czp];
    dg[c] = __double2bfloat16(g - 1.0);
  }
}

// W = D^1/2 = D D^-1/2 per cell (FP32; unit: over the power of two of the first cell's, so that the
// preconditioner, which CG knows up to a factor only, stays in the FP32 range), and with rho the scaled fixed-point iteration's weight rho W
// (each null: not stored).  rho comes from the density itself, or where a context was set up for the
// density form from the two FP32 parts kept there (48 bits; kappa / s = 2^e0).
__global__ void k_weights(const double* __restrict__ rho, const float* __restrict__ rho32,
                          const float* __restrict__ rho_lo, const double* __restrict__ dsc, double is2,
                          const double* __restrict__ dg, const double* __restrict__ sinv, long long n, bool unit,
                          float* __restrict__ omega, float* __restrict__ rho_w, const int* bad, int gen) {
  if (rejected(bad, gen)) return;
  const double one = unit ? ldexp(1.0, -(ilogb(dg[0]) / 2)) : 1.0;
  const double scale = rho || !rho_w ? 1.0 : dsc[0] * is2;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    const double w = dg[c] * sinv[c];
    if (omega) omega[c] = __double2float_rn(w * one);
    if (rho_w) {
      const double r = rho ? rho[c] : ((double)rho32[c] + (double)rho_lo[c]) * scale;
      rho_w[c] = __double2float_rn(r * w);
    }
  }
}

// ---- host launchers ---------------------------------------------------------------------------

static int flat_grid(long long n) {
  long long b = (n + 1023) / 1024;
  if (b > kSMs * 8) b = kSMs * 8;
  return (int)(b < 1 ? 1 : b);
}

// z chunks: one plane per block on small grids (the shortest chains), else about six blocks per
// SM slot, so that the reload of the plane below at a chunk's start stays rare.
static dim3 pair_grid(int nx, int ny, int nz) {
  const long long pairs = (long long)nx / 2 * ny;
  const long long gx = (pairs + kSetupThreads - 1) / kSetupThreads;
  long long zc = (long long)kSMs * 48 / gx;
  if (zc > nz) zc = nz;
  if (zc > 65535) zc = 65535;
  if (zc < 1) zc = 1;
  return dim3((unsigned)gx, (unsigned)zc);
}

cudaError_t launch_check_density(const double* rho, long long n, int gen, int* bad, cudaStream_t s) {
  k_check_density<<<flat_grid(n), 256, 0, s>>>(rho, n, gen, bad);
  return cudaGetLastError();
}

cudaError_t launch_build_coefficients(const double* rho, int nx, int ny, int nz, double hx,
                                      double hy, double hz, int duct, double* bx, double* by,
                                      double* bz, double* sinv, double* dg, float* rho32,
                                      float* rho_lo, double* dsc, double s2, const int* bad,
                                      int* far, int gen, cudaStream_t s) {
  const dim3 g = pair_grid(nx, ny, nz);
  auto factor = [](double h) {
    FaceFactor f;
    f.c = 2.0 / (h * h);
    f.e = std::ilogb(f.c);
    const double m = std::ldexp(f.c, -f.e);
    f.h = (float)m;
    if (f.h >= 2.f) f.h = 2.f - 0x1p-23f;
    f.l = (float)(m - (double)f.h);
    if (f.e < -800 || f.e > 800) f.e = kSlow;
    return f;
  };
  k_faces<<<g, kSetupThreads, 0, s>>>(rho, nx, ny, nz, factor(hx), factor(hy), factor(hz), duct, bx,
                                      by, bz, rho32, rho_lo, dsc, s2, bad, far, gen);
  k_diag<<<g, kSetupThreads, 0, s>>>(bx, by, bz, nx, ny, nz, sinv, dg, bad, gen);
  return cudaGetLastError();
}

cudaError_t launch_sinv(const double* dg, long long n, double* sinv, cudaStream_t s) {
  k_sinv<<<flat_grid(n), 256, 0, s>>>(dg, n, sinv);
  return cudaGetLastError();
}

cudaError_t launch_scaled(int prec, const double* bx, const double* by, const double* bz,
                          const double* sinv, int nx, int ny, int nz, void* sx, void* sy, void* sz,
                          void* sd, const int* bad, int gen, cudaStream_t s) {
  const dim3 g = pair_grid(nx, ny, nz);
  if (prec == PREC_FP64)
    k_scaled<double><<<g, kSetupThreads, 0, s>>>(bx, by, bz, sinv, nx, ny, nz, (double*)sx,
                                                 (double*)sy, (double*)sz, bad, gen);
  else if (prec == PREC_MIXED)
    k_scaled<float><<<g, kSetupThreads, 0, s>>>(bx, by, bz, sinv, nx, ny, nz, (float*)sx,
                                                (float*)sy, (float*)sz, bad, gen);
  else {
    k_scaled<__nv_bfloat16><<<g, kSetupThreads, 0, s>>>(bx, by, bz, sinv, nx, ny, nz,
                                                        (__nv_bfloat16*)sx, (__nv_bfloat16*)sy,
                                                        (__nv_bfloat16*)sz, bad, gen);
    k_diag_correction<<<flat_grid((long long)nx * ny * nz), 256, 0, s>>>(
        (const __nv_bfloat16*)sx, (const __nv_bfloat16*)sy, (const __nv_bfloat16*)sz, sinv, nx, ny,
        nz, (__nv_bfloat16*)sd, bad, gen);
  }
  return cudaGetLastError();
}

cudaError_t launch_weights(const double* rho, const double* dg, const double* sinv, long long n,
                           bool unit, float* omega, float* rho_w, const int* bad, int gen, cudaStream_t s) {
  k_weights<<<flat_grid(n), 256, 0, s>>>(rho, nullptr, nullptr, nullptr, 1.0, dg, sinv, n, unit, omega,
                                          rho_w, bad, gen);
  return cudaGetLastError();
}

cudaError_t launch_rho_weight(const float* rho32, const float* rho_lo, const double* dsc, double s2,
                              const double* dg, const double* sinv, long long n, float* rho_w,
                              cudaStream_t s) {
  k_weights<<<flat_grid(n), 256, 0, s>>>(nullptr, rho32, rho_lo, dsc, 1.0 / s2, dg, sinv, n, false,
                                          nullptr, rho_w, nullptr, 0);
  return cudaGetLastError();
}

}  // namespace vdp
