// vdp_device.cuh -- device code shared by the solver's translation units (vdp_kernels.cu and
// vdp_spectral.cu): deterministic partial sums, the last-unit ticket, the phase transitions of
// the per-instance state machine, and the state snapshot.  Internal to libvdp.
#pragma once

#include "vdp_internal.cuh"

namespace vdp {

// Conversions between binary64 and binary32 by repacking the IEEE 754 fields with integer
// operations: on this GPU the conversion instructions run on the FP64 pipe (2 results per clock
// per SM), which FP64 kernels otherwise spend a large share of their time in.
//   to binary32: exponent rebiased (1023 -> 127), the 23 leading fraction bits kept (rounding
//                toward zero), magnitudes below the binary32 normal range flushed to zero and
//                above it (infinities, NaNs) sent to infinity -- adequate for a preconditioner
//                input, which the FP32 transforms round anyway;
//   to binary64: exact for every binary32 normal number and zero (subnormals flush to zero).
__device__ __forceinline__ float narrow(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ffu) - 1023 + 127;
  const unsigned frac = ((hi & 0xfffffu) << 3) | (lo >> 29);
  const unsigned bits = e <= 0 ? sign : (e >= 255 ? (sign | 0x7f800000u) : (sign | ((unsigned)e << 23) | frac));
  return __uint_as_float(bits);
}
__device__ __forceinline__ double widen(float v) {
  const unsigned b = __float_as_uint(v);
  const unsigned sign = b & 0x80000000u, e = (b >> 23) & 0xffu, frac = b & 0x7fffffu;
  const unsigned hi = e == 0 ? sign : (sign | ((e + 1023u - 127u) << 20) | (frac >> 3));
  const unsigned lo = e == 0 ? 0u : (frac << 29);
  return __hiloint2double((int)hi, (int)lo);
}
// to binary32 of v times 2^p, the same way
__device__ __forceinline__ float narrow_pow2(double v, int p) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ffu) - 1023 + 127 + p;
  const unsigned frac = ((hi & 0xfffffu) << 3) | (lo >> 29);
  const unsigned bits = e <= 0 ? sign : (e >= 255 ? (sign | 0x7f800000u) : (sign | ((unsigned)e << 23) | frac));
  return __uint_as_float(bits);
}

// v times 2^p to binary64 (results in the normal range)
__device__ __forceinline__ double widen_scaled(float v, int p) {
  const unsigned b = __float_as_uint(v);
  const unsigned sign = b & 0x80000000u, e = (b >> 23) & 0xffu, frac = b & 0x7fffffu;
  const unsigned hi = e == 0 ? sign : (sign | ((e + 1023u - 127u + (unsigned)p) << 20) | (frac >> 3));
  return __hiloint2double((int)hi, (int)(e == 0 ? 0u : frac << 29));
}

// approximate reciprocal (1 ulp)
__device__ __forceinline__ float rcp_approx(float s) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(s));
  return y;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---- reductions: per-unit partial slots, last unit reduces them in a fixed order --------------

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block reduction of NS per-thread partials of type A into slot k of this unit:
// part[k * nunits + unit], always in the same order (threads without cells add zeros), so the
// block size does not show.  FP32 partials, and blocks of more than kDirectThreads: a shuffle tree
// per warp, the warp totals combined in FP64.  FP64 partials: through shared memory, a lane adding
// its column of the block's warps before one shuffle tree -- a warp-wide FP64 addition holds this
// GPU's FP64 pipe for 16 cycles, and a tree in every warp cost more of them than the update of
// four cells per thread.
template <int NS, class A>
__device__ __forceinline__ void store_partials_by_warp(const A (&v)[NS], double* part, int nunits,
                                                       int unit) {
  __shared__ double red[kMaxThreads / 32][NS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  A w[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) w[k] = warp_sum(v[k]);
  __syncthreads();  // red[] may still be read by a previous use
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NS; ++k) red[warp][k] = (double)w[k];
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      double s = lane < nwarps ? red[lane][k] : 0.0;
      s = warp_sum(s);
      if (lane == 0) part[k * nunits + unit] = s;
    }
  }
}

// 32 lanes' sums of a column of up to eight warps, then over the lanes
__device__ __forceinline__ double column_sum(const double* col, int nwarps) {
  static_assert(kDirectThreads == 256 && kFlatThreads == 256, "eight warps");
  const int lane = threadIdx.x & 31;
  double c[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) c[w] = w < nwarps ? col[w * 32 + lane] : 0.0;
  return warp_sum(((c[0] + c[1]) + (c[2] + c[3])) + ((c[4] + c[5]) + (c[6] + c[7])));
}

template <int NS>
__device__ __forceinline__ void store_partials_by_column(const double (&v)[NS], double* part,
                                                         int nunits, int unit) {
  __shared__ double col[NS][kDirectThreads];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  __syncthreads();  // col[] may still be read by a previous use
#pragma unroll
  for (int k = 0; k < NS; ++k) col[k][threadIdx.x] = v[k];
  __syncthreads();
  for (int k = warp; k < NS; k += nwarps) {
    const double s = column_sum(col[k], nwarps);
    if (lane == 0) part[k * nunits + unit] = s;
  }
}

template <int NS, class A>
__device__ __forceinline__ void store_partials(const A (&v)[NS], double* part, int nunits,
                                               int unit) {
  if constexpr (sizeof(A) == 8)
    store_partials_by_column<NS>(v, part, nunits, unit);
  else
    store_partials_by_warp<NS, A>(v, part, nunits, unit);
}

// Returns true in every thread of the unit that arrives last for its instance.
__device__ __forceinline__ bool arrive_last(unsigned int* ticket, int nunits) {
  __shared__ int last;
  __syncthreads();  // every warp's partials are written
  if (threadIdx.x == 0) {
    __threadfence();  // ... and visible before this unit's ticket
    unsigned t = atomicAdd(ticket, 1u);
    last = (t == (unsigned)nunits - 1u);
    if (last) __threadfence();
  }
  __syncthreads();
  return last != 0;
}

// Fixed-order sums of the first ns slots over all units, for thread 0.  A slot is summed by 128
// lanes, each adding the slots lane, lane + 128, ... in index order with eight loads in flight,
// then a fixed shuffle tree per 32 lanes, then the four totals in order.  The (slot, 32 lanes)
// pairs are spread over the block's warps, so the slots are summed side by side; the order does
// not depend on the block size, so an instance sums identically whatever launch it runs in.  The
// FP64 pipe takes a warp's addition in 64 cycles per scheduler: four warps, one a scheduler, and
// only thread 0 adds the totals (eight warps and every thread: 3000 cycles instead of 1500).
static __device__ __noinline__ void block_sum_slots(const double* part, int nunits, int ns,
                                                    double (&S)[kSlots]) {
  constexpr int U = 8, LANES = 128, G = LANES / 32;
  __shared__ double wsum[kSlots][G];
  const int lane = threadIdx.x & 31;
  for (int q = threadIdx.x >> 5; q < ns * G; q += blockDim.x >> 5) {
    const double* slot = part + (long long)(q / G) * nunits;
    double s = 0.0;
    int i = (q % G) * 32 + lane;
    for (; i + (U - 1) * LANES < nunits; i += U * LANES) {
      double v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = __ldcg(slot + i + u * LANES);
#pragma unroll
      for (int u = 0; u < U; ++u) s += v[u];
    }
    double v[U];
#pragma unroll
    for (int u = 0; u < U - 1; ++u) v[u] = i + u * LANES < nunits ? __ldcg(slot + i + u * LANES) : 0.0;
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
      if (i - lane + u * LANES < nunits) s += v[u];  // uniform in the warp
    s = warp_sum(s);
    if (lane == 0) wsum[q / G][q % G] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 0; k < ns; ++k) S[k] = (wsum[k][0] + wsum[k][1]) + (wsum[k][2] + wsum[k][3]);
}

__device__ __forceinline__ int exponent_of(double v) {  // biased exponent field
  return (__double2hiint(v) >> 20) & 0x7ff;
}
// Mantissa of a positive normal v as an FP32 value in [1, 2) (truncated to 23 fraction bits).
__device__ __forceinline__ float mantissa_f(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  return __uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29));
}
// FP32 value y in (0, 2) times 2^p as FP64, by integer operations (no FP64 conversion).
__device__ __forceinline__ double widen_pow2(float y, int p) {
  const unsigned b = __float_as_uint(y);
  const unsigned e = (b >> 23) + 1023u - 127u + (unsigned)p;
  return __hiloint2double((int)((e << 20) | ((b & 0x7fffffu) >> 3)), (int)(b << 29));
}
// Exponents that neither the seed nor the products can push out of the normal range.
__device__ __forceinline__ bool mid_range(double v) {
  const int e = exponent_of(v);
  return e > 200 && e < 1846;
}
// c / s in FP64 for s > 0 in the middle of the binary64 range: the FP32 approximation of 1/s as the
// seed Y, e = 1 - s Y (|e| < 2^-21.4), c/s = w (1 + e + e^2), w = c Y; relative error below
// 2^-52.  Five FP64 instructions; the division takes more than ten, each 64 cycles after the other.
__device__ __forceinline__ double quotient(double c, double s) {
  if (!mid_range(s)) return c / s;
  const double Y = widen_pow2(rcp_approx(mantissa_f(s)), 1023 - exponent_of(s));
  const double e = fma(-s, Y, 1.0);
  const double w = c * Y;
  return fma(w, fma(e, e, e), w);
}

// Powers of two for what FP32 holds, where the root mean square of f - <f> (fn2: an FP64 sum), or of
// rt = D^-1/2 r of an FP32 inner solve (rrt, summed in FP32), lies so far out that squares, or what an
// inner solve leaves of them, would leave the FP32 range: both are then brought to about one (D from the
// first cell).  false: none.  Solves in ordinary units have none; a power of two would not change their
// results either, but the repeated residual costs time.
__device__ __forceinline__ bool set_scales(const InstDesc& I, InstState* st, double fn2, double rrt) {
  const double n = (double)I.ncell;
  if (I.mode != 0 || !(fn2 > 0.0) || !isfinite(fn2)) return false;
  const int e = ilogb(fn2 / n) / 2;
  const bool fp32 = st->precision != PREC_FP64;
  if (e >= -30 && e <= 40 && (!fp32 || (rrt > 0x1p-60 * n && rrt < 0x1p80 * n))) return false;
  st->rexp = -e;
  if (fp32) st->texp = ilogb(I.dg[0]) / 2 - e;
  return st->rexp != 0 || st->texp != 0;
}

// ---- phase transitions (run by thread 0 of the last unit) -------------------------------------

static __device__ __noinline__ void transition(const InstDesc& I, InstState* st, int phase,
                                               const double (&S)[kSlots]) {
  st->sweeps += 1;
  if (st->fault && phase != PH_FINAL) {  // a bounded wait expired: stop with what p holds
    st->status = 6;                      // VDP_ETIMEOUT
    st->phase = PH_FINAL;
    return;
  }
  switch (phase) {
    case PH_MEANF:
      st->mu_f = S[0] / (double)I.ncell;
      st->f2 = (double)I.ncell * st->mu_f * st->mu_f;
      st->first_res = 1;
      st->phase = PH_RES64;
      break;
    case PH_RES64: {
      const double rr64 = st->rexp ? ldexp(S[0], -2 * st->rexp) : S[0], rrt = S[1];
      const bool first = st->first_res != 0;
      if (st->first_res) st->sum_p = S[2];  // later: summed by the correction sweep
      if (st->first_res) {
        st->fn2 = S[3];
        st->first_res = 0;
      }
      st->outer += 1;
      const double fn2 = st->fn2;
      if (fn2 <= 1e-28 * st->f2) {  // f is constant up to the rounding of its mean: p = 0
        st->zero_sol = 1;
        st->rel_res = 0.0;
        st->phase = PH_FINAL;
        break;
      }
      if (first && st->rexp == 0 && st->texp == 0 && set_scales(I, st, fn2, rrt)) {
        // the sweep is repeated with the scaled variables (p, and what it adds, are as they were)
        st->first_res = 1;
        st->outer -= 1;
        break;
      }
      const double rel = sqrt(rr64 / fn2);
      st->rel_res = rel;
      if (!isfinite(rel)) {
        st->status = 5;  // VDP_EBREAKDOWN
        st->phase = PH_FINAL;
      } else if (rel <= st->tol) {
        st->phase = PH_FINAL;
      } else if (st->iters >= st->max_iter) {
        st->status = 4;  // VDP_ENOTCONV
        st->phase = PH_FINAL;
      } else if (rrt == 0.0) {  // residual below the inner type's range: cannot refine further
        st->status = 4;
        st->phase = PH_FINAL;
      } else if (I.pc == PC_FIXED && rel > 1e4) {  // the paper's iteration is diverging (the
        st->status = 4;                              // density varies too much for it)
        st->phase = PH_FINAL;
      } else {
        // How far the FP64 residual fell during the last inner solve compared with the scaled
        // inner residual; the next inner target is tightened by it (at least 1).
        if (st->outer > 1 && st->inner_ratio > 0.0) {
          const double obs = sqrt(rr64 / st->rr64_prev) / st->inner_ratio;
          st->eta = fmax(1.0, fmin(obs, 1e6));
        }
        double tau = 0.5 * st->tol * sqrt(fn2 / rr64) / st->eta;
        if (st->precision != PREC_FP64) tau = fmax(tau, st->inner_tol);
        tau = fmin(tau, 0.5);
        st->tau2 = tau * tau;
        st->rr64_prev = rr64;
        st->rr = rrt;
        st->rr0 = rrt;
        st->rz = rrt;
        st->beta = 0.0;
        st->inner_iters = 0;
        st->cheb_j = 1;
        st->phase = I.pc == PC_CHEB ? PH_CHEB : (I.pc >= PC_SPECTRAL ? PH_SPEC : PH_STENCIL);
      }
      st->rr64 = rr64;
      break;
    }
    case PH_STENCIL: {
      const double dq = S[0];
      if (I.pc == PC_FIXED) {
        // the paper's iteration: the stencil sweep has also applied the update x += z,
        // rt -= At z and summed <rt, rt> (S[0]); continue as after an update sweep
        phase = PH_UPDATE;
        goto after_update;
      } else if (dq > 0.0 && isfinite(dq)) {
        st->alpha = quotient(I.pc != PC_JACOBI ? st->rz : st->rr, dq);
        st->phase = PH_UPDATE;
      } else if (st->inner_iters > 0) {
        // loss of curvature at the end of an inner solve: hand the iterate to the refinement
        st->inner_ratio = sqrt(st->rr / st->rr0);
        st->phase = PH_CORRECT;
      } else {
        st->status = 5;
        st->phase = PH_FINAL;
      }
      break;
    }
    case PH_UPDATE:
    after_update: {
      const double rn = S[0];
      st->inner_iters += 1;
      st->iters += 1;
      if (!isfinite(rn)) {
        st->status = 5;
        st->phase = PH_FINAL;
      } else if (rn <= st->tau2 * st->rr0 || st->iters >= st->max_iter ||
                 st->inner_iters >= st->inner_max ||
                 (I.pc == PC_FIXED && rn > 1e8 * st->rr0)) {  // a diverging iteration stops
        st->inner_ratio = sqrt(rn / st->rr0);
        st->phase = PH_CORRECT;
      } else if (I.pc != PC_JACOBI) {  // preconditioned: z = M^-1 rt first, then beta from <rt, z>
        st->rr = rn;
        st->cheb_j = 1;
        st->phase = I.pc == PC_CHEB ? PH_CHEB : PH_SPEC;
      } else {
        st->beta = quotient(rn, st->rr);
        st->rr = rn;
        st->rz = rn;
        st->parity ^= 1;
        st->phase = PH_STENCIL;
      }
      break;
    }
    case PH_CHEB:
    case PH_SPEC: {
      if (I.pc == PC_FIXED) {  // z = the scaled update of the paper's iteration
        st->beta = 0.0;
        st->phase = PH_STENCIL;
        break;
      }
      if (phase == PH_CHEB && st->cheb_j < I.cheb_k - 1) {
        st->cheb_j += 1;
        break;
      }
      const double rz = I.form && st->rexp ? ldexp(S[0], -2 * st->rexp) : S[0];
      if (!(rz > 0.0) || !isfinite(rz)) {  // the preconditioner must stay positive definite
        if (st->inner_iters > 0) {
          st->inner_ratio = sqrt(st->rr / st->rr0);
          st->phase = PH_CORRECT;
        } else {
          st->status = 5;
          st->phase = PH_FINAL;
        }
        break;
      }
      if (st->inner_iters == 0) {
        st->beta = 0.0;
      } else {
        st->beta = quotient(rz, st->rz);
        st->parity ^= 1;
      }
      st->rz = rz;
      st->phase = PH_STENCIL;
      break;
    }
    case PH_CORRECT:
      st->sum_p = S[0];  // sum of the corrected p (for the gauge at the end)
      st->p_set = 1;
      st->phase = PH_RES64;
      break;
    case PH_FINAL:
      st->phase = PH_DONE;
      if (I.remaining) atomicSub(I.remaining, 1);
      break;
    default:
      break;
  }
}

static_assert(sizeof(InstState) % 16 == 0, "the state is copied in 16-byte words");
__device__ __forceinline__ void load_state(const InstState* st, InstState& s) {
  const int4* a = reinterpret_cast<const int4*>(st);
  int4* b = reinterpret_cast<int4*>(&s);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(InstState) / 16); ++i) b[i] = __ldcg(a + i);
}
__device__ __forceinline__ void store_state(InstState* st, const InstState& s) {
  int4* a = reinterpret_cast<int4*>(st);
  const int4* b = reinterpret_cast<const int4*>(&s);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(InstState) / 16); ++i) __stcg(a + i, b[i]);
}

// partial-sum slots each phase produces
__device__ __forceinline__ int phase_slots(int phase) {
  switch (phase) {
    case PH_MEANF: return 1;
    case PH_RES64: return 4;
    case PH_STENCIL:
    case PH_UPDATE:
    case PH_CORRECT:
    case PH_CHEB:
    case PH_SPEC: return 1;
    default: return 0;
  }
}

// nunits units arrive; their partial slots were written by nparts units (default: the same),
// which lets a sweep of several kernels reduce what an earlier kernel of the sweep stored.
__device__ __forceinline__ void finish_sweep(const InstDesc& I, InstState* st, int phase,
                                             int nunits, int nparts = 0, bool sums = true) {
  if (nparts <= 0) nparts = nunits;
  if (arrive_last(I.ticket, nunits)) {  // uniform in the block
    double S[kSlots] = {0.0, 0.0, 0.0, 0.0};
    if (sums) block_sum_slots(I.part, nparts, phase_slots(phase), S);
    if (threadIdx.x == 0) {
      // the whole state in one go (its words are independent loads past L1), the transition on
      // the copy, and back: field by field it was a chain of a dozen trips to L2
      InstState s;
      load_state(st, s);
      transition(I, &s, phase, S);
      store_state(st, s);
      *I.ticket = 0u;
      __threadfence();
    }
  }
}

// The block's copy of an instance's state, read once per block: the words are loaded past L1 (in
// the persistent kernel another SM may have written them moments ago) by the first threads and
// handed on through shared memory.  When every warp of every block read the fields itself, a sweep
// of 1000 blocks sent 100000 requests to the one L2 slice that holds them (the update of a
// 112 x 100 x 90 grid took 25 us with 250 blocks and 32 us with 1000).  Every thread calls it.
__device__ __forceinline__ const InstState& block_state(const InstState* st) {
  __shared__ InstState s;
  __syncthreads();  // a previous copy may still be in use
  if (threadIdx.x < sizeof(InstState) / 16)
    reinterpret_cast<int4*>(&s)[threadIdx.x] = __ldcg(reinterpret_cast<const int4*>(st) + threadIdx.x);
  __syncthreads();
  return s;
}

}  // namespace vdp
