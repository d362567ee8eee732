// vdp_resident.cu -- a whole solve in one cooperative launch, for grids whose sweeps are shorter than
// a kernel launch.
//
// A solve is a chain of sweeps, each needing the one before complete: six launches per iteration of
// the fixed-point method (two more return at once), three per Jacobi iteration.  On a 32^3 grid the
// passes themselves take about a microsecond each and a launch in a graph three to four, so the
// chain is launch bound (32^3: 480 us for 11 iterations; 40 x 37 x 29 FP64 Jacobi: 25 us an
// iteration).  Here the blocks stay resident (cooperative launch), every block runs its share of
// each sweep's units, and a counter in global memory separates the sweeps.  What a sweep costs then
// is trips to L2, 0.5 - 0.7 us each on this GPU, so there are as few as possible in a chain: the
// arrival (a releasing reduction, no answer awaited), the poll, and the partial sums, which every
// block reads and adds for itself -- each block keeps its own copy of the solve's state in shared
// memory and makes the same transition on it.  (With one block summing, moving the state in global
// memory on and releasing the others, a sweep took 10 us instead of 4.)  The partials alternate
// between two halves of the slot array: a block may be a barrier ahead of one that still reads.
//
// Units, partial slots, the order of the sums and the arithmetic of every sweep are those of the
// separate kernels (vdp_sweeps.cuh, vdp_density.cuh, vdp_fft.cuh), so the result is the same bit
// for bit; data that other blocks wrote are read by plain loads, never through the read-only path.
// All waits are bounded: one that expires sets the fault word, which the other waits look at too, and
// ends the launch; the host reports VDP_ETIMEOUT, and a batch starts the member again.
#include <cuda_runtime.h>

#include <mutex>

#include "vdp_density.cuh"
#include "vdp_device.cuh"
#include "vdp_fft.cuh"
#include "vdp_internal.cuh"
#include "vdp_launch.h"
#include "vdp_sweeps.cuh"

namespace vdp {

namespace {

constexpr int kResThreads = 256;
constexpr int kResidentSlots = kSlots * kSMs * 8;  // half of the smallest partial-slot array

// ---- the grid barrier -----------------------------------------------------------------------------

struct GridBarrier {
  ResidentCtl* ctl;
  unsigned target;  // arrivals of all barriers so far, this one included
  unsigned long long limit_ns;

  __device__ __forceinline__ static unsigned load_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
  }

  // Every block's writes before it are visible to every block after it.  false: the wait gave up.
  __device__ __forceinline__ bool sync() {
    target += gridDim.x;
    bool ok = true;
    __syncthreads();
    if (threadIdx.x == 0) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->count) : "memory");
      unsigned polls = 0;
      uint64_t t0 = 0;
      while ((int)(load_acquire(&ctl->count) - target) < 0) {
        if ((++polls & 255u) == 0) {
          const uint64_t now = global_ns();
          if (t0 == 0) t0 = now;
          if (now - t0 > limit_ns || __ldcg(&ctl->fault) != 0) {
            atomicExch(&ctl->fault, 1);
            ok = false;
            break;
          }
        }
      }
    }
    return __syncthreads_and(ok) != 0;
  }
};

// ---- the spectral passes ----------------------------------------------------------------------------

// Rows of an X pass: groups of `per` rows per block and round, spread over all blocks.
__device__ __forceinline__ int rows_each(int rows, int most) {
  const int per = (rows + gridDim.x - 1) / (int)gridDim.x;
  return per < most ? per : most;
}

// The passes and sweeps are separate functions (not inlined), each with its own register allocation;
// one body held them all in 128 registers with kilobytes of spills and took minutes to compile.
// The mirrored row transforms serve both boundary conditions: without the mirror no pair lies in a
// second half.
template <int M1, int M2>
__device__ __noinline__ void x_forward(const SpecArgs& a, const Tables& tb, float2* buf) {
  constexpr int RY = rows_per_block<M1, M2>(), SX = x_row_stride<M1, M2>();
  const int rows = a.ny * a.nz, per = rows_each(rows, RY);
  const int t = threadIdx.x % M1, r = threadIdx.x / M1;
  for (int g = blockIdx.x; (long long)g * per < rows; g += gridDim.x) {
    const long long row = (long long)g * per + r;
    const bool live = r < per && row < rows;
    float2* out = a.spec + row * a.nxp;
    x_fwd_rows<float, M1, M2, true>(a, tb, buf + (r < RY ? r : 0) * SX,
                                  static_cast<const float*>(a.in) + row * a.nxd, row, live, t,
                                  [&](int k, float2 X) { out[k] = X; }, [] {});
    __syncthreads();
  }
}

template <int M1, int M2, bool WEIGHT>
__device__ __noinline__ void x_inverse(const SpecArgs& a, const Tables& tb, float2* buf) {
  constexpr int RY = inv_rows_per_block<M1, M2>(), SB = pad_stride(M2 * (M1 + 1));
  const int rows = a.ny * a.nz, per = rows_each(rows, RY);
  const int t = threadIdx.x % M1, r = threadIdx.x / M1;
  for (int g = blockIdx.x; (long long)g * per < rows; g += gridDim.x) {
    const long long row = (long long)g * per + r;
    const bool live = r < per && row < rows;
    x_inv_rows<float, M1, M2, true, WEIGHT>(a, tb, buf + (r < RY ? r : 0) * SB,
                                             a.spec + (live ? row : 0) * a.nxp, row, live, t, [] {});
    __syncthreads();
  }
}

// Tiles of the Y (WHICH 0 forward, 1 inverse) or Z (2) lines: M1 x 8 threads per tile, several
// tiles side by side in a block.  Steps, exchange layout and arithmetic of k_spec_y and k_spec_z;
// a thread loads its inputs itself.  Z stores <rt, z> as k_spec_z does (part, or null: not
// needed), its blocks (zunits) played by the thread groups.
template <int M1, int M2, int WHICH>
__device__ __noinline__ void lines(const SpecArgs& a, const Tables& tb, const float2* w, const float* lz,
                                   float2* buf, double* part) {
  constexpr bool INV = WHICH == 1, ENERGY = WHICH == 2;
  constexpr int NT = M1 * kTX, SUBS = kResThreads / NT;
  constexpr int R = (M2 + M1 - 1) / M1;
  __shared__ double col[ENERGY ? kResThreads : 1];
  const int sub = threadIdx.x / NT, lt = threadIdx.x - sub * NT;
  const int c = lt % kTX, t = lt / kTX;
  float2* sm = buf + (sub < SUBS ? sub : 0) * line_buffer<M1, M2>();
  const int tiles = a.nxp / kTX;
  const int ntile = tiles * (WHICH == 2 ? a.ny : a.nz);
  const int m = a.nx / 2;
  const long long es = WHICH == 2 ? (long long)a.ny * a.nxp : a.nxp;
  const int nv = ENERGY ? a.zunits : ntile;  // groups of tiles v, v + nv, ...
  for (int v0 = blockIdx.x; v0 < nv; v0 += gridDim.x * SUBS) {
    const int v = v0 + gridDim.x * sub;
    const bool mine = sub < SUBS && v < nv;
    double energy_sum = 0.0;
    for (int j = 0; j * nv < ntile; ++j) {
      const int tile = v + j * nv;
      const bool live = mine && tile < ntile;
      const int line = tile / tiles, kx = (tile - line * tiles) * kTX + c;  // kz (Y) or ky (Z)
      float2* g = a.spec + (WHICH == 2 ? (long long)line * a.nxp : (long long)line * a.ny * a.nxp) + kx;
      if (live) {
        float2 x[M2], y[M2];
#pragma unroll
        for (int j2 = 0; j2 < M2; ++j2) x[j2] = g[(t + M1 * j2) * es];
        dft<M2, 0, 1, INV>(x, y);
#pragma unroll
        for (int k2 = 0; k2 < M2; ++k2) {
          const float2 r = w[t * k2];
          sm[tx<M1>(k2, t, c)] = k2 == 0 || t == 0 ? y[k2] : (INV ? cmulc(y[k2], r) : cmul(y[k2], r));
        }
      }
      __syncthreads();
      if (WHICH != 2) {
        if (live) {
#pragma unroll
          for (int rr = 0; rr < R; ++rr) {
            const int k2 = t + M1 * rr;
            if (k2 < M2) {
              float2 u[M1], o[M1];
#pragma unroll
              for (int j1 = 0; j1 < M1; ++j1) u[j1] = sm[tx<M1>(k2, j1, c)];
              dft<M1, 0, 1, INV>(u, o);
#pragma unroll
              for (int k1 = 0; k1 < M1; ++k1) g[(k2 + M2 * k1) * es] = o[k1];
            }
          }
        }
        __syncthreads();  // the exchange is reused by the next tile
        continue;
      }
      const bool pad = kx > m;
      const float lxy = !live || pad ? 0.f : tb.lx[kx] + tb.ly[line];
      const float wkx = (kx == 0 || kx == m) ? 1.f : 2.f;
      float energy = 0.f;
      if (live) {
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
          const int k2 = t + M1 * rr;
          if (k2 < M2) {
            float2 u[M1], o[M1];
#pragma unroll
            for (int j1 = 0; j1 < M1; ++j1) u[j1] = sm[tx<M1>(k2, j1, c)];
            dft<M1, 0, 1, false>(u, o);
#pragma unroll
            for (int k1 = 0; k1 < M1; ++k1) {
              const float lam = lxy + lz[k2 + M2 * k1];
              const float s = (lam > 0.f && !pad) ? __fdividef(a.scale, lam) : 0.f;
              energy = fmaf(wkx * s, fmaf(o[k1].x, o[k1].x, o[k1].y * o[k1].y), energy);
              o[k1] = cscale(o[k1], s);
            }
            dft<M1, 0, 1, true>(o, u);
#pragma unroll
            for (int l2 = 0; l2 < M1; ++l2)
              sm[tx<M1>(k2, l2, c)] = l2 == 0 || k2 == 0 ? u[l2] : cmulc(u[l2], w[k2 * l2]);
          }
        }
        if (part) energy_sum += (double)energy;
      }
      __syncthreads();
      if (live) {
        float2 x[M2], o[M2];
#pragma unroll
        for (int k2 = 0; k2 < M2; ++k2) x[k2] = sm[tx<M1>(k2, t, c)];
        dft<M2, 0, 1, true>(x, o);
#pragma unroll
        for (int l1 = 0; l1 < M2; ++l1) g[(t + M1 * l1) * es] = o[l1];
      }
      __syncthreads();
    }
    if (ENERGY && part) {  // the group's partial, in the order of store_partials
      col[threadIdx.x] = energy_sum * (double)a.ewt;
      __syncthreads();
      if (mine && lt < 32) {
        const double s = column_sum(col + sub * NT, NT / 32);
        if (lt == 0) part[v] = s;
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ void x_forward_any(const SpecArgs& a, const Tables& tb, float2* buf) {
  switch (a.nx / 2) {
    case 16: x_forward<4, 4>(a, tb, buf); break;
    case 24: x_forward<4, 6>(a, tb, buf); break;
    case 32: x_forward<4, 8>(a, tb, buf); break;
    case 48: x_forward<6, 8>(a, tb, buf); break;
    case 64: x_forward<8, 8>(a, tb, buf); break;
    case 96: x_forward<8, 12>(a, tb, buf); break;
    case 128: x_forward<8, 16>(a, tb, buf); break;
    default: x_forward<16, 16>(a, tb, buf); break;
  }
}

template <bool WEIGHT>
__device__ __forceinline__ void x_inverse_any(const SpecArgs& a, const Tables& tb, float2* buf) {
  switch (a.nx / 2) {
    case 16: x_inverse<4, 4, WEIGHT>(a, tb, buf); break;
    case 24: x_inverse<4, 6, WEIGHT>(a, tb, buf); break;
    case 32: x_inverse<4, 8, WEIGHT>(a, tb, buf); break;
    case 48: x_inverse<6, 8, WEIGHT>(a, tb, buf); break;
    case 64: x_inverse<8, 8, WEIGHT>(a, tb, buf); break;
    case 96: x_inverse<8, 12, WEIGHT>(a, tb, buf); break;
    case 128: x_inverse<8, 16, WEIGHT>(a, tb, buf); break;
    default: x_inverse<16, 16, WEIGHT>(a, tb, buf); break;
  }
}

template <int WHICH>
__device__ __forceinline__ void lines_any(int n, const SpecArgs& a, const Tables& tb, const float2* w,
                                          const float* lz, float2* buf, double* part) {
  switch (n) {
    case 32: lines<4, 8, WHICH>(a, tb, w, lz, buf, part); break;
    case 48: lines<4, 12, WHICH>(a, tb, w, lz, buf, part); break;
    case 64: lines<8, 8, WHICH>(a, tb, w, lz, buf, part); break;
    case 96: lines<8, 12, WHICH>(a, tb, w, lz, buf, part); break;
    case 128: lines<8, 16, WHICH>(a, tb, w, lz, buf, part); break;
    case 192: lines<12, 16, WHICH>(a, tb, w, lz, buf, part); break;
    default: lines<16, 16, WHICH>(a, tb, w, lz, buf, part); break;
  }
}

constexpr int kMaxLine = 256;  // lines of the Y and Z passes here (512 only in the separate kernels)

// Tables in shared memory, copied once: W_m, W_nx, W_ny, W_nz, then the z eigenvalues.
__device__ Tables shared_tables(const SpecArgs& a, float2* st, const float2*& wy, const float2*& wz,
                                const float*& lz, float2*& work) {
  Tables tb = tables(a);
  const int m = a.nx / 2, n = 2 * m + 1 + a.ny + a.nz;
  for (int k = threadIdx.x; k < n; k += blockDim.x) st[k] = a.tw[k];
  float* l = reinterpret_cast<float*>(st + n);
  for (int k = threadIdx.x; k < a.nz; k += blockDim.x) l[k] = tb.lz[k];
  __syncthreads();
  tb.wm = st;
  tb.wr = st + m;
  wy = st + 2 * m + 1;
  wz = wy + a.ny;
  lz = l;
  work = st + (n + (a.nz + 1) / 2 + 1) / 2 * 2;
  return tb;
}

size_t table_bytes(int nx, int ny, int nz) {
  const int n = nx + 1 + ny + nz;
  return sizeof(float2) * (size_t)((n + (nz + 1) / 2 + 1) / 2 * 2);
}

// ---- the solve ------------------------------------------------------------------------------------

// What the instance runs: Jacobi CG, the fixed-point iteration or spectral CG.  The last two run in the
// density form in FP64 and in the scaled form in FP32, Jacobi CG always in the scaled form.
enum ResidentKind { R_JACOBI = 0, R_FIXED = 1, R_SPECTRAL = 2 };

template <class T, bool DENS>
__device__ __noinline__ void unit_res64(const InstDesc& I, const InstState& sn, int u,
                                        double* slots) {
  double acc[kSlots] = {0.0, 0.0, 0.0, 0.0};
  sweep_res64_direct<T, DENS>(I, &sn, u, acc);
  store_partials<kSlots, double>(acc, slots, I.nunits, u);
}

template <class T, int KIND>
__device__ __noinline__ void unit_stencil(const InstDesc& I, const InstState& sn, int u, double* slots) {
  T part[1] = {0};
  if constexpr (KIND == R_FIXED) {
    sweep_stencil_direct<T, T, false, 2, false>(I, &sn, u, part[0]);
  } else {
    if (sn.inner_iters > 0)
      sweep_stencil_direct<T, T, false, 1, false>(I, &sn, u, part[0]);
    else
      sweep_stencil_direct<T, T, false, 0, false>(I, &sn, u, part[0]);
  }
  store_partials<1, T>(part, slots, I.nunits, u);
}

// The FP64 density sweep has four cells per thread where the layout counts two: two units, first
// and second, side by side in a block (second < 0: one).
template <bool FIXED>
__device__ __noinline__ void two_units_density64(const InstDesc& I, const InstState& sn, int first,
                                                 int second, ulonglong2* stages, double* slots) {
  __shared__ double col[kResThreads];
  const int half = threadIdx.x / kDensity64Threads, thread = threadIdx.x % kDensity64Threads;
  const int u = half ? second : first;
  double part = 0.0;
  if (u >= 0) sweep_density64<FIXED, false>(I, sn, u, part, stages, thread);
  __syncthreads();
  col[threadIdx.x] = part;
  __syncthreads();
  if (thread < 32 && u >= 0) {
    const double s = column_sum(col + half * kDensity64Threads, kDensity64Threads / 32);
    if (thread == 0) slots[u] = s;
  }
}

template <class T, bool DENS>
__device__ __noinline__ void unit_flat(const InstDesc& I, const InstState& sn, int phase, int u,
                                       double* slots) {
  const long long c0 = flat_begin(I, u), c1 = flat_begin(I, u + 1);
  if (phase == PH_UPDATE) {
    T part[1] = {0};
    sweep_update<T>(I, &sn, c0, c1, part[0]);
    store_partials<1, T>(part, slots, I.nunits_f, u);
  } else if (phase == PH_FINAL) {
    sweep_final(I, &sn, c0, c1);
  } else {
    double sum[1] = {0.0};
    if (phase == PH_MEANF)
      sweep_meanf(I, c0, c1, sum[0]);
    else
      sweep_correct<T, DENS>(I, c0, c1, sn.p_set == 0, sn.texp, sum[0]);
    store_partials<1, double>(sum, slots, I.nunits_f, u);
  }
}

// Place of a phase in a round of the separate launches: residual, preconditioner, stencil, flat sweeps.
__device__ __forceinline__ int round_place(int phase) {
  return phase == PH_RES64 ? 0 : phase == PH_SPEC ? 1 : phase == PH_STENCIL ? 2 : 3;
}

template <class T, int KIND>
__global__ void __launch_bounds__(kResThreads, sizeof(T) == 8 && KIND != R_JACOBI ? 1 : 2)
    k_resident(const InstDesc* desc, const __grid_constant__ SpecArgs spec, ResidentCtl* ctl,
               unsigned max_rounds) {
  constexpr bool SPEC = KIND != R_JACOBI, DENS = SPEC && sizeof(T) == 8;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(16) unsigned char desc_bytes[sizeof(InstDesc)];
  for (int k = threadIdx.x; k < (int)(sizeof(InstDesc) / 4); k += blockDim.x)
    reinterpret_cast<unsigned*>(desc_bytes)[k] = __ldcg(reinterpret_cast<const unsigned*>(desc) + k);
  __syncthreads();
  const InstDesc& I = *reinterpret_cast<const InstDesc*>(desc_bytes);
  __shared__ InstState sn;  // this block's copy of the state; all blocks' copies stay equal
  if (threadIdx.x < sizeof(InstState) / 16)
    reinterpret_cast<int4*>(&sn)[threadIdx.x] = __ldcg(reinterpret_cast<const int4*>(I.st) + threadIdx.x);
  Tables tb{};
  const float2 *wy = nullptr, *wz = nullptr;
  const float* lz = nullptr;
  float2* work = reinterpret_cast<float2*>(smem);
  if constexpr (SPEC) tb = shared_tables(spec, reinterpret_cast<float2*>(smem), wy, wz, lz, work);
  ulonglong2* stages = reinterpret_cast<ulonglong2*>(work);
  __syncthreads();
  GridBarrier bar{ctl, __ldcg(&ctl->extra), __ldcg(&ctl->limit_ns)};
  bool ok = true;
  unsigned rounds = 0;
  int place = 3;
  for (unsigned done = 0; ok; ++done) {
    int phase = sn.phase;
    if (phase >= PH_DONE) break;
    if (round_place(phase) <= place && rounds++ == max_rounds) break;
    place = round_place(phase);
    double* slots = I.part + (done & 1u) * kResidentSlots;
    int nparts = I.nunits;
    bool applied = false;  // the preconditioner's sweep was part of this round
    if (SPEC && phase == PH_SPEC) {
      x_forward_any(spec, tb, work);
      if (!(ok = bar.sync())) break;
      lines_any<0>(spec.ny, spec, tb, wy, nullptr, work, slots);
      if (!(ok = bar.sync())) break;
      lines_any<2>(spec.nz, spec, tb, wz, lz, work, KIND == R_SPECTRAL ? slots : nullptr);
      if (!(ok = bar.sync())) break;
      lines_any<1>(spec.ny, spec, tb, wy, nullptr, work, slots);
      if (!(ok = bar.sync())) break;
      x_inverse_any<!DENS>(spec, tb, work);  // scaled form: z = W x
      if (KIND == R_FIXED) {  // always followed by the sweep: one transition for both
        if (!(ok = bar.sync())) break;
        applied = true;
        phase = PH_STENCIL;
        place = round_place(phase);
      } else {
        nparts = spec.zunits;
      }
    }
    if (phase == PH_RES64) {
      for (int u = blockIdx.x; u < I.nunits; u += gridDim.x) unit_res64<T, DENS>(I, sn, u, slots);
    } else if (phase == PH_STENCIL) {
      if constexpr (DENS) {
        for (int u = blockIdx.x; u < I.nunits; u += 2 * gridDim.x)
          two_units_density64<KIND == R_FIXED>(I, sn, u, u + gridDim.x < I.nunits ? u + gridDim.x : -1,
                                               stages, slots);
      } else {
        for (int u = blockIdx.x; u < I.nunits; u += gridDim.x)
          unit_stencil<T, KIND>(I, sn, u, slots);
      }
    } else if (phase != PH_SPEC) {
      nparts = I.nunits_f;
      for (int u = blockIdx.x; u < I.nunits_f; u += gridDim.x) unit_flat<T, DENS>(I, sn, phase, u, slots);
    }
    if (!(ok = bar.sync())) break;
    double S[kSlots] = {0.0, 0.0, 0.0, 0.0};
    block_sum_slots(slots, nparts, phase_slots(phase), S);
    if (threadIdx.x == 0) {
      if (applied) transition(I, &sn, PH_SPEC, S);
      transition(I, &sn, phase, S);
    }
    __syncthreads();
  }
  if (!ok && threadIdx.x == 0) {  // a wait expired: the sweep is incomplete, the solve ends
    sn.status = 6;                  // VDP_ETIMEOUT
    sn.phase = PH_DONE;
  }
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x < sizeof(InstState) / 16)
    __stcg(reinterpret_cast<int4*>(I.st) + threadIdx.x, reinterpret_cast<const int4*>(&sn)[threadIdx.x]);
}

using ResidentKernel = void (*)(const InstDesc*, const SpecArgs, ResidentCtl*, unsigned);

ResidentKernel resident_kernel(int prec, int kind) {
  if (prec == PREC_FP64)
    return kind == R_JACOBI  ? k_resident<double, R_JACOBI>
           : kind == R_FIXED ? k_resident<double, R_FIXED>
                             : k_resident<double, R_SPECTRAL>;
  return kind == R_JACOBI  ? k_resident<float, R_JACOBI>
         : kind == R_FIXED ? k_resident<float, R_FIXED>
                           : k_resident<float, R_SPECTRAL>;
}

int resident_kind(const InstDesc& d) {
  return d.pc == PC_JACOBI ? R_JACOBI : d.pc == PC_FIXED ? R_FIXED : R_SPECTRAL;
}

// Shared memory of the transforms' buffers: 40 KB of rows at most, and the tiles of 256 threads.
size_t line_bytes(int n) {
  switch (n) {
    case 32: return sizeof(float2) * 8 * line_buffer<4, 8>();
    case 48: return sizeof(float2) * 8 * line_buffer<4, 12>();
    case 64: return sizeof(float2) * 4 * line_buffer<8, 8>();
    case 96: return sizeof(float2) * 4 * line_buffer<8, 12>();
    case 128: return sizeof(float2) * 4 * line_buffer<8, 16>();
    case 192: return sizeof(float2) * 2 * line_buffer<12, 16>();
    default: return sizeof(float2) * 2 * line_buffer<16, 16>();
  }
}

size_t resident_smem(int prec, int kind, const SpecArgs& a) {
  if (kind == R_JACOBI) return 0;
  size_t b = 40960;
  for (int n : {a.ny, a.nz})
    if (line_bytes(n) > b) b = line_bytes(n);
  if (prec == PREC_FP64 && density64_smem(kResThreads) > b) b = density64_smem(kResThreads);
  return table_bytes(a.nx, a.ny, a.nz) + b;
}

constexpr int kMaxDevices = 64;

}  // namespace

// Where the line lies (us a solve to 1e-9, resident and in a graph of launches): FP32 fixed point 64^3
// 440 and 554, 96^3 640 and 643, 128 x 96 x 96 672 and 683, 128 x 128 x 96 850 and 803, 128^3 980 and
// 925; FP64 fixed point 64^3 390 and 506, 96^3 750 and 728, 128 x 96 x 96 784 and 751; spectral CG FP32
// 96^3 1314 and 1343, 128 x 96 x 96 1452 and 1427, FP64 64^3 860 and 1073, 96^3 1589 and 1526; Jacobi FP32
// 96^3 9918 and 12437, 128 x 96 x 96 12559 and 14297, FP64 17367 and 18645, 24908 and 24921.
bool resident_supported(const InstDesc& d, int prec) {
  if (prec == PREC_MIXED_BF16 || d.mode != 0 || d.ncell > kResidentCells ||
      kSlots * d.nunits > kResidentSlots || d.nunits_f > kResidentSlots)
    return false;
  if (d.pc == PC_JACOBI) return d.form == 0;
  return d.form == (prec == PREC_FP64 ? 1 : 0) && (d.pc == PC_FIXED || d.pc == PC_SPECTRAL) && d.ny <= kMaxLine && d.nz <= kMaxLine;
}

cudaError_t launch_resident(int prec, const InstDesc& d, const InstDesc* desc, const SpecArgs& spec,
                            ResidentCtl* ctl, unsigned max_rounds, int max_blocks, cudaStream_t s) {
  const int kind = resident_kind(d);
  if (kind != R_JACOBI && spec.zunits > kResidentSlots) return cudaErrorInvalidValue;
  const ResidentKernel k = resident_kernel(prec, kind);
  const size_t smem = resident_smem(prec, kind, spec);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  static std::mutex mu;
  static int sms[kMaxDevices];  // 0: this device's set-up is still to do
  {
    std::lock_guard<std::mutex> lk(mu);
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (sms[dev] == 0) {
      for (int p : {PREC_FP64, PREC_MIXED})
        for (int q : {R_FIXED, R_SPECTRAL})
          if ((e = cudaFuncSetAttribute((const void*)resident_kernel(p, q),
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024)) !=
              cudaSuccess)
            return e;
      if ((e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    }
  }
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kResThreads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // as many blocks as the widest sweep has units, at most what is resident at once
  int most = d.nunits > d.nunits_f ? d.nunits : d.nunits_f;
  if (kind != R_JACOBI) {
    const int tiles = spec.nxp / kTX * (spec.ny > spec.nz ? spec.ny : spec.nz);
    if (tiles > most) most = tiles;
  }
  int grid = per_sm * sms[dev];
  if (grid > most) grid = most;
  if (max_blocks > 0 && grid > max_blocks) grid = max_blocks;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kResThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // all blocks resident: the barrier is safe
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[] = {(void*)&desc, (void*)&spec, (void*)&ctl, (void*)&max_rounds};
  return cudaLaunchKernelExC(&cfg, (const void*)k, args);
}

}  // namespace vdp
