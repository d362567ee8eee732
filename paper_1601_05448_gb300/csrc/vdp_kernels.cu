// vdp_kernels.cu -- sm_103a kernels of libvdp.
//
// Problem (Sec. 3.4 of Pouransari, Mortazavi & Mani, arXiv:1601.05448): div((1/rho) grad p) = f
// on a uniform triply periodic staggered grid (Sec. 3.1, Sec. 3.2 case 1), discretised in
// conservative face-flux form with 1/rho on a face taken from the arithmetic mean of the two
// adjacent cell densities (the averaging App. B applies to rho off the cell centres), and
// f replaced by f - <f> (the compatibility constant chi' of App. A).
//
// Solver.  With A the FP64 operator and D its (negated) diagonal, the inner Krylov solver works
// on the Jacobi-scaled system  At = D^-1/2 (-A) D^-1/2  (unit diagonal, off-diagonal -bt with
// bt = b sinv_l sinv_r on each face).  Conjugate gradients on At is Jacobi-preconditioned CG in
// scaled variables, with one coefficient stream fewer and fewer FP64 operations per cell.  An
// outer FP64 loop evaluates the true residual r = (f - <f>) - A p, hands rt = D^-1/2 r to the
// inner solver (FP64, or FP32 with FP32/BF16 coefficients), and applies p -= D^-1/2 x.
//
// The preconditioned residual z (Chebyshev polynomial or the spectral passes of
// vdp_spectral.cu) replaces rt as the stencil sweep's source; the paper's fixed-point iteration
// runs as the same sweeps with beta = 0 and alpha = 1.
//
// Kernels (the coefficient builders are in vdp_setup.cu): three sweep kernels, each advancing every
// instance whose phase is of its kind (see vdp_internal.cuh): k_res64_direct (FP64 residual),
// k_stencil_direct (search direction, stencil product and <d, q>; Chebyshev sweeps in its
// CHEBOK variant) and k_flat (element-wise phases).  The direct sweeps march each work unit
// through a z chunk with three planes in registers: a thread owns 16 bytes of one row, takes
// its x neighbours from the adjacent lanes by warp shuffle and the rows above and below from
// L1/L2, and waits on no other warp.  k_stencil_tma is the TMA-staged variant (cp.async.bulk
// row blocks into a shared-memory ring, mbarrier completion with bounded waits, one block
// barrier per plane), kept as an option; k_persistent runs all of them for a batch.
#include "vdp_device.cuh"
#include "vdp_internal.cuh"
#include "vdp_launch.h"
#include "vdp_sweeps.cuh"

namespace vdp {

// ---- small helpers ----------------------------------------------------------------------------

template <class T> __device__ __forceinline__ T from_double_rn(double v);
template <> __device__ __forceinline__ double from_double_rn<double>(double v) { return v; }
template <> __device__ __forceinline__ float from_double_rn<float>(double v) {
  return __double2float_rn(v);
}

// global row index of ring row ry (0 = halo row above the tile, ty + 1 = halo row below)
__device__ __forceinline__ int ring_gy(int ry, int y0, int ny) {
  int gy = y0 + ry - 1;
  if (gy < 0) gy += ny;
  if (gy >= ny) gy -= ny;
  return gy;
}

// ---- TMA bulk copies and mbarriers (inline PTX) -----------------------------------------------

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// order this thread's earlier generic-proxy shared accesses before later async-proxy (TMA) ones
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for phase `parity` of an mbarrier, giving up after ~2 s (returns false); no hang.
__device__ __noinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (global_ns() - t0 > 2000000000ull) return false;
  }
}

// ---- unit geometry -------------------------------------------------------------------------------

struct Seg {
  int y0, ty;   // row tile: first row, rows
  int z0, nzs;  // first plane, planes
};

// Calls fn(seg) for the z run of work unit `unit`: row tile unit % uy, z chunk unit / uy.  Units
// that run at the same time share z chunks, so the halo rows one unit reads are the rows its
// neighbours stream at about the same moment (L2 hits rather than DRAM re-reads).
template <class F>
__device__ __forceinline__ void for_each_segment(const InstDesc& I, int unit, F&& fn) {
  const int tile = unit % I.uy, chunk = unit / I.uy;
  Seg s;
  s.y0 = tile * I.ty;
  s.ty = min(I.ty, I.ny - s.y0);
  s.z0 = (int)((long long)chunk * I.nz / I.zc);
  s.nzs = (int)((long long)(chunk + 1) * I.nz / I.zc) - s.z0;
  if (s.nzs > 0) fn(s);
}

// ---- the stencil sweep: TMA-fed z march -----------------------------------------------------------


template <class T, class BT>
struct StageLayout {
  int nx, ty;
  __device__ __forceinline__ size_t r_off() const { return 0; }
  __device__ __forceinline__ size_t o_off() const { return (size_t)(ty + 2) * nx * sizeof(T); }
  __device__ __forceinline__ size_t bx_off() const { return (size_t)2 * (ty + 2) * nx * sizeof(T); }
  __device__ __forceinline__ size_t by_off() const { return bx_off() + (size_t)ty * nx * sizeof(BT); }
  __device__ __forceinline__ size_t bz_off() const {
    return by_off() + (size_t)(ty + 1) * nx * sizeof(BT);
  }
  __device__ __forceinline__ size_t bd_off() const { return bz_off() + (size_t)ty * nx * sizeof(BT); }
};

// Issue part `part` (0..3) of the bulk copies of plane `j` (j = -1 .. nzs) of segment `sg` into
// stage buffer `buf`; lane 0 of warps 0..3 issue one part each, so the four arrive on the stage's
// mbarrier (count 4) with their own byte counts.  Part 0: rt rows (tile + one halo row above and
// below); 1: d_old rows (when the direction recurrence needs it); 2: x and y coefficients;
// 3: z coefficients (+ BF16 diagonal correction).  Plane -1 needs only rt / d_old (it supplies d
// below the segment); plane nzs needs rt / d_old and the z coefficients (its low z face is the
// high face of the last plane).
template <class T, class BT>
__device__ __forceinline__ void issue_part(int part, const InstDesc& I, const Seg& sg, int j,
                                           unsigned char* buf, uint64_t* bar, const T* rt,
                                           const T* dold, bool use_old, const BT* sx,
                                           const BT* sy, const BT* sz, const BT* sd) {
  const StageLayout<T, BT> L{I.nx, I.ty};
  int zg = sg.z0 + j;
  if (zg < 0) zg += I.nz;
  if (zg >= I.nz) zg -= I.nz;
  const int nx = I.nx;
  const long long plane = (long long)zg * I.ny;
  const uint32_t rowT = nx * sizeof(T), rowB = nx * sizeof(BT);
  if (part <= 1) {
    const T* src = part == 0 ? rt : dold;
    if (part == 1 && !use_old) {
      mbar_arrive_expect_tx(bar, 0);
      return;
    }
    const int top = ring_gy(0, sg.y0, I.ny), bot = ring_gy(sg.ty + 1, sg.y0, I.ny);
    unsigned char* R = buf + (part == 0 ? L.r_off() : L.o_off());
    mbar_arrive_expect_tx(bar, (uint32_t)(sg.ty + 2) * rowT);
    bulk_g2s(R, src + (plane + top) * nx, rowT, bar);
    bulk_g2s(R + rowT, src + (plane + sg.y0) * nx, sg.ty * rowT, bar);
    bulk_g2s(R + (sg.ty + 1) * rowT, src + (plane + bot) * nx, rowT, bar);
  } else if (part == 2) {
    if (!(j >= 0 && j < sg.nzs)) {
      mbar_arrive_expect_tx(bar, 0);
      return;
    }
    mbar_arrive_expect_tx(bar, (uint32_t)(2 * sg.ty + 1) * rowB);
    bulk_g2s(buf + L.bx_off(), sx + (plane + sg.y0) * nx, sg.ty * rowB, bar);
    unsigned char* BY = buf + L.by_off();
    if (sg.y0 + sg.ty < I.ny) {
      bulk_g2s(BY, sy + (plane + sg.y0) * nx, (sg.ty + 1) * rowB, bar);
    } else {  // the row below the tile wraps to row 0
      bulk_g2s(BY, sy + (plane + sg.y0) * nx, sg.ty * rowB, bar);
      bulk_g2s(BY + sg.ty * rowB, sy + plane * nx, rowB, bar);
    }
  } else {
    const bool need_z = j >= 0, need_d = CoefTraits<BT>::kDiag && j >= 0 && j < sg.nzs;
    mbar_arrive_expect_tx(bar, (uint32_t)((need_z ? sg.ty : 0) + (need_d ? sg.ty : 0)) * rowB);
    if (need_z) bulk_g2s(buf + L.bz_off(), sz + (plane + sg.y0) * nx, sg.ty * rowB, bar);
    if (need_d) bulk_g2s(buf + L.bd_off(), sd + (plane + sg.y0) * nx, sg.ty * rowB, bar);
  }
}

// d = rt + beta d_old in place over all ring rows of a stage
template <class T>
__device__ __forceinline__ void form_direction(T* R, const T* O, int cells, T beta) {
  constexpr int V = VecW<T>::V;
  for (int v = threadIdx.x; v < cells / V; v += blockDim.x) {
    T a[V], b[V];
    VecIO<T, V>::ld(R + v * V, a);
    VecIO<T, V>::ld(O + v * V, b);
#pragma unroll
    for (int k = 0; k < V; ++k) a[k] = fma(beta, b[k], a[k]);
    VecIO<T, V>::st(R + v * V, a);
  }
}

// One z march per segment.  Iteration k (plane k of the segment) forms d two planes ahead
// (plane k + 2, stage k + 3) while it applies the stencil to plane k from the stages of planes
// k - 1, k, k + 1, so one block barrier per plane separates the two; the barrier also frees the
// stage of plane k - 1, which thread 0 then refills with plane k - 1 + S.  S >= 4 stages.
template <class T, class BT>
__device__ void sweep_stencil(const InstDesc& I, InstState* st, int unit, T& part,
                              unsigned char* smem) {
  constexpr int V = VecW<T>::V;
  constexpr bool kDiag = CoefTraits<BT>::kDiag;
  __shared__ __align__(8) uint64_t bars[kMaxStages];
  __shared__ int timed_out;
  const int S = I.stages;
  const int nx = I.nx;
  const StageLayout<T, BT> L{nx, I.ty};
  const size_t sbytes = stage_bytes(nx, I.ty, sizeof(T), sizeof(BT), kDiag);
  const T beta = (T)st->beta;
  const bool use_old = st->inner_iters > 0;
  const T* rt = static_cast<const T*>(I.r);
  const T* dold = static_cast<const T*>(st->parity ? I.d1 : I.d0);
  T* dnew = static_cast<T*>(st->parity ? I.d0 : I.d1);
  T* q = static_cast<T*>(I.q);
  const BT* sx = static_cast<const BT*>(I.sx);
  const BT* sy = static_cast<const BT*>(I.sy);
  const BT* sz = static_cast<const BT*>(I.sz);
  const BT* sd = static_cast<const BT*>(I.sd);

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) mbar_init(&bars[s], 4);  // four issuing lanes arrive per fill
    fence_mbar_init();
    timed_out = 0;
  }
  __syncthreads();
  uint32_t parity = 0;  // bit s: phase parity of the next completion of stage s
  T sum[V];
#pragma unroll
  for (int k = 0; k < V; ++k) sum[k] = 0;

  auto stage_ptr = [&](int jj) { return smem + (size_t)(jj % S) * sbytes; };
  auto wait_stage = [&](int jj) {
    const int s = jj % S;
    if (!timed_out && !mbar_wait(&bars[s], (parity >> s) & 1u)) timed_out = 1;
    parity ^= 1u << s;
  };
  auto ready = [&](int jj, int ring_cells) {  // wait for stage jj and form d in it
    wait_stage(jj);
    if (use_old) {
      unsigned char* b = stage_ptr(jj);
      form_direction<T>(reinterpret_cast<T*>(b + L.r_off()),
                        reinterpret_cast<const T*>(b + L.o_off()), ring_cells, beta);
    }
  };

  for_each_segment(I, unit, [&](const Seg& sg) {
    const int np = sg.nzs + 2;  // planes -1 .. nzs, stage index jj = j + 1
    const int ring_cells = (sg.ty + 2) * nx;
    const int part = threadIdx.x >> 5;  // issuing lanes: lane 0 of warps 0..3
    const bool issuer = (threadIdx.x & 31) == 0 && part < 4;
    if (issuer) {
      fence_proxy_async_smem();  // stage buffers were last touched by ordinary loads/stores
      for (int jj = 0; jj < min(S, np); ++jj)
        issue_part<T, BT>(part, I, sg, jj - 1, stage_ptr(jj), &bars[jj % S], rt, dold, use_old, sx,
                          sy, sz, sd);
    }
    ready(0, ring_cells);  // plane -1
    ready(1, ring_cells);  // plane 0
    ready(2, ring_cells);  // plane 1 (exists: np >= 3)
    __syncthreads();
    const int vrow = nx / V;
    const int own = sg.ty * vrow;  // vectors in the tile's own rows
    for (int k = 0; k < sg.nzs; ++k) {
      const int z = sg.z0 + k;
      if (k + 3 < np) ready(k + 3, ring_cells);  // plane k + 2
      const unsigned char* bm = stage_ptr(k);
      const unsigned char* bc = stage_ptr(k + 1);
      const unsigned char* bp = stage_ptr(k + 2);
      const T* Dm = reinterpret_cast<const T*>(bm + L.r_off());
      const T* Dc = reinterpret_cast<const T*>(bc + L.r_off());
      const T* Dp = reinterpret_cast<const T*>(bp + L.r_off());
      const BT* Bx = reinterpret_cast<const BT*>(bc + L.bx_off());
      const BT* By = reinterpret_cast<const BT*>(bc + L.by_off());
      const BT* Bz = reinterpret_cast<const BT*>(bc + L.bz_off());
      const BT* Bd = reinterpret_cast<const BT*>(bc + L.bd_off());
      const BT* Bzp = reinterpret_cast<const BT*>(bp + L.bz_off());
      for (int v = threadIdx.x; v < own; v += blockDim.x) {
        const int row = v / vrow;               // 0 .. ty-1
        const int x0 = (v - row * vrow) * V;
        const int o = (row + 1) * nx;           // ring row of this tile row
        const int ob = row * nx;                // coefficient row
        T dc[V], du[V], dd[V], dzm[V], dzp[V];
        T bx[V], by[V], byd[V], bz[V], bzp[V], bd[V];
        VecIO<T, V>::ld(Dc + o + x0, dc);
        VecIO<T, V>::ld(Dc + o - nx + x0, du);
        VecIO<T, V>::ld(Dc + o + nx + x0, dd);
        VecIO<T, V>::ld(Dm + o + x0, dzm);
        VecIO<T, V>::ld(Dp + o + x0, dzp);
        CoefIO<BT, T, V>::ld(Bx + ob + x0, bx);
        CoefIO<BT, T, V>::ld(By + ob + x0, by);
        CoefIO<BT, T, V>::ld(By + ob + nx + x0, byd);
        CoefIO<BT, T, V>::ld(Bz + ob + x0, bz);
        CoefIO<BT, T, V>::ld(Bzp + ob + x0, bzp);
        if (kDiag) CoefIO<BT, T, V>::ld(Bd + ob + x0, bd);
        const int xl = x0 == 0 ? nx - 1 : x0 - 1;
        const int xr = x0 + V == nx ? 0 : x0 + V;
        const T dl = Dc[o + xl], dr = Dc[o + xr];
        const T bxr = (T)ld1(Bx + ob + xr);
        T qv[V];
#pragma unroll
        for (int k2 = 0; k2 < V; ++k2) {
          const T left = k2 == 0 ? dl : dc[k2 - 1];
          const T right = k2 == V - 1 ? dr : dc[k2 + 1];
          const T bright = k2 == V - 1 ? bxr : bx[k2 + 1];
          T a = dc[k2];
          if (kDiag) a = fma(bd[k2], dc[k2], a);
          a = fma(-bx[k2], left, a);
          a = fma(-bright, right, a);
          a = fma(-by[k2], du[k2], a);
          a = fma(-byd[k2], dd[k2], a);
          a = fma(-bz[k2], dzm[k2], a);
          a = fma(-bzp[k2], dzp[k2], a);
          qv[k2] = a;
          sum[k2] = fma(dc[k2], a, sum[k2]);
        }
        const long long g = ((long long)z * I.ny + sg.y0 + row) * nx + x0;
        VecIO<T, V>::st(dnew + g, dc);
        VecIO<T, V>::st(q + g, qv);
      }
      fence_proxy_async_smem();  // this thread's shared accesses before the refill's TMA writes
      __syncthreads();           // stage k (plane k - 1) is free; plane k + 2 is formed
      if (issuer && k + S < np) {
        issue_part<T, BT>(part, I, sg, k + S - 1, stage_ptr(k + S), &bars[(k + S) % S], rt, dold,
                          use_old, sx, sy, sz, sd);
      }
    }
  });
  if (timed_out && threadIdx.x == 0) atomicExch(&st->fault, 1);
  T tot = 0;
#pragma unroll
  for (int k = 0; k < V; ++k) tot += sum[k];
  part = tot;
}

// ---- the FP64 residual sweep (a few times per solve): z march through a three-plane ring ---------

// zero: the solve starts from p = 0 and p has not been written yet (it is not read)
__device__ __forceinline__ void fill_p(const InstDesc& I, const Seg& sg, double* ring, int stride,
                                       int slot, int zg, bool zero) {
  const int nx = I.nx;
  const int cells = (sg.ty + 2) * nx;
  const long long pz = (long long)zg * nx * I.ny;
  double* dst = ring + slot * stride;
  for (int m = threadIdx.x; m < cells; m += blockDim.x) {
    const int ry = m / nx, x = m - ry * nx;
    dst[m] = zero ? 0.0 : I.p[pz + (long long)ring_gy(ry, sg.y0, I.ny) * nx + x];
  }
}

// r = (f - <f>) - A p; rt = D^-1/2 r in the inner type; sums of r^2, rt^2, p and, on the first
// call, (f - <f>)^2
template <class T>
__device__ void sweep_res64(const InstDesc& I, const InstState* st, int unit,
                            double (&acc)[kSlots], double* ring) {
  const int nx = I.nx, ny = I.ny, nz = I.nz;
  const int stride = (I.ty + 2) * nx;
  const long long plane = (long long)nx * ny;
  const double mu = st->mu_f;
  const bool first = st->first_res != 0;
  const bool zero = st->p_set == 0;  // from p = 0, before the first correction
  T* rt = static_cast<T*>(I.r);
  double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
  for_each_segment(I, unit, [&](const Seg& sg) {
    int zm = sg.z0 - 1;
    if (zm < 0) zm += nz;
    __syncthreads();  // ring reuse across segments
    fill_p(I, sg, ring, stride, 0, zm, zero);
    fill_p(I, sg, ring, stride, 1, sg.z0, zero);
    const int own = sg.ty * nx;
    for (int k = 0; k < sg.nzs; ++k) {
      const int z = sg.z0 + k;
      const int zp = z + 1 == nz ? 0 : z + 1;
      const int sm = k % 3, sc = (k + 1) % 3, sp = (k + 2) % 3;
      fill_p(I, sg, ring, stride, sp, zp, zero);
      __syncthreads();
      const double* Rm = ring + sm * stride;
      const double* Rc = ring + sc * stride;
      const double* Rp = ring + sp * stride;
      for (int m = threadIdx.x; m < own; m += blockDim.x) {
        const int ry = m / nx + 1, x = m - (ry - 1) * nx;
        const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
        const int gy = sg.y0 + ry - 1;
        const int gyp = gy + 1 == ny ? 0 : gy + 1;
        const long long row = (long long)z * plane + (long long)gy * nx;
        const long long c = row + x;
        const int o = ry * nx;
        const double pc = Rc[o + x];
        double ap = __ldg(I.bx + row + xp) * (Rc[o + xp] - pc) - __ldg(I.bx + c) * (pc - Rc[o + xm]);
        ap += __ldg(I.by + (long long)z * plane + (long long)gyp * nx + x) * (Rc[o + nx + x] - pc) -
              __ldg(I.by + c) * (pc - Rc[o - nx + x]);
        ap += __ldg(I.bz + (long long)zp * plane + (long long)gy * nx + x) * (Rp[o + x] - pc) -
              __ldg(I.bz + c) * (pc - Rm[o + x]);
        const double f0 = __ldg(I.rhs + c) - mu;
        const double r = f0 - ap;
        const T tv = from_double_rn<T>(__ldg(I.sinv + c) * r);
        rt[c] = tv;
        a0 = fma(r, r, a0);
        a1 = fma((double)tv, (double)tv, a1);
        a2 += pc;
        if (first) a3 = fma(f0, f0, a3);
      }
      __syncthreads();
    }
  });
  acc[0] = a0;
  acc[1] = a1;
  acc[2] = a2;
  acc[3] = a3;
}

// ---- the step kernels ----------------------------------------------------------------------------
// One sweep per launch for every instance of the batch whose phase is of the kernel's kind: the
// stencil kind (RES64, STENCIL: shared-memory z march, stencil units) or the flat kind (MEANF,
// UPDATE, CORRECT, FINAL: streaming, flat units).  The host alternates the two kinds; a launch
// whose instances are all in the other kind's phase exits at once.

// One stencil-kind unit of instance I: WHICH = 0 handles the RES64 and STENCIL phases, 1 only
// STENCIL, 2 only RES64; a no-op for other phases.
// KIND (direct form): 0 = CG sweeps only (the Chebyshev sweep compiled out, so the kernel keeps
// the register budget of the plain stencil sweep), 1 = CG and Chebyshev sweeps, 2 = the
// fixed-point iteration's sweep only.  The persistent batch kernel uses 1.
// PERSIST: that kernel's units, in which every thread reads the state words that it needs: a block runs
// units one after the other there, and handing the state on through shared memory cost each of them two
// barriers (64 grids of 32^3 mixed 12.3 ms, now 11.8, FP64 24.4 and 23.4; 32 of 64^3 79.0 and 75.7).
template <class T, class BT, int MODE, int WHICH = 0, int KIND = 1, bool PERSIST = false>
__device__ __forceinline__ void stencil_kind_unit(const InstDesc& I, int unit,
                                                  unsigned char* smem_raw) {
  InstState* st = I.st;
  InstState own;
  if (PERSIST) load_state(st, own);
  const InstState& sn = PERSIST ? own : block_state(st);
  const int phase = sn.phase;  // decides whether this unit has work
  if (phase != PH_RES64 && phase != PH_STENCIL && phase != PH_CHEB) return;
  if ((WHICH == 1 && phase == PH_RES64) || (WHICH == 2 && phase != PH_RES64)) return;
  if ((MODE != 0 || KIND != 1) && phase == PH_CHEB) return;  // direct form, KIND 1 only
  if (I.form != 0) return;  // the density form has its own kernels
  if (WHICH != 1 && phase == PH_RES64) {
    double acc[kSlots] = {0.0, 0.0, 0.0, 0.0};
    if (MODE == 0)
      sweep_res64_direct<T>(I, &sn, unit, acc);
    else
      sweep_res64<T>(I, &sn, unit, acc, reinterpret_cast<double*>(smem_raw));
    if constexpr (MODE == 0)
      store_partials<kSlots, double>(acc, I.part, I.nunits, unit);
    else  // blocks of up to 512 threads, and hardly any static shared memory left
      store_partials_by_warp<kSlots, double>(acc, I.part, I.nunits, unit);
  } else if (WHICH != 2) {
    T part[1] = {0};
    if constexpr (MODE != 0) {
      sweep_stencil<T, BT>(I, st, unit, part[0], smem_raw);
    } else if constexpr (KIND == 2) {
      sweep_stencil_direct<T, BT, false, 2>(I, &sn, unit, part[0]);
    } else {
      if (KIND == 1 && phase == PH_CHEB)
        sweep_stencil_direct<T, BT, KIND == 1, 0>(I, &sn, unit, part[0]);
      else if (I.pc == PC_FIXED)  // the persistent kernel runs every kind of instance
        sweep_stencil_direct<T, BT, false, 2>(I, &sn, unit, part[0]);
      else if (sn.inner_iters > 0)
        sweep_stencil_direct<T, BT, false, 1>(I, &sn, unit, part[0]);
      else
        sweep_stencil_direct<T, BT, false, 0>(I, &sn, unit, part[0]);
    }
    if constexpr (MODE == 0)
      store_partials<1, T>(part, I.part, I.nunits, unit);
    else
      store_partials_by_warp<1, T>(part, I.part, I.nunits, unit);
  }
  finish_sweep(I, st, phase, I.nunits);
}

// One flat-kind unit (MEANF, UPDATE, CORRECT or FINAL phase) of instance I.
template <class T, bool PERSIST = false>
__device__ __forceinline__ void flat_kind_unit(const InstDesc& I, int unit) {
  InstState* st = I.st;
  InstState own;
  if (PERSIST) load_state(st, own);
  const InstState& sn = PERSIST ? own : block_state(st);
  const int phase = sn.phase;
  if (phase != PH_MEANF && phase != PH_UPDATE && phase != PH_CORRECT && phase != PH_FINAL) return;
  const long long c0 = flat_begin(I, unit), c1 = flat_begin(I, unit + 1);
  switch (phase) {
    case PH_MEANF: {
      double sum[1] = {0.0};
      sweep_meanf(I, c0, c1, sum[0]);
      store_partials<1, double>(sum, I.part, I.nunits_f, unit);
      break;
    }
    case PH_UPDATE: {
      T part[1] = {0};
      sweep_update<T>(I, &sn, c0, c1, part[0]);
      store_partials<1, T>(part, I.part, I.nunits_f, unit);
      break;
    }
    case PH_CORRECT: {
      double ps[1] = {0.0};
      if (sizeof(T) == 8 && I.form)
        sweep_correct<T, sizeof(T) == 8>(I, c0, c1, sn.p_set == 0, sn.texp, ps[0]);
      else
        sweep_correct<T, false>(I, c0, c1, sn.p_set == 0, sn.texp, ps[0]);
      store_partials<1, double>(ps, I.part, I.nunits_f, unit);
      break;
    }
    default: sweep_final(I, &sn, c0, c1); break;
  }
  finish_sweep(I, st, phase, I.nunits_f);
}

// Direct register march, STENCIL phase only: at most 256 threads, three units per SM (24 warps
// keep enough loads in flight).
#ifndef VDP_DIRECT_MIN_BLOCKS
#define VDP_DIRECT_MIN_BLOCKS 2
#endif
// Units per SM the register budget is sized for: three (80 registers, no spills) for every kind;
// measured at 256^3 against two units with the unconstrained allocation: FP64 CG sweep 315 ->
// 307 us, FP64 fused fixed-point sweep 299 -> 284 us.
template <class T, int KIND> struct DirectOcc { static constexpr int kMinBlocks = VDP_DIRECT_MIN_BLOCKS + 1; };

template <class T, class BT, int KIND>
__global__ void __launch_bounds__(kDirectThreads, DirectOcc<T, KIND>::kMinBlocks) k_stencil_direct(
    const InstDesc* __restrict__ insts, const UnitRef* __restrict__ units) {
  const UnitRef ur = units[blockIdx.x];
  stencil_kind_unit<T, BT, 0, 1, KIND>(insts[ur.inst], ur.unit, nullptr);
}

// Direct register march, RES64 phase only (a few launches per solve do work; the kernel has its
// own register allocation so that the FP64 residual does not limit the stencil's occupancy).
// Units per SM: three for the FP64 inner type (80 registers, no spills), two for FP32 (whose
// variant would spill at three).
template <class T> struct Res64Occ { static constexpr int kMinBlocks = IsF64<T>::value ? 3 : 2; };

template <class T>
__global__ void __launch_bounds__(kDirectThreads, Res64Occ<T>::kMinBlocks) k_res64_direct(
    const InstDesc* __restrict__ insts, const UnitRef* __restrict__ units) {
  const UnitRef ur = units[blockIdx.x];
  stencil_kind_unit<T, T, 0, 2>(insts[ur.inst], ur.unit, nullptr);
}

// The same for the instances in the density form (FP64).
__global__ void __launch_bounds__(kDirectThreads, Res64Occ<double>::kMinBlocks) k_res64_density(
    const InstDesc* __restrict__ insts, const UnitRef* __restrict__ units) {
  const UnitRef ur = units[blockIdx.x];
  const InstDesc& I = insts[ur.inst];
  InstState* st = I.st;
  const InstState& sn = block_state(st);
  if (sn.phase != PH_RES64 || I.form == 0) return;
  double acc[kSlots] = {0.0, 0.0, 0.0, 0.0};
  sweep_res64_direct<double, true>(I, &sn, ur.unit, acc);
  store_partials<kSlots, double>(acc, I.part, I.nunits, ur.unit);
  finish_sweep(I, st, PH_RES64, I.nunits);
}

// TMA-staged pipeline
template <class T, class BT>
__global__ void __launch_bounds__(kMaxThreads) k_stencil_tma(const InstDesc* __restrict__ insts,
                                                             const UnitRef* __restrict__ units) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const UnitRef ur = units[blockIdx.x];
  stencil_kind_unit<T, BT, 1>(insts[ur.inst], ur.unit, smem_raw);
}

template <class T>
__global__ void __launch_bounds__(kFlatThreads, 4) k_flat(const InstDesc* __restrict__ insts,
                                                          const UnitRef* __restrict__ units) {
  const UnitRef ur = units[blockIdx.x];
  flat_kind_unit<T>(insts[ur.inst], ur.unit);
}

// Grid-wide barrier of the persistent kernel (all CTAs co-resident: cooperative launch).  Bounded:
// after the batch's wait limit (2 s by default) it gives up, sets the fault word and returns
// false, so a lost arrival ends the launch with an error status instead of a hang.
__device__ bool grid_sync(BatchCtl* ctl) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned int* vgen = &ctl->gen;
    const unsigned int gen = *vgen;
    __threadfence();
    const unsigned int arrived = atomicAdd(&ctl->count, 1u) + 1u;
    const unsigned long long limit = ctl->limit_ns;
    ok = 1;
    if (arrived == gridDim.x + ctl->extra) {
      ctl->count = 0u;
      __threadfence();
      atomicAdd(&ctl->gen, 1u);
    } else {
      const uint64_t t0 = global_ns();
      while (*vgen == gen) {
        if (global_ns() - t0 > limit) {
          atomicExch(&ctl->fault, 1);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// The batch engine's persistent kernel: `pairs` rounds of (stencil-kind sweep of every
// instance, grid barrier, flat-kind sweep of every instance, grid barrier), units distributed
// over the resident CTAs; stops early once every instance is done.
template <class T, class BT>
__global__ void __launch_bounds__(kDirectThreads, VDP_DIRECT_MIN_BLOCKS)
    k_persistent(const InstDesc* __restrict__ insts, const UnitRef* __restrict__ sunits, int ns,
                 const UnitRef* __restrict__ funits, int nf, int pairs, BatchCtl* ctl) {
  for (int it = 0; it < pairs; ++it) {
    // uniform: `remaining` only changes in flat sweeps, and every CTA reads it after a barrier
    if (*(volatile int*)&ctl->remaining <= 0) break;
    for (int u = blockIdx.x; u < ns; u += gridDim.x) {
      const UnitRef ur = sunits[u];
      stencil_kind_unit<T, BT, 0, 0, 1, true>(insts[ur.inst], ur.unit, nullptr);
    }
    if (!grid_sync(ctl)) return;
    for (int u = blockIdx.x; u < nf; u += gridDim.x) {
      const UnitRef ur = funits[u];
      flat_kind_unit<T, true>(insts[ur.inst], ur.unit);
    }
    if (!grid_sync(ctl)) return;
  }
}

// Copies the state of n instances into a contiguous array (one D2H copy for the host).
__global__ void k_gather_states(const InstDesc* __restrict__ insts, int n, InstState* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = *insts[i].st;  // a separate launch: the solver kernels have finished
}

// Per-solve initialisation of one instance's state.
__global__ void k_init(InstDesc* desc, const double* rhs, double* p, double tol, double inner_tol,
                       int max_iter, int inner_max, int use_guess, int precision,
                       ResidentCtl* ctl) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  desc->rhs = rhs;
  desc->p = p;
  InstState* st = desc->st;
  InstState s;
  memset(&s, 0, sizeof(s));
  s.phase = PH_MEANF;
  s.status = 0;
  s.max_iter = max_iter;
  s.inner_max = inner_max;
  s.use_guess = use_guess;
  s.p_set = use_guess ? 1 : 0;
  s.precision = precision;
  s.tol = tol;
  s.inner_tol = inner_tol;
  s.eta = 1.0;
  *st = s;
  *desc->ticket = 0u;
  if (ctl) {
    ctl->count = 0u;
    ctl->fault = 0;
    ctl->extra = 0u;
    ctl->limit_ns = kResidentWaitNs;
  }
}

// ---- one operator application -----------------------------------------------------------------------

// out = A p (FP64)
__global__ void k_apply(const double* __restrict__ bx, const double* __restrict__ by,
                        const double* __restrict__ bz, const double* __restrict__ p, int nx, int ny,
                        int nz, double* __restrict__ out) {
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
    const double pc = p[c];
    out[c] = bx[cxp] * (p[cxp] - pc) - bx[c] * (pc - p[cxm]) + by[cyp] * (p[cyp] - pc) -
             by[c] * (pc - p[cym]) + bz[czp] * (p[czp] - pc) - bz[c] * (pc - p[czm]);
  }
}

// ---- host launchers ---------------------------------------------------------------------------

static int grid_for(long long n) {
  long long b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  if (b < 1) b = 1;
  return (int)b;
}

cudaError_t launch_apply(const double* bx, const double* by, const double* bz, const double* p,
                         int nx, int ny, int nz, double* out, cudaStream_t s) {
  const long long n = (long long)nx * ny * nz;
  k_apply<<<grid_for(n), 256, 0, s>>>(bx, by, bz, p, nx, ny, nz, out);
  return cudaGetLastError();
}

cudaError_t launch_init(InstDesc* desc, const double* rhs, double* p, double tol, double inner_tol,
                        int max_iter, int inner_max, int use_guess, int precision,
                        ResidentCtl* ctl, cudaStream_t s) {
  k_init<<<1, 32, 0, s>>>(desc, rhs, p, tol, inner_tol, max_iter, inner_max, use_guess,
                          precision, ctl);
  return cudaGetLastError();
}

template <int KIND>
static void* direct_fn(int prec) {
  if (prec == PREC_FP64) return (void*)k_stencil_direct<double, double, KIND>;
  if (prec == PREC_MIXED) return (void*)k_stencil_direct<float, float, KIND>;
  return (void*)k_stencil_direct<float, __nv_bfloat16, KIND>;
}

static void* stencil_fn(int prec, int mode, int kind) {
  if (mode == 0) return kind == 2 ? direct_fn<2>(prec) : kind == 1 ? direct_fn<1>(prec) : direct_fn<0>(prec);
  if (prec == PREC_FP64) return (void*)k_stencil_tma<double, double>;
  if (prec == PREC_MIXED) return (void*)k_stencil_tma<float, float>;
  return (void*)k_stencil_tma<float, __nv_bfloat16>;
}

cudaError_t prepare_step(int prec, int mode, size_t smem_bytes) {
  if (mode == 0) return cudaSuccess;  // the direct sweeps use no dynamic shared memory
  return cudaFuncSetAttribute(stencil_fn(prec, mode, 0),
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
}

cudaError_t launch_res64(int prec, int form, const InstDesc* desc, const UnitRef* units, int nunits,
                         int threads, cudaStream_t s) {
  if (form)
    k_res64_density<<<nunits, threads, 0, s>>>(desc, units);
  else if (prec == PREC_FP64)
    k_res64_direct<double><<<nunits, threads, 0, s>>>(desc, units);
  else
    k_res64_direct<float><<<nunits, threads, 0, s>>>(desc, units);
  return cudaGetLastError();
}

cudaError_t launch_stencil(int prec, int mode, int kind, const InstDesc* desc,
                           const UnitRef* units, int nunits, int threads, size_t smem_bytes,
                           cudaStream_t s) {
  if (kind >= kSweepDensityCg) return launch_density(kind, desc, units, nunits, threads, s);
  void* fn = stencil_fn(prec, mode, kind);
  void* args[] = {(void*)&desc, (void*)&units};
  return cudaLaunchKernel(fn, dim3(nunits), dim3(threads), args, smem_bytes, s);
}

static void* persistent_fn(int prec) {
  if (prec == PREC_FP64) return (void*)k_persistent<double, double>;
  if (prec == PREC_MIXED) return (void*)k_persistent<float, float>;
  return (void*)k_persistent<float, __nv_bfloat16>;
}

cudaError_t persistent_grid(int prec, int* grid) {
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, persistent_fn(prec),
                                                                kDirectThreads, 0);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *grid = per_sm * sms;
  return cudaSuccess;
}

cudaError_t launch_persistent(int prec, const InstDesc* desc, const UnitRef* sunits, int ns,
                              const UnitRef* funits, int nf, int pairs, BatchCtl* ctl, int grid,
                              cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kDirectThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // all CTAs co-resident: the grid barrier is safe
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[] = {(void*)&desc, (void*)&sunits, (void*)&ns, (void*)&funits, (void*)&nf,
                  (void*)&pairs, (void*)&ctl};
  return cudaLaunchKernelExC(&cfg, persistent_fn(prec), args);
}

// The body of a solve's device-side loop ends with this kernel: it keeps the loop going while
// the solve is unfinished and the round count rounds[0] is below its bound and the launch's own
// limit rounds[1] (0: none).
__global__ void k_continue(const InstState* st, cudaGraphConditionalHandle handle, unsigned* rounds,
                           unsigned max_rounds) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    const unsigned r = rounds[0] + 1u, limit = rounds[1];
    rounds[0] = r;
    const bool more = __ldcg(&st->phase) < PH_DONE && r < max_rounds && (limit == 0u || r < limit);
    cudaGraphSetConditional(handle, more ? 1u : 0u);
  }
}

__global__ void k_start_rounds(unsigned* rounds, unsigned limit) {
  rounds[0] = 0u;
  rounds[1] = limit;
}

__global__ void k_start_resident(ResidentCtl* ctl, unsigned extra, unsigned long long limit_ns) {
  ctl->count = 0u;
  ctl->fault = 0;
  ctl->extra = extra;
  ctl->limit_ns = limit_ns;
}

cudaError_t launch_start_resident(ResidentCtl* ctl, unsigned extra, unsigned long long limit_ns, cudaStream_t s) {
  k_start_resident<<<1, 1, 0, s>>>(ctl, extra, limit_ns);
  return cudaGetLastError();
}

cudaError_t launch_start_rounds(unsigned* rounds, unsigned limit, cudaStream_t s) {
  k_start_rounds<<<1, 1, 0, s>>>(rounds, limit);
  return cudaGetLastError();
}

cudaError_t launch_continue(const InstState* st, cudaGraphConditionalHandle handle,
                            unsigned* rounds, unsigned max_rounds, cudaStream_t s) {
  k_continue<<<1, 32, 0, s>>>(st, handle, rounds, max_rounds);
  return cudaGetLastError();
}

cudaError_t launch_gather(const InstDesc* desc, int n, InstState* out, cudaStream_t s) {
  k_gather_states<<<(n + 127) / 128, 128, 0, s>>>(desc, n, out);
  return cudaGetLastError();
}

cudaError_t launch_flat(int prec, const InstDesc* desc, const UnitRef* units, int nunits,
                        cudaStream_t s) {
  if (prec == PREC_FP64)
    k_flat<double><<<nunits, kFlatThreads, 0, s>>>(desc, units);
  else
    k_flat<float><<<nunits, kFlatThreads, 0, s>>>(desc, units);
  return cudaGetLastError();
}

}  // namespace vdp
