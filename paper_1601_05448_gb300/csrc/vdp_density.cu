// vdp_density.cu -- kernels of the density form's sweeps (vdp_density.cuh says what they compute and
// why): one launch per sweep.
#include "vdp_density.cuh"
#include "vdp_launch.h"

namespace vdp {

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

// The same in FP64: four cells per thread of the FP64 layout's two, so half its threads; three
// blocks of 128 threads per SM (168 registers).
template <bool FIXED>
__global__ void __launch_bounds__(kDensity64Threads, 3)
    k_density64(const InstDesc* __restrict__ insts, const UnitRef* __restrict__ units) {
  extern __shared__ __align__(16) ulonglong2 slots[];
  const UnitRef ur = units[blockIdx.x];
  const InstDesc& I = insts[ur.inst];
  InstState* st = I.st;
  const InstState& sn = block_state(st);
  if (sn.phase != PH_STENCIL || I.form == 0 || (I.pc == PC_FIXED) != FIXED) return;
  double part[1] = {0.0};
  sweep_density64<FIXED>(I, sn, ur.unit, part[0], slots);
  store_partials<1, double>(part, I.part, I.nunits, ur.unit);
  finish_sweep(I, st, PH_STENCIL, I.nunits);
}

cudaError_t prepare_density() {
  struct {
    const void* fn;
    size_t smem;
  } const k[] = {{(const void*)k_density<true>, density_smem(true, kDirectThreads)},
                 {(const void*)k_density<false>, density_smem(false, kDirectThreads)},
                 {(const void*)k_density64<true>, density64_smem(kDensity64Threads)},
                 {(const void*)k_density64<false>, density64_smem(kDensity64Threads)}};
  for (const auto& e : k) {
    const cudaError_t r = cudaFuncSetAttribute(e.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)e.smem);
    if (r != cudaSuccess) return r;
  }
  return cudaSuccess;
}

cudaError_t launch_density(int prec, int kind, const InstDesc* desc, const UnitRef* units,
                           int nunits, int threads, cudaStream_t s) {
  const bool fixed = kind == kSweepDensityFixed;
  if (prec == PREC_FP64) {
    const int t = (threads / 2 + 31) / 32 * 32;  // whole warps; threads beyond the tile are idle
    if (fixed)
      k_density64<true><<<nunits, t, density64_smem(t), s>>>(desc, units);
    else
      k_density64<false><<<nunits, t, density64_smem(t), s>>>(desc, units);
  } else if (fixed) {
    k_density<true><<<nunits, threads, density_smem(true, threads), s>>>(desc, units);
  } else {
    k_density<false><<<nunits, threads, density_smem(false, threads), s>>>(desc, units);
  }
  return cudaGetLastError();
}

}  // namespace vdp
