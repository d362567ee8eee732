// vdp_density.cu -- kernels of the density form's sweeps (vdp_density.cuh says what they compute and
// why): one launch per sweep.
#include "vdp_density.cuh"
#include "vdp_launch.h"

namespace vdp {

// STENCIL phase of the instances in the density form: FIXED the fixed-point iteration, else CG.
// Four cells per thread of the FP64 layout's two, so half its threads; three blocks of 128 threads
// per SM (168 registers).
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
  for (const void* fn : {(const void*)k_density64<true>, (const void*)k_density64<false>}) {
    const cudaError_t r = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)density64_smem(kDensity64Threads));
    if (r != cudaSuccess) return r;
  }
  return cudaSuccess;
}

cudaError_t launch_density(int kind, const InstDesc* desc, const UnitRef* units, int nunits,
                           int threads, cudaStream_t s) {
  const int t = (threads / 2 + 31) / 32 * 32;  // whole warps; threads beyond the tile are idle
  if (kind == kSweepDensityFixed)
    k_density64<true><<<nunits, t, density64_smem(t), s>>>(desc, units);
  else
    k_density64<false><<<nunits, t, density64_smem(t), s>>>(desc, units);
  return cudaGetLastError();
}

}  // namespace vdp
