// vdp_launch.h -- host-side launchers of the kernels in vdp_kernels.cu, vdp_setup.cu
// and vdp_density.cu (internal to libvdp).
#pragma once

#include <cuda_runtime.h>

#include "vdp_internal.cuh"

namespace vdp {

// vdp_setup.cu.  The check stores gen in *bad when an entry is <= 0 or not finite; the launches
// that take (bad, gen) then write nothing (null: not gated).
cudaError_t launch_check_density(const double* rho, long long n, int gen, int* bad, cudaStream_t s);
// face coefficients on the low faces (spacings h_d; duct: no flux through the x ends) and D; with
// sinv also D^-1/2, with rho32 the density form's FP32 density, what it rounds off (rho_lo) and
// dsc[0] = kappa = 2^e0 s, and far[0] = gen where these do not hold the density
cudaError_t launch_build_coefficients(const double* rho, int nx, int ny, int nz, double hx,
                                      double hy, double hz, int duct, double* bx, double* by,
                                      double* bz, double* sinv, double* dg, float* rho32,
                                      float* rho_lo, double* dsc, double s2, const int* bad,
                                      int* far, int gen, cudaStream_t s);
cudaError_t launch_sinv(const double* dg, long long n, double* sinv, cudaStream_t s);
cudaError_t launch_scaled(int prec, const double* bx, const double* by, const double* bz,
                          const double* sinv, int nx, int ny, int nz, void* sx, void* sy, void* sz,
                          void* sd, const int* bad, int gen, cudaStream_t s);
// W = D^1/2 (omega; unit: over the first cell's power of two) and rho W (rho_w, the scaled fixed-point iteration's input weight); null: not
// stored.  launch_rho_weight takes rho from the density form's fields instead.
cudaError_t launch_weights(const double* rho, const double* dg, const double* sinv, long long n,
                           bool unit, float* omega, float* rho_w, const int* bad, int gen, cudaStream_t s);
cudaError_t launch_rho_weight(const float* rho32, const float* rho_lo, const double* dsc, double s2,
                              const double* dg, const double* sinv, long long n, float* rho_w,
                              cudaStream_t s);
cudaError_t launch_apply(const double* bx, const double* by, const double* bz, const double* p,
                         int nx, int ny, int nz, double* out, cudaStream_t s);
// ctl: also the control words of a resident solve (or null)
cudaError_t launch_init(InstDesc* desc, const double* rhs, double* p, double tol, double inner_tol,
                        int max_iter, int inner_max, int use_guess, int precision,
                        ResidentCtl* ctl, cudaStream_t s);
cudaError_t prepare_step(int prec, int mode, size_t smem_bytes);
// mode 0 only: the FP64 residual sweep (its own kernel, launched before each stencil launch) of
// the instances in the scaled (form 0) or the density form (1)
cudaError_t launch_res64(int prec, int form, const InstDesc* desc, const UnitRef* units, int nunits,
                         int threads, cudaStream_t s);
// kind (direct sweep variants): 0 = CG, 1 = CG and Chebyshev preconditioner sweeps (PH_CHEB),
// 2 = the fixed-point iteration; the density form's sweeps (vdp_density.cu); stencil_kind(d)
// picks it for an instance
constexpr int kSweepDensityCg = 3, kSweepDensityFixed = 4;
inline int stencil_kind(const InstDesc& d) {
  if (d.form) return d.pc == PC_FIXED ? kSweepDensityFixed : kSweepDensityCg;
  return d.pc == PC_FIXED ? 2 : (d.pc == PC_CHEB ? 1 : 0);
}
cudaError_t prepare_density();  // shared-memory limits on the current device
cudaError_t launch_density(int kind, const InstDesc* desc, const UnitRef* units, int nunits,
                           int threads, cudaStream_t s);
cudaError_t launch_stencil(int prec, int mode, int kind, const InstDesc* desc,
                           const UnitRef* units, int nunits, int threads, size_t smem_bytes,
                           cudaStream_t s);
cudaError_t launch_flat(int prec, const InstDesc* desc, const UnitRef* units, int nunits,
                        cudaStream_t s);

// vdp_resident.cu: the whole solve in one cooperative launch, for grids of at most kResidentCells
// cells.  spec: the solve's spectral arguments (unused by Jacobi CG); stops after max_rounds rounds, a
// round being what one pass of the separate launches (residual, preconditioner, stencil, flat) advances;
// at most max_blocks blocks (0: as many as are resident).  The control words are set before, by
// launch_init or launch_start_resident.
struct SpecArgs;
bool resident_supported(const InstDesc& d, int prec);
cudaError_t launch_resident(int prec, const InstDesc& d, const InstDesc* desc, const SpecArgs& spec,
                            ResidentCtl* ctl, unsigned max_rounds, int max_blocks, cudaStream_t s);

cudaError_t persistent_grid(int prec, int* grid);
cudaError_t launch_persistent(int prec, const InstDesc* desc, const UnitRef* sunits, int ns,
                              const UnitRef* funits, int nf, int pairs, BatchCtl* ctl, int grid,
                              cudaStream_t s);
cudaError_t launch_gather(const InstDesc* desc, int n, InstState* out, cudaStream_t s);
cudaError_t launch_start_resident(ResidentCtl* ctl, unsigned extra, unsigned long long limit_ns, cudaStream_t s);
// before a device-side loop: rounds = {0, limit} (limit 0: none)
cudaError_t launch_start_rounds(unsigned* rounds, unsigned limit, cudaStream_t s);
// device-side solve loop: sets the WHILE condition `handle` to continue while the instance is
// unfinished and fewer than max_rounds loop iterations have run (*rounds counts them)
cudaError_t launch_continue(const InstState* st, cudaGraphConditionalHandle handle,
                            unsigned* rounds, unsigned max_rounds, cudaStream_t s);

}  // namespace vdp
