// vdp_spectral.cu -- the constant-coefficient spectral inverse (Sec. 3.4) on sm_103a, used as a
// preconditioner of the inner conjugate-gradient solve and exposed as vdp_inverse_laplacian.
//
// The paper solves the variable-density equation by repeated constant-coefficient Poisson
// solves done with FFTs.  Here the same operator, the inverse of the 7-point Laplacian L_h on
// the periodic grid (eigenvalues -sum_d 4 sin^2(pi k_d / n_d) / h_d^2, zero mode removed), is
// applied to the Jacobi-scaled inner residual as
//     z = W (-L_h)^-1 W rt,   W = D^1/2 (D: diagonal of the variable-coefficient operator),
// which is the constant-coefficient inverse in unscaled variables.  Between the smallest and the
// largest face value of 1/rho the variable operator is bounded by multiples of -L_h, so the
// preconditioned condition number is at most the density ratio, whatever the grid size.
//
// Five passes over a half spectrum S[kz][ky][kx] (kx = 0 .. nx/2, complex FP32, row pitch nxp):
//   X+  each row of nx reals is read as nx/2 complex pairs (in the scaled form weighted by W; the
//       density form, vdp_density.cuh, has no weights), transformed by a complex FFT of length
//       nx/2 and unpacked into the nx/2 + 1 bins of the real transform;
//   Y+  complex FFTs along y of tiles of 8 consecutive kx columns;
//   Z   FFT along z, division by the eigenvalue (and by nx ny nz), inverse FFT along z: the
//       whole z line is in the block, so the solve costs one pass;
//   Y-  inverse FFTs along y;
//   X-  the real inverse transform of each row, (weighted by W and) stored as z; in the solve the
//       last unit to finish also sums the <rt, z> partials of Z (spectral CG) and moves the solve
//       to its next phase (the same fixed-order reduction as every other sweep).
// Every line FFT is a four-step factorisation n = M1 x M2 (both products of 2 and 3, at most
// 32): M2-point DFTs in registers, twiddles W_n^(j1 k2), an exchange through shared memory,
// M1-point DFTs in registers.  Global accesses are coalesced: rows are contiguous in the X
// passes and the Y/Z tiles read 8 consecutive complex values (64 bytes) per line element.
// One application moves about 41 bytes per cell (FP32 input, no weights; with weights 49).  At 512^3 X
// takes 185 us a launch (with weights X+ 242, X- 256), Y 191 (0.87 of the copy bandwidth each) and Z, which does two transforms per element, 315
// (0.53).  At 256^3 the spectrum stays in L2 and nothing is saturated (ncu: issue 42-58 %, shared
// memory 28-54 %, DRAM 28-43 %; 15-20 warps per SM): X 33 (with
// weights 36 and 40), Y 26, Z 36 us.  In every pass the
// first tile's copies and the tables are under way while the solve's phase is read.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "vdp.h"
#include "vdp_device.cuh"
#include "vdp_fft.cuh"
#include "vdp_internal.cuh"
#include "vdp_spectral.h"

namespace vdp {

// X+ with one group of RY rows per block, everything loaded at its use: the weighted FP32 rows whose
// transform has 512 values.  512^3: 261 us; with the rows staged as below, their weights then waited for
// behind a few large blocks, 293 (256^3: 45.5 and 36 the other way round).
template <class T, int M1, int M2, bool MIRROR>
__global__ void __launch_bounds__(M1 * rows_per_block<M1, M2>(), 1024 / (M1 * rows_per_block<M1, M2>()))
    k_spec_x_fwd(SpecArgs a) {
  constexpr int RY = rows_per_block<M1, M2>();
  constexpr int SX = x_row_stride<M1, M2>();
  __shared__ float2 sx[RY * SX];  // per row: the exchange, then the transformed row
  if (!spec_active(a)) return;
  const Tables tb = tables(a);
  const int t = threadIdx.x % M1, r = threadIdx.x / M1;
  const long long row = (long long)a.z0 * a.ny + (long long)blockIdx.x * RY + r;
  const bool live = row < (long long)a.z1 * a.ny;
  float2* out = a.spec + row * a.nxp;
  x_fwd_rows<T, M1, M2, MIRROR>(a, tb, sx + r * SX, static_cast<const T*>(a.in) + row * a.nxd, row, live, t,
                                 [&](int k, float2 X) { out[k] = X; }, [] {});
}

// X+ of FP64 rows on a persistent grid: groups of RY rows (group = block, block + grid, ...) of
// the planes [z0, z1), tables in shared memory; at least 768 resident threads per SM (80
// registers a thread).  The 512^3 FP64 solve: 47.3 ms against 49.2 ms with one group of rows
// per block and the tables read through L1.
template <class T, int M1, int M2, bool MIRROR>
__global__ void __launch_bounds__(M1 * rows_per_block<M1, M2>(), 768 / (M1 * rows_per_block<M1, M2>()))
    k_spec_x_fwd_persistent(SpecArgs a) {
  constexpr int RY = rows_per_block<M1, M2>();
  constexpr int SX = x_row_stride<M1, M2>();
  __shared__ float2 sx[RY * SX];  // per row: the exchange, then the transformed row
  __shared__ float2 stab[2 * M1 * M2 + 1];
  if (!spec_active(a)) return;
  const Tables tb = x_tables_shared<M1, M2>(a, stab);
  const int t = threadIdx.x % M1, r = threadIdx.x / M1;
  const long long rows = (long long)(a.z1 - a.z0) * a.ny;
  for (long long g = blockIdx.x; g * RY < rows; g += gridDim.x) {
    const long long row = (long long)a.z0 * a.ny + g * RY + r;
    const bool live = g * RY + r < rows;
    float2* out = a.spec + row * a.nxp;
    x_fwd_rows<T, M1, M2, MIRROR>(a, tb, sx + r * SX, static_cast<const T*>(a.in) + row * a.nxd, row, live,
                                   t, [&](int k, float2 X) { out[k] = X; }, [] {});
    __syncthreads();  // the row buffers are reused by the next group
  }
}

// X+ of FP32 rows on a persistent grid, the group's rows copied to shared memory while the group
// before is transformed (an FP32 row of the solve's own fields starts on a 16-byte boundary; FP64 rows
// may be a caller's).  Loading them at their use, 512^3 took 204 us, the 256 x 128 x 128 duct 24;
// now 185 and 20.
template <int M1, int M2, bool MIRROR>
__global__ void __launch_bounds__(M1 * inv_rows_per_block<M1, M2>()) k_spec_x_fwd_staged(SpecArgs a) {
  constexpr int RY = inv_rows_per_block<M1, M2>();
  constexpr int SX = x_row_stride<M1, M2>();
  constexpr int m = M1 * M2, SR = pad_stride(m);
  __shared__ float2 sx[RY * SX];                // per row: the exchange, then the transformed row
  __shared__ __align__(16) float2 sr[RY * SR];  // the group's rows, fetched ahead
  __shared__ float2 stab[2 * m + 1];
  const long long rows = (long long)(a.z1 - a.z0) * a.ny, first = (long long)a.z0 * a.ny;
  const int pieces = a.nxd / 4;
  auto fetch = [&](long long g) {
    const int n = (int)(rows - g * RY < RY ? rows - g * RY : RY);
    const float* src = static_cast<const float*>(a.in) + (first + g * RY) * a.nxd;
    for (int q = threadIdx.x; q < n * pieces; q += M1 * RY) {  // the rows follow one another
      const int r = q / pieces;
      cp_async16(sr + r * SR + 2 * (q - r * pieces), src + 4 * (long long)q);
    }
    cp_async_commit();
  };
  long long g = blockIdx.x;
  if (g * RY < rows) fetch(g);
  const Tables tb = x_tables_shared<M1, M2>(a, stab);
  if (!spec_active(a)) return cp_async_wait_all();
  const int t = threadIdx.x % M1, r = threadIdx.x / M1;
  for (; g * RY < rows; g += gridDim.x) {
    const long long row = first + g * RY + r;
    float2* out = a.spec + row * a.nxp;
    cp_async_wait_all();
    __syncthreads();  // the rows are there, and the row buffers of the group before have been read
    x_fwd_rows<float, M1, M2, MIRROR>(
        a, tb, sx + r * SX, reinterpret_cast<const float*>(sr + r * SR), row, g * RY + r < rows, t,
        [&](int k, float2 X) { out[k] = X; },
        [&] { if ((g + gridDim.x) * RY < rows) fetch(g + gridDim.x); });
  }
}

// X- on a persistent grid: groups of RY rows (group = block, block + grid, ...), tables in
// shared memory, the group's rows copied there while the group before is transformed: each bin is
// read twice (k and nx/2 - k), which through L1 cost 76 % of its rate and left 8 stall cycles per
// issue on the loads (256^3: 35 us, now 33; 512^3 201 and 185).
template <class T, int M1, int M2, bool MIRROR, bool WEIGHT>
__global__ void __launch_bounds__(M1 * inv_rows_per_block<M1, M2>())
    k_spec_x_inv_persistent(SpecArgs a) {
  constexpr int RY = inv_rows_per_block<M1, M2>();
  constexpr int SB = pad_stride(M2 * (M1 + 1));
  constexpr int m = M1 * M2, SR = pad_stride(m + 1), kPieces = m / 2 + 1;
  __shared__ float2 sb[RY * SB];                 // the exchange
  __shared__ __align__(16) float2 sr[RY * SR];   // the group's rows, fetched ahead
  __shared__ float2 stab[2 * m + 1];
  const long long rows = (long long)(a.z1 - a.z0) * a.ny, first = (long long)a.z0 * a.ny;
  auto fetch = [&](long long g) {
    const int n = (int)(rows - g * RY < RY ? rows - g * RY : RY);
    const float2* src = a.spec + (first + g * RY) * a.nxp;
    for (int q = threadIdx.x; q < n * kPieces; q += M1 * RY) {
      const int r = q / kPieces, p = 2 * (q - r * kPieces);
      cp_async16(sr + r * SR + p, src + (long long)r * a.nxp + p);
    }
    cp_async_commit();
  };
  long long g = blockIdx.x;
  if (g * RY < rows) fetch(g);
  const Tables tb = x_tables_shared<M1, M2>(a, stab);
  if (!spec_active(a)) return cp_async_wait_all();
  const int t = threadIdx.x % M1, r = threadIdx.x / M1;
  for (; g * RY < rows; g += gridDim.x) {
    cp_async_wait_all();
    __syncthreads();  // the rows are there, and the exchange of the group before has been read
    const bool live = g * RY + r < rows;
    x_inv_rows<T, M1, M2, MIRROR, WEIGHT>(a, tb, sb + r * SB, sr + r * SR, first + g * RY + r, live, t,
                                            [&] { if ((g + gridDim.x) * RY < rows) fetch(g + gridDim.x); });
  }
  if (a.st) {  // the solve: the last block of the application's X- launches completes the
               // preconditioner sweep, in spectral CG with <rt, z> from the partial sums of Z
    const InstDesc& I = *a.I;
    finish_sweep(I, I.st, PH_SPEC, a.xunits, a.zunits, (a.f32 & kEnergy) != 0);
  }
}

// ---- Y and Z: tiles of TX consecutive kx columns, whole lines -----------------------------------

// Y: at least 512 resident threads per SM (at most 128 registers a thread); lines of 512: four
// blocks of 128 threads.  Z: at least 640 (96 registers, a few bytes spilled): at 512^3 Z
// 352 -> 327 us with five blocks per SM, while Y at five (or six) blocks ran 191 -> 209 us.
template <int M1> struct LineOcc { static constexpr int kMinBlocks = (512 + M1 * kTX - 1) / (M1 * kTX); };
template <int M1> struct ZOcc { static constexpr int kMinBlocks = (640 + M1 * kTX - 1) / (M1 * kTX); };

template <int M1, int M2>
constexpr size_t y_smem() {  // tile buffer, twiddles W_ny^k
  return sizeof(float2) * (size_t)(line_buffer<M1, M2>() + M1 * M2);
}

// Y pass (forward or inverse), in place.  Tiles are (column tile, kz); a persistent grid walks
// them (tile = block, block + grid, ...).  The twiddles W_ny^k are copied to shared memory once
// per block; a tile's copies go out as soon as the previous tile's exchange is read, so they
// overlap its step B and stores.  Step A: M2-point DFTs over j2 (thread (t, c)), twiddles, the
// exchange; step B: M1-point DFTs over j1 by owner k2, element k2 + M2 k1 stored.
template <int M1, int M2, bool INV>
__global__ void __launch_bounds__(M1 * kTX, LineOcc<M1>::kMinBlocks) k_spec_y(SpecArgs a) {
  constexpr int R = (M2 + M1 - 1) / M1;
  constexpr int n = M1 * M2;
  constexpr int S = pad_stride(M1 * kTX);
  extern __shared__ __align__(16) float2 ybuf[];
  float2* sm = ybuf;                          // the tile
  float2* wy = ybuf + line_buffer<M1, M2>();  // W_ny^k, k < ny
  const Tables tb = tables(a);
  const int c = threadIdx.x % kTX, t = threadIdx.x / kTX;
  const int tiles = a.nxp / kTX;
  const int ntile = tiles * (a.z1 - a.z0);
  const long long es = a.nxp;  // element stride along y
  auto base = [&](int tile) {
    return a.spec + (long long)(a.z0 + tile / tiles) * a.ny * a.nxp + (tile % tiles) * kTX;
  };
  int tile = blockIdx.x;
  if (tile < ntile) fetch_tile<M1, M2>(sm, base(tile), es);
  for (int k = threadIdx.x; k < n; k += M1 * kTX) wy[k] = tb.wy[k];
  if (!spec_active(a)) return cp_async_wait_all();
  for (; tile < ntile; tile += gridDim.x) {
    cp_async_wait_all();  // this thread's copies of the tile have landed
    __syncthreads();      // ... and every other thread's (and the twiddles are in place)
    {
      float2 v[M2], y[M2];
#pragma unroll
      for (int j2 = 0; j2 < M2; ++j2) v[j2] = sm[j2 * S + t * kTX + c];
      dft<M2, 0, 1, INV>(v, y);
      __syncthreads();  // every input slot is read before the exchange overwrites it
#pragma unroll
      for (int k2 = 0; k2 < M2; ++k2) {
        const float2 w = wy[t * k2];
        sm[tx<M1>(k2, t, c)] = k2 == 0 || t == 0 ? y[k2] : (INV ? cmulc(y[k2], w) : cmul(y[k2], w));
      }
    }
    __syncthreads();
    float2 u[R][M1];
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
      const int k2 = t + M1 * rr;
      if (k2 < M2) {
#pragma unroll
        for (int j1 = 0; j1 < M1; ++j1) u[rr][j1] = sm[tx<M1>(k2, j1, c)];
      }
    }
    __syncthreads();  // the tile is read: the next tile's copies may go out
    if (tile + (int)gridDim.x < ntile) fetch_tile<M1, M2>(sm, base(tile + gridDim.x), es);
    float2* g = base(tile) + c;
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
      const int k2 = t + M1 * rr;
      if (k2 < M2) {
        float2 o[M1];
        dft<M1, 0, 1, INV>(u[rr], o);
#pragma unroll
        for (int k1 = 0; k1 < M1; ++k1) g[(k2 + M2 * k1) * es] = o[k1];
      }
    }
  }
}

// Z pass: forward FFT along z, scale by sign / (N lambda), inverse FFT along z.  Tiles are
// (column tile, ky); a persistent grid walks them (tile = block, block + grid, ...).  The twiddles
// W_nz^k and the z eigenvalues are copied to shared memory once per block (every lookup of a
// thread is then a shared-memory load: the table loads from L1 were the pass's main stall), and
// the copies of a tile's nz x 8 values go out as soon as the previous tile's values are read, so
// they overlap its inverse transform and stores.  Element e = t + M1 j2 of column c arrives at
// slot (j2, t, c); forward: A (M2-point over j2, thread (t, c)) writes slot (k2, t, c), B
// (M1-point over j1 = t) leaves owner k2 with X[k2 + M2 k1]; the owner scales and runs A' (M1-
// point over k1) and writes back to the slots it read, (k2, l2), so B -> scaling -> A' needs no
// barrier and keeps no line in registers across one; B' (M2-point over k2) reads slots (k2, t).
// In spectral CG (ENERGY) it also stores this block's part of <y, (-L_h)^-1 y> = sum_k |Y(k)|^2 s(k)
// (Parseval; y = W rt, the half spectrum counting kx = 1 .. nx/2 - 1 twice), which is <rt, z>:
// FP32 per tile, summed over the block's tiles in FP64, always in the same order.  The fixed-point
// iteration has no use for it: without, 512^3 327 -> 315 us, 256^3 38.2 -> 35.8.
template <int M1, int M2>
constexpr size_t z_smem() {  // tile buffer, twiddles W_nz^k, eigenvalues lz
  return sizeof(float2) * (size_t)(line_buffer<M1, M2>() + M1 * M2) + sizeof(float) * (size_t)(M1 * M2);
}

template <int M1, int M2, bool ENERGY>
__global__ void __launch_bounds__(M1 * kTX, ZOcc<M1>::kMinBlocks) k_spec_z(SpecArgs a) {
  constexpr int R = (M2 + M1 - 1) / M1;
  constexpr int n = M1 * M2;
  constexpr int S = pad_stride(M1 * kTX);
  extern __shared__ __align__(16) float2 zbuf[];
  float2* sm = zbuf;                         // the tile
  float2* wz = zbuf + line_buffer<M1, M2>();  // W_nz^k, k < nz
  float* lz = reinterpret_cast<float*>(wz + n);
  const Tables tb = tables(a);
  const int c = threadIdx.x % kTX, t = threadIdx.x / kTX;
  const int tiles = a.nxp / kTX;
  const int ntile = tiles * a.ny;
  const long long es = (long long)a.ny * a.nxp;  // element stride along z
  const int m = a.nx / 2;
  auto fetch = [&](int tile) {
    fetch_tile<M1, M2>(sm, a.spec + (long long)(tile / tiles) * a.nxp + (tile % tiles) * kTX, es);
  };
  int tile = blockIdx.x;
  if (tile < ntile) fetch(tile);
  for (int k = threadIdx.x; k < n; k += M1 * kTX) {
    wz[k] = tb.wz[k];
    lz[k] = tb.lz[k];
  }
  if (!spec_active(a)) return cp_async_wait_all();
  double energy_sum = 0.0;
  for (; tile < ntile; tile += gridDim.x) {
    cp_async_wait_all();  // this thread's copies of the tile have landed
    __syncthreads();      // ... and every other thread's (and the tables are in place)
    const int ky = tile / tiles, kx = (tile % tiles) * kTX + c;
    {
      float2 v[M2], y[M2];
#pragma unroll
      for (int j2 = 0; j2 < M2; ++j2) v[j2] = sm[j2 * S + t * kTX + c];
      dft<M2, 0, 1, false>(v, y);
      __syncthreads();  // every input slot is read before the exchange overwrites it
#pragma unroll
      for (int k2 = 0; k2 < M2; ++k2)
        sm[tx<M1>(k2, t, c)] = k2 == 0 || t == 0 ? y[k2] : cmul(y[k2], wz[t * k2]);
    }
    __syncthreads();
    const bool pad = kx > m;  // padding columns of the row pitch: set to 0
    const float lxy = pad ? 0.f : tb.lx[kx] + tb.ly[ky];
    const float wkx = (kx == 0 || kx == m) ? 1.f : 2.f;  // conjugate partners of the half spectrum
    float energy = 0.f;
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
          // zero mode removed; the quotient is the hardware's approximate one (2 ulp)
          const float s = (lam > 0.f && !pad) ? __fdividef(a.scale, lam) : 0.f;
          if (ENERGY) energy = fmaf(wkx * s, fmaf(o[k1].x, o[k1].x, o[k1].y * o[k1].y), energy);
          o[k1] = cscale(o[k1], s);
        }
        dft<M1, 0, 1, true>(o, u);
#pragma unroll
        for (int l2 = 0; l2 < M1; ++l2)
          sm[tx<M1>(k2, l2, c)] = l2 == 0 || k2 == 0 ? u[l2] : cmulc(u[l2], wz[k2 * l2]);
      }
    }
    if (ENERGY) energy_sum += (double)energy;
    __syncthreads();
    float2 w[M2];
#pragma unroll
    for (int k2 = 0; k2 < M2; ++k2) w[k2] = sm[tx<M1>(k2, t, c)];
    __syncthreads();  // the tile is read: the next tile's copies may go out
    if (tile + (int)gridDim.x < ntile) fetch(tile + gridDim.x);
    float2 o[M2];
    dft<M2, 0, 1, true>(w, o);
    float2* g = a.spec + (long long)ky * a.nxp + kx;
#pragma unroll
    for (int l1 = 0; l1 < M2; ++l1) g[(t + M1 * l1) * es] = o[l1];
  }
  if (ENERGY) {
    const double part[1] = {energy_sum * (double)a.ewt};
    store_partials<1, double>(part, a.I->part, gridDim.x, blockIdx.x);
  }
}

// ---- host side ----------------------------------------------------------------------------------

namespace {

// n = M1 x M2 for the supported line lengths (0 = unsupported)
void factor(int n, int* m1, int* m2) {
  switch (n) {
    case 16: *m1 = 4; *m2 = 4; return;
    case 24: *m1 = 4; *m2 = 6; return;
    case 32: *m1 = 4; *m2 = 8; return;
    case 48: *m1 = 6; *m2 = 8; return;  // x rows; y and z lines use 4 x 12 (warp-sized blocks)
    case 64: *m1 = 8; *m2 = 8; return;
    case 96: *m1 = 8; *m2 = 12; return;
    case 128: *m1 = 8; *m2 = 16; return;
    case 192: *m1 = 12; *m2 = 16; return;
    case 256: *m1 = 16; *m2 = 16; return;
    case 512: *m1 = 16; *m2 = 32; return;
    default: *m1 = 0; *m2 = 0; return;
  }
}

using SpecKernel = void (*)(SpecArgs);

constexpr int kXDirect = 256;  // nx / 2 of the weighted FP32 rows that k_spec_x_fwd transforms

template <class T>
SpecKernel x_kernel(int m, bool inverse, bool mirror, bool weight, int* threads) {
  int m1, m2;
  factor(m, &m1, &m2);
#define VDP_X(M1, M2)                                                                       \
  if (m1 == M1 && m2 == M2) {                                                               \
    *threads = M1 * (inverse || sizeof(T) == 4 ? inv_rows_per_block<M1, M2>()                \
                                               : rows_per_block<M1, M2>());                  \
    if (inverse && weight)                                                                  \
      return mirror ? k_spec_x_inv_persistent<T, M1, M2, true, true>                        \
                    : k_spec_x_inv_persistent<T, M1, M2, false, true>;                      \
    if (inverse)                                                                            \
      return mirror ? k_spec_x_inv_persistent<T, M1, M2, true, false>                       \
                    : k_spec_x_inv_persistent<T, M1, M2, false, false>;                     \
    if constexpr (sizeof(T) == 4 && M1 * M2 == kXDirect)                                    \
      if (weight) {                                                                         \
        *threads = M1 * rows_per_block<M1, M2>();                                           \
        return mirror ? k_spec_x_fwd<T, M1, M2, true> : k_spec_x_fwd<T, M1, M2, false>;     \
      }                                                                                     \
    if constexpr (sizeof(T) == 8)                                                           \
      return mirror ? k_spec_x_fwd_persistent<T, M1, M2, true>                              \
                    : k_spec_x_fwd_persistent<T, M1, M2, false>;                            \
    else                                                                                    \
      return mirror ? k_spec_x_fwd_staged<M1, M2, true> : k_spec_x_fwd_staged<M1, M2, false>; \
  }
  VDP_X(4, 4) VDP_X(4, 6) VDP_X(4, 8) VDP_X(6, 8) VDP_X(8, 8) VDP_X(8, 12) VDP_X(8, 16)
  VDP_X(16, 16)
#undef VDP_X
  return nullptr;
}

int x_rows_per_block(int m, bool half) {
  int m1, m2;
  factor(m, &m1, &m2);
#define VDP_R(M1, M2) \
  if (m1 == M1 && m2 == M2) return half ? inv_rows_per_block<M1, M2>() : rows_per_block<M1, M2>();
  VDP_R(4, 4) VDP_R(4, 6) VDP_R(4, 8) VDP_R(6, 8) VDP_R(8, 8) VDP_R(8, 12) VDP_R(8, 16)
  VDP_R(16, 16)
#undef VDP_R
  return 0;
}

SpecKernel yz_kernel(int n, int which, int* threads, size_t* smem = nullptr) {
  // which: 0 = Y+, 1 = Y-, 2 = Z, 3 = Z with the energy; smem: the pass's dynamic shared memory
  int m1, m2;
  factor(n, &m1, &m2);
  if (n == 48) {  // blocks of M1 * 8 threads: a whole number of warps for the block reduction
    m1 = 4;
    m2 = 12;
  }
#define VDP_YZ(M1, M2)                                                                  \
  if (m1 == M1 && m2 == M2) {                                                           \
    *threads = M1 * kTX;                                                                \
    if (smem) *smem = which >= 2 ? z_smem<M1, M2>() : y_smem<M1, M2>();               \
    return which == 0 ? k_spec_y<M1, M2, false> : which == 1 ? k_spec_y<M1, M2, true>   \
           : which == 2 ? k_spec_z<M1, M2, false> : k_spec_z<M1, M2, true>;             \
  }
  VDP_YZ(4, 8) VDP_YZ(4, 12) VDP_YZ(8, 8) VDP_YZ(8, 12) VDP_YZ(8, 16) VDP_YZ(12, 16)
  VDP_YZ(16, 16) VDP_YZ(16, 32)
#undef VDP_YZ
  return nullptr;
}

// Resident blocks per SM of the Y+ / Y- / Z passes for each supported line length, per device
// (filled when the spectral passes are first prepared on the device): a persistent grid is that
// times the SMs.
constexpr int kLineLengths[] = {32, 48, 64, 96, 128, 192, 256, 512};
constexpr int kLineCount = sizeof(kLineLengths) / sizeof(kLineLengths[0]);
constexpr int kMaxDevices = 64;
int g_per_sm[kMaxDevices][4][kLineCount];

int current_device() {
  int dev = -1;
  return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices ? dev : -1;
}

int line_index(int n) {
  for (int i = 0; i < kLineCount; ++i)
    if (kLineLengths[i] == n) return i;
  return -1;
}

// Resident blocks per SM of the X kernels, per device (filled with the line tables).
std::vector<std::pair<SpecKernel, int>> g_x_per_sm[kMaxDevices];
constexpr int kXHalfLengths[] = {16, 24, 32, 48, 64, 96, 128, 256};  // nx / 2

bool x_f64(int prec, bool inv, const SpecArgs& a) {
  return prec == PREC_FP64 && !(a.f32 & (inv ? kOutF32 : kInF32));
}

SpecKernel x_pass_kernel(int prec, bool inv, const SpecArgs& a, int* threads) {
  const int m = a.nx / 2;
  const bool weight = inv ? a.omega_out != nullptr : a.omega_in != nullptr;
  return x_f64(prec, inv, a) ? x_kernel<double>(m, inv, a.mirror != 0, weight, threads)
                             : x_kernel<float>(m, inv, a.mirror != 0, weight, threads);
}

// Grid of an X pass over `rows` rows: a persistent grid for the persistent forms (0 if not
// prepared), else one block per group of rows.
long long x_grid(int prec, bool inv, const SpecArgs& a, long long rows) {
  int threads = 0;
  if (!inv && a.omega_in && a.nx / 2 == kXDirect && !x_f64(prec, inv, a)) {
    const int ry = x_rows_per_block(kXDirect, false);
    return (rows + ry - 1) / ry;
  }
  const SpecKernel k = x_pass_kernel(prec, inv, a, &threads);
  const int dev = current_device(), ry = x_rows_per_block(a.nx / 2, inv || !x_f64(prec, inv, a));
  if (!k || dev < 0 || ry <= 0) return 0;
  int per_sm = 0;
  for (const auto& e : g_x_per_sm[dev])
    if (e.first == k) per_sm = e.second;
  if (per_sm < 1) return 0;
  const long long groups = (rows + ry - 1) / ry, grid = (long long)per_sm * kSMs;
  return groups < grid ? groups : grid;
}

// Persistent grid of a Y (which 0, 1) or Z (2) pass over `tiles` tiles: 0 if not prepared.
long long line_grid(int which, int n, long long tiles) {
  const int dev = current_device(), i = line_index(n);
  const int per_sm = dev >= 0 && i >= 0 ? g_per_sm[dev][which][i] : 0;
  if (per_sm < 1) return 0;
  const long long grid = (long long)per_sm * kSMs;
  return tiles < grid ? tiles : grid;
}

bool x_supported(int nx) {
  if (nx % 2) return false;
  int threads = 0;
  return x_kernel<float>(nx / 2, false, false, false, &threads) != nullptr;
}

bool yz_supported(int n) {
  int threads = 0;
  return n != 16 && n != 24 && yz_kernel(n, 0, &threads) != nullptr;
}

}  // namespace

bool spectral_supported(int nx, int ny, int nz) {
  return x_supported(nx) && yz_supported(ny) && yz_supported(nz);
}

int spectral_pitch(int nx) { return ((nx / 2 + 1 + kTX - 1) / kTX) * kTX; }

size_t spectral_table_floats(int nx, int ny, int nz) {
  const int m = nx / 2;
  return 2 * (size_t)(2 * m + 1 + ny + nz) + (size_t)(m + 1 + ny + nz);
}

void spectral_tables(int nx, int ny, int nz, double hx, double hy, double hz,
                     std::vector<float>& out) {
  const int m = nx / 2;
  out.assign(spectral_table_floats(nx, ny, nz), 0.f);
  size_t i = 0;
  auto roots = [&](int n, int count) {
    for (int k = 0; k < count; ++k) {
      const double ang = -2.0 * M_PI * (double)k / (double)n;
      out[i++] = (float)std::cos(ang);
      out[i++] = (float)std::sin(ang);
    }
  };
  roots(m, m);
  roots(nx, m + 1);
  roots(ny, ny);
  roots(nz, nz);
  auto eig = [&](int n, int count, double h) {
    for (int k = 0; k < count; ++k) {
      const double s = std::sin(M_PI * (double)k / (double)n);
      out[i++] = (float)(4.0 * s * s / (h * h));
    }
  };
  eig(nx, m + 1, hx);
  eig(ny, ny, hy);
  eig(nz, nz, hz);
}

cudaError_t spectral_prepare() {
  cudaError_t e = cudaSuccess;
  const int dev = current_device();
  if (dev < 0) e = cudaErrorInvalidDevice;
  // the Y and Z passes' tile buffer and tables: dynamic shared memory (37 and 41 KB for lines
  // of 512), then the resident blocks per SM that size their persistent grids
  for (int which = 0; which < 4 && e == cudaSuccess; ++which)
    for (int i = 0; i < kLineCount && e == cudaSuccess; ++i) {
      int threads = 0;
      size_t smem = 0;
      const SpecKernel k = yz_kernel(kLineLengths[i], which, &threads, &smem);
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      int per_sm = 0;
      if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem);
      if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
      if (e == cudaSuccess) g_per_sm[dev][which][i] = per_sm;
    }
  // the X kernels (static shared memory): resident blocks per SM, for the persistent grids
  g_x_per_sm[dev < 0 ? 0 : dev].clear();
  for (const int m : kXHalfLengths)
    for (int v = 0; v < 16 && e == cudaSuccess; ++v) {
      const bool f64 = v & 1, inv = v & 2, mirror = v & 4, weight = v & 8;
      if (weight && !inv) continue;
      int threads = 0, per_sm = 0;
      const SpecKernel k = f64 ? x_kernel<double>(m, inv, mirror, weight, &threads)
                               : x_kernel<float>(m, inv, mirror, weight, &threads);
      if (!k) continue;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, 0);
      if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
      if (e == cudaSuccess) g_x_per_sm[dev].push_back({k, per_sm});
    }
  return e;
}

cudaError_t launch_spectral_pass(int prec, int pass, const SpecArgs& a, cudaStream_t s) {
  int threads = 0;
  size_t smem = 0;
  SpecKernel k = nullptr;
  unsigned grid = 0;
  if (a.z0 < 0 || a.z1 > a.nz || a.z0 >= a.z1) return cudaErrorInvalidValue;
  switch (pass) {
    case SPEC_X_FWD:
    case SPEC_X_INV: {
      const bool inv = pass == SPEC_X_INV;
      k = x_pass_kernel(prec, inv, a, &threads);
      grid = (unsigned)x_grid(prec, inv, a, (long long)a.ny * (a.z1 - a.z0));
      break;
    }
    case SPEC_Y_FWD:
    case SPEC_Y_INV: {
      const int which = pass == SPEC_Y_FWD ? 0 : 1;
      k = yz_kernel(a.ny, which, &threads, &smem);
      grid = (unsigned)line_grid(which, a.ny, (long long)(a.nxp / kTX) * (a.z1 - a.z0));
      break;
    }
    case SPEC_Z:
      k = yz_kernel(a.nz, a.f32 & kEnergy ? 3 : 2, &threads, &smem);
      grid = (unsigned)spectral_units(a.nx, a.ny, a.nz);
      break;
    default:
      break;
  }
  if (!k || !grid) return cudaErrorInvalidValue;
  k<<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

// Slabs only on request: measured on the 512^3 mixed solve (half spectrum 553 MB), slabs of
// 128, 64 and 32 planes made one application 12 %, 20 % and 34 % slower than the whole grid --
// the passes gain less from the L2 hand-over than they lose to the extra launches and tails.
int spectral_slab_planes(int nx, int ny, int nz, int req) {
  (void)nx;
  (void)ny;
  return req > 0 && req < nz ? req : nz;
}

void spectral_schedule(int nz, int slab, std::vector<SpecLaunch>& out) {
  out.clear();
  if (slab < 1) slab = nz;
  for (int z0 = 0; z0 < nz; z0 += slab) {
    const int z1 = z0 + slab < nz ? z0 + slab : nz;
    out.push_back(SpecLaunch{SPEC_X_FWD, z0, z1});
    out.push_back(SpecLaunch{SPEC_Y_FWD, z0, z1});
  }
  out.push_back(SpecLaunch{SPEC_Z, 0, nz});
  for (int z0 = 0; z0 < nz; z0 += slab) {
    const int z1 = z0 + slab < nz ? z0 + slab : nz;
    out.push_back(SpecLaunch{SPEC_Y_INV, z0, z1});
    out.push_back(SpecLaunch{SPEC_X_INV, z0, z1});
  }
}

int spectral_xinv_units(int prec, const SpecArgs& a, int slab) {
  if (slab < 1) slab = a.nz;
  long long u = 0;
  for (int z0 = 0; z0 < a.nz; z0 += slab) {
    const int z1 = z0 + slab < a.nz ? z0 + slab : a.nz;
    u += x_grid(prec, true, a, (long long)a.ny * (z1 - z0));
  }
  return (int)u;
}

SpecArgs spectral_launch_args(int prec, const SpecArgs& a, const SpecLaunch& l, int slab) {
  SpecArgs b = a;
  b.z0 = l.z0;
  b.z1 = l.z1;
  b.xunits = spectral_xinv_units(prec, a, slab);
  return b;
}

cudaError_t launch_spectral_apply(int prec, const SpecArgs& a, int slab, cudaStream_t s) {
  std::vector<SpecLaunch> sched;
  spectral_schedule(a.nz, slab, sched);
  for (const SpecLaunch& l : sched) {
    const cudaError_t e = launch_spectral_pass(prec, l.pass, spectral_launch_args(prec, a, l, slab), s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int spectral_units(int nx, int ny, int nz) {  // CTAs of the Z pass (they store <rt, z> parts)
  return (int)line_grid(3, nz, (long long)(spectral_pitch(nx) / kTX) * ny);
}

}  // namespace vdp
