// vdp_fft.cuh -- device code of the line transforms of the spectral passes, shared by the passes
// (vdp_spectral.cu) and the resident solve (vdp_resident.cu): register DFTs, the row transforms of
// X+ and X-, and the tile layout of the Y and Z lines.  Internal to libvdp.
#pragma once

#include "vdp_device.cuh"
#include "vdp_internal.cuh"
#include "vdp_spectral.h"

namespace vdp {

// ---- complex arithmetic and small DFTs in registers ---------------------------------------------

// Complex sums, differences and real scalings as one paired FP32 instruction (add / sub / mul
// .rn.f32x2: both lanes rounded as the scalar operation would round them); the FFT butterflies
// are mostly these (Z issues the most instructions per byte of all passes).
#define VDP_F32X2(op)                                                                        \
  "{\n .reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n " op        \
  ".rn.f32x2 rd, ra, rb;\n mov.b64 {%0, %1}, rd;\n}"
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
  float2 r;
  asm(VDP_F32X2("add") : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  float2 r;
  asm(VDP_F32X2("sub") : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 cscale(float2 a, float s) {
  float2 r;
  asm(VDP_F32X2("mul") : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(s), "f"(s));
  return r;
}
#undef VDP_F32X2
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}

// exp(-2 pi i k / 96), 0 <= k < 96: the roots of unity of every register DFT size used here (all
// divide 96).  k is a constant after unrolling, so each root is an immediate operand (from a table in
// constant memory the Z pass ran 128^3 in 13.1 us instead of 12.5).
__device__ __forceinline__ float quarter_cos(int j) {  // cos(2 pi j / 96), j = 0 .. 24
  switch (j) {
    case 0: return 1.0f; case 1: return 0.997858942f; case 2: return 0.991444886f;
    case 3: return 0.980785251f; case 4: return 0.965925813f; case 5: return 0.94693011f;
    case 6: return 0.923879504f; case 7: return 0.896872759f; case 8: return 0.866025388f;
    case 9: return 0.831469595f; case 10: return 0.793353319f; case 11: return 0.751839817f;
    case 12: return 0.707106769f; case 13: return 0.659345806f; case 14: return 0.60876143f;
    case 15: return 0.555570245f; case 16: return 0.5f; case 17: return 0.442288697f;
    case 18: return 0.382683426f; case 19: return 0.321439475f; case 20: return 0.258819044f;
    case 21: return 0.195090324f; case 22: return 0.130526185f; case 23: return 0.0654031262f;
    case 24: return 0.0f;
  }
  return 0.f;
}
__device__ __forceinline__ float cos96(int k) {
  const int j = k > 48 ? 96 - k : k;
  return j <= 24 ? quarter_cos(j) : -quarter_cos(48 - j);
}
__device__ __forceinline__ float2 root96(int k) { return make_float2(cos96(k), -cos96((k + 72) % 96)); }

// v * W_M^k with W = exp(-2 pi i / M) (INV: the conjugate root).  k and M are constants after
// unrolling, so the trivial roots cost nothing and the others are immediates.
template <bool INV>
__device__ __forceinline__ float2 rot(float2 v, int k, int M) {
  k %= M;
  if (k == 0) return v;
  if (2 * k == M) return make_float2(-v.x, -v.y);
  if (4 * k == M) return INV ? make_float2(-v.y, v.x) : make_float2(v.y, -v.x);
  if (4 * k == 3 * M) return INV ? make_float2(v.y, -v.x) : make_float2(-v.y, v.x);
  const float2 w = root96((96 / M) * k);
  return cmul(v, INV ? cconj(w) : w);
}

// y[k] = sum_j x[O + S j] W_M^(j k), k < M: recursive decimation in time (radix 2, then 3).
template <int M, int O, int S, bool INV, int N>
__device__ __forceinline__ void dft(const float2 (&x)[N], float2 (&y)[M]) {
  static_assert(O + S * (M - 1) < N, "dft reads outside its input");
  if constexpr (M == 1) {
    y[0] = x[O];
  } else if constexpr (M % 2 == 0) {
    constexpr int H = M / 2;
    float2 e[H], o[H];
    dft<H, O, 2 * S, INV>(x, e);
    dft<H, O + S, 2 * S, INV>(x, o);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const float2 t = rot<INV>(o[k], k, M);
      y[k] = cadd(e[k], t);
      y[k + H] = csub(e[k], t);
    }
  } else {
    static_assert(M % 3 == 0, "register DFT sizes are products of 2 and 3");
    constexpr int T = M / 3;
    constexpr float kS3 = 0.86602540378443864676f;  // sin(pi / 3)
    float2 a[T], b[T], c[T];
    dft<T, O, 3 * S, INV>(x, a);
    dft<T, O + S, 3 * S, INV>(x, b);
    dft<T, O + 2 * S, 3 * S, INV>(x, c);
#pragma unroll
    for (int k = 0; k < T; ++k) {
      const float2 tb = rot<INV>(b[k], k, M), tc = rot<INV>(c[k], 2 * k, M);
      const float2 s = cadd(tb, tc), d = csub(tb, tc);
      const float2 m = make_float2(a[k].x - 0.5f * s.x, a[k].y - 0.5f * s.y);
      // forward: W_3 = -1/2 - i sin(pi/3); (tb - tc) times -i sin(pi/3) (+i for the inverse)
      const float2 j = INV ? make_float2(-kS3 * d.y, kS3 * d.x) : make_float2(kS3 * d.y, -kS3 * d.x);
      y[k] = cadd(a[k], s);
      y[k + T] = cadd(m, j);
      y[k + 2 * T] = csub(m, j);
    }
  }
}

// ---- table layout ---------------------------------------------------------------------------------

struct Tables {
  const float2* wm;  // W_m^k, m = nx / 2
  const float2* wr;  // W_nx^k, k = 0 .. m
  const float2* wy;  // W_ny^k
  const float2* wz;  // W_nz^k
  const float* lx;   // 4 sin^2(pi k / nx) / hx^2, k = 0 .. m
  const float* ly;
  const float* lz;
};

__device__ __forceinline__ Tables tables(const SpecArgs& a) {
  const int m = a.nx / 2;
  Tables t;
  t.wm = a.tw;
  t.wr = a.tw + m;
  t.wy = a.tw + 2 * m + 1;
  t.wz = a.tw + 2 * m + 1 + a.ny;
  t.lx = a.lam;
  t.ly = a.lam + m + 1;
  t.lz = a.lam + m + 1 + a.ny;
  return t;
}

// In the solve every pass first checks that the instance is in the spectral phase (one L2
// load per block: thread 0's, handed on by the barrier); the stand-alone inverse passes
// st = nullptr and always runs.  Every thread calls it.
__device__ __forceinline__ bool spec_active(const SpecArgs& a) {
  if (a.st == nullptr) return true;
  return __syncthreads_or(threadIdx.x == 0 && __ldcg(&a.st->phase) == PH_SPEC) != 0;
}

template <class T> struct Pair;
template <> struct Pair<float> {
  static __device__ __forceinline__ float2 ld(const float* p) { return *reinterpret_cast<const float2*>(p); }
  static __device__ __forceinline__ void st(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
  static __device__ __forceinline__ void ld2(const float* p, float& a, float& b) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    a = v.x;
    b = v.y;
  }
};
template <> struct Pair<double> {
  static __device__ __forceinline__ float2 ld(const double* p) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    return make_float2(narrow(v.x), narrow(v.y));
  }
  static __device__ __forceinline__ void st(double* p, float2 v) {
    *reinterpret_cast<double2*>(p) = make_double2(widen(v.x), widen(v.y));
  }
  static __device__ __forceinline__ void ld2(const double* p, double& a, double& b) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    a = v.x;
    b = v.y;
  }
};

// Shared-memory row strides (in complex values) congruent to 8 modulo 16: the four rows (or
// line groups) a warp touches then fall on alternating halves of the 32 banks.
__host__ __device__ constexpr int pad_stride(int len) { return ((len + 7) / 16) * 16 + 8; }

// Shared memory of one row in the X passes: the four-step exchange, reused for the whole
// transformed row (X+ unpack).
template <int M1, int M2>
constexpr int x_row_stride() {
  return pad_stride(M2 * (M1 + 1)) > pad_stride(M1 * M2 + 1) ? pad_stride(M2 * (M1 + 1))
                                                              : pad_stride(M1 * M2 + 1);
}

// Rows per block of the X passes: at most 256 threads and about 40 KB of shared memory, and a
// multiple of 32 threads (the block reduction works on whole warps).
template <int M1, int M2>
constexpr int rows_per_block() {
  for (int ry = 256 / M1; ry > 1; --ry)
    if ((M1 * ry) % 32 == 0 && 8 * ry * x_row_stride<M1, M2>() <= 40960) return ry;
  return 32;  // not reached for the supported sizes
}

// Rows per block of X- (register bound: half the rows of X+, so that more blocks share an SM).
template <int M1, int M2>
constexpr int inv_rows_per_block() {
  for (int ry = 256 / M1; ry > 1; --ry)
    if ((M1 * ry) % 32 == 0 &&
        8 * ry * (pad_stride(M2 * (M1 + 1)) + pad_stride(M1 * M2 + 1)) <= 40960)
      return ry;
  return 32;  // not reached for the supported sizes
}

// The four-step exchange of one line through shared memory: step A's thread j1 writes its
// M2 outputs to [k2][j1], step B's thread k2 reads them back; rows of M1 + 1 values keep the
// step B reads (stride M1 + 1) free of bank conflicts.
template <int M1>
__device__ __forceinline__ int ex(int k2, int j1) { return k2 * (M1 + 1) + j1; }

// 16-byte asynchronous copy global -> shared (cached in L2 only), and its group wait: the copies
// hold no registers while in flight, so a block can fetch its next tile while it finishes this
// one.  wait_group is a hardware wait for this thread's own copies (no spin loop).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// ---- X+ : real rows -> half spectrum -----------------------------------------------------------

// The X+ transform of RY rows (one per group of M1 threads: t = lane in the row, r = row in the
// group), row `row` of the grid in thread group r; `ra` is the row's shared buffer of SX values
// (the exchange, then the transformed row); `in` its cells (global or shared memory).  store(k, X)
// receives bin k of the row's half spectrum for k < nxp (zero beyond nx/2); read() is called once
// every thread of the block has read its part of `in`.  Every thread of the block calls it
// (barriers).
template <class T, int M1, int M2, bool MIRROR, class Store, class Read>
__device__ __forceinline__ void x_fwd_rows(const SpecArgs& a, const Tables& tb, float2* ra, const T* in,
                                           long long row, bool live, int t, Store&& store, Read&& read) {
  constexpr int m = M1 * M2;
  float2* rb = ra;
  // step A: M2-point DFTs over j2 of z[t + M1 j2] = (x[2j], x[2j+1]) * W
  if (live) {
    const float* om = a.omega_in ? a.omega_in + row * a.nxd : nullptr;
    float2 v[M2], y[M2];
#pragma unroll
    for (int j2 = 0; j2 < M2; ++j2) {
      const int j = t + M1 * j2;
      // pair j of the transformed row; mirrored rows read their second half backwards:
      // cells (2j, 2j + 1) of the extension are cells (q + 1, q) of the row, q = 2 nxd - 2 - 2j
      const bool back = MIRROR && 2 * j >= a.nxd;
      const int q = back ? 2 * a.nxd - 2 - 2 * j : 2 * j;
      float2 z = Pair<T>::ld(in + q);
      if (om) {
        const float2 w = *reinterpret_cast<const float2*>(om + q);
        z = make_float2(z.x * w.x, z.y * w.y);
      }
      v[j2] = back ? make_float2(z.y, z.x) : z;
    }
    dft<M2, 0, 1, false>(v, y);
#pragma unroll
    for (int k2 = 0; k2 < M2; ++k2)
      ra[ex<M1>(k2, t)] = k2 == 0 || t == 0 ? y[k2] : cmul(y[k2], tb.wm[t * k2]);
  }
  __syncthreads();
  read();
  // step B: M1-point DFTs over j1 -> Z[k2 + M2 k1]; the exchange is read completely before the
  // transformed row overwrites it
  constexpr int R = (M2 + M1 - 1) / M1;
  float2 u[R][M1];
  if (live) {
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
      const int k2 = t + M1 * rr;
      if (k2 < M2) {
#pragma unroll
        for (int j1 = 0; j1 < M1; ++j1) u[rr][j1] = ra[ex<M1>(k2, j1)];
      }
    }
  }
  __syncthreads();
  if (live) {
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
      const int k2 = t + M1 * rr;
      if (k2 < M2) {
        float2 o[M1];
        dft<M1, 0, 1, false>(u[rr], o);
#pragma unroll
        for (int k1 = 0; k1 < M1; ++k1) rb[k2 + M2 * k1] = o[k1];
      }
    }
  }
  __syncthreads();
  // unpack: X[k] = E + W_nx^k O, X[m - k] = conj(E - W_nx^k O) with E = (Z[k] + conj Z[m-k]) / 2,
  // O = (Z[k] - conj Z[m-k]) / 2i: both bins of a pair from one pair of values
  if (live) {
    auto bins = [&](int k) {
      const float2 p = rb[k], q = cconj(rb[k == 0 ? 0 : m - k]);
      const float2 e = cscale(cadd(p, q), 0.5f), d = cscale(csub(p, q), 0.5f);
      const float2 o = cmul(tb.wr[k], make_float2(d.y, -d.x));
      store(k, cadd(e, o));
      if (k != m / 2) store(m - k, cconj(csub(e, o)));
    };
#pragma unroll
    for (int i = 0; i < M2 / 2; ++i) bins(t + M1 * i);
    if (t == 0) bins(m / 2);
    for (int k = m + 1 + t; k < a.nxp; k += M1) store(k, make_float2(0.f, 0.f));
  }
}

// The X tables W_m^k (k < m) and W_nx^k (k <= m) copied to the block's shared memory (every
// lookup of a row transform is then a shared-memory load); returns the tables with them.
template <int M1, int M2>
__device__ __forceinline__ Tables x_tables_shared(const SpecArgs& a, float2* st) {
  constexpr int m = M1 * M2;
  Tables tb = tables(a);
  for (int k = threadIdx.x; k < 2 * m + 1; k += blockDim.x) st[k] = k < m ? tb.wm[k] : tb.wr[k - m];
  __syncthreads();
  tb.wm = st;
  tb.wr = st + m;
  return tb;
}

// ---- X- : half spectrum -> real rows, z = W x ----------------------------------------------------

// The X- transform of one row per group of M1 threads: `src` is the row of the half spectrum
// (global or shared memory), `rb` the group's shared exchange buffer; z = W x is stored to row
// `row` of a.out; read() is called once every thread of the block has read its part of src.
// Every thread of the block calls it (barrier).
template <class T, int M1, int M2, bool MIRROR, bool WEIGHT, class Read>
__device__ __forceinline__ void x_inv_rows(const SpecArgs& a, const Tables& tb, float2* rb,
                                           const float2* src, long long row, bool live, int t,
                                           Read&& read) {
  constexpr int m = M1 * M2;
  // the output weights of this thread's cells are loaded first, so that their latency overlaps
  // the transforms (cells 2l, 2l + 1 with l = k2 + M2 k1, k2 = t, t + M1, ...)
  constexpr int R = (M2 + M1 - 1) / M1;
  float2 wv[R][M1];
  if constexpr (WEIGHT) {
    const float* om = a.omega_out + row * a.nxd;
#pragma unroll
    for (int rr = 0; rr < R; ++rr)
#pragma unroll
      for (int k1 = 0; k1 < M1; ++k1) {
        const int k2 = t + M1 * rr;
        const int l = k2 + M2 * k1;
        wv[rr][k1] = make_float2(1.f, 1.f);
        if (live && k2 < M2 && (!MIRROR || 2 * l < a.nxd))
          wv[rr][k1] = *reinterpret_cast<const float2*>(om + 2 * l);
      }
  }
  // Z'[k] = (X[k] + conj X[m-k]) + i conj(W_nx^k) (X[k] - conj X[m-k]); inverse M2-point DFTs.
  // Both X[k] and X[m-k] are read straight from the spectrum: for a fixed j2 the lanes of a row
  // read consecutive values, ascending and descending.
  if (live) {
    float2 xa[M2], xb[M2];
#pragma unroll
    for (int j2 = 0; j2 < M2; ++j2) {
      const int k = t + M1 * j2;
      xa[j2] = src[k];
      xb[j2] = src[m - k];
    }
    float2 v[M2], y[M2];
#pragma unroll
    for (int j2 = 0; j2 < M2; ++j2) {
      const int k = t + M1 * j2;
      const float2 p = xa[j2], q = cconj(xb[j2]);
      const float2 e = cadd(p, q);
      const float2 o = cmulc(csub(p, q), tb.wr[k]);
      v[j2] = make_float2(e.x - o.y, e.y + o.x);
    }
    dft<M2, 0, 1, true>(v, y);
#pragma unroll
    for (int k2 = 0; k2 < M2; ++k2)
      rb[ex<M1>(k2, t)] = k2 == 0 || t == 0 ? y[k2] : cmulc(y[k2], tb.wm[t * k2]);
  }
  __syncthreads();
  read();
  if (live) {
    T* out = static_cast<T*>(a.out) + row * a.nxd;
#pragma unroll
    for (int rr = 0; rr < R; ++rr) {
      const int k2 = t + M1 * rr;
      if (k2 >= M2) break;
      float2 u[M1], o[M1];
#pragma unroll
      for (int j1 = 0; j1 < M1; ++j1) u[j1] = rb[ex<M1>(k2, j1)];
      dft<M1, 0, 1, true>(u, o);
#pragma unroll
      for (int k1 = 0; k1 < M1; ++k1) {
        const int l = k2 + M2 * k1;  // cells 2l, 2l + 1 of the row
        if (MIRROR && 2 * l >= a.nxd) continue;  // the second half is the reflection
        Pair<T>::st(out + 2 * l, WEIGHT ? make_float2(o[k1].x * wv[rr][k1].x, o[k1].y * wv[rr][k1].y)
                                        : o[k1]);
      }
    }
  }
}

// ---- Y and Z: tiles of TX consecutive kx columns, whole lines -----------------------------------

constexpr int kTX = 8;  // columns per tile (64 bytes of each line element)

// shared-memory index of line element e (of a tile column c) when lines are grouped by g
// elements: groups of g * kTX values padded to a stride = 8 (mod 16)
template <int G>
__device__ __forceinline__ int tx(int group, int e, int c) {
  return group * pad_stride(G * kTX) + e * kTX + c;
}

// Tiles of the Y and Z passes: nz (or ny) line elements of kTX columns.  Element e = t + M1 j2 of
// column c is copied to slot (j2, t, c) of the tile buffer, the layout step A reads; step A
// writes the exchange to slots (k2, t, c) of the same buffer.
template <int M1, int M2>
constexpr int line_buffer() { return M2 * pad_stride(M1 * kTX); }  // complex values of one tile
// Copies of the tile of n = M1 x M2 line elements at g (element stride es) into the buffer sm:
// 4 pieces of 16 bytes per element, spread over the block's threads; one commit group.
template <int M1, int M2>
__device__ __forceinline__ void fetch_tile(float2* sm, const float2* g, long long es) {
  constexpr int S = pad_stride(M1 * kTX);
  for (int q = threadIdx.x; q < 4 * M1 * M2; q += M1 * kTX) {
    const int e = q >> 2, part = q & 3;
    cp_async16(sm + (e / M1) * S + (e % M1) * kTX + 2 * part, g + e * es + 2 * part);
  }
  cp_async_commit();
}

}  // namespace vdp
