// lsp_long.cu -- one object on its whole grid by one large nonuniform FFT.
//
// lsp_transform.cu spreads every observation again for each run of 2048 bins
// and gives each run to one CTA.  For one object that wastes work when it has
// many observations (1e5 on 1e6 bins: 489 spreads of each) and leaves SMs idle
// when it has few.  Here the observations are spread once, by all SMs, onto
// one periodic grid of Mg = 2^p >= 2 N_f cells in global memory, and one
// transform of Mg points gives all bins:
//
//   spread  8 (FP32) or 16 (FP64) lanes per observation add the window to the
//           grid of 64-bit fixed-point cells {Z re, Z im, W re, W im} (one
//           32-byte sector) with integer atomics: the order does not matter,
//           repeats are bit-identical.  A cell of W is at most N, one of Z at
//           most sqrt(N sum y^2), so the scales need no pass of their own;
//   pass 1  transforms of length M1 over the cells n1 M2 + n2 of each n2,
//           times e^{2 pi i n2 k1 / Mg}, to t[n2][k1] (Mg = M1 M2);
//   pass 2  transforms of length M2 over n2 of each k1: bin offsets
//           k1 + M1 k2; powers to a row;
//   rows    re-evaluates ill-conditioned bins, writes the periodogram and the
//           runs' maxima, and (first maximum) the peak.
//
// Measured (GB300, prepared plans): 1e5 observations on 1e6 bins FP32 127 us
// (direct 23 400, run by run 1480); FP64 1000 on 1e5 82 us (direct 1404), 5e4 on
// 5e5 175 us (direct 300 000).  Up to N_f = 1e5 the FP64 time
// is the latency of the two passes' dependent two-float chains.  At 1e6 bins
// the FP32 kernels take 22 (spread), 55 (pass 1), 17 (pass 2) and 12 us (rows):
// pass 1 is bound by its access pattern, not by bytes -- M1 = 4096 leaves one
// column a tile, so each lane reads a lone 32-byte cell 16 KB from its
// neighbour's (L1 data pipe 69 %, 245 MB through L2 in 55 us).
//
// Both passes are the register transform of lsp_fft.cuh over tiles of 4096
// cells: 4096 / L columns of length L = 256 R.  The grid stays in L2 (67 MB
// for 1e6 bins).  FP64 runs in two-float numbers like lsp_transform_f64.cu,
// with the same window, Z and W in the two halves of a 512-thread CTA.
#include <cstring>

#include "../../include/lsp.h"
#include "lsp_fft.cuh"
#include "lsp_launch.h"
#include "lsp_peak.cuh"

namespace lsp {

namespace {

#define LSP_TF_TABLES_LONG
#include "lsp_transform_tables.inc"
#include "lsp_window_dd.cuh"

constexpr int kThreads = 256;

// y_exponent for FP32 factors: 2^-e has to be finite (magnitudes below 2^-126
// keep their bits, which the product with 2^126 makes normal).
__device__ __forceinline__ int y_exponent_f32(double sum_y2) { return max(y_exponent(sum_y2), -126); }

// ------------------------------------------------------------------- spread
__global__ void __launch_bounds__(kThreads) spread_f32(const RecF32* __restrict__ rec, const ObjInfo* __restrict__ obj,
                                                       uint32_t kc, int lg, long long* __restrict__ cells) {
  const ObjInfo oi = obj[0];
  const int n = oi.flags ? 0 : oi.n;
  const int lane = threadIdx.x & 31, r = lane & 7;
  const int j0 = (blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * 32;
  if (j0 >= n) return;
  f2_t poly[9];
#pragma unroll
  for (int d = 0; d < 9; ++d) poly[d] = dup_<f2_t>(__ldg(&kTfPoly[d * 8 + r]));
  const float y_sc = (float)pow2(-y_exponent_f32(oi.sum_y2)), z_one = (float)pow2(z_bits(n)), w_one = (float)pow2(w_bits(n));
  float zr = 0.f, zi = 0.f, wr = 0.f, wi = 0.f, uz = 0.f, uw = 0.f;
  uint32_t cz = 0u, cw = 0u;
  const uint32_t mask = (1u << lg) - 1u;
  const int j = j0 + lane;
  if (j < n) {
    const uint4* q = reinterpret_cast<const uint4*>(rec + oi.begin + j);
    const uint4 r0 = __ldg(q), r1 = __ldg(q + 1);
    float s, c;
    sincospif(__int2float_rn((int)phase_hi32(r0.w, r1.x, r1.y, kc)) * 4.656612873077393e-10f, &s, &c);
    const float ys = __uint_as_float(r0.x) * y_sc;
    zr = ys * c * z_one;
    zi = ys * s * z_one;
    wr = (c - s) * (c + s) * w_one;
    wi = 2.0f * c * s * w_one;
    const uint64_t b = (uint64_t)r1.x << 32 | r1.y, b2 = b << 1;
    cz = (uint32_t)(b >> (64 - lg)) - 3u;
    cw = (uint32_t)(b2 >> (64 - lg)) - 3u;
    uz = fmaf(__uint2float_rn((uint32_t)(b << lg >> 32)), 2.3283064365386963e-10f, -0.5f);
    uw = fmaf(__uint2float_rn((uint32_t)(b2 << lg >> 32)), 2.3283064365386963e-10f, -0.5f);
  }
  for (int i = lane >> 3; i < 32; i += 4) {
    const float a0 = __shfl_sync(0xffffffffu, zr, i), a1 = __shfl_sync(0xffffffffu, zi, i);
    const float a2 = __shfl_sync(0xffffffffu, wr, i), a3 = __shfl_sync(0xffffffffu, wi, i);
    const f2_t u = f2_pack(__shfl_sync(0xffffffffu, uz, i), __shfl_sync(0xffffffffu, uw, i));
    const uint32_t lz = (__shfl_sync(0xffffffffu, cz, i) + (uint32_t)r) & mask;
    const uint32_t lw = (__shfl_sync(0xffffffffu, cw, i) + (uint32_t)r) & mask;
    f2_t w2 = poly[8];
#pragma unroll
    for (int d = 7; d >= 0; --d) w2 = f2_fma(w2, u, poly[d]);
    float wz, ww;
    f2_unpack(w2, wz, ww);
    if (j0 + i < n) {
      add_cell(cells + 4 * (int64_t)lz, fixed_of(wz * a0));
      add_cell(cells + 4 * (int64_t)lz + 1, fixed_of(wz * a1));
      add_cell(cells + 4 * (int64_t)lw + 2, fixed_of(ww * a2));
      add_cell(cells + 4 * (int64_t)lw + 3, fixed_of(ww * a3));
    }
  }
}

__global__ void __launch_bounds__(kThreads) spread_f64(const RecF64* __restrict__ rec, const ObjInfo* __restrict__ obj,
                                                       uint64_t kc, int lg, long long* __restrict__ cells) {
  const ObjInfo oi = obj[0];
  const int n = oi.flags ? 0 : oi.n;
  const int lane = threadIdx.x & 31;
  const int j0 = (blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * 32;
  if (j0 >= n) return;
  const float one[2] = {(float)pow2(z_bits(n)), (float)pow2(w_bits(n))};
  const int j = j0 + lane < n ? j0 + lane : j0;
  const ObsD o = obs_of(rec[oi.begin + j], kc, lg, pow2(-y_exponent(oi.sum_y2)));
  spread_warp(o, min(32, n - j0), (1u << lg) - 1u, one, [&](int t, uint32_t l, long long re, long long im) {
    add_cell(cells + 4 * (int64_t)l + 2 * t, re);
    add_cell(cells + 4 * (int64_t)l + 2 * t + 1, im);
  });
}

// ------------------------------------------------------------------- passes
template <typename T>
__device__ __forceinline__ void dft8(Cx<T>& x0, Cx<T>& x1, Cx<T>& x2, Cx<T>& x3, Cx<T>& x4, Cx<T>& x5, Cx<T>& x6,
                                     Cx<T>& x7) {
  constexpr double h = 0.70710678118654752440;
  Cx<T> e0 = x0, e1 = x2, e2 = x4, e3 = x6, o0 = x1, o1 = x3, o2 = x5, o3 = x7;
  dft4(e0, e1, e2, e3);
  dft4(o0, o1, o2, o3);
  o1 = cmul(o1, twiddle<T>(h, h));
  o3 = cmul(o3, twiddle<T>(-h, h));
  x0 = e0 + o0;
  x4 = e0 - o0;
  x1 = e1 + o1;
  x5 = e1 - o1;
  x2 = add_i(e2, o2);
  x6 = sub_i(e2, o2);
  x3 = e3 + o3;
  x7 = e3 - o3;
}

template <typename T> struct Tables;
template <> struct Tables<f2_t> {
  static __device__ __forceinline__ float2 unit(uint32_t i) { return __ldg(&kUnit[i]); }
  static __device__ __forceinline__ float2 fine(uint32_t i) { return __ldg(&kFine[i]); }
};
template <> struct Tables<dd> {
  static __device__ __forceinline__ float4 unit(uint32_t i) { return __ldg(&kUnitD[i]); }
  static __device__ __forceinline__ float4 fine(uint32_t i) { return __ldg(&kFineD[i]); }
};

// Transforms of length L = 256 R of a tile of 4096 values, B = 16 / R columns.
// On entry thread tid = u B + col holds x[a] = element 16 R a + u of column
// col; on return thread tid = 16 p + r holds, for column col and s < R, the
// value k = p + 16 r + 256 s at x[slot<R>(s, col)].  buf: 4096 complex words
// used by these 256 threads; starts with a barrier.
template <int R>
__device__ __forceinline__ constexpr int slot(int s, int col) {
  return R == 16 ? 4 * (s & 3) + (s >> 2) : s * (16 / R) + col;
}
template <typename T, int R>
__device__ __forceinline__ void fft_tile(Cx<T> (&x)[16], Cx<T>* buf, int tid) {
  constexpr int B = 16 / R;
  const int u = tid / B, d = (tid & 15) / B;  // afterwards e = d B + col
  fft_two_passes<false>(  // run once per CTA: rolled, the loop's spills cost more (5e4 on 5e5: 195 -> 202 us)
      x, buf, tid, [&](int p) { return Tables<T>::unit((uint32_t)(p * u * B)); },
      [&](int r) { return Tables<T>::unit((uint32_t)(r * d * (256 / R)) & 4095u); });
  if constexpr (R == 2) {
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const Cx<T> a = x[c], b = x[8 + c];
      x[c] = a + b;
      x[8 + c] = a - b;
    }
  } else if constexpr (R == 4) {
#pragma unroll
    for (int c = 0; c < 4; ++c) dft4(x[c], x[4 + c], x[8 + c], x[12 + c]);
  } else if constexpr (R == 8) {
#pragma unroll
    for (int c = 0; c < 2; ++c) dft8(x[c], x[2 + c], x[4 + c], x[6 + c], x[8 + c], x[10 + c], x[12 + c], x[14 + c]);
  } else if constexpr (R == 16) {
    dft16(x);
  }
}

__device__ __forceinline__ Cx<f2_t> load_cell(const long long* cells, int64_t i, int, f2_t) {
  const longlong2* q = reinterpret_cast<const longlong2*>(cells + 4 * i);
  const longlong2 z = __ldcs(q), w = __ldcs(q + 1);
  return {f2_pack(float_of_int(z.x), float_of_int(w.x)), f2_pack(float_of_int(z.y), float_of_int(w.y))};
}
__device__ __forceinline__ Cx<dd> load_cell(const long long* cells, int64_t i, int half, dd) {
  const longlong2 z = __ldcs(reinterpret_cast<const longlong2*>(cells + 4 * i) + half);
  return {dd_of_int(z.x), dd_of_int(z.y)};
}

// Pass 1.  FP32: one CTA per tile, Z and W packed.  FP64: blockIdx.y = 0 (Z)
// or 1 (W), each with its own t.
template <typename T, int R>
__global__ void __launch_bounds__(kThreads, 2) pass1_kernel(const long long* __restrict__ cells, int lg, int m2,
                                                            Cx<T>* __restrict__ t) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  constexpr int B = 16 / R, M1 = 256 * R;
  const int tid = threadIdx.x, u = tid / B;
  const int n2 = blockIdx.x * B + tid % B;
  Cx<T> x[16];
#pragma unroll
  for (int a = 0; a < 16; ++a)
    x[a] = load_cell(cells, (int64_t)(16 * R * a + u) * m2 + n2, (int)blockIdx.y, T());
  fft_tile<T, R>(x, reinterpret_cast<Cx<T>*>(dyn_smem), tid);
  Cx<T>* const out = t + ((int64_t)blockIdx.y << lg);
  const int p = tid >> 4, r = tid & 15;
#pragma unroll
  for (int s = 0; s < R; ++s) {
#pragma unroll
    for (int c = 0; c < B; ++c) {
      const int k1 = p + 16 * r + 256 * s, n = blockIdx.x * B + c;
      // e^{2 pi i n k1 / Mg}: the index' top 12 bits and the rest, in units of 2^-24
      const uint32_t e = (uint32_t)(n * k1) << (24 - lg);
      Cx<T> v = cmul(x[slot<R>(s, c)], Tables<T>::unit((e >> 12) & 4095u));
      v = cmul(v, Tables<T>::fine(e & 4095u));
      put(out, n * M1 + k1, v);
    }
  }
}

__device__ __forceinline__ float deconv(float z, float) {
  float v = __ldg(&kDeconvPoly[8]);
#pragma unroll
  for (int d = 7; d >= 0; --d) v = fmaf(v, z, __ldg(&kDeconvPoly[d]));
  return v;
}
__device__ __forceinline__ dd deconv(dd z) {
  float2 c = __ldg(&kDeconvPolyD[16]);
  dd v{c.x, c.y};
#pragma unroll
  for (int d = 15; d >= 0; --d) {
    c = __ldg(&kDeconvPolyD[d]);
    v = add_(mul_(v, z), dd{c.x, c.y});
  }
  return v;
}

// Pass 2, FP32: powers of the bins k1 + M1 k2 - Mg (k2 in the upper half) +
// kc into row[] (-1: re-evaluate).
template <int R>
__global__ void __launch_bounds__(kThreads, 2) pass2_f32(const Cx<f2_t>* __restrict__ t, int lg, int m1, int kc, int n_f,
                                                         const ObjInfo* __restrict__ obj, float* __restrict__ row) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  constexpr int B = 16 / R, M2 = 256 * R;
  const int tid = threadIdx.x, u = tid / B;
  Cx<f2_t> x[16];
#pragma unroll
  for (int a = 0; a < 16; ++a) x[a] = get(t, (16 * R * a + u) * m1 + (int)blockIdx.x * B + tid % B);
  fft_tile<f2_t, R>(x, reinterpret_cast<Cx<f2_t>*>(dyn_smem), tid);
  const ObjInfo oi = obj[0];
  const int n = oi.flags ? 0 : oi.n;
  const f2_t inv = f2_pack((float)pow2(-z_bits(n)), (float)pow2(-w_bits(n)));
  const float nf = (float)oi.n;
  // the magnitudes' power of two comes back with the normalisation, in FP64 range
  const double y_inv = pow2(y_exponent_f32(oi.sum_y2));
  const float scale = (float)(oi.norm_scale * y_inv * y_inv);
  const int p = tid >> 4, r = tid & 15;
  const float xi4 = (float)pow2(2 - lg);  // 4 / Mg
#pragma unroll
  for (int s = 0; s < R; ++s) {
    const int k2 = p + 16 * r + 256 * s;
    const int m = m1 * k2 + (int)blockIdx.x * B - (k2 >= M2 / 2 ? 1 << lg : 0);
    const int bin = m + kc;
    if (bin < 0 || bin >= n_f) continue;
    float v[B];
#pragma unroll
    for (int c = 0; c < B; ++c) {
      const float xi = (float)(m + c) * xi4;
      const float f1 = deconv(xi * xi, 0.0f);
      const f2_t f = f2_mul(f2_pack(f1, f1), inv);
      float zr, wr, zi, wi;
      f2_unpack(f2_mul(x[slot<R>(s, c)].re, f), zr, wr);
      f2_unpack(f2_mul(x[slot<R>(s, c)].im, f), zi, wi);
      bool ill;
      const float pw = scale * power_zw(zr, zi, wr, wi, nf, ill);
      v[c] = ill ? -1.0f : pw;
    }
    if constexpr (B >= 4) {
#pragma unroll
      for (int c = 0; c < B; c += 4) *reinterpret_cast<float4*>(row + bin + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
    } else {
#pragma unroll
      for (int c = 0; c < B; ++c) row[bin + c] = v[c];
    }
  }
}

// Pass 2, FP64: threads 0 .. 255 transform Z's tile, 256 .. 511 W's; then all
// of them share the powers.
template <int R>
__global__ void __launch_bounds__(2 * kThreads, 1) pass2_f64(const Cx<dd>* __restrict__ t, int lg, int m1, int kc, int n_f,
                                                             const ObjInfo* __restrict__ obj, double* __restrict__ row) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  constexpr int B = 16 / R, M2 = 256 * R;
  Cx<dd>* const buf = reinterpret_cast<Cx<dd>*>(dyn_smem);
  const int half = threadIdx.x >> 8, tid = threadIdx.x & 255, u = tid / B;
  {
    const Cx<dd>* const in = t + ((int64_t)half << lg);
    Cx<dd> x[16];
#pragma unroll
    for (int a = 0; a < 16; ++a) x[a] = get(in, (16 * R * a + u) * m1 + (int)blockIdx.x * B + tid % B);
    fft_tile<dd, R>(x, buf + half * 4096, tid);
    __syncthreads();
    // word (s, c) of thread tid at 256 (s B + c) + tid
#pragma unroll
    for (int s = 0; s < R; ++s)
#pragma unroll
      for (int c = 0; c < B; ++c) put(buf + half * 4096, 256 * (s * B + c) + tid, x[slot<R>(s, c)]);
  }
  __syncthreads();
  const ObjInfo oi = obj[0];
  const int n = oi.flags ? 0 : oi.n;
  const float z_inv = (float)pow2(-z_bits(n)), w_inv = (float)pow2(-w_bits(n));
  const double y_inv = pow2(y_exponent(oi.sum_y2));
  const double scale = oi.norm_scale * y_inv * y_inv;
  const dd nd = dd_of((double)oi.n);
  const int p = tid >> 4, r = tid & 15;
#pragma unroll 1
  for (int q = half * 8; q < half * 8 + 8; ++q) {
    const int s = q / B, c = q % B;
    const int k2 = p + 16 * r + 256 * s;
    const int m = m1 * k2 + (int)blockIdx.x * B + c - (k2 >= M2 / 2 ? 1 << lg : 0);
    const int bin = m + kc;
    if (bin < 0 || bin >= n_f) continue;
    const float xs = (float)pow2(2 - lg);
    const dd xi = dd{(float)m * xs, 0.0f};  // |m| < 2^24: exact
    const dd f = deconv(mul_(xi, xi));
    const dd fz{f.hi * z_inv, f.lo * z_inv}, fw{f.hi * w_inv, f.lo * w_inv};
    const Cx<dd> z = get(buf, 256 * q + tid), w = get(buf + 4096, 256 * q + tid);
    bool ill;
    const dd v = power_dd(Cx<dd>{mul_(z.re, fz), mul_(z.im, fz)}, Cx<dd>{mul_(w.re, fw), mul_(w.im, fw)}, nd, ill);
    row[bin] = ill ? -1.0 : scale * dd_double(v);
  }
}

// --------------------------------------------------------------------- rows
__device__ __forceinline__ void fix_row(float (&pv)[8], uint32_t k0, int64_t n_f, const RecF32* rec, const ObjInfo& oi) {
  uint32_t bad = 0u;
#pragma unroll
  for (int m = 0; m < 8; ++m)
    if (pv[m] < 0.0f && (int64_t)k0 + m < n_f) bad |= 1u << m;
  fix_ill_conditioned<8>(pv, bad, k0, rec, oi.begin, oi.n, oi.norm_scale);
}
__device__ __forceinline__ void fix_row(double (&pv)[8], uint32_t k0, int64_t n_f, const RecF64* rec, const ObjInfo& oi) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    unsigned mask = __ballot_sync(0xffffffffu, pv[m] < 0.0 && (int64_t)k0 + m < n_f);
    while (mask) {
      const int l = __ffs(mask) - 1;
      mask &= mask - 1;
      const uint32_t k = __shfl_sync(0xffffffffu, k0 + (uint32_t)m, l);
      const double q = exact_power_warp64(rec, oi.begin, oi.n, k, oi.norm_scale);
      if (lane == l) pv[m] = q;
    }
  }
}

template <typename Rec, typename Real>
__global__ void __launch_bounds__(kThreads) rows_kernel(const Real* __restrict__ row, TransformParamsOf<Rec, Real> p) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  __shared__ double red_p[32];
  __shared__ int64_t red_k[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const ObjInfo oi = p.obj[0];
  const int64_t kc0 = (int64_t)blockIdx.x * kTfBins;
  const uint32_t k0 = (uint32_t)kc0 + 8u * (uint32_t)tid;
  Real pv[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) pv[m] = !oi.flags && (int64_t)k0 + m < p.n_f ? row[k0 + m] : Real(0);
  fix_row(pv, k0, p.n_f, p.rec, oi);
  if (p.power_out) store_row<8>(p.power_out, (int64_t)k0, pv, p.n_f);
  if constexpr (sizeof(Real) == 4)
    chunk_results_f32<8>(pv, k0, kc0, p.n_f, p.best + blockIdx.x, p.cand ? p.cand + blockIdx.x : nullptr,
                         reinterpret_cast<float*>(dyn_smem), reinterpret_cast<unsigned long long*>(red_p));
  else
    chunk_results<double, 8>(pv, (int64_t)k0, kc0, p.n_f, p.best + blockIdx.x, p.cand ? p.cand + blockIdx.x : nullptr,
                             reinterpret_cast<double*>(dyn_smem), red_p, red_k);
  // first maximum: the last CTA to finish writes the peak
  if (!p.peaks) return;
  __shared__ bool s_last;
  if (tid == 0) {  // thread 0 wrote this CTA's results
    __threadfence();
    s_last = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last || warp != 0) return;
  __threadfence();
  double bp = 0.0;
  int64_t bk = -1;
  for (uint32_t c = lane; c < gridDim.x; c += 32) {
    const double q = __ldcg(&p.best[c].p);
    const int64_t k = __ldcg(&p.best[c].k);
    if (better(q, k, bp, bk)) {
      bp = q;
      bk = k;
    }
  }
  warp_best(bp, bk);
  if (lane == 0) p.peaks[0] = make_peak(bk, bp, p.f_min, p.df, oi.flags);
}

template <typename Kern, typename... Args>
cudaError_t go(Kern kern, dim3 grid, int threads, size_t dyn, cudaStream_t st, Args... args) {
  cudaError_t e = allow_dyn_smem(kern, dyn);
  if (e != cudaSuccess) return e;
  kern<<<grid, threads, dyn, st>>>(args...);
  return cudaGetLastError();
}

template <typename T>
cudaError_t pass1(const LongPlan& lp, const long long* cells, Cx<T>* t, cudaStream_t st) {
  const int r1 = (1 << (lp.lg - lp.lg2)) / 256;
  const dim3 grid((1u << lp.lg) / 4096u, sizeof(T) == 8 && std::is_same<T, dd>::value ? 2u : 1u);
  const size_t dyn = 4096 * sizeof(Cx<T>);
  const int m2 = 1 << lp.lg2;
  switch (r1) {
    case 1: return go(pass1_kernel<T, 1>, grid, kThreads, dyn, st, cells, lp.lg, m2, t);
    case 2: return go(pass1_kernel<T, 2>, grid, kThreads, dyn, st, cells, lp.lg, m2, t);
    case 4: return go(pass1_kernel<T, 4>, grid, kThreads, dyn, st, cells, lp.lg, m2, t);
    case 8: return go(pass1_kernel<T, 8>, grid, kThreads, dyn, st, cells, lp.lg, m2, t);
    case 16: return go(pass1_kernel<T, 16>, grid, kThreads, dyn, st, cells, lp.lg, m2, t);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

bool long_plan(int prec, int64_t n_f, LongPlan* lp) {
  int lg = 16;
  while (lg <= kLongMaxLog2 && ((int64_t)1 << (lg - 1)) < n_f + 32) ++lg;
  if (lg > kLongMaxLog2) return false;
  lp->lg = lg;
  lp->lg2 = lg <= 20 ? 8 : lg - 12;
  lp->kc = (int32_t)(n_f / 2) & ~15;  // pass 2 stores groups of up to 16 bins from multiples of 16
  const size_t m = (size_t)1 << lg;
  lp->cell_bytes = m * 32;
  lp->t_bytes = m * (prec ? 32 : 16);
  lp->row_bytes = ((size_t)n_f + 32) * (prec ? 8 : 4);
  return true;
}

cudaError_t launch_long32(const LongPlan& lp, const TransformParams& p, int64_t max_n, void* cells, void* t, void* row,
                          cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(cells, 0, lp.cell_bytes, st);
  if (e != cudaSuccess) return e;
  long long* c = (long long*)cells;
  e = go(spread_f32, dim3((unsigned)((max_n + kThreads - 1) / kThreads)), kThreads, 0, st, p.rec, p.obj, (uint32_t)lp.kc,
         lp.lg, c);
  if (e == cudaSuccess) e = pass1<f2_t>(lp, c, (Cx<f2_t>*)t, st);
  if (e != cudaSuccess) return e;
  const dim3 grid((1u << lp.lg) / 4096u);
  const size_t dyn = 4096 * 16;
  const int m1 = 1 << (lp.lg - lp.lg2), n_f = (int)p.n_f;
  const Cx<f2_t>* tt = (const Cx<f2_t>*)t;
  switch (lp.lg2) {
    case 8: e = go(pass2_f32<1>, grid, kThreads, dyn, st, tt, lp.lg, m1, lp.kc, n_f, p.obj, (float*)row); break;
    case 9: e = go(pass2_f32<2>, grid, kThreads, dyn, st, tt, lp.lg, m1, lp.kc, n_f, p.obj, (float*)row); break;
    case 10: e = go(pass2_f32<4>, grid, kThreads, dyn, st, tt, lp.lg, m1, lp.kc, n_f, p.obj, (float*)row); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  return go(rows_kernel<RecF32, float>, dim3((unsigned)p.n_chunks), kThreads, (4 * (kThreads / 32) + 2) * sizeof(float),
            st, (const float*)row, p);
}

cudaError_t launch_long64(const LongPlan& lp, const TransformParams64& p, int64_t max_n, void* cells, void* t, void* row,
                          cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(cells, 0, lp.cell_bytes, st);
  if (e != cudaSuccess) return e;
  long long* c = (long long*)cells;
  e = go(spread_f64, dim3((unsigned)((max_n + kThreads - 1) / kThreads)), kThreads, 0, st, p.rec, p.obj, (uint64_t)lp.kc,
         lp.lg, c);
  if (e == cudaSuccess) e = pass1<dd>(lp, c, (Cx<dd>*)t, st);
  if (e != cudaSuccess) return e;
  const dim3 grid((1u << lp.lg) / 4096u);
  const size_t dyn = 2 * 4096 * 16;
  const int m1 = 1 << (lp.lg - lp.lg2), n_f = (int)p.n_f;
  const Cx<dd>* tt = (const Cx<dd>*)t;
  switch (lp.lg2) {
    case 8: e = go(pass2_f64<1>, grid, 2 * kThreads, dyn, st, tt, lp.lg, m1, lp.kc, n_f, p.obj, (double*)row); break;
    case 9: e = go(pass2_f64<2>, grid, 2 * kThreads, dyn, st, tt, lp.lg, m1, lp.kc, n_f, p.obj, (double*)row); break;
    case 10: e = go(pass2_f64<4>, grid, 2 * kThreads, dyn, st, tt, lp.lg, m1, lp.kc, n_f, p.obj, (double*)row); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  return go(rows_kernel<RecF64, double>, dim3((unsigned)p.n_chunks), kThreads, (size_t)kThreads * 8 * 8, st,
            (const double*)row, p);
}

}  // namespace lsp
