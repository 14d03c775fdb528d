// lsp_fft.cuh -- the 4096-point transform of the transform kernels (internal).
//
// One CTA of 256 threads, 16 points per thread, 4096 = 16^3: three register
// passes with two exchanges through shared memory, e^{+2 pi i jk / 4096},
// outputs only for the half of the frequencies inside a run of bins.  The
// element type T is f2_t (two FP32 transforms side by side in packed f32x2
// halves, sharing every twiddle), float, or dd (two-float numbers of about 48
// bits, the FP64 path).
#pragma once

#include <cstring>
#include <type_traits>

#include "lsp_common.cuh"

namespace lsp {

// ------------------------------------------------------------ arithmetic on
// f32x2 pairs (two transforms at once) or single floats
__device__ __forceinline__ f2_t add_(f2_t a, f2_t b) {
  f2_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2_t sub_(f2_t a, f2_t b) { return f2_fma(b, 0xbf800000bf800000ull, a); }
__device__ __forceinline__ float add_(float a, float b) { return a + b; }
__device__ __forceinline__ float sub_(float a, float b) { return a - b; }
__device__ __forceinline__ f2_t mul_(f2_t a, f2_t b) { return f2_mul(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return a * b; }
__device__ __forceinline__ f2_t fma_(f2_t a, f2_t b, f2_t c) { return f2_fma(a, b, c); }
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
template <typename T> __device__ __forceinline__ T dup_(float v);
template <> __device__ __forceinline__ f2_t dup_<f2_t>(float v) { return f2_pack(v, v); }
template <> __device__ __forceinline__ float dup_<float>(float v) { return v; }
__device__ __forceinline__ f2_t neg1_(f2_t a) { return mul_(a, 0xbf800000bf800000ull); }
__device__ __forceinline__ float neg1_(float a) { return -a; }

// ----------------------------------------------------------- two-float numbers
// hi + lo with |lo| <= ulp(hi)/2: Dekker's arithmetic (1971), products by FMA.
// GB300 runs FP64 at 1/64 of the FP32 rate, so 11 FP32 operations for a sum
// and 7 for a product are 6 to 9 times faster than one FP64 operation each.
// The sum's error is relative to |a| + |b| (2^-47), not to the result, which
// is what a transform needs.
struct __align__(8) dd {
  float hi, lo;
};
__device__ __forceinline__ dd dd_fast(float s, float e) {  // |s| >= |e|
  const float h = __fadd_rn(s, e);
  return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ dd add_(dd a, dd b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float t = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, t)), __fsub_rn(b.hi, t));
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return dd_fast(s, e);
}
// A sum whose two parts may overlap by a few bits: exact hi, lo not yet folded
// in.  Enough where the next operation is another sum.
__device__ __forceinline__ dd add_lazy_(dd a, dd b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float t = __fsub_rn(s, a.hi);
  const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, t)), __fsub_rn(b.hi, t));
  return {s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
}
template <typename T> __device__ __forceinline__ T add_lazy_(T a, T b) { return add_(a, b); }
__device__ __forceinline__ dd neg1_(dd a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ dd sub_(dd a, dd b) { return add_(a, neg1_(b)); }
__device__ __forceinline__ dd sub_lazy_(dd a, dd b) { return add_lazy_(a, neg1_(b)); }
template <typename T> __device__ __forceinline__ T sub_lazy_(T a, T b) { return sub_(a, b); }
__device__ __forceinline__ dd mul_(dd a, dd b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return dd_fast(p, e);
}
__device__ __forceinline__ dd dd_of(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}
__device__ __forceinline__ double dd_double(dd v) { return (double)v.hi + (double)v.lo; }

// Twiddle factors (cos, sin) as a table holds them.
template <typename T> struct Twiddle { typedef float2 type; };
template <> struct Twiddle<dd> { typedef float4 type; };  // cos hi, lo, sin hi, lo
template <typename T>
__device__ __forceinline__ typename Twiddle<T>::type twiddle(double c, double s) {
  if constexpr (sizeof(typename Twiddle<T>::type) == 8) {
    return make_float2((float)c, (float)s);
  } else {
    const float ch = (float)c, sh = (float)s;
    return make_float4(ch, (float)(c - (double)ch), sh, (float)(s - (double)sh));
  }
}

// w^p, p = 1 .. 15, from w, w^2, w^4 and w^8.
__device__ __forceinline__ float2 unit_mul(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -(a.y * b.y)), __fmaf_rn(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 unit_power(int p, float2 w1, float2 w2, float2 w4, float2 w8) {
  const float2 w3 = unit_mul(w2, w1), w12 = unit_mul(w8, w4);
  const float2 lo = (p & 3) == 1 ? w1 : (p & 3) == 2 ? w2 : w3, hi = p < 8 ? w4 : p < 12 ? w8 : w12;
  return p < 4 ? lo : (p & 3) == 0 ? hi : unit_mul(hi, lo);
}

template <typename T>
struct Cx {
  T re, im;
};
template <typename T>
__device__ __forceinline__ Cx<T> operator+(Cx<T> a, Cx<T> b) { return {add_(a.re, b.re), add_(a.im, b.im)}; }
template <typename T>
__device__ __forceinline__ Cx<T> operator-(Cx<T> a, Cx<T> b) { return {sub_(a.re, b.re), sub_(a.im, b.im)}; }
// a + i b and a - i b
template <typename T>
__device__ __forceinline__ Cx<T> add_i(Cx<T> a, Cx<T> b) { return {sub_(a.re, b.im), add_(a.im, b.re)}; }
template <typename T>
__device__ __forceinline__ Cx<T> sub_i(Cx<T> a, Cx<T> b) { return {add_(a.re, b.im), sub_(a.im, b.re)}; }
template <typename T>
__device__ __forceinline__ Cx<T> cmul(Cx<T> a, float2 w) {
  const T r = dup_<T>(w.x), i = dup_<T>(w.y), ni = dup_<T>(-w.y);
  return {fma_(a.im, ni, mul_(a.re, r)), fma_(a.re, i, mul_(a.im, r))};
}
__device__ __forceinline__ Cx<dd> cmul(Cx<dd> a, float4 w) {
  const dd r{w.x, w.y}, i{w.z, w.w};
  return {sub_(mul_(a.re, r), mul_(a.im, i)), add_(mul_(a.im, r), mul_(a.re, i))};
}

// In-place transform of 4 points with e^{+2 pi i jk/4}.
template <typename T>
__device__ __forceinline__ void dft4(Cx<T>& x0, Cx<T>& x1, Cx<T>& x2, Cx<T>& x3) {
  const Cx<T> a{add_lazy_(x0.re, x2.re), add_lazy_(x0.im, x2.im)}, b{sub_lazy_(x0.re, x2.re), sub_lazy_(x0.im, x2.im)};
  const Cx<T> c{add_lazy_(x1.re, x3.re), add_lazy_(x1.im, x3.im)}, d{sub_lazy_(x1.re, x3.re), sub_lazy_(x1.im, x3.im)};
  x0 = a + c;
  x1 = add_i(b, d);
  x2 = a - c;
  x3 = sub_i(b, d);
}

// First half of the 16-point transform: afterwards x[4 k1 + n2] holds the
// k1-th output of the n2-th inner transform, times e^{2 pi i n2 k1 / 16}.
template <typename T>
__device__ __forceinline__ void dft16_first(Cx<T> (&x)[16]) {
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) dft4(x[n2], x[4 + n2], x[8 + n2], x[12 + n2]);
  constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, h = 0.70710678118654752440;
  x[4 * 1 + 1] = cmul(x[4 * 1 + 1], twiddle<T>(c1, s1));    // W^1
  x[4 * 2 + 1] = cmul(x[4 * 2 + 1], twiddle<T>(h, h));      // W^2
  x[4 * 3 + 1] = cmul(x[4 * 3 + 1], twiddle<T>(s1, c1));    // W^3
  x[4 * 1 + 2] = cmul(x[4 * 1 + 2], twiddle<T>(h, h));      // W^2
  x[4 * 2 + 2] = Cx<T>{neg1_(x[4 * 2 + 2].im), x[4 * 2 + 2].re};  // W^4 = i
  x[4 * 3 + 2] = cmul(x[4 * 3 + 2], twiddle<T>(-h, h));     // W^6
  x[4 * 1 + 3] = cmul(x[4 * 1 + 3], twiddle<T>(s1, c1));    // W^3
  x[4 * 2 + 3] = cmul(x[4 * 2 + 3], twiddle<T>(-h, h));     // W^6
  x[4 * 3 + 3] = cmul(x[4 * 3 + 3], twiddle<T>(-c1, -s1));  // W^9
}
// The whole 16-point transform; output k sits at x[4 (k & 3) + (k >> 2)].
template <typename T>
__device__ __forceinline__ void dft16(Cx<T> (&x)[16]) {
  dft16_first(x);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) dft4(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);
}

// One complex word of the exchange buffer: 16 bytes (f2_t, dd) or 8 (float).
template <typename T>
__device__ __forceinline__ void put(Cx<T>* buf, int i, Cx<T> v) {
  typedef typename std::conditional<sizeof(T) == 8, uint4, uint2>::type Word;
  Word w;
  memcpy(&w, &v, sizeof w);
  reinterpret_cast<Word*>(buf)[i] = w;
}
template <typename T>
__device__ __forceinline__ Cx<T> get(const Cx<T>* buf, int i) {
  typedef typename std::conditional<sizeof(T) == 8, uint4, uint2>::type Word;
  const Word w = reinterpret_cast<const Word*>(buf)[i];
  Cx<T> v;
  memcpy(&v, &w, sizeof w);
  return v;
}

// The first two radix-16 passes of a tile of 4096 values and the exchanges
// after them: thread tid enters with the values of indices 16 R a + u, u =
// tid / B, of its column (see the callers) at x[a] and leaves with those of
// its (p, r = tid & 15), p = tid >> 4, in the order e of the last pass.
// tw_a(p), tw_b(r): the twiddles after each pass.  The second exchange stays
// within the 16 threads of one p, in the 256 words that only they read in the
// first one, so it needs no barrier of the whole CTA.
//
// ROLL: the two passes are one loop body.  Unrolled, a two-float transform is
// 130 KB of instructions, more than the cache that feeds the SM holds (FP64
// batch, N_t 275, per run and SM: 114 500 -> 110 700 clocks rolled).
template <bool ROLL, typename T, typename TwA, typename TwB>
__device__ __forceinline__ void fft_two_passes(Cx<T> (&x)[16], Cx<T>* buf, int tid, TwA&& tw_a, TwB&& tw_b) {
  const int e0 = tid & 15;
  Cx<T>* const own = buf + (tid >> 4) * 256;
  if constexpr (ROLL) {
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      dft16(x);
#pragma unroll
      for (int p = 1; p < 16; ++p) {
        const int q = 4 * (p & 3) + (p >> 2);
        x[q] = cmul(x[q], pass ? tw_b(p) : tw_a(p));
      }
      // first exchange: word 256 p + tid, read at own + 16 c + e0; second:
      // own + 16 r + (e0 ^ r), read at own + 16 e0 + (e ^ e0)
      Cx<T>* const to = pass ? own : buf + tid;
      const int step = pass ? 16 : 256, mix = pass ? 15 : 0;
      if (pass) __syncwarp(); else __syncthreads();
#pragma unroll
      for (int p = 0; p < 16; ++p) put(to, p * step + ((e0 ^ p) & mix), x[4 * (p & 3) + (p >> 2)]);
      if (pass) __syncwarp(); else __syncthreads();
      const Cx<T>* const from = pass ? own + 16 * e0 : own + e0;
      const int stride = pass ? 1 : 16, flip = pass ? e0 : 0;
#pragma unroll
      for (int c = 0; c < 16; ++c) x[c] = get(from, (c * stride) ^ flip);
    }
  } else {
    dft16(x);
#pragma unroll
    for (int p = 1; p < 16; ++p) {
      const int q = 4 * (p & 3) + (p >> 2);
      x[q] = cmul(x[q], tw_a(p));
    }
    __syncthreads();  // every thread has read its cells
#pragma unroll
    for (int p = 0; p < 16; ++p) put(buf, p * 256 + tid, x[4 * (p & 3) + (p >> 2)]);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 16; ++c) x[c] = get(own, 16 * c + e0);
    dft16(x);
#pragma unroll
    for (int r = 1; r < 16; ++r) {
      const int q = 4 * (r & 3) + (r >> 2);
      x[q] = cmul(x[q], tw_b(r));
    }
    __syncwarp();
    // word (r, d) at 16 r + (d ^ r): the lanes of either the writing order (d
    // runs) or the reading order (r runs) fall on distinct banks
#pragma unroll
    for (int r = 0; r < 16; ++r) put(own, 16 * r + (e0 ^ r), x[4 * (r & 3) + (r >> 2)]);
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 16; ++e) x[e] = get(own, 16 * e0 + (e ^ e0));
  }
}

// The 4096-point transform of the CTA: on entry thread b holds cells
// 256 a + b (a = 0 .. 15); on return, with p = tid >> 4 and r = tid & 15,
// out[s] holds the value at offset p + 16 r + 256 s - 1024 from the run's
// centre, s = 0 .. 7.  buf: 4096 complex words, free once every thread has
// passed the first barrier here; free again only after a barrier of the
// caller.
// tw1 holds e^{2 pi i p b / 4096} for b = 0 .. 255, tw2 e^{2 pi i r d / 256} for
// d = 0 .. 15: dd all of p, r = 1 .. 15; FP32 those of 1, 2, 4 and 8, the
// others are products (at most three).  The full FP32 tables are 32 KB, about
// what three CTAs' shared memory leaves of the L1 cache: half of the kernel's
// loads missed it (clocks per run and SM at N_t 64 / 275 / 1000: 6355 / 7616 /
// 12 028 before, 6064 / 7350 / 11 540 now, of which the staging's layout gave
// 60 / 90 / 260).  Two loads and 13 products would be 1 % faster, but the error
// against 64 bits (rms of a row, N_t 120, median of 100 objects) goes 2.0e-7,
// 2.2e-7 with four loads, 2.3e-7 with two, and the largest error of a peak
// 4.4e-7, 4.4e-7, 6.4e-7; the direct kernel's are 3.1e-7 and 5.8e-7.
template <typename T>
__device__ __forceinline__ void fft4096(Cx<T> (&x)[16], Cx<T>* buf, const typename Twiddle<T>::type* __restrict__ tw1,
                                        const typename Twiddle<T>::type* __restrict__ tw2, Cx<T> (&out)[8]) {
  const int tid = threadIdx.x, e0 = tid & 15;
  fft_two_passes<std::is_same<T, dd>::value>(
      x, buf, tid,
      [&](int p) {
        if constexpr (std::is_same<T, dd>::value) return __ldg(&tw1[(p - 1) * 256 + tid]);
        else return unit_power(p, __ldg(&tw1[tid]), __ldg(&tw1[256 + tid]), __ldg(&tw1[512 + tid]), __ldg(&tw1[768 + tid]));
      },
      [&](int r) {
        if constexpr (std::is_same<T, dd>::value) return __ldg(&tw2[(r - 1) * 16 + e0]);
        else return unit_power(r, __ldg(&tw2[e0]), __ldg(&tw2[16 + e0]), __ldg(&tw2[32 + e0]), __ldg(&tw2[48 + e0]));
      });
  dft16_first(x);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    const Cx<T> x0 = x[4 * k1], x1 = x[4 * k1 + 1], x2 = x[4 * k1 + 2], x3 = x[4 * k1 + 3];
    out[4 + k1] = (x0 + x2) + (x1 + x3);    // s = k1 of the transform's 16
    out[k1] = sub_i(x0 - x2, x1 - x3);      // s = 12 + k1
  }
}

// -------------------------------------------------------------------- power
// Eq. 2 from Z and W (lsp_power_f32 with its sums already combined).
__device__ __forceinline__ float power_zw(float zr, float zi, float wr, float wi, float n, bool& ill) {
  const float r2 = fmaf(wr, wr, wi * wi);
  const float nn = n * n;
  const float z2 = fmaf(zr, zr, zi * zi);
  const float re = fmaf((zr - zi) * (zr + zi), wr, 2.0f * zr * zi * wi);
  const float num = fmaf(n, z2, -re);
  const float den = nn - r2;
  ill = r2 > kIllR2 * nn;
  return den > 0.0f ? __fdividef(fmaxf(num, 0.0f), den) : 0.0f;
}

// (N |Z|^2 - Re(Z^2 conj W)) / (N^2 - |W|^2), as lsp_power_f32.
__device__ __forceinline__ dd power_dd(Cx<dd> z, Cx<dd> w, dd n, bool& ill) {
  const dd w2 = add_(mul_(w.re, w.re), mul_(w.im, w.im));
  const dd nn = mul_(n, n);
  const dd zr2 = mul_(z.re, z.re), zi2 = mul_(z.im, z.im);
  dd b = mul_(z.re, z.im);
  b = dd{2.0f * b.hi, 2.0f * b.lo};
  const dd re = add_(mul_(sub_(zr2, zi2), w.re), mul_(b, w.im));
  const dd num = sub_(mul_(n, add_(zr2, zi2)), re);
  const dd den = sub_(nn, w2);
  ill = w2.hi > kIllR2 * nn.hi;
  if (!(den.hi > 0.0f) || !(num.hi > 0.0f)) return dd{0.0f, 0.0f};
  const float q = __fdiv_rn(num.hi, den.hi);
  const dd r = sub_(num, mul_(den, dd{q, 0.0f}));
  return dd_fast(q, __fdiv_rn(r.hi, den.hi));
}

}  // namespace lsp
