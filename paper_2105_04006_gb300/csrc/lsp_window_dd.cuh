// lsp_window_dd.cuh -- 64-bit fixed-point grid cells and the 16-cell window in
// two-float numbers (internal; included inside the translation unit's unnamed
// namespace, after the tables).
// Window value of cell r - 7 for an observation at (sub, v).
__device__ __forceinline__ dd window(uint32_t sub, dd v, int r) {
  const float2* c = kTfPolyD + (6 * sub) * 16 + r;
  const float2 c0 = __ldg(c), c1 = __ldg(c + 16), c2 = __ldg(c + 32), c3 = __ldg(c + 48);
  const float c4 = __ldg(&c[64].x), c5 = __ldg(&c[80].x);
  dd q = add_(dd{c3.x, c3.y}, dd{fmaf(c5, v.hi, c4) * v.hi, 0.0f});
  q = add_(mul_(q, v), dd{c2.x, c2.y});
  q = add_(mul_(q, v), dd{c1.x, c1.y});
  return add_(mul_(q, v), dd{c0.x, c0.y});
}

// Magnitudes are scaled by 2^-e, sum y^2 <= 2^2e: then a cell of Z is at most
// sum |y| <= sqrt(N) <= 2^((count_bits + 1) / 2) and one of W at most N.
__device__ __forceinline__ int y_exponent(double sum_y2) {
  return (((int)(__double_as_longlong(sum_y2) >> 52) & 0x7ff) - 1023) / 2 + 1;
}
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }
__device__ __forceinline__ int count_bits(int n) { return 32 - __clz(n); }  // n < 2^count_bits
__device__ __forceinline__ int z_bits(int n) { return 61 - (count_bits(n) + 1) / 2; }  // cells are in units of 2^-bits
__device__ __forceinline__ int w_bits(int n) { return 61 - count_bits(n); }

__device__ __forceinline__ void add_cell(long long* cell, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long*>(cell), (unsigned long long)v);
}

// Conversions between floats and the 64-bit cells by 32-bit ones: the 64-bit
// conversions run at the FP64 pipe's rate.
//
// A float below 2^61 as an integer, rounded: its part above 2^30 is exact.
__device__ __forceinline__ long long fixed_of(float v) {
  const float top = rintf(v * 9.313225746154785e-10f);  // 2^-30
  return ((long long)__float2int_rn(top) << 30) + __float2int_rn(fmaf(top, -1073741824.0f, v));
}
// A two-float number times 2^s (below 2^61).
__device__ __forceinline__ long long fixed_of(dd v, float two_s) {
  return fixed_of(v.hi * two_s) + fixed_of(v.lo * two_s);
}
// A cell as a two-float number.  Upper word: rounded and remainder (zero below
// 2^24); lower word: its upper 24 bits and the other 8, each exact (taken as
// one float its 8 dropped bits left a cell of few upper bits with 37 in all:
// 6e-13 instead of 7e-15 at N_t 5e4).
__device__ __forceinline__ dd dd_of_int(long long v) {
  const int h = (int)(v >> 32);
  const uint32_t low = (uint32_t)v;
  const float hf = __int2float_rn(h), rest = __int2float_rn(h - __float2int_rn(hf));
  const float s = hf * 4294967296.0f, l = __uint2float_rn(low >> 8) * 256.0f;
  const float t = __fadd_rn(s, l), u = __fsub_rn(t, s);
  const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, u)), __fsub_rn(l, u));
  return {t, __fadd_rn(e, fmaf(rest, 4294967296.0f, __uint2float_rn(low & 255u)))};
}
// ... and as a float.
__device__ __forceinline__ float float_of_int(long long v) {
  return fmaf(__int2float_rn((int)(v >> 32)), 4294967296.0f, __uint2float_rn((uint32_t)v));
}

// What an observation adds to the two grids of 2^lg cells: amplitudes times
// e^{i phase} (Z: re, im; W: re, im), first cells, sub-intervals and places.
struct ObsD {
  dd a[4];
  dd v[2];
  uint32_t cell[2], sub[2];
};
__device__ __forceinline__ ObsD obs_of(const RecF64& q, uint64_t kc, int lg, double y_sc) {
  ObsD o;
  double c, s;
  seed_sincos_f64(q.a + kc * q.b, c, s);
  const double ys = q.y * y_sc;
  o.a[0] = dd_of(ys * c);
  o.a[1] = dd_of(ys * s);
  o.a[2] = dd_of((c - s) * (c + s));
  o.a[3] = dd_of(2.0 * c * s);
#pragma unroll
  for (int t = 0; t < 2; ++t) {  // place of Z (b) and W (2 b): cell, 6 bits of sub-interval, 24 + 22 of place
    const uint64_t b = q.b << t, f = b << lg;
    o.cell[t] = (uint32_t)(b >> (64 - lg)) - 7u;
    o.sub[t] = (uint32_t)(f >> 58);
    const float hi = (float)((uint32_t)(f >> 34) & 0xffffffu) * 5.9604644775390625e-8f;   // 2^-24
    const float lo = (float)((uint32_t)(f >> 12) & 0x3fffffu) * 1.4210854715202004e-14f;  // 2^-46
    o.v[t] = dd{hi - 0.5f, lo};
  }
  return o;
}
// Spreads the observations that lanes 0 .. nt - 1 of the warp hold, two at a
// time, 16 lanes each: add(t, cell, re, im) for t = 0 (Z), 1 (W), in units of
// one[t].
template <typename Add>
__device__ __forceinline__ void spread_warp(const ObsD& o, int nt, uint32_t mask, const float (&one)[2], Add&& add) {
  const int lane = threadIdx.x & 31, r = lane & 15;
  auto bcast = [&](dd x, int i) { return dd{__shfl_sync(0xffffffffu, x.hi, i), __shfl_sync(0xffffffffu, x.lo, i)}; };
#pragma unroll 1
  for (int i0 = 0; i0 < nt; i0 += 2) {
    const int i = i0 + (lane >> 4);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const dd w = window(__shfl_sync(0xffffffffu, o.sub[t], i & 31), bcast(o.v[t], i & 31), r);
      const uint32_t l = (__shfl_sync(0xffffffffu, o.cell[t], i & 31) + (uint32_t)r) & mask;
      const dd re = mul_(w, bcast(o.a[2 * t], i & 31)), im = mul_(w, bcast(o.a[2 * t + 1], i & 31));
      if (i < nt) add(t, l, fixed_of(re, one[t]), fixed_of(im, one[t]));
    }
  }
}
