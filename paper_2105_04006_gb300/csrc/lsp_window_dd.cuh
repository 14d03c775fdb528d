// lsp_window_dd.cuh -- the 16-cell window in two-float numbers (internal;
// included inside the translation unit's unnamed namespace, after the tables).
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
