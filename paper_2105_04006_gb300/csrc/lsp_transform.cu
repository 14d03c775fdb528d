// lsp_transform.cu -- the trig sums of a run of bins by a nonuniform FFT
// (FP32 paths).
//
// What it computes: for an object and a run of 2048 consecutive grid bins
// k = kc + m, m = -1024 .. 1023, the two sums Eq. 2 needs (see lsp_power),
//   Z_k = sum_j y_j e^{i phi_jk},  W_k = sum_j e^{2 i phi_jk},
//   phi_jk = 2 pi (a_j + k b_j) cycles as in the records,
// (generalized periodogram: sums weighted by u_j and w_j, and W_k by w_j),
// the power of every bin and the run's maxima.
//
// Why: evaluated pair by pair (lsp_main_impl.cuh) every (observation, bin)
// costs 8 FP32 operations, and that kernel already issues them at 0.9 of the
// pipe's rate.  Over a run of evenly spaced bins the same sums are a Fourier
// transform of the observations taken at uneven places b_j: spread each one
// over the 8 nearest cells of a periodic grid of 4096 cells with a
// Kaiser-Bessel window, transform the grid, divide by the window's own
// transform.  A bin then costs about 200 operations plus 0.1 per observation
// instead of 8 per observation.
//
// Measured (GB300): 10 000 survey light curves (N_t 50 .. 500) on 1e5 bins
// 11.8 ms against 64.7 ms with the direct kernel, 1e5 observations on 1e6
// bins 1.48 ms against 23.4 ms.  A run of 2048 bins takes an SM 6060 clocks at
// N_t 64, 7350 at 275, 11540 at 1000 (top-3 8 % more, generalized 1.6 times);
// what bounds it is the L1 data pipe (71 % busy: the FFT's exchanges, the
// spread's atomics), with issue at 60 % and the FMA pipe at 52 %.
//
// Accuracy: the window's aliasing is at most 1.6e-7 (5e-8 rms) of the largest
// amplitude near the run, the FP32 transform adds about as much; the cells'
// rounding adds about 2.4 sqrt(N_t) 2^-30 of the largest sum of |weights| over 16
// neighbouring cells (1e-7 at N_t 4096 if all lie there, 2e-6 at 1e6).  The
// direct kernel's largest error of a power was the larger in emulations of N_t
// 300 .. 1e6 over years, a month or one night with equal or lognormal error
// bars, but for rows whose errors are below 1e-7 on both sides (its SFU seeds are
// good to 2^-21.4, its FP32 sums to about 4e-8 sqrt(N_t)).
// Phases are the records' 64-bit fixed-point ones.
//
// How:
//   - one CTA of 256 threads per (object, run), persistent, from a queue;
//   - the grid is accumulated in 32-bit fixed point with shared-memory
//     integer atomics: integer addition is associative, so the result does
//     not depend on the order of the adds (bit-identical repeats), any time
//     order and any clustering of the observations run at the same speed,
//     and 8 lanes per observation hit 8 consecutive banks.  The scale is the
//     largest one that cannot overflow: |weights| are summed per 8 cells
//     first, and an observation's window covers at most two neighbouring
//     groups (TfCounter);
//   - lane r of an octet always adds the r-th cell, so the window polynomial
//     of its cell stays in 9 registers;
//   - 4096 = 16^3: three register passes of 16 points per thread with two
//     exchanges through the (then free) grid memory; Z and W ride in the two
//     halves of packed f32x2 registers and share every twiddle; the last pass
//     computes only the 8 of 16 outputs that lie inside the run.
#include <type_traits>

#include "../../include/lsp.h"
#include "lsp_fft.cuh"
#include "lsp_launch.h"
#include "lsp_peak.cuh"

namespace lsp {

namespace {

#define LSP_TF_TABLES_F32
#include "lsp_transform_tables.inc"

constexpr int kM = 4096;                 // grid cells
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
// A word of padding per 8 powers: the lanes fall on distinct banks both in the
// transform's order (18 apart) and in runs of eight (9 apart).  Together with
// the staged words in rows of 32: 11 733 -> 11 470 clocks a run at N_t 1000.
constexpr size_t kPowers = kTfBins + kTfBins / 8;
static_assert(kTfBins == kM / 2 && kTfBins == kThreads * 8 && kTfGroups == kM / 8, "run length");

// Objects of many observations add their window values with an offset in
// (-1/2, 1/2) before the rounding, different for every value and set by its
// index alone.  A unit of a cell is up to N 2^-30 of one observation's weight:
// rounded to nearest, the window's tails lose up to half a unit each, in the
// same direction where the observations share few cells, and the error of a
// sum grows like N / 2^30 of it; with the offsets the errors cancel and it
// grows like sqrt(N).  Emulated, 1e6 observations in a month: error of a power
// 3.8e-5 without, 1.7e-6 with the offsets (direct kernel 1.2e-5; generalized,
// lognormal errors: 8.4e-5, 1.6e-6, 2.3e-3).  At 4096 the two are level.
constexpr int kTfOffsets = 4096;
__device__ __forceinline__ uint32_t scramble(uint32_t x) {
  x *= 0x9e3779b1u;  // 2^32 / golden ratio
  x ^= x >> 16;
  x *= 0x9e3779b1u;
  return x ^ (x >> 15);
}
__device__ __forceinline__ void rounding_offsets(uint32_t i, float (&d)[6]) {
  const uint32_t x = scramble(i), z = scramble(x + 1u);
  auto byte = [](uint32_t v) { return __uint_as_float(0x3f800000u | (v & 0xffu) << 15) - 1.498046875f; };
  d[0] = byte(x);
  d[1] = byte(x >> 8);
  d[2] = byte(x >> 16);
  d[3] = byte(x >> 24);
  d[4] = byte(z);
  d[5] = byte(z >> 8);
}

__device__ __forceinline__ f2_t cells_f2(const int32_t* a, const int32_t* b, int i) {
  return f2_pack(__int2float_rn(a[i]), __int2float_rn(b[i]));
}

// Shared memory: grid planes (the exchange buffer after the grid is read),
// staged observations (group sums before, the run's powers after them).
template <bool GLS>
struct Smem {
  static constexpr int kPlanes = GLS ? 6 : 4;
  static constexpr int kStage = GLS ? 48 : 32;  // bytes per staged observation
  static constexpr size_t grid = (size_t)kPlanes * kM * 4;
  static constexpr size_t stage = (size_t)kThreads * kStage > kPowers * 4 ? (size_t)kThreads * kStage : kPowers * 4;
  static constexpr size_t total = grid + stage;
  static_assert(stage >= TfCounter<GLS>::kWords * 4, "the group sums use the staging area");
};

template <bool GLS>
__global__ void __launch_bounds__(kThreads, GLS ? 2 : 3) transform_kernel(TransformParams p) {
  using S = Smem<GLS>;
  constexpr int kW = GLS ? 4 : 2;  // grid planes: Z (re, im), with errors C, then W
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  int32_t* const plane = reinterpret_cast<int32_t*>(dyn_smem);
  unsigned char* const stage = dyn_smem + S::grid;
  __shared__ unsigned long long red[32];
  __shared__ float s_edge[4 * kWarps + 2];
  __shared__ uint32_t s_max[4][kWarps];
  __shared__ uint32_t s_item;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n_items = p.n_items_dev ? *p.n_items_dev : p.n_items;
  const uint32_t n_chunks = (uint32_t)p.n_chunks;
  auto clear_grid = [&]() {
    int4* g4 = reinterpret_cast<int4*>(plane);
#pragma unroll
    for (int i = 0; i < S::kPlanes * kM / 4 / kThreads; ++i) g4[tid + i * kThreads] = make_int4(0, 0, 0, 0);
  };
  clear_grid();

  uint32_t ticket = blockIdx.x;  // first item static, then one ticket ahead (as in main_f32_packed_body)
  for (;;) {
    if (tid == 0) s_item = ticket;
    __syncthreads();  // also: the grid is clear
    const uint32_t item = s_item;
    if (item >= n_items) break;
    if (tid == 0) ticket = gridDim.x + atomicAdd(p.queue, 1u);
    const uint32_t chunk = item % n_chunks;
    const uint32_t orank = item / n_chunks;
    const int64_t o = p.order_back ? (int64_t)p.order_back[-(int64_t)orank]
                                   : p.order ? (int64_t)p.order[orank] : (int64_t)orank;
    const ObjInfo oi = p.obj[o];
    // bins of this item lie in [kc0, kend): the run inside the grid, or the object's window
    const int64_t kc0 = p.win_start ? (int64_t)p.win_start[o] : (int64_t)chunk * kTfBins;
    const int64_t kend = p.win_start && kc0 + p.win_len < p.n_f ? kc0 + p.win_len : p.n_f;
    const uint32_t kc = (uint32_t)kc0 + kTfBins / 2;
    const int n = oi.flags ? 0 : oi.n;  // flagged objects: zero power
    const uint4* rec = reinterpret_cast<const uint4*>(p.rec + oi.begin);

    // ---- fixed-point scales: the records kernel's, or counted here
    TfScale sc;
    if (p.have_scale) {
      sc = tf_scale_of(oi);
    } else {
      uint32_t* const count = reinterpret_cast<uint32_t*>(stage);
      for (int i = tid; i < TfCounter<GLS>::kWords; i += kThreads) count[i] = 0u;
      __syncthreads();
      TfCounter<GLS> counter(count, oi);
      for (uint32_t j = tid; j < (uint32_t)n; j += kThreads) {
        const uint4 r0 = __ldg(rec + 2 * (size_t)j), r1 = __ldg(rec + 2 * (size_t)j + 1);
        counter.add(__uint_as_float(r0.x), __uint_as_float(r1.w), r1.x, r1.y);
      }
      __syncthreads();
      sc = counter.template scale<kWarps>(s_max);  // its barrier ends the use of the sums
    }
    const float y_sc = sc.y, w_sc = sc.w, c_sc = sc.c;

    // ---- spread: each warp takes an eighth of the observations, 32 at a
    // time: a lane each for the phase, then an octet of lanes each for the 8
    // cells
    {
      // window coefficients of this lane's cell (not kept across the transform:
      // their 18 registers are what lets three CTAs share an SM)
      f2_t poly[9];
#pragma unroll
      for (int d = 0; d < 9; ++d) poly[d] = dup_<f2_t>(__ldg(&kTfPoly[d * 8 + (lane & 7)]));
      const uint32_t j1 = (uint32_t)((int64_t)n * (warp + 1) / kWarps);
      unsigned char* const mine = stage + (size_t)warp * 32 * S::kStage;
      auto spread = [&](auto offsets) {
        for (uint32_t jb = (uint32_t)((int64_t)n * warp / kWarps); jb < j1; jb += 32) {
          const uint32_t j = jb + lane;
          if (j < j1) {
            const uint4 r0 = __ldg(rec + 2 * (size_t)j), r1 = __ldg(rec + 2 * (size_t)j + 1);
            const uint32_t ph = phase_hi32(r0.w, r1.x, r1.y, kc);
            float s, c;
            sincospif(__int2float_rn((int)ph) * 4.656612873077393e-10f, &s, &c);  // 2^-31 half-cycles
            const float ys = __uint_as_float(r0.x) * y_sc;
            const float ws = GLS ? __uint_as_float(r1.w) * w_sc : w_sc;
            // position in cells, 12 bits of cell and 32 of fraction
            const uint32_t fz = (r1.x << 12) | (r1.y >> 20), b2 = (r1.x << 1) | (r1.y >> 31), lo2 = r1.y << 1;
            const uint32_t fw = (b2 << 12) | (lo2 >> 20);
            const float uz = fmaf(__uint2float_rn(fz), 2.3283064365386963e-10f, -0.5f);
            const float uw = fmaf(__uint2float_rn(fw), 2.3283064365386963e-10f, -0.5f);
            float4* st = reinterpret_cast<float4*>(mine) + lane;  // word w of an observation at 32 w: no bank twice
            st[0] = make_float4(uz, uw, __uint_as_float((r1.x >> 20) - 3u), __uint_as_float((b2 >> 20) - 3u));
            st[32] = make_float4(ys * c, ys * s, ws * (c - s) * (c + s), ws * 2.0f * c * s);
            if (GLS) {
              const float cs = __uint_as_float(r1.w) * c_sc;
              st[64] = make_float4(cs * c, cs * s, 0.0f, 0.0f);
            }
          }
          __syncwarp();
          const int nt = (int)min(32u, j1 - jb);
#pragma unroll 2
          for (int i = lane >> 3; i < nt; i += 4) {
            const float4* st = reinterpret_cast<const float4*>(mine) + i;
            const float4 at = st[0], v = st[32];
            const f2_t u = f2_pack(at.x, at.y);
            f2_t w2 = poly[8];
#pragma unroll
            for (int d = 7; d >= 0; --d) w2 = f2_fma(w2, u, poly[d]);
            float wz, ww;
            f2_unpack(w2, wz, ww);
            const int lz = (int)(__float_as_uint(at.z) + (uint32_t)(lane & 7)) & (kM - 1);
            const int lw = (int)(__float_as_uint(at.w) + (uint32_t)(lane & 7)) & (kM - 1);
            float d[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            if constexpr (decltype(offsets)::value) rounding_offsets(8u * (jb + i) + (lane & 7), d);
            atomicAdd(&plane[0 * kM + lz], __float2int_rn(fmaf(wz, v.x, d[0])));
            atomicAdd(&plane[1 * kM + lz], __float2int_rn(fmaf(wz, v.y, d[1])));
            atomicAdd(&plane[kW * kM + lw], __float2int_rn(fmaf(ww, v.z, d[2])));
            atomicAdd(&plane[(kW + 1) * kM + lw], __float2int_rn(fmaf(ww, v.w, d[3])));
            if (GLS) {
              const float4 q = st[64];
              atomicAdd(&plane[2 * kM + lz], __float2int_rn(fmaf(wz, q.x, d[4])));
              atomicAdd(&plane[3 * kM + lz], __float2int_rn(fmaf(wz, q.y, d[5])));
            }
          }
          __syncwarp();
        }
      };
      if (n < kTfOffsets) spread(std::false_type{});  // two loops: the test inside one took 0.5 % of a batch's time
      else spread(std::true_type{});
    }
    __syncthreads();

    // ---- transform, power
    float* const pw = reinterpret_cast<float*>(stage);
    const float scale = oi.norm_scale_f;
    if constexpr (!GLS) {
      Cx<f2_t> x[16], out[8];
#pragma unroll
      for (int a = 0; a < 16; ++a) {
        const int i = 256 * a + tid;
        x[a] = Cx<f2_t>{cells_f2(plane, plane + 2 * kM, i), cells_f2(plane + kM, plane + 3 * kM, i)};
      }
      fft4096(x, reinterpret_cast<Cx<f2_t>*>(plane), kTfTw1, kTfTw2, out);
      const f2_t inv = f2_pack(1.0f / y_sc, 1.0f / w_sc);
      const float nf = (float)oi.n;
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const int i = (tid >> 4) + (tid >> 7) + 18 * (tid & 15) + 288 * s;  // bin b = p + 16 r + 256 s at b + b / 8
        const float dc = __ldg(&kTfDeconv[256 * s + tid]);
        const f2_t f = f2_mul(inv, f2_pack(dc, dc));
        float zr, wr, zi, wi;
        f2_unpack(f2_mul(out[s].re, f), zr, wr);
        f2_unpack(f2_mul(out[s].im, f), zi, wi);
        bool ill;
        const float v = scale * power_zw(zr, zi, wr, wi, nf, ill);
        pw[i] = ill ? -1.0f : v;  // powers are >= 0: marks the bin for FP64
      }
    } else {
      // (Y, C) in packed halves through the first four planes' memory, then W
      // alone, whose planes lie past it
      Cx<f2_t> out[8];
      Cx<float> outw[8];
      {
        Cx<f2_t> x[16];
#pragma unroll
        for (int a = 0; a < 16; ++a) {
          const int i = 256 * a + tid;
          x[a] = Cx<f2_t>{cells_f2(plane, plane + 2 * kM, i), cells_f2(plane + kM, plane + 3 * kM, i)};
        }
        fft4096(x, reinterpret_cast<Cx<f2_t>*>(plane), kTfTw1, kTfTw2, out);
      }
      {
        Cx<float> x[16];
#pragma unroll
        for (int a = 0; a < 16; ++a) {
          const int i = kW * kM + 256 * a + tid;
          x[a] = Cx<float>{__int2float_rn(plane[i]), __int2float_rn(plane[kM + i])};
        }
        fft4096(x, reinterpret_cast<Cx<float>*>(plane), kTfTw1, kTfTw2, outw);
      }
      const f2_t inv = f2_pack(1.0f / y_sc, 1.0f / c_sc);
      const float inv_w = 1.0f / w_sc, wsum = oi.wsum_f, yy = (float)oi.sum_y2;
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const int i = (tid >> 4) + (tid >> 7) + 18 * (tid & 15) + 288 * s;  // bin b = p + 16 r + 256 s at b + b / 8
        const float dc = __ldg(&kTfDeconv[256 * s + tid]);
        const f2_t f = f2_mul(inv, f2_pack(dc, dc));
        float yr, cr, yi, ci;
        f2_unpack(f2_mul(out[s].re, f), yr, cr);
        f2_unpack(f2_mul(out[s].im, f), yi, ci);
        const float wr = outw[s].re * (inv_w * dc), wi = outw[s].im * (inv_w * dc);
        bool ill;
        const float v = scale * gls_power<float>(yr, yi, cr, ci, 0.5f * (wsum + wr), 0.5f * wi, wsum, yy,
                                                 EpsRel<float>::v, ill);
        pw[i] = ill ? -1.0f : v;
      }
    }
    __syncthreads();

    // ---- eight consecutive bins per thread from here on
    float pv[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) pv[m] = pw[9 * tid + m];
    clear_grid();  // for the next item: every thread is past the transform
    const uint32_t k0 = (uint32_t)kc0 + 8u * (uint32_t)tid;
    uint32_t bad = 0u;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      if (pv[m] < 0.0f && (int64_t)k0 + m < kend) bad |= 1u << m;
      if (oi.flags) pv[m] = 0.0f;
    }
    if (oi.flags) bad = 0u;
    if constexpr (GLS)
      fix_ill_conditioned_gls<8>(pv, bad, k0, p.rec, oi);
    else
      fix_ill_conditioned<8>(pv, bad, k0, p.rec, oi.begin, oi.n, oi.norm_scale);
    if (p.power_out) store_row<8>(p.power_out + o * p.n_f, (int64_t)k0, pv, kend);
    const int64_t res = o * (int64_t)n_chunks + chunk;
    chunk_results_f32<8>(pv, k0, kc0, kend, p.best + res, p.cand ? p.cand + res : nullptr, s_edge, red);
  }

  // ---- one object, first maximum: the last CTA to finish writes the peak
  if (!p.peaks) return;
  __shared__ bool s_last;
  if (tid == 0) {  // thread 0 wrote this CTA's run results
    __threadfence();
    s_last = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last || warp != 0) return;
  __threadfence();
  double bp = 0.0;
  int64_t bk = -1;
  for (uint32_t c = lane; c < n_items; c += 32) {
    const double q = __ldcg(&p.best[c].p);
    const int64_t k = __ldcg(&p.best[c].k);
    if (better(q, k, bp, bk)) {
      bp = q;
      bk = k;
    }
  }
  warp_best(bp, bk);
  if (lane == 0) p.peaks[0] = make_peak(bk, bp, p.f_min, p.df, p.obj[0].flags);
}

}  // namespace

int transform_blocks_per_sm64();

int transform_blocks_per_sm(int prec, int gls) {
  if (prec) return gls ? 0 : transform_blocks_per_sm64();
  return gls ? blocks_per_sm(transform_kernel<true>, kThreads, Smem<true>::total)
             : blocks_per_sm(transform_kernel<false>, kThreads, Smem<false>::total);
}

cudaError_t launch_transform(const TransformParams& p, int gls, int grid, cudaStream_t stream) {
  auto go = [&](auto kern, size_t dyn) {
    cudaError_t e = allow_dyn_smem(kern, dyn);
    if (e != cudaSuccess) return e;
    kern<<<grid, kThreads, dyn, stream>>>(p);
    return cudaGetLastError();
  };
  return gls ? go(transform_kernel<true>, Smem<true>::total) : go(transform_kernel<false>, Smem<false>::total);
}

}  // namespace lsp
