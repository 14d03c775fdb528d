// lsp_transform_f64.cu -- the trig sums of a run of bins by a nonuniform FFT,
// FP64 path (see lsp_transform.cu for the method).
//
// GB300 runs FP64 at 1/64 of the FP32 rate, so a transform in FP64 registers
// would take 160 000 clocks a run on an SM; this kernel computes in two-float
// numbers (dd, lsp_fft.cuh: about 48 bits) on the FP32 pipe instead.
//
// Accuracy: the window spans 16 cells, its aliasing is below 5e-15 and its
// piecewise polynomial below 9e-15 of its peak, two-float sums are good to
// 2^-47; Z and W come out within about 1e-14 of their norm.  Bins whose
// denominator nearly vanishes (N - R < 5 % N) are re-evaluated with FP64
// sums from the exact phases.  Both are below the rounding that the FP64
// pairwise kernel's chains of 16 accumulate.
//
// Measured (GB300): 200 survey light curves (N_t 50 .. 500) on 1e5 bins 3.3 ms
// against 64 ms with the direct kernel; N_t 8 0.64 | 1.34, 12 0.65 | 1.62, 64
// 0.73 | 5.3 ms (60 objects).
//
// Differences from the FP32 kernel:
//   - Z and W one after the other through one grid of two-float cells; Z's
//     outputs wait in shared memory;
//   - cells are floating-point, so the order of the adds matters: tiles of
//     256 observations are sorted by their first cell (rank by counting, ties
//     by index) and every cell gathers its own contributions in that order.
//     Repeats are bit-identical, and clustered observations cost no more than
//     spread-out ones as long as they fill more than a few cells;
//   - window values: 64 sub-intervals per cell, degree 5, the two leading
//     coefficients (below 2^-27) in single floats;
//   - magnitudes are scaled by a power of two (|y|^2 <= sum y^2) into the
//     FP32 exponent range, and back in the power's last FP64 product.
#include <cstring>

#include "../../include/lsp.h"
#include "lsp_fft.cuh"
#include "lsp_launch.h"
#include "lsp_peak.cuh"

namespace lsp {

namespace {

#define LSP_TF_TABLES_F64
#include "lsp_transform_tables.inc"
#include "lsp_window_dd.cuh"

constexpr int kM = 4096;
constexpr int kThreads = 256;
constexpr int kTile = 256;  // observations staged at a time
static_assert(kTfBins == kM / 2 && kTfBins == kThreads * 8, "run length");

struct __align__(16) StagedObs {
  dd re, im;      // amplitude times e^{i phase}
  dd v;           // place inside the sub-interval, -1/2 .. 1/2
  uint32_t sub;   // sub-interval
  int32_t cell;   // first cell of the window
};
static_assert(sizeof(StagedObs) == 32, "two 16-byte words");

constexpr size_t kGridBytes = (size_t)kM * sizeof(Cx<dd>);       // also: powers of the run
constexpr size_t kZBytes = (size_t)kTfBins * sizeof(Cx<dd>);     // Z's outputs
constexpr size_t kStageBytes = (size_t)kTile * sizeof(StagedObs);
constexpr size_t kKeyBytes = (size_t)kTile * 4;                  // sort keys
constexpr size_t kStartBytes = (size_t)(kM / 16) * 4;            // first observation of each 16 cells
constexpr size_t kSmem = kGridBytes + kZBytes + kStageBytes + kKeyBytes + kStartBytes;
static_assert(kM / 16 == kThreads, "one start per thread");

__global__ void __launch_bounds__(kThreads, 2) transform64_kernel(TransformParams64 p) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  Cx<dd>* const grid = reinterpret_cast<Cx<dd>*>(dyn_smem);
  Cx<dd>* const s_z = reinterpret_cast<Cx<dd>*>(dyn_smem + kGridBytes);
  StagedObs* const stage = reinterpret_cast<StagedObs*>(dyn_smem + kGridBytes + kZBytes);
  uint32_t* const s_key = reinterpret_cast<uint32_t*>(dyn_smem + kGridBytes + kZBytes + kStageBytes);
  int32_t* const s_start = reinterpret_cast<int32_t*>(s_key + kTile);
  double* const pw = reinterpret_cast<double*>(dyn_smem);
  __shared__ double red_p[32];
  __shared__ int64_t red_k[32];
  __shared__ uint32_t s_item;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n_items = p.n_items_dev ? *p.n_items_dev : p.n_items;
  const uint32_t n_chunks = (uint32_t)p.n_chunks;

  uint32_t ticket = blockIdx.x;  // first item static, then one ticket ahead (as in main_f32_packed_body)
  for (;;) {
    if (tid == 0) s_item = ticket;
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= n_items) break;
    if (tid == 0) ticket = gridDim.x + atomicAdd(p.queue, 1u);
    const uint32_t chunk = item % n_chunks;
    const uint32_t orank = item / n_chunks;
    const int64_t o = p.order_back ? (int64_t)p.order_back[-(int64_t)orank] : (int64_t)orank;
    const ObjInfo oi = p.obj[o];
    const int64_t kc0 = (int64_t)chunk * kTfBins;
    const uint64_t kc = (uint64_t)kc0 + kTfBins / 2;
    const int n = oi.flags ? 0 : oi.n;  // flagged objects: zero power
    const RecF64* rec = p.rec + oi.begin;
    // 2^-e bounds the magnitudes by 1: |y| <= sqrt(sum y^2) < 2^e
    const int e = (((int)(__double_as_longlong(oi.sum_y2) >> 52) & 0x7ff) - 1023) / 2 + 1;
    const double y_sc = __longlong_as_double((long long)(1023 - e) << 52);

#pragma unroll 1
    for (int tr = 0; tr < 2; ++tr) {  // Z, then W
      {
        uint4* g4 = reinterpret_cast<uint4*>(grid);
#pragma unroll
        for (int i = 0; i < kM / kThreads; ++i) g4[tid + i * kThreads] = make_uint4(0u, 0u, 0u, 0u);
      }
      for (int ts = 0; ts < n; ts += kTile) {
        const int j = ts + tid, nt = min(kTile, n - ts);
        StagedObs st;
        uint32_t key = 0xffffffffu;
        if (j < n) {
          const RecF64 r = rec[j];
          const uint64_t ph = r.a + kc * r.b, b = tr ? r.b << 1 : r.b;
          double c, s;
          seed_sincos_f64(tr ? ph << 1 : ph, c, s);
          if (!tr) {
            const double ys = r.y * y_sc;
            c *= ys;
            s *= ys;
          }
          st.re = dd_of(c);
          st.im = dd_of(s);
          // 12 bits of cell, 6 of sub-interval, 46 of place: 24 and 22 exactly in two floats
          st.cell = (int32_t)(((uint32_t)(b >> 52) - 7u) & (kM - 1));
          st.sub = (uint32_t)(b >> 46) & 63u;
          const float hi = (float)((uint32_t)(b >> 22) & 0xffffffu) * 5.9604644775390625e-8f;  // 2^-24
          const float lo = (float)((uint32_t)b & 0x3fffffu) * 1.4210854715202004e-14f;         // 2^-46
          st.v = dd{hi - 0.5f, lo};
          key = (uint32_t)st.cell << 8 | (uint32_t)tid;
        }
        s_key[tid] = key;
        __syncthreads();  // keys; on the first tile also: the grid is clear
        int rank = 0;
        for (int i = 0; i < (nt + 3) / 4; ++i) {
          const uint4 k = reinterpret_cast<const uint4*>(s_key)[i];
          rank += (int)(k.x < key) + (int)(k.y < key) + (int)(k.z < key) + (int)(k.w < key);
        }
        if (j < n) stage[rank] = st;
        __syncthreads();
        {  // first sorted observation whose cell is at least 16 tid
          int lo = 0, hi = nt;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (stage[mid].cell < 16 * tid) lo = mid + 1;
            else hi = mid;
          }
          s_start[tid] = lo;
        }
        __syncthreads();
#pragma unroll 1
        for (int a = 0; a < kM / kThreads; ++a) {
          const int l = kThreads * a + tid;  // contributions: first cells l - 15 .. l, around the end
          Cx<dd> acc{{0.0f, 0.0f}, {0.0f, 0.0f}};
          bool any = false;
          auto add = [&](int i) {
            const StagedObs q = stage[i];
            const dd w = window(q.sub, q.v, (l - q.cell) & (kM - 1));
            acc = acc + Cx<dd>{mul_(w, q.re), mul_(w, q.im)};
            any = true;
          };
          const int from = l - 15;
          if (from < 0) {
            int i = s_start[(from + kM) >> 4];
            while (i < nt && stage[i].cell < from + kM) ++i;
            for (; i < nt; ++i) add(i);
          }
          int i = s_start[(from < 0 ? 0 : from) >> 4];
          while (i < nt && stage[i].cell < from) ++i;
          for (; i < nt && stage[i].cell <= l; ++i) add(i);
          if (any) put(grid, l, get(grid, l) + acc);
        }
        __syncthreads();
      }
      if (n <= 0) __syncthreads();  // the grid is clear
      Cx<dd> x[16], out[8];
#pragma unroll
      for (int a = 0; a < 16; ++a) x[a] = get(grid, 256 * a + tid);
      fft4096(x, grid, kTfTwD1, kTfTwD2, out);
      if (!tr) {
#pragma unroll
        for (int s = 0; s < 8; ++s) put(s_z, 256 * s + tid, out[s]);
      }
      __syncthreads();  // every thread is past its reads of the grid
      if (tr) {
        const dd nd = dd_of((double)oi.n);
        const double scale = oi.norm_scale / y_sc / y_sc;
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const float2 t = __ldg(&kTfDeconvD[256 * s + tid]);
          const dd dc{t.x, t.y};
          const Cx<dd> z = get(s_z, 256 * s + tid);
          bool ill;
          const dd v = power_dd(Cx<dd>{mul_(z.re, dc), mul_(z.im, dc)},
                                Cx<dd>{mul_(out[s].re, dc), mul_(out[s].im, dc)}, nd, ill);
          // bin p + 16 r + 256 s, padded by one word per 16; -1 marks it for re-evaluation
          pw[(tid >> 4) + 17 * (tid & 15) + 272 * s] = ill ? -1.0 : scale * dd_double(v);
        }
      }
    }
    __syncthreads();

    double pv[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) pv[m] = oi.flags ? 0.0 : pw[8 * tid + (tid >> 1) + m];
    const uint32_t k0 = (uint32_t)kc0 + 8u * (uint32_t)tid;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      unsigned mask = __ballot_sync(0xffffffffu, pv[m] < 0.0 && (int64_t)k0 + m < p.n_f);
      while (mask) {
        const int l = __ffs(mask) - 1;
        mask &= mask - 1;
        const uint32_t k = __shfl_sync(0xffffffffu, k0 + (uint32_t)m, l);
        const double q = exact_power_warp64(p.rec, oi.begin, oi.n, k, oi.norm_scale);
        if (lane == l) pv[m] = q;
      }
    }
    if (p.power_out) store_row<8>(p.power_out + o * p.n_f, (int64_t)k0, pv, p.n_f);
    __syncthreads();  // pw is free for the chunk's results
    const int64_t res = o * (int64_t)n_chunks + chunk;
    chunk_results<double, 8>(pv, (int64_t)k0, kc0, p.n_f, p.best + res, p.cand ? p.cand + res : nullptr, pw, red_p,
                             red_k);
  }

  // one object, first maximum: the last CTA to finish writes the peak
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

int transform_blocks_per_sm64() {
  return blocks_per_sm(transform64_kernel, kThreads, kSmem);
}

cudaError_t launch_transform64(const TransformParams64& p, int grid, cudaStream_t stream) {
  cudaError_t e = allow_dyn_smem(transform64_kernel, kSmem);
  if (e != cudaSuccess) return e;
  transform64_kernel<<<grid, kThreads, kSmem, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace lsp
