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
// sums from the exact phases.  Against quadruple precision the powers are as
// exact as the FP64 pairwise kernel's from N_t 60 on and on grids of 20 000 bins
// and more, where what both share (the mean, the phases of late bins) sets the
// error; at N_t 8 on 3000 bins it is 3e-15 against 3e-16.
//
// Measured (GB300): 200 survey light curves (N_t 50 .. 500) on 1e5 bins 2.6 ms
// against 64 ms with the direct kernel; a run on one SM 60 000 clocks plus 89
// an observation; 60 objects of N_t 8 0.61 | 1.34, 12 0.59 | 1.62, 64 0.63 |
// 5.3 ms (transform | direct).  Bound by instruction issue (55 %, two CTAs of
// 128 registers; 64 bytes spilled, 292 read back).
//
// Differences from the FP32 kernel:
//   - cells are 64-bit fixed point (a cell of W is at most N, one of Z at most
//     sqrt(N sum y^2)).  Shared memory has no 64-bit add of its own, so each
//     CTA's 128 KB of cells lie in global memory (in L2: 40 MB for all CTAs)
//     and take integer reductions there; any time order and any clustering
//     run at the same speed and repeats are bit-identical.  (Gathered per cell
//     from sorted observations in shared memory instead, the spread took 190
//     clocks an observation, lanes waiting for the fullest cell.)
//   - Z and W are transformed one after the other; Z's outputs wait in shared
//     memory;
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
constexpr int kWarps = kThreads / 32;
constexpr int kLog2M = 12;
static_assert(kTfBins == kM / 2 && kTfBins == kThreads * 8 && kM == 1 << kLog2M, "run length");

constexpr size_t kBufBytes = (size_t)kM * sizeof(Cx<dd>);     // exchange buffer; later the powers of the run
constexpr size_t kZBytes = (size_t)kTfBins * sizeof(Cx<dd>);  // Z's outputs
constexpr size_t kSmem = kBufBytes + kZBytes;
static_assert(kTf64CellBytes == 4 * kM * sizeof(long long), "four planes of cells per CTA");

__global__ void __launch_bounds__(kThreads, 2) transform64_kernel(TransformParams64 p) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  Cx<dd>* const buf = reinterpret_cast<Cx<dd>*>(dyn_smem);
  Cx<dd>* const s_z = reinterpret_cast<Cx<dd>*>(dyn_smem + kBufBytes);
  // this CTA's cells: planes Z re, Z im, W re, W im; zero between runs
  long long* const cells = p.cells + (int64_t)blockIdx.x * (4 * kM);
  double* const pw = reinterpret_cast<double*>(dyn_smem);
  __shared__ double red_p[32];
  __shared__ int64_t red_k[32];
  __shared__ uint32_t s_item;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n_items = p.n_items_dev ? *p.n_items_dev : p.n_items;
  const uint32_t n_chunks = (uint32_t)p.n_chunks;

  for (int i = tid; i < 4 * kM / 2; i += kThreads) reinterpret_cast<longlong2*>(cells)[i] = make_longlong2(0, 0);
  __threadfence();

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
    const double y_sc = pow2(-y_exponent(oi.sum_y2));
    {  // spread: each warp takes an eighth of the observations
      const float one[2] = {(float)pow2(z_bits(n)), (float)pow2(w_bits(n))};
      const uint32_t j1 = (uint32_t)((int64_t)n * (warp + 1) / kWarps);
      for (uint32_t jb = (uint32_t)((int64_t)n * warp / kWarps); jb < j1; jb += 32) {
        const ObsD ob = obs_of(rec[jb + lane < j1 ? jb + lane : jb], kc, kLog2M, y_sc);
        spread_warp(ob, (int)min(32u, j1 - jb), kM - 1, one, [&](int t, uint32_t l, long long re, long long im) {
          add_cell(cells + (2 * t) * kM + l, re);
          add_cell(cells + (2 * t + 1) * kM + l, im);
        });
      }
    }
    __threadfence();
    __syncthreads();  // every reduction has reached L2
    const float z_inv = (float)pow2(-z_bits(n)), w_inv = (float)pow2(-w_bits(n));

#pragma unroll 1
    for (int tr = 0; tr < 2; ++tr) {  // Z, then W
      Cx<dd> x[16], out[8];
#pragma unroll
      for (int a = 0; a < 16; ++a) {
        long long* const c = cells + 2 * tr * kM + 256 * a + tid;
        x[a] = Cx<dd>{dd_of_int(__ldcg(c)), dd_of_int(__ldcg(c + kM))};
        c[0] = 0;
        c[kM] = 0;
      }
      fft4096(x, buf, kTfTwD1, kTfTwD2, out);
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
          const dd dz{t.x * z_inv, t.y * z_inv}, dw{t.x * w_inv, t.y * w_inv};
          const Cx<dd> z = get(s_z, 256 * s + tid);
          bool ill;
          const dd v = power_dd(Cx<dd>{mul_(z.re, dz), mul_(z.im, dz)},
                                Cx<dd>{mul_(out[s].re, dw), mul_(out[s].im, dw)}, nd, ill);
          // bin p + 16 r + 256 s, padded by one word per 16; -1 marks it for re-evaluation
          pw[(tid >> 4) + 17 * (tid & 15) + 272 * s] = ill ? -1.0 : scale * dd_double(v);
        }
      }
    }
    __threadfence();  // the cleared cells, before the next run's reductions
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
