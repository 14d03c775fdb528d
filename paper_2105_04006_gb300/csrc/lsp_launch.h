// lsp_launch.h -- host-side launchers of the library's kernels (internal).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "lsp_common.cuh"

struct lsp_peak;

namespace lsp {

// Opts a kernel in to `dyn` bytes of dynamic shared memory where its static
// and dynamic shared memory together pass the 48 KB available by default.
template <typename Kern>
inline cudaError_t allow_dyn_smem(Kern kern, size_t dyn) {
  if (dyn == 0) return cudaSuccess;  // static shared memory alone never passes it
  if (dyn <= 48 * 1024) {
    cudaFuncAttributes a{};
    cudaError_t e = cudaFuncGetAttributes(&a, kern);
    if (e != cudaSuccess) return e;
    if (dyn + a.sharedSizeBytes <= 48 * 1024) return cudaSuccess;
  }
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
}

int current_sm_count();  // of the current device, asked of the runtime once (152 on an error)

// CTAs of a kernel resident per SM (0 on an error), asked of the runtime once
// per device, kernel and shape: the query costs several microseconds, as much
// as the smallest calls' kernels.
int cached_blocks_per_sm(const void* kern, int threads, size_t dyn);
template <typename Kern>
inline int blocks_per_sm(Kern* kern, int threads, size_t dyn) {
  return cached_blocks_per_sm(reinterpret_cast<const void*>(kern), threads, dyn);
}

// Prologue, Section 2 (zero-mean magnitudes) and the per-observation phase
// data of the grid recurrences (rotation step, three-term coefficients).  y is float (y64 = false) or double.
// gls: weighted statistics / records of the generalized periodogram (dy
// NULL: unit weights).
cudaError_t launch_stats(const double* t, const void* y, bool y64, const int64_t* offsets,
                         int64_t n_obj, int64_t total_nt, int center, int norm, ObjInfo* obj,
                         cudaStream_t stream, bool gls = false, const void* dy = nullptr,
                         void* slices_ws = nullptr, uint32_t* ticket = nullptr);
// Scratch of the one-object statistics pass (slices_ws of launch_stats): with
// it, and a zeroed ticket word, one object without offsets is reduced by
// many CTAs; without it by one.
size_t stats_slices_bytes(int64_t total_nt);
// tf_min > 0 (batches, FP32 records of float magnitudes): also the transform
// path's scales of objects of at least tf_min observations (tf_scale_of).
cudaError_t launch_records(const double* t, const void* y, bool y64, ObjInfo* obj,
                           int64_t n_obj, int64_t max_nt_single, double f_min, double df,
                           bool rec64, void* rec, cudaStream_t stream, bool gls = false,
                           const void* dy = nullptr, int tf_min = 0);
// One object of at most kFusedMaxNt observations: statistics and records in
// one launch, which also clears the four work-counter words at `queue` (no
// memset, no ticket).  Every CTA redoes the object's FP64 statistics, about
// 3.5 clocks per observation on one SM at GB300's FP64 rate, which caps it.
constexpr int64_t kFusedMaxNt = 2048;
cudaError_t launch_single_prologue(const double* t, const void* y, bool y64, int64_t n, int center, int norm,
                                   double f_min, double df, bool rec64, ObjInfo* obj, void* rec, uint32_t* queue,
                                   cudaStream_t stream, bool gls = false, const void* dy = nullptr);
// The work-queue order: objects by N_t (counting sort), the longest and the
// shortest alternating.
cudaError_t launch_lpt_order(const ObjInfo* obj, int64_t n_obj, uint32_t* hist, int32_t* order,
                             cudaStream_t stream);

// Main kernel variants.
struct MainLaunch {
  int prec;      // 0 FP32, 1 FP64
  int packed;    // FP32 only
  int k_reseed;  // chain length K
  int fpt;       // frequencies per thread (packed: 2K; scalar: K)
  int gls = 0;   // generalized periodogram kernels
  int abl = 0;   // ablation kernel: trig + 3 * staging (lsp_config), 0 = production
  int threads;
  int grid;      // persistent CTAs
  int top;       // 1: top-k candidates
  const void* rec;
  const ObjInfo* obj;
  const int32_t* order;
  void* power_out;
  void* part;
  ChunkBest* best;
  ChunkCand* cand;
  uint32_t* queue;
  int64_t n_f;
  int32_t n_chunks;
  int32_t split;
  int64_t n_items;
  const uint32_t* n_items_dev = nullptr;  // device item count (overrides n_items)
  const int32_t* win_start = nullptr;     // per-object window origins (packed FP32 kernels)
  int32_t win_len = 0;
};
bool main_variant_exists(int prec, int packed, int k_reseed, int fpt, int gls = 0, int abl = 0);
cudaError_t launch_main(const MainLaunch& ml, cudaStream_t stream);
// CTAs of the main variant resident per SM (0 if the variant does not exist).
int main_blocks_per_sm(int prec, int packed, int k_reseed, int fpt, int threads, int top, int gls = 0,
                      int abl = 0);
size_t main_dyn_smem(int prec, int fpt, int threads, int top);

// Transform path (lsp_transform.cu): the trig sums of runs of kTfBins bins by
// a nonuniform FFT; FP32 (standard and generalized periodogram) and FP64
// (standard).
constexpr int kTfBins = 2048;
constexpr size_t kTf64CellBytes = 4 * 4096 * 8;
template <typename Rec, typename Real>
struct TransformParamsOf {
  const Rec* rec;
  const ObjInfo* obj;
  const int32_t* order = nullptr;       // object list, read forwards, or
  const int32_t* order_back = nullptr;  // its last word, read backwards (neither: identity)
  Real* power_out;      // nullable, n_obj x n_f
  ChunkBest* best;
  ChunkCand* cand;       // nullable: only with top_k > 1
  uint32_t* queue;       // zeroed work counter
  const uint32_t* n_items_dev;  // device item count (overrides n_items)
  uint32_t n_items;
  int32_t n_chunks;      // runs per object
  long long* cells = nullptr;  // FP64: kTf64CellBytes per CTA
  int32_t have_scale;    // the records kernel left the scales (batches)
  // FP32: per-object windows instead of runs from 0 (n_chunks = 1, one item
  // per object): bins [win_start[o], win_start[o] + win_len) of the grid
  const int32_t* win_start = nullptr;
  int32_t win_len = 0;
  int64_t n_f;
  // one object, first maximum only: the peak is written by the last CTA
  // (ticket: a zeroed word); NULL: a finalize launch follows
  lsp_peak* peaks;
  double f_min, df;
  uint32_t* ticket;
};
typedef TransformParamsOf<RecF32, float> TransformParams;
typedef TransformParamsOf<RecF64, double> TransformParams64;
cudaError_t launch_transform(const TransformParams& p, int gls, int grid, cudaStream_t stream);
cudaError_t launch_transform64(const TransformParams64& p, int grid, cudaStream_t stream);
int transform_blocks_per_sm(int prec, int gls);  // 0: no such kernel
// One object on its whole grid by one large transform (lsp_long.cu).
constexpr int kLongMaxLog2 = 22;
struct LongPlan {
  int lg, lg2;   // log2 of the transform's length and of its second pass's
  int32_t kc;    // the bin at offset 0
  size_t cell_bytes, t_bytes, row_bytes;  // scratch
};
bool long_plan(int prec, int64_t n_f, LongPlan* lp);  // false: the grid is too long
// p: rec, obj, power_out, best, cand, n_chunks, n_f, peaks, f_min, df, ticket;
// max_n: an upper bound of the object's observations.
cudaError_t launch_long32(const LongPlan& lp, const TransformParams& p, int64_t max_n, void* cells, void* t, void* row,
                          cudaStream_t stream);
cudaError_t launch_long64(const LongPlan& lp, const TransformParams64& p, int64_t max_n, void* cells, void* t,
                          void* row, cudaStream_t stream);
// The work lists of a batch that takes both paths: objects of at least
// `n_min` observations (the transform) from the back of order[], the others
// (the direct kernel) from its front, each list by decreasing N_t;
// items[0] and items[1] receive the two lists' lengths times n_chunks.
cudaError_t launch_split_order(const ObjInfo* obj, int64_t n_obj, int n_min, int n_chunks, uint32_t* hist,
                               int32_t* order, uint32_t* items, cudaStream_t stream);

// Split-N_t combine (single object; gls: the generalized periodogram's six
// sums in stride-8 slots): sums the partial sums in a fixed order,
// evaluates the power, stores it (optional) and reduces chunk results; with
// peaks, no candidates and a zeroed ticket word it also writes the first
// maximum (no finalize launch needed).
constexpr int kCombineThreads = 256;
#ifndef LSP_COMBINE_PER_THREAD
#define LSP_COMBINE_PER_THREAD 1
#endif
constexpr int kCombinePerThread = LSP_COMBINE_PER_THREAD;
cudaError_t launch_combine(int prec, const void* part, int split, int64_t n_f, const ObjInfo* obj,
                           const void* rec, void* power_out, ChunkBest* best, ChunkCand* cand,
                           cudaStream_t stream, lsp_peak* peaks = nullptr, double f_min = 0.0,
                           double df = 0.0, uint32_t* ticket = nullptr, bool gls = false);

// Per-object peaks from the chunk results.
cudaError_t launch_finalize(const ObjInfo* obj, const ChunkBest* best, const ChunkCand* cand,
                            int64_t n_obj, int n_chunks, int top_k, double f_min, double df,
                            lsp_peak* peaks, cudaStream_t stream);

// First maximum of stored periodograms (no workspace: the peak records hold
// the reduction state).
cudaError_t launch_argmax_period(const void* power, bool p64, int64_t n_obj, int64_t n_f,
                                 double f_min, double df, lsp_peak* peaks, cudaStream_t stream);

// Autotuner error gate helpers.
cudaError_t launch_f32_to_f64(const float* a, double* b, int64_t n, cudaStream_t stream);
cudaError_t launch_max_abs_diff(const float* a, const double* b, int64_t n, double* out,
                                cudaStream_t stream);
// out[r] = max_i |a[r n + i] - b[r n + i]| for each of `rows` rows.
cudaError_t launch_row_max_abs_diff(const float* a, const double* b, int64_t rows, int64_t n, double* out,
                                    cudaStream_t stream);
// score[i] = max over the grid of |sum_j exp(2 pi i 2 f_k t_j)| / N for the
// observations t[begin[i] .. begin[i] + count[i]) (device arrays).
cudaError_t launch_window_score(const double* t, const int64_t* begin, const int64_t* count, int n_list,
                                double f_min, double df, int64_t n_f, float* score, cudaStream_t stream);

}  // namespace lsp
