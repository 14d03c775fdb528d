// lsp_peak.cuh -- the peak record of a grid bin (internal).
#pragma once

#include "../../include/lsp.h"
#include "lsp_common.cuh"

namespace lsp {

__device__ __forceinline__ lsp_peak make_peak(int64_t k, double p, double f_min, double df,
                                              int flags) {
  lsp_peak pk;
  pk.flags = flags;
  pk.reserved = 0;
  if (flags || k < 0) {
    pk.idx = -1;
    pk.power = 0.0;
    pk.freq = 0.0;
    pk.period = 0.0;
  } else {
    pk.idx = k;
    pk.power = p;
    pk.freq = __dadd_rn(f_min, __dmul_rn((double)k, df));  // f_min + k df, two roundings
    pk.period = 1.0 / pk.freq;
  }
  return pk;
}

}  // namespace lsp
