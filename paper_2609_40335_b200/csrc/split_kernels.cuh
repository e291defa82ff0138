// Split of fp32 operands into two bf16 terms for the tensor-core path of DP_F32 inputs.
#pragma once

#include "dp_common.cuh"

namespace dpg {

// the operand that the clipped sums scale is the narrower one: A, unless it is wider than G
inline bool a_is_scaled(const dp_linear_desc& L) { return L.d <= L.p; }

// operand width rounded up to 8 columns (a 16-byte pitch for the TMA tensor maps)
inline int split_padded(int c) { return (c + 7) / 8 * 8; }
// bytes of one split operand: (2, B, T, padded(c)) bf16, the high terms of all examples, then the low ones
inline size_t split_bytes(long long rows, int c) {
  return align_up(size_t(rows) * 2 * size_t(split_padded(c)) * 2, 256);
}

struct SplitJob {
  const float* src;
  int64_t lds;
  int c;                 // columns
  bool scaled;           // multiply example i by clip[i] first
  void* dst;
};
// all jobs in as few launches as the parameter block allows; clip may be NULL if no job is scaled
dp_status launch_split(const SplitJob* jobs, int n, int B, int T, const float* clip, cudaStream_t st);

}  // namespace dpg
