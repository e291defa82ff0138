// fp32 operands on the bf16 tensor cores: every fp32 value x is split into two bf16 terms,
//   hi = bf16(x),  lo = bf16(x - hi),   x = hi + lo up to 2^-17 |x|,
// and a product x*y is taken as hi*hi' + hi*lo' + lo*hi' (the dropped lo*lo' is below 2^-16 of the
// product) -- three tensor-core products with fp32 accumulation instead of one, the same idea as
// the "3 x TF32" scheme with 16 instead of 21 mantissa bits, far inside the 1e-4 the fp32 path has
// to meet, and at three bf16 MMAs cheaper than three TF32 MMAs (which run at half the bf16 rate).
//
// An operand is stored once, the high terms of all examples and behind them the low ones (as many bytes as the fp32
// original); the Gram and G^T A kernels pick the plane of each side of each product by the tensor map's outer
// coordinate, and a contraction over tokens finds the rows of all examples in one piece.  (Widened copies [hi | hi | lo] and [hi | lo | hi] took three to six times the
// workspace and traffic and, the workspace being sized for one layer, a dozen launches per layer:
// 24 layers and a head of DistilGPT2 at B = 8, T = 128 took 236 launches, now 12.)
// For the clipped sum the clip factor R_i (Eq. 7) multiplies the narrower operand in fp32 BEFORE the
// split, so the GEMM itself runs unscaled and no bf16 rounding of R_i * g occurs.  In a whole step the other
// operand's planes are those of the norms, where the workspace holds all layers: 999 -> 865 us (DistilGPT2,
// B = 8, T = 128, the second split 180 -> 44).
#include <cuda_bf16.h>

#include <algorithm>

#include "dp_common.cuh"
#include "split_kernels.cuh"

namespace dpg {

namespace {

constexpr int kMaxJobs = 208;          // tensors per launch (parameter block)
constexpr int kChunksPerBlock = 1024;  // 8-column chunks per block of 256 threads

struct SplitTensor {
  const float* src;
  __nv_bfloat16* dst;
  long long lds;
  int c, per_row;                      // columns, 8-column chunks per row
  int block_begin, scaled;
};
struct SplitParams {
  SplitTensor t[kMaxJobs];
  int n, T;
  long long rows;                      // B * T
  const float* clip;
};

// HBM-bound: 4 bytes read and 4 written per element, 32 + 32 per thread and step
__global__ void __launch_bounds__(256)
split_kernel(const __grid_constant__ SplitParams P) {
  int lo = 0, hi = P.n - 1;            // the tensor this block belongs to
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (int(blockIdx.x) >= P.t[mid].block_begin) lo = mid; else hi = mid - 1;
  }
  const SplitTensor& S = P.t[lo];
  const bool vec = ((reinterpret_cast<uintptr_t>(S.src) & 15) == 0) && ((S.lds & 3) == 0);
  const long long total = P.rows * S.per_row;
  const long long first = (long long)(int(blockIdx.x) - S.block_begin) * kChunksPerBlock;
  const size_t plane = size_t(P.rows) * S.per_row * 8;     // elements of the high terms
  const long long row0 = first / S.per_row;                // the block's first row and chunk in it
  const unsigned off0 = unsigned(first - row0 * S.per_row);
#pragma unroll
  for (int k = 0; k < kChunksPerBlock / 256; ++k) {
    const unsigned off = off0 + k * 256 + threadIdx.x;
    const unsigned dr = off / unsigned(S.per_row);
    if (first + k * 256 + threadIdx.x >= total) break;
    const unsigned r = unsigned(row0) + dr;                // token row i*T + t
    const int col = int(off - dr * S.per_row) * 8;
    float v[8];
    load8<float>(S.src + (long long)r * S.lds + col, S.c - col, vec, v);      // columns >= c read as zero
    if (S.scaled) {
      const float f = __ldg(P.clip + r / unsigned(P.T));
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] *= f;
    }
    uint4 h, l;
    __nv_bfloat162* h2 = reinterpret_cast<__nv_bfloat162*>(&h);
    __nv_bfloat162* l2 = reinterpret_cast<__nv_bfloat162*>(&l);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      h2[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
      const float2 b = __bfloat1622float2(h2[j]);
      l2[j] = __floats2bfloat162_rn(v[2 * j] - b.x, v[2 * j + 1] - b.y);
    }
    __nv_bfloat16* d = S.dst + size_t(r) * S.per_row * 8 + col;
    *reinterpret_cast<uint4*>(d) = h;
    *reinterpret_cast<uint4*>(d + plane) = l;
  }
}

}  // namespace

dp_status launch_split(const SplitJob* jobs, int n, int B, int T, const float* clip, cudaStream_t st) {
  for (int j0 = 0; j0 < n; j0 += kMaxJobs) {
    SplitParams P;
    P.n = std::min(n - j0, kMaxJobs);
    P.T = T; P.rows = (long long)B * T; P.clip = clip;
    long long blocks = 0;
    for (int k = 0; k < P.n; ++k) {
      const SplitJob& J = jobs[j0 + k];
      SplitTensor& S = P.t[k];
      S.src = J.src; S.dst = static_cast<__nv_bfloat16*>(J.dst); S.lds = J.lds; S.c = J.c;
      S.per_row = split_padded(J.c) / 8; S.scaled = J.scaled ? 1 : 0; S.block_begin = int(blocks);
      blocks += (P.rows * S.per_row + kChunksPerBlock - 1) / kChunksPerBlock;
    }
    if (blocks > 0x7fffffffLL) return DP_ERR_UNSUPPORTED;
    split_kernel<<<(unsigned)blocks, 256, 0, st>>>(P);
    DP_LAUNCH_OK();
  }
  return DP_OK;
}

}  // namespace dpg
