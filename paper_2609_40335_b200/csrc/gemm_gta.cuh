// Declarations for the tensor-core G^T A kernels (clipped sum and DIRECT per-example norm).
#pragma once

#include "dp_common.cuh"
#include "fma_kernels.cuh"
#include "ghost_plan.cuh"

namespace dpg {

// Layers per launch: what fits the 32 764-byte parameter block (two tensor maps and 56 bytes per layer).
// GPT-2 medium's 97 layers have to fit: a second launch cost a second partly filled last wave.
constexpr int kGtaMaxLayers = 102;

// Plain data: copied into kernel parameters.
struct GtaLayer {
  float* out;             // (M, N) destination when the K range is not split
  float* partial;         // [nsplit][M][N] planes when it is
  long long ldo;
  int M, N;               // p, d
  int item_begin;
  int col_begin;          // square-sum mode: first partial-sum column of this layer
  int prescaled;          // 1: the clip factors were applied to this layer's narrow operand beforehand
  float noise_amp;        // sigma*C of the fused noise, negative = none
  uint32_t tensor_id;     // noise stream id of this output tensor
};

// Fused Gaussian mechanism of a grouped call (host side).
struct GtaNoise {
  float amp, scale;
  uint64_t seed;
  uint32_t step;
  const uint32_t* tensor_ids;   // [n_layers]
};

// How a clipped sum walks its contraction.  The token rows of a batch lie one after the other (row i*T + t, one
// pitch), so the tensor map has them as one dimension and a K step is 64 consecutive rows whatever examples they
// belong to; the scaler warps look up a clip factor per row where a step holds several.  Steps that end with
// their example instead were filled up with zeros: at T = 203 84 steps of 64 for 21 examples, 67 now; at T = 77 two
// steps an example, at T = 16 one, three quarters of it zeros.  The step of DistilGPT2 with all its parameters at B = 21, T = 203
// 1383 -> 1295 us, of GPT-2 small at B = 3, T = 77 349 -> 344; at B = 32, T = 128 (the same steps) 940 -> 945, within the runs'
// differences.  Scaling row by row costs more, so the batch is walked whole only where that saves a sixth of the steps (7 layers
// of d = 576 at B = 23, T = 57, 21 steps or 23: step 232 us against 217).  Coordinates are 32-bit: a batch of 2^31 rows
// keeps steps per example.
struct GtaRows {
  int B, T;                // planes along K, rows of each, as the tensor map has them
  int scaled_rows, scaled_steps;   // scaling: all rows, or 0 and the steps of an example where each has its own
};
inline GtaRows gta_rows(int B, int T, int terms) {
  const long long rows = (long long)B * T;
  const int steps = (T + 63) / 64;
  if ((T % 64 == 0 || terms > 1) && rows <= 0x7fffffffLL - 64) return {1, int(rows), 0, steps};      // no factors by row
  if (rows > 0x7fffffffLL - 64 || 6 * ((rows + 63) / 64) > 5LL * B * steps) return {B, T, 0, steps};
  return {1, int(rows), int(rows), steps};
}

// Clip factors of a K step's rows: lane k holds those of rows k and k + 32; `one`: they are all the same.
struct RowFactors { float lo, hi; bool one; };
// step: K step of the contraction; rows: all token rows, 0: `tsteps` steps belong to each example, as always without kByRow:
// kernels that never meet several examples in a step are compiled without the code for them, whose mere presence costs
// more than its use saves (4 GPT-2-small layers at B = 88, T = 272 346 us without, 365 with).  The lanes look their
// rows up only where a step holds several examples.
template <bool kByRow>
__device__ __forceinline__ RowFactors row_factors(const float* clip, int step, int lane, int T, int rows, int tsteps) {
  if (!kByRow || rows == 0) {
    const float r = __ldg(clip + step / tsteps);
    return {r, r, true};
  }
  const unsigned first = unsigned(step) * 64u, ex = first / unsigned(T);
  if (first + 64u <= (ex + 1u) * unsigned(T)) {
    const float r = __ldg(clip + ex);
    return {r, r, true};
  }
  const unsigned last = unsigned(rows) - 1u, mine = first + unsigned(lane);
  return {__ldg(clip + min(mine, last) / unsigned(T)), __ldg(clip + min(mine + 32u, last) / unsigned(T)), false};
}

// One warp multiplies a 16 KiB operand part (two boxes of 64 rows x 128 bytes; the 128-byte swizzle moves 16-byte
// chunks inside a row only) by its rows' factors.  r = r_hi + r_lo with both parts in bf16 (16 mantissa bits in
// total); x*r is formed as fma(x, r_hi, x*r_lo) on packed bf16 pairs: one rounding of the exact x*r_hi plus a tiny
// correction, i.e. the correctly rounded bf16 product up to 2^-17 relative.  16-byte chunks, eight at a time.
__device__ __forceinline__ void scale_part(uint4* part, float r, int lane) {
  const __nv_bfloat16 rh = __float2bfloat16_rn(r);
  const __nv_bfloat16 rl = __float2bfloat16_rn(r - __bfloat162float(rh));
  const __nv_bfloat162 rh2 = __halves2bfloat162(rh, rh), rl2 = __halves2bfloat162(rl, rl);
  uint4* x = part + lane;
#pragma unroll 1
  for (int c0 = 0; c0 < 32; c0 += 8) {
    uint4 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = x[(c0 + q) * 32];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      __nv_bfloat162* e = reinterpret_cast<__nv_bfloat162*>(&v[q]);
#pragma unroll
      for (int k = 0; k < 4; ++k) e[k] = __hfma2(e[k], rh2, __hmul2(e[k], rl2));
      x[(c0 + q) * 32] = v[q];
    }
  }
}

// The same with a factor per row.  Out of line: inside the scalers' loop it cost the steps that need none of it more.
static __device__ __noinline__ void scale_rows(uint4* part, float lo, float hi, int lane) {
  auto split = [](float x) {                       // r_hi in the low half, r_lo in the high one
    const __nv_bfloat16 h = __float2bfloat16_rn(x), l = __float2bfloat16_rn(x - __bfloat162float(h));
    return uint32_t(__bfloat16_as_ushort(h)) | (uint32_t(__bfloat16_as_ushort(l)) << 16);
  };
  auto pair = [](uint32_t w, uint32_t sel) {
    const uint32_t b = __byte_perm(w, w, sel);
    return *reinterpret_cast<const __nv_bfloat162*>(&b);
  };
  const uint32_t w_lo = split(lo), w_hi = split(hi);
  uint4* x = part + lane;
  // chunk 32 i + lane of a box lies in row 4 i + lane / 8: four rows of both boxes at a time
#pragma unroll 1
  for (int i0 = 0; i0 < 16; i0 += 4) {
    const uint32_t mine = i0 & 8 ? w_hi : w_lo;
    uint4 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = x[(i0 + (q >> 1) + 16 * (q & 1)) * 32];
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      const uint32_t w = __shfl_sync(0xffffffffu, mine, (4 * (i0 + (q >> 1)) + (lane >> 3)) & 31);
      const __nv_bfloat162 rh2 = pair(w, 0x1010), rl2 = pair(w, 0x3232);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        __nv_bfloat162* e = reinterpret_cast<__nv_bfloat162*>(&v[q + h]);
#pragma unroll
        for (int k = 0; k < 4; ++k) e[k] = __hfma2(e[k], rh2, __hmul2(e[k], rl2));
        x[(i0 + (q >> 1) + 16 * h) * 32] = v[q + h];
      }
    }
  }
}

// terms = 3: the operands are planes of high and, behind them all, of low bf16 terms (fp32 inputs) and a product
// takes three K steps per 64 tokens; terms = 1: plain bf16 operands.
//
// Order of a contraction's K steps.  With three terms, first lo hi' and hi lo' of all its 64-token blocks, then
// hi hi' of all: an MMA rounds its sum towards zero, by as much as the sum is large, and while the small products
// are added the sum is 2^-8 of its final size.  Block by block, every product of the three rounded the whole sum: error of
// 25 layers of DistilGPT2's shapes against 64 bits 9.1e-6 at 2048 tokens, 2.8e-5 at 16384; in this order 5.1e-6 and 1.0e-5 (4.5e-6
// is the operands' own).  The fp32 step of DistilGPT2 at B = 8, T = 128 takes 876 us in this order, 868 in the other.
// kSplit: three terms.  A template, since the producers' loop is part of every stage's round trip: with the terms looked up
// at run time the step of GPT-2 medium at B = 16, T = 128 came out 0.4 % slower than with a fixed order, in this form 0.4 % faster.
template <bool kSplit>
struct GtaWalk {
  int ex, ts, tblocks;                 // plane (example, or all of them), block in it, blocks per plane
  int term = 0, ex0 = 0, ts0 = 0, left = 0;      // split: which product, where the contraction starts, blocks left in this round

  // blocks [b0, b1), counted from plane `first`
  __device__ __forceinline__ GtaWalk(int first, int b0, int b1, int tblocks_) : tblocks(tblocks_) {
    ex = first + b0 / tblocks;
    ts = b0 % tblocks;
    if (kSplit) { ex0 = ex; ts0 = ts; left = b1 - b0; }
  }
  __device__ __forceinline__ void next() {
    if (kSplit && term == 0) { term = 1; return; }
    if (++ts == tblocks) { ts = 0; ++ex; }
    if (!kSplit || term != 1) return;
    term = 0;
    if (--left == 0) { ex = ex0; ts = ts0; term = 2; }
  }
  // plane of the A or G operand; `low`: the first plane of low terms
  __device__ __forceinline__ int plane(bool is_a, int low) const { return kSplit && term == (is_a ? 0 : 1) ? ex + low : ex; }
};

long long gta_tiles(const dp_linear_desc& L);           // output tiles of one layer
bool gta_prescales(const dp_linear_desc& L);            // terms = 1: a scaled copy goes into the scratch, for TMA to read
int gta_choose_nsplit(long long tiles, int B, int T, int terms, int sms);
// scratch of a grouped call behind the clip factors: K-split planes (if any) and, terms = 1, the
// pre-scaled copies of very narrow operands
// ample: planes of as many splits as if K steps ended with their examples, at least as many; room in which more layers go together
size_t gta_partial_bytes(const dp_linear_desc* layers, int n_layers, int B, int T, int terms, int sms, bool ample = false);

// One persistent launch over the output tiles of all layers (plus split-K reduces if needed).
dp_status launch_clip_accumulate_tc(const dp_linear_desc* layers, int n_layers, int B, int T, int terms,
                                    const float* clip, float* const* outs, const int64_t* ldos,
                                    float beta, const GtaNoise* noise, float* partial_ws,
                                    int* dev_status, cudaStream_t st);

// Items of two output tiles sharing an operand, for calls with tiles enough (gemm_gta_big.cu).
struct GtaBigJob {
  const void* A;
  int64_t lda;
  const void* G;
  int64_t ldg;
  int d, p;
  float* out;
  int64_t ldo;
  int prescaled;
  float noise_amp;        // sigma*C of the fused noise, negative = none
  uint32_t tensor_id;
};
dp_status launch_gta_big(const GtaBigJob* jobs, int n, int B, int T, int terms, const float* clip, float beta,
                         const GtaNoise* noise, int* dev_status, cudaStream_t st);

dp_status launch_direct_norm_tc(const dp_linear_desc* layers, const GhostPlan& plan, int B, int T, int terms,
                                float* partials, int* dev_status, cudaStream_t st);

}  // namespace dpg
