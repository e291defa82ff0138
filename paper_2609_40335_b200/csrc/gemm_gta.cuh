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

// terms = 3: the operands are (2B, T, .) planes of high and low bf16 terms (fp32 inputs) and a product
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
  int ex, ts, tblocks;                 // example, block in it, blocks per example
  int term = 0, ex0 = 0, ts0 = 0, left = 0;      // split: which product, where the contraction starts, blocks left in this round

  // blocks [b0, b1), counted from example `first`
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
  // plane of the A or G operand
  __device__ __forceinline__ int plane(bool is_a) const { return kSplit ? 2 * ex + (term == (is_a ? 0 : 1)) : ex; }
};

long long gta_tiles(const dp_linear_desc& L);           // output tiles of one layer
bool gta_prescales(const dp_linear_desc& L);            // terms = 1: a scaled copy goes into the scratch, for TMA to read
int gta_choose_nsplit(long long tiles, int B, int T, int terms, int sms);
// scratch of a grouped call behind the clip factors: K-split planes (if any) and, terms = 1, the
// pre-scaled copies of very narrow operands
size_t gta_partial_bytes(const dp_linear_desc* layers, int n_layers, int B, int T, int terms, int sms);

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
