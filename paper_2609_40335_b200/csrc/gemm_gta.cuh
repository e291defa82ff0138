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
long long gta_tiles(const dp_linear_desc& L);           // output tiles of one layer
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
