// Declarations of the fp32-FMA launchers (fma_kernels.cu), the embedding launchers
// (embed_kernels.cu) and the noise launcher (noise_kernel.cu).
#pragma once

#include "dp_common.cuh"

namespace dpg {

dp_status launch_norms_fma(const dp_linear_desc& L, dp_dtype dt, int mode, int B, int T, float* sq,
                           cudaStream_t st, bool overwrite = false);
// ghost norms of layers[index[0 .. n)] in one launch: partial sums [B][n_per], gram_fma_partials per layer
int gram_fma_partials(const dp_linear_desc& L, int T);
// a layer by itself whose norm launch_norms_fma forms faster, without the launch that adds up partial sums (d = p = 768:
// 6.4 against 7.2 us at T = 1, 39 against 42 at T = 31)
bool gram_alone_fma(const dp_linear_desc& L, int T);
dp_status launch_gram_norms_fma(const dp_linear_desc* layers, const int* index, int n, dp_dtype dt, int B, int T,
                                float* partials, int n_per, cudaStream_t st);
// clipped sums of layers[index[0 .. n)]; noise: added onto them (inside the kernel where d is a multiple
// of 4), NULL = none
struct GtaNoise;
dp_status launch_clip_accumulate_fma(const dp_linear_desc* layers, const int* index, int n, dp_dtype dt, int B, int T,
                                     const float* clip, float* const* outs, const int64_t* ldos, float beta,
                                     const GtaNoise* noise, cudaStream_t st);
// partials: [B * ceil(T/16)] floats, example-major
dp_status launch_cross_term_fma(const int* ids, const void* Ge, int64_t ldge, const void* Al,
                                int64_t ldal, const void* Gl, int64_t ldgl, dp_dtype dt, int B,
                                int T, int d, int V, float* partials, int* dev_status,
                                cudaStream_t st);
// extra: added to sq first, the sum written to `sum` (which may be sq)
dp_status launch_clip_factors(const float* sq, int B, float C, float* clip, float* norms,
                              cudaStream_t st, const float* extra = nullptr, float* sum = nullptr);
// Partial sums of squared norms that a step has left in workspaces: [B][n_per] floats each.
struct NormSource { const float* partials; int n_per; float factor; float* plain_out; };
struct NormSources {
  NormSource src[6];
  int n_main, n;             // src[0 .. n_main) are added up, src[n_main .. n) are, then the two sums
};
dp_status launch_finish_norms(const NormSources& S, int B, float C, float* sq, float* clip, float* norms,
                              cudaStream_t st);

// embedding
constexpr int kEmbedMaxT = 4096;
constexpr int kEmbedColsPerBlock = 256;
dp_status launch_embed_norms(const int* ids, const void* G, int64_t ldg, dp_dtype dt, int B, int T,
                             int d, int V, int parts, float* partials, int* first_occ,
                             int* dev_status, cudaStream_t st);
int embed_norm_parts(int B, int T, int d);      // partial sums per (example, 256-column slab)
struct EmbedSortWs {
  int* totals;      // [V], [ceil(V / 1024)] and [chunks][V]: tokens per id, per 1024 ids, per chunk and id
  int* seg;         // [V+1]
  int* perm;        // [B*T]
  int* rank;        // [B*T]  rank of a token among the equal ids of its chunk
};
constexpr int kSortChunk = 1024;
// One block sorts by itself in one launch instead of four, but its walk over the tokens and its scan over the ids are
// serial.  One block and chunks, Zipf ids, replayed as a graph: 5.8 and 8.5 us at 64 tokens and 1000 ids, 14.7 and 16.4 at 2048 and
// 4000; 18.9 and 16.8 at 2048 and 8192, 11.2 and 8.2 at 64 and 8192, 22.6 and 17.7 at 3072 and 8192.  The line over the ids lies where a
// small step still gains: launched call by call the three launches are 8 us of the host's time, which bounds it (34 -> 42 us at
// 64 tokens and 4500 ids).
constexpr int kSortOneBlock = 2048, kSortOneBlockIds = 8192;
inline bool sort_in_one_block(int n, int V) { return n <= kSortOneBlock && V <= kSortOneBlockIds; }
// Chunks whose counts a token adds up when it is placed; with more, sort_prefix_kernel adds them up once: 22.7 us with it
// against 21.9 at 4 chunks, 24.9 against 25.4 at 16, 55 against 77 at 64, 0.84 against 14.7 ms at 1024 (V = 50257).
constexpr int kSortWalk = 8;
dp_status launch_clear(void* p, size_t bytes, cudaStream_t st);
dp_status launch_embed_sort(const int* ids, int n, int V, const EmbedSortWs& ws, int* dev_status,
                            cudaStream_t st);
dp_status launch_embed_scatter(const int* ids, const void* G, int64_t ldg, dp_dtype dt, int n,
                               int T, int d, int V, const float* clip, const int* perm,
                               const int* seg, float* out, int64_t ldo, float beta, float scale,
                               bool clear, float* long_part, cudaStream_t st,
                               int* dev_status = nullptr);
dp_status launch_bounds_probe(long long idx, long long n, int* dev_status, cudaStream_t st);
// bytes of the per-chunk partial sums of long segments: [chunks][2][d] floats
size_t embed_scatter_partial_bytes(long long n, int d);

// logical (rows, cols) tensor with row pitch ld; element j = row*cols + col of the stream.
// fill: write scale*amp*z without reading out (first_quad: add mode only).
dp_status launch_add_noise(float* out, long long rows, int cols, long long ld, bool fill, float amp,
                           float scale, uint64_t seed, uint32_t tensor_id, uint32_t step,
                           cudaStream_t st, long long first_quad = 0);

dp_status launch_noise_error_scan(float t_max, double* out3, cudaStream_t st);

}  // namespace dpg
