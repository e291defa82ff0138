// fp32-FMA kernels for linear layers: the DP_F32 path (fp32 tensors need better than TF32
// accuracy) and the cross-check path for DP_BF16.  Any shape, no alignment rules.
//   ghost  : sq[i] += sum_{t,s} (a_t.a_s)(g_t.g_s)            (Eq. 4 - Eq. 5 over T tokens)
//   direct : sq[i] += sum_{r,c} (sum_t G[t,r] A[t,c])^2
//   clipped sum: out = beta*out + sum_i R_i G_i^T A_i          (inner sum of Eq. 3)
#include <algorithm>

#include "dp_common.cuh"
#include "fma_kernels.cuh"
#include "gemm_gta.cuh"
#include "noise_device.cuh"

namespace dpg {

namespace {

// One block per example, one warp per pair of tokens at a time.  Bound by the latency of its loads and
// reductions: 1024 threads against 256 at B = 4, T = 16, d = p = 64: 15.1 -> 7.5 us.
constexpr int kNormThreads = 1024;

// sum over the pairs of tokens of one example of (a_t.a_s over columns [a0, a1)) * (g_t.g_s over [g0, g1)); in thread 0
template <typename T>
__device__ __forceinline__ float pairs_sum(const T* Ai, long long lda, int a0, int a1, const T* Gi, long long ldg, int g0, int g1,
                                           int Tn, float* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const long long npairs = (long long)Tn * (Tn + 1) / 2;
  float acc = 0.f;
  int t = 0, s = 0;                       // pair index -> (t, s), s >= t, walked incrementally
  long long cur = 0;
  for (long long pr = w; pr < npairs; pr += nw) {
    while (cur < pr) {                    // advance the (t, s) cursor to pair pr
      const long long left = Tn - s - 1;  // pairs left in row t after (t, s)
      const long long jump = pr - cur;
      if (jump <= left) { s += (int)jump; cur = pr; }
      else { cur += left + 1; ++t; s = t; }
    }
    float da = 0.f, dg = 0.f;
#pragma unroll 4
    for (int k = a0 + lane; k < a1; k += 32) da = fmaf(to_f32(Ai[t * lda + k]), to_f32(Ai[s * lda + k]), da);
#pragma unroll 4
    for (int k = g0 + lane; k < g1; k += 32) dg = fmaf(to_f32(Gi[t * ldg + k]), to_f32(Gi[s * ldg + k]), dg);
    da = warp_sum(da);
    dg = warp_sum(dg);
    acc += (t == s ? 1.f : 2.f) * da * dg;
  }
  return block_sum(lane == 0 ? acc : 0.f, red);
}

template <typename T>
__global__ void __launch_bounds__(kNormThreads)
ghost_norm_fma_kernel(const T* __restrict__ A, long long lda, int d,
                                      const T* __restrict__ G, long long ldg, int p, int Tn,
                                      float* __restrict__ sq, int overwrite) {
  __shared__ float red[32];
  const int i = blockIdx.x;
  const float tot = pairs_sum(A + size_t(i) * Tn * lda, lda, 0, d, G + size_t(i) * Tn * ldg, ldg, 0, p, Tn, red);
  if (threadIdx.x == 0) sq[i] = (overwrite ? 0.f : sq[i]) + tot;
}

template <typename T>
__global__ void __launch_bounds__(kNormThreads)
direct_norm_fma_kernel(const T* __restrict__ A, long long lda, int d,
                                       const T* __restrict__ G, long long ldg, int p, int Tn,
                                       float* __restrict__ sq, int overwrite) {
  __shared__ float red[32];
  const int i = blockIdx.x;
  const T* Ai = A + size_t(i) * Tn * lda;
  const T* Gi = G + size_t(i) * Tn * ldg;
  const long long n = (long long)d * p;
  float acc = 0.f;
  for (long long e = threadIdx.x; e < n; e += blockDim.x) {
    const int r = int(e / d), c = int(e - (long long)r * d);
    float v = 0.f;
    for (int t = 0; t < Tn; ++t) v = fmaf(to_f32(Gi[t * ldg + r]), to_f32(Ai[t * lda + c]), v);
    acc = fmaf(v, v, acc);
  }
  const float tot = block_sum(acc, red);
  if (threadIdx.x == 0) sq[i] = (overwrite ? 0.f : sq[i]) + tot;
}

// Clipped sums of several layers in one launch.  kTile x kTile output tile per block of 256 threads, kStep
// token rows per shared-memory step; the rows of the next step are in flight while a step is multiplied,
// 16-byte shared loads feed 16 FMAs each pair (bound by FMAs; 4-byte loads bound it by shared memory).
// The noise of Eq. 3 (amp >= 0) is drawn here where a Philox counter covers four columns of one row (d a
// multiple of 4).  Tiles of 64 where they fill the chip; 32 where that many would leave SMs idle.  A last step of few rows ends
// with them, and a thread's outputs leave in one store: 768 -> 50257 at one token 71 -> 52 us (64 before the one launch).
// B = 4, T = 16, d = p = 64, sum and noise: 10.0 + 2.1 -> 5.5 us in one launch instead of two.
constexpr int kFmaMaxLayers = 64;
struct FmaSumLayer {
  const void *A, *G;
  float* out;
  long long lda, ldg, ldo;
  int d, p, tile_begin, tiles_n;
  float amp;                 // sigma*C of the fused noise, negative = none
  uint32_t tensor_id;
};
struct FmaSumParams {
  FmaSumLayer layer[kFmaMaxLayers];
  int n, B, T;
  const float* clip;
  float beta, scale;
  NoiseKeys keys;
  uint32_t step;
  const uint32_t* step_dev;
};

// last entry whose `begin` is not above `at`
template <typename L, typename F>
__device__ __forceinline__ const L& find_layer(const L* layer, int n, int at, F begin) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (at >= begin(layer[mid])) lo = mid; else hi = mid - 1;
  }
  return layer[lo];
}

template <typename T, int kTile>
__global__ void __launch_bounds__(256)
clip_accumulate_fma_kernel(const __grid_constant__ FmaSumParams P) {
  constexpr int kStep = 1024 / kTile, kPer = 4;            // rows per step; values per thread and operand
  constexpr int kRowsApart = 256 / kTile;                  // rows between a thread's values
  constexpr int kR = kTile / 16;                           // outputs per thread and direction
  __shared__ __align__(16) float Gs[kStep][kTile + 4];
  __shared__ __align__(16) float As[kStep][kTile + 4];
  const FmaSumLayer& L = find_layer(P.layer, P.n, int(blockIdx.x), [](const FmaSumLayer& x) { return x.tile_begin; });
  const int tile = int(blockIdx.x) - L.tile_begin;
  const int m0 = tile / L.tiles_n * kTile, n0 = tile % L.tiles_n * kTile;
  const T* A = static_cast<const T*>(L.A);
  const T* G = static_cast<const T*>(L.G);
  const int d = L.d, p = L.p, Tn = P.T;
  const long long lda = L.lda, ldg = L.ldg;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int lr = threadIdx.x / kTile, lc = threadIdx.x % kTile;
  const long long K = (long long)P.B * Tn;
  float acc[kR][kR] = {};
  float g[kPer], a[kPer];
  int ex = lr / Tn, t = lr - ex * Tn;                      // example and token of this thread's first row
  auto load = [&](long long k0) {
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const long long k = k0 + lr + kRowsApart * j;
      int e = ex, tt = t + kRowsApart * j;
      while (tt >= Tn) { tt -= Tn; ++e; }
      g[j] = 0.f; a[j] = 0.f;
      if (k < K) {
        if (m0 + lc < p) g[j] = P.clip[e] * to_f32(G[k * ldg + m0 + lc]);
        if (n0 + lc < d) a[j] = to_f32(A[k * lda + n0 + lc]);
      }
    }
    t += kStep;
    while (t >= Tn) { t -= Tn; ++ex; }
  };
  load(0);
  for (long long k0 = 0; k0 < K; k0 += kStep) {
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      Gs[lr + kRowsApart * j][lc] = g[j];
      As[lr + kRowsApart * j][lc] = a[j];
    }
    __syncthreads();
    if (k0 + kStep < K) load(k0 + kStep);
    auto product = [&](int kk) {
      float gv[kR], av[kR];
      if constexpr (kR == 4) {
        const float4 x = *reinterpret_cast<const float4*>(&Gs[kk][ty * 4]), y = *reinterpret_cast<const float4*>(&As[kk][tx * 4]);
        gv[0] = x.x; gv[1] = x.y; gv[2] = x.z; gv[3] = x.w;
        av[0] = y.x; av[1] = y.y; av[2] = y.z; av[3] = y.w;
      } else {
        const float2 x = *reinterpret_cast<const float2*>(&Gs[kk][ty * 2]), y = *reinterpret_cast<const float2*>(&As[kk][tx * 2]);
        gv[0] = x.x; gv[1] = x.y;
        av[0] = y.x; av[1] = y.y;
      }
#pragma unroll
      for (int r = 0; r < kR; ++r)
#pragma unroll
        for (int c = 0; c < kR; ++c) acc[r][c] = fmaf(gv[r], av[c], acc[r][c]);
    };
    if (K - k0 >= kStep) {
#pragma unroll
      for (int kk = 0; kk < kStep; ++kk) product(kk);
    } else {
#pragma unroll 4
      for (int kk = 0; kk < int(K - k0); ++kk) product(kk);      // the rest is zeros
    }
    __syncthreads();
  }
  const float amp = L.amp;
  const uint32_t step = amp >= 0.f ? effective_step(P.step, P.step_dev) : 0u;
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    const int row = m0 + ty * kR + r, col = n0 + tx * kR;
    if (row >= p || col >= d) continue;
    float* o = L.out + size_t(row) * L.ldo + col;
    if (P.beta != 0.f) {
#pragma unroll
      for (int c = 0; c < kR; ++c) if (col + c < d) acc[r][c] += o[c];
    }
    if (amp >= 0.f) {
      float z[4];                                          // d % 4 == 0: all in one row
      normals4(((unsigned long long)row * d + col) >> 2, P.keys, L.tensor_id, step, z);
#pragma unroll
      for (int c = 0; c < kR; ++c)
        acc[r][c] = noised(acc[r][c], kR == 4 ? z[c] : z[c + (col & 2)], amp, P.scale);
    }
    // a thread's outputs lie side by side: stored one by one they are a quarter of a sector each
    if (col + kR <= d && (reinterpret_cast<uintptr_t>(o) & (4 * kR - 1)) == 0) {
      if constexpr (kR == 4) *reinterpret_cast<float4*>(o) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
      else *reinterpret_cast<float2*>(o) = make_float2(acc[r][0], acc[r][1]);
    } else {
#pragma unroll
      for (int c = 0; c < kR; ++c) if (col + c < d) o[c] = acc[r][c];
    }
  }
}

// Ghost norms of several layers in one launch, in fp32: a work item is the product of one pair (ti <= tj) of
// 32-token tiles of the two Gram matrices of a (layer, example), over all columns of the narrower operand
// and a chunk of the wider one's (the product is linear in each).  256 threads, 2 x 2 entries each; columns
// go through shared memory 32 at a time, transposed, the next 32 in flight.  Bound by shared-memory
// loads.  With one block per example, a warp per pair of tokens and, as for the sums, a launch per layer the
// step of three blocks of d = 64 with V = 8064 at B = 2, T = 29 took 616 us, now 72; five of d = 640 at B = 16, T = 26
// 2918, now 1010 (most of it the sums' FMAs).  Those kernels remain for a workspace without room for the
// partial sums.
// Very short sequences (gram_by_pairs) fill little of a tile, whose walk over the columns takes as long as ever: there an
// item is all pairs of tokens, a warp each (gram_pairs_fma_kernel): one layer of 768 -> 3072 at B = 4, T = 16 67 -> 23 us, 24 layers of
// DistilGPT2 at B = 32, T = 16 364 -> 194 (829 with a launch per layer).
constexpr int kGramTile = 32, kGramChunk = 2048;     // tokens per tile; columns per item of the wider operand
struct FmaNormLayer {
  const void *A, *G;
  long long lda, ldg;
  int d, p, nsplit, item_begin, col_begin;
};
struct FmaNormParams {
  FmaNormLayer layer[kFmaMaxLayers];
  int n, B, T, nt, ntp, n_per;
  float* partials;           // [B][n_per]
};

// entries (2 ty .. 2 ty + 1) x (2 tx .. 2 tx + 1) of the product of two 32-row tiles over columns [c0, c1)
template <typename T>
__device__ __forceinline__ void gram_tile(const T* X, long long ld, int ri, int rj, int rows, int c0, int c1,
                                          float (&s)[2][2], float (*xi)[kGramTile + 2], float (*xj)[kGramTile + 2]) {
  const int lr = threadIdx.x >> 5, lc = threadIdx.x & 31;          // rows lr, lr + 8, ...
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const bool two = ri != rj;
  float u[4], v[4];
  auto load = [&](int c) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = lr + 8 * j;
      const bool in = c + lc < c1;
      u[j] = in && ri + r < rows ? to_f32(X[(ri + r) * ld + c + lc]) : 0.f;
      v[j] = two && in && rj + r < rows ? to_f32(X[(rj + r) * ld + c + lc]) : 0.f;
    }
  };
  s[0][0] = s[0][1] = s[1][0] = s[1][1] = 0.f;
  load(c0);
  for (int c = c0; c < c1; c += 32) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      xi[lc][lr + 8 * j] = u[j];
      if (two) xj[lc][lr + 8 * j] = v[j];
    }
    __syncthreads();
    if (c + 32 < c1) load(c + 32);
    float (*y)[kGramTile + 2] = two ? xj : xi;
    float part[2][2] = {};                                         // 32 columns by themselves: shorter chains
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const float2 p = *reinterpret_cast<const float2*>(&xi[k][2 * ty]), q = *reinterpret_cast<const float2*>(&y[k][2 * tx]);
      part[0][0] = fmaf(p.x, q.x, part[0][0]);
      part[0][1] = fmaf(p.x, q.y, part[0][1]);
      part[1][0] = fmaf(p.y, q.x, part[1][0]);
      part[1][1] = fmaf(p.y, q.y, part[1][1]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) s[e >> 1][e & 1] += part[e >> 1][e & 1];
    __syncthreads();
  }
}

template <typename T>
__global__ void __launch_bounds__(256, 4)
gram_norm_fma_kernel(const __grid_constant__ FmaNormParams P) {
  __shared__ __align__(16) float xi[32][kGramTile + 2], xj[32][kGramTile + 2];
  __shared__ float red[32];
  const FmaNormLayer& L = find_layer(P.layer, P.n, int(blockIdx.x), [](const FmaNormLayer& x) { return x.item_begin; });
  int local = int(blockIdx.x) - L.item_begin;
  const int sp = local % L.nsplit;
  local /= L.nsplit;
  const int tp = local % P.ntp, i = local / P.ntp;
  int ti = 0, rem = tp;                                            // tile pairs row by row, tj >= ti
  while (rem >= P.nt - ti) { rem -= P.nt - ti; ++ti; }
  const int ri = ti * kGramTile, rj = (ti + rem) * kGramTile;
  const T* A = static_cast<const T*>(L.A) + size_t(i) * P.T * L.lda;
  const T* G = static_cast<const T*>(L.G) + size_t(i) * P.T * L.ldg;
  const bool wide_g = L.p >= L.d;
  const int lo = sp * kGramChunk, hi = min(wide_g ? L.p : L.d, lo + kGramChunk);
  float sa[2][2], sg[2][2];
  gram_tile(A, L.lda, ri, rj, P.T, wide_g ? 0 : lo, wide_g ? L.d : hi, sa, xi, xj);
  gram_tile(G, L.ldg, ri, rj, P.T, wide_g ? lo : 0, wide_g ? hi : L.p, sg, xi, xj);
  float acc = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) acc = fmaf(sa[e >> 1][e & 1], sg[e >> 1][e & 1], acc);
  const float tot = block_sum(acc, red);
  if (threadIdx.x == 0) P.partials[size_t(i) * P.n_per + L.col_begin + tp * L.nsplit + sp] = ri == rj ? tot : 2.f * tot;
}

template <typename T>
__global__ void __launch_bounds__(kNormThreads)
gram_pairs_fma_kernel(const __grid_constant__ FmaNormParams P) {
  __shared__ float red[32];
  const FmaNormLayer& L = find_layer(P.layer, P.n, int(blockIdx.x), [](const FmaNormLayer& x) { return x.item_begin; });
  const int local = int(blockIdx.x) - L.item_begin, sp = local % L.nsplit, i = local / L.nsplit;
  const bool wide_g = L.p >= L.d;
  const int lo = sp * kGramChunk, hi = min(wide_g ? L.p : L.d, lo + kGramChunk);
  const float tot = pairs_sum(static_cast<const T*>(L.A) + size_t(i) * P.T * L.lda, L.lda, wide_g ? 0 : lo, wide_g ? L.d : hi,
                              static_cast<const T*>(L.G) + size_t(i) * P.T * L.ldg, L.ldg, wide_g ? lo : 0, wide_g ? hi : L.p, P.T, red);
  if (threadIdx.x == 0) P.partials[size_t(i) * P.n_per + L.col_begin + sp] = tot;
}

// <g_in_i, g_out_i> = sum_{t,s} G_lm[i,s,id_t] * (g_emb_t . a_lm_s)   (expansion of Eq. 11's
// inner product); one block per (example, 16-token slab of t), one warp per (t, s) pair.
template <typename T>
__global__ void cross_term_fma_kernel(const int* __restrict__ ids, const T* __restrict__ Ge,
                                      long long ldge, const T* __restrict__ Al, long long ldal,
                                      const T* __restrict__ Gl, long long ldgl, int Tn, int d, int V,
                                      int slabs, float* __restrict__ partials,
                                      int* __restrict__ dev_status) {
  __shared__ float red[32];
  const int i = blockIdx.x / slabs, slab = blockIdx.x % slabs;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int t_lo = slab * 16, t_hi = min(Tn, t_lo + 16);
  float acc = 0.f;
  for (int t = t_lo; t < t_hi; ++t) {
    const int id = ids[size_t(i) * Tn + t];
    if (id < 0 || id >= V) {
      if (threadIdx.x == 0 && dev_status) atomicOr(dev_status, DP_DEV_BAD_ID);
      continue;
    }
    const T* g = Ge + (size_t(i) * Tn + t) * ldge;
    for (int s = w; s < Tn; s += nw) {
      const T* a = Al + (size_t(i) * Tn + s) * ldal;
      float dot = 0.f;
      for (int k = lane; k < d; k += 32) dot = fmaf(to_f32(g[k]), to_f32(a[k]), dot);
      dot = warp_sum(dot);
      acc = fmaf(to_f32(Gl[(size_t(i) * Tn + s) * ldgl + id]), dot, acc);
    }
  }
  const float tot = block_sum(lane == 0 ? acc : 0.f, red);
  if (threadIdx.x == 0) partials[blockIdx.x] = tot;
}

// extra: added to sq first
__global__ void clip_factors_kernel(const float* sq, const float* __restrict__ extra, float* sum,
                                    int B, float C, float* __restrict__ clip, float* __restrict__ norms) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B) return;
  float s = sq[i];
  if (extra) { s += extra[i]; sum[i] = s; }
  if (clip) clip[i] = clip_from_sq(s, C);
  if (norms) norms[i] = __fsqrt_rn(s);
}

// All partial sums of a step's norms and Eq. 7, one warp per example: the additions, and their order, of
// reduce_partials_kernel once per source and clip_factors_kernel.  A launch in the chain between the norm
// kernels and the GEMM takes 5 to 6 us with its gap: the step of one 64 x 64 layer 51.7 -> 49.1 us, DistilGPT2 B = 32, T = 128 896 -> 887.
__global__ void __launch_bounds__(128)
finish_norms_kernel(const __grid_constant__ NormSources S, int B, float C, float* __restrict__ sq,
                    float* __restrict__ clip, float* __restrict__ norms) {
  const int i = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= B) return;
  float total[2] = {0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    if (k >= S.n) break;
    const NormSource& q = S.src[k];
    const float* p = q.partials + size_t(i) * q.n_per;
    float s = 0.f;
#pragma unroll 8
    for (int j = lane; j < q.n_per; j += 32) s += p[j];
    s = warp_sum(s);
    if (q.plain_out && lane == 0) q.plain_out[i] = s;
    if (k < S.n_main) total[0] += q.factor * s; else total[1] += q.factor * s;
  }
  if (lane == 0) {
    const float s = total[0] + total[1];
    sq[i] = s;
    if (clip) clip[i] = clip_from_sq(s, C);
    if (norms) norms[i] = __fsqrt_rn(s);
  }
}

}  // namespace

template <typename T>
static dp_status norms_fma_t(const dp_linear_desc& L, int mode, int B, int Tn, float* sq,
                             cudaStream_t st, int overwrite) {
  if (mode == DP_NORM_GHOST)
    ghost_norm_fma_kernel<T><<<B, kNormThreads, 0, st>>>((const T*)L.A, L.lda, L.d, (const T*)L.G, L.ldg,
                                               L.p, Tn, sq, overwrite);
  else
    direct_norm_fma_kernel<T><<<B, kNormThreads, 0, st>>>((const T*)L.A, L.lda, L.d, (const T*)L.G, L.ldg,
                                                L.p, Tn, sq, overwrite);
  DP_LAUNCH_OK();
  return DP_OK;
}

dp_status launch_norms_fma(const dp_linear_desc& L, dp_dtype dt, int mode, int B, int T, float* sq,
                           cudaStream_t st, bool overwrite) {
  return dt == DP_F32 ? norms_fma_t<float>(L, mode, B, T, sq, st, overwrite)
                      : norms_fma_t<__nv_bfloat16>(L, mode, B, T, sq, st, overwrite);
}

dp_status launch_clip_accumulate_fma(const dp_linear_desc* layers, const int* index, int n, dp_dtype dt, int B, int T,
                                     const float* clip, float* const* outs, const int64_t* ldos, float beta,
                                     const GtaNoise* noise, cudaStream_t st) {
  long long wide_tiles = 0;
  for (int k = 0; k < n; ++k)
    wide_tiles += (long long)ceil_div(layers[index[k]].d, 64) * ceil_div(layers[index[k]].p, 64);
  const int tile = wide_tiles >= sm_count() ? 64 : 32;
  for (int k0 = 0; k0 < n; k0 += kFmaMaxLayers) {
    FmaSumParams P;
    P.n = std::min(n - k0, kFmaMaxLayers);
    P.B = B; P.T = T; P.clip = clip; P.beta = beta; P.scale = noise ? noise->scale : 1.f;
    P.keys = expand_noise_keys(noise ? noise->seed : 0);
    P.step = noise ? noise->step : 0; P.step_dev = g_step_dev;
    long long tiles = 0;
    for (int k = 0; k < P.n; ++k) {
      const int l = index[k0 + k];
      const dp_linear_desc& D = layers[l];
      const bool fused = noise && D.d % 4 == 0;
      P.layer[k] = {D.A, D.G, outs[l], D.lda, D.ldg, ldos[l], D.d, D.p, int(tiles), ceil_div(D.d, tile),
                    fused ? noise->amp : -1.f, noise ? noise->tensor_ids[l] : 0u};
      tiles += (long long)ceil_div(D.d, tile) * ceil_div(D.p, tile);
    }
    if (tiles > 0x7fffffffLL) return DP_ERR_UNSUPPORTED;
    const unsigned grid = (unsigned)tiles;
    if (dt == DP_F32) {
      if (tile == 64) clip_accumulate_fma_kernel<float, 64><<<grid, 256, 0, st>>>(P);
      else clip_accumulate_fma_kernel<float, 32><<<grid, 256, 0, st>>>(P);
    } else {
      if (tile == 64) clip_accumulate_fma_kernel<__nv_bfloat16, 64><<<grid, 256, 0, st>>>(P);
      else clip_accumulate_fma_kernel<__nv_bfloat16, 32><<<grid, 256, 0, st>>>(P);
    }
    DP_LAUNCH_OK();
    for (int k = 0; k < P.n && noise; ++k) {
      const int l = index[k0 + k];
      if (layers[l].d % 4 == 0) continue;
      const dp_status s = launch_add_noise(outs[l], layers[l].p, layers[l].d, ldos[l], false, noise->amp, noise->scale,
                                           noise->seed, noise->tensor_ids[l], noise->step, st);
      if (s != DP_OK) return s;
    }
  }
  return DP_OK;
}

int gram_fma_partials(const dp_linear_desc& L, int T) {
  const int nt = ceil_div(T, kGramTile);
  return nt * (nt + 1) / 2 * ceil_div(std::max(L.d, L.p), kGramChunk);
}

// All pairs of tokens per item, or tiles.  A tile takes about as long whatever the tokens, pairs do not (d = p = 64: 6.4 and 7.6 us at 8
// tokens, 7.8 and 7.7 at 12; 24 layers of DistilGPT2 at B = 32: 255 and 370 at 20, about 340 and 374 at 24).
static bool gram_by_pairs(int T, int widest) { return T <= (widest >= 512 ? 24 : 12); }

bool gram_alone_fma(const dp_linear_desc& L, int T) { return std::max(L.d, L.p) >= 512 && gram_fma_partials(L, T) == 1; }

dp_status launch_gram_norms_fma(const dp_linear_desc* layers, const int* index, int n, dp_dtype dt, int B, int T,
                                float* partials, int n_per, cudaStream_t st) {
  int col = 0, widest = 0;
  for (int k = 0; k < n; ++k) widest = std::max(widest, std::max(layers[index[k]].d, layers[index[k]].p));
  const bool pairs = gram_by_pairs(T, widest);
  for (int k0 = 0; k0 < n; k0 += kFmaMaxLayers) {
    FmaNormParams P;
    P.n = std::min(n - k0, kFmaMaxLayers);
    P.B = B; P.T = T; P.nt = ceil_div(T, kGramTile); P.ntp = P.nt * (P.nt + 1) / 2;
    P.n_per = n_per; P.partials = partials;
    long long items = 0;
    for (int k = 0; k < P.n; ++k) {
      const dp_linear_desc& D = layers[index[k0 + k]];
      const int nsplit = ceil_div(std::max(D.d, D.p), kGramChunk);
      P.layer[k] = {D.A, D.G, D.lda, D.ldg, D.d, D.p, nsplit, int(items), col};
      items += (long long)B * P.ntp * nsplit;
      col += P.ntp * nsplit;
    }
    if (items > 0x7fffffffLL) return DP_ERR_UNSUPPORTED;
    if (pairs) {
      if (dt == DP_F32) gram_pairs_fma_kernel<float><<<(unsigned)items, kNormThreads, 0, st>>>(P);
      else gram_pairs_fma_kernel<__nv_bfloat16><<<(unsigned)items, kNormThreads, 0, st>>>(P);
    } else {
      if (dt == DP_F32) gram_norm_fma_kernel<float><<<(unsigned)items, 256, 0, st>>>(P);
      else gram_norm_fma_kernel<__nv_bfloat16><<<(unsigned)items, 256, 0, st>>>(P);
    }
    DP_LAUNCH_OK();
  }
  return DP_OK;
}

dp_status launch_cross_term_fma(const int* ids, const void* Ge, int64_t ldge, const void* Al,
                                int64_t ldal, const void* Gl, int64_t ldgl, dp_dtype dt, int B,
                                int T, int d, int V, float* partials, int* dev_status,
                                cudaStream_t st) {
  const int slabs = ceil_div(T, 16);
  if (dt == DP_F32)
    cross_term_fma_kernel<float><<<B * slabs, 256, 0, st>>>(ids, (const float*)Ge, ldge,
                                                          (const float*)Al, ldal, (const float*)Gl,
                                                          ldgl, T, d, V, slabs, partials, dev_status);
  else
    cross_term_fma_kernel<__nv_bfloat16><<<B * slabs, 256, 0, st>>>(
        ids, (const __nv_bfloat16*)Ge, ldge, (const __nv_bfloat16*)Al, ldal,
        (const __nv_bfloat16*)Gl, ldgl, T, d, V, slabs, partials, dev_status);
  DP_LAUNCH_OK();
  return DP_OK;
}

dp_status launch_clip_factors(const float* sq, int B, float C, float* clip, float* norms,
                              cudaStream_t st, const float* extra, float* sum) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&launch_clip_factors)))
    DP_CUDA_OK(prefer_max_shared(clip_factors_kernel));
  clip_factors_kernel<<<ceil_div(B, 128), 128, 0, st>>>(sq, extra, sum, B, C, clip, norms);
  DP_LAUNCH_OK();
  return DP_OK;
}

dp_status launch_finish_norms(const NormSources& S, int B, float C, float* sq, float* clip, float* norms,
                              cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&launch_finish_norms)))
    DP_CUDA_OK(prefer_max_shared(finish_norms_kernel));
  finish_norms_kernel<<<ceil_div(B, 4), 128, 0, st>>>(S, B, C, sq, clip, norms);
  DP_LAUNCH_OK();
  return DP_OK;
}

}  // namespace dpg
