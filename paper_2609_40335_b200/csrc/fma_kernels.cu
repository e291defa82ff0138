// fp32-FMA kernels for linear layers: the DP_F32 path (fp32 tensors need better than TF32
// accuracy) and the cross-check path for DP_BF16.  Any shape, no alignment rules.
//   ghost  : sq[i] += sum_{t,s} (a_t.a_s)(g_t.g_s)            (Eq. 4 - Eq. 5 over T tokens)
//   direct : sq[i] += sum_{r,c} (sum_t G[t,r] A[t,c])^2
//   clipped sum: out = beta*out + sum_i R_i G_i^T A_i          (inner sum of Eq. 3)
#include "dp_common.cuh"
#include "fma_kernels.cuh"
#include "gemm_gta.cuh"
#include "noise_device.cuh"

namespace dpg {

namespace {

// One block per example, one warp per pair of tokens at a time.  Bound by the latency of its loads and
// reductions: 1024 threads against 256 at B = 4, T = 16, d = p = 64: 15.1 -> 7.5 us.
constexpr int kNormThreads = 1024;

template <typename T>
__global__ void __launch_bounds__(kNormThreads)
ghost_norm_fma_kernel(const T* __restrict__ A, long long lda, int d,
                                      const T* __restrict__ G, long long ldg, int p, int Tn,
                                      float* __restrict__ sq, int overwrite) {
  __shared__ float red[32];
  const int i = blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const T* Ai = A + size_t(i) * Tn * lda;
  const T* Gi = G + size_t(i) * Tn * ldg;
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
    for (int k = lane; k < d; k += 32) da = fmaf(to_f32(Ai[t * lda + k]), to_f32(Ai[s * lda + k]), da);
#pragma unroll 4
    for (int k = lane; k < p; k += 32) dg = fmaf(to_f32(Gi[t * ldg + k]), to_f32(Gi[s * ldg + k]), dg);
    da = warp_sum(da);
    dg = warp_sum(dg);
    acc += (t == s ? 1.f : 2.f) * da * dg;
  }
  const float tot = block_sum(lane == 0 ? acc : 0.f, red);
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

// kTile x kTile output tile per block of 256 threads, kStep token rows per shared-memory step; the rows of
// the next step are in flight while a step is multiplied.  The noise of Eq. 3 (amp >= 0) is drawn here
// where a Philox counter covers four columns of one row (d a multiple of 4).  Tiles of 64 where they fill the
// chip; 32 where that many would leave SMs idle.  B = 4, T = 16, d = p = 64, sum and noise: 10.0 + 2.1 -> 5.5 us in one
// launch instead of two.
template <typename T, int kTile>
__global__ void __launch_bounds__(256)
clip_accumulate_fma_kernel(const T* __restrict__ A, long long lda, int d, const T* __restrict__ G,
                           long long ldg, int p, int B, int Tn, const float* __restrict__ clip,
                           float* __restrict__ out, long long ldo, float beta, float amp, float scale,
                           const __grid_constant__ NoiseKeys keys, uint32_t tensor_id, uint32_t step,
                           const uint32_t* __restrict__ step_dev) {
  constexpr int kStep = 1024 / kTile, kPer = 4;            // rows per step; values per thread and operand
  constexpr int kRowsApart = 256 / kTile;                  // rows between a thread's values
  constexpr int kR = kTile / 16;                           // outputs per thread and direction
  __shared__ float Gs[kStep][kTile + 1];
  __shared__ float As[kStep][kTile + 1];
  const int m0 = blockIdx.y * kTile, n0 = blockIdx.x * kTile;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int lr = threadIdx.x / kTile, lc = threadIdx.x % kTile;
  const long long K = (long long)B * Tn;
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
        if (m0 + lc < p) g[j] = clip[e] * to_f32(G[k * ldg + m0 + lc]);
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
#pragma unroll
    for (int kk = 0; kk < kStep; ++kk) {
      float gv[kR], av[kR];
#pragma unroll
      for (int j = 0; j < kR; ++j) { gv[j] = Gs[kk][ty * kR + j]; av[j] = As[kk][tx * kR + j]; }
#pragma unroll
      for (int r = 0; r < kR; ++r)
#pragma unroll
        for (int c = 0; c < kR; ++c) acc[r][c] = fmaf(gv[r], av[c], acc[r][c]);
    }
    __syncthreads();
  }
  if (amp >= 0.f) step = effective_step(step, step_dev);
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    const int row = m0 + ty * kR + r, col = n0 + tx * kR;
    if (row >= p || col >= d) continue;
    float* o = out + size_t(row) * ldo + col;
    if (beta != 0.f) {
#pragma unroll
      for (int c = 0; c < kR; ++c) if (col + c < d) acc[r][c] += o[c];
    }
    if (amp >= 0.f) {
      float z[4];                                          // d % 4 == 0: all in one row
      normals4(((unsigned long long)row * d + col) >> 2, keys, tensor_id, step, z);
#pragma unroll
      for (int c = 0; c < kR; ++c)
        acc[r][c] = noised(acc[r][c], kR == 4 ? z[c] : z[c + (col & 2)], amp, scale);
    }
#pragma unroll
    for (int c = 0; c < kR; ++c) if (col + c < d) o[c] = acc[r][c];
  }
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

__global__ void clip_factors_kernel(const float* __restrict__ sq, int B, float C,
                                    float* __restrict__ clip, float* __restrict__ norms) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B) return;
  const float s = sq[i];
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

namespace {

template <typename T, int kTile>
dp_status clip_fma_t(const dp_linear_desc& L, int B, int Tn, const float* clip, float* out, int64_t ldo,
                     float beta, const GtaNoise* noise, uint32_t tensor_id, cudaStream_t st) {
  const dim3 grid(ceil_div(L.d, kTile), ceil_div(L.p, kTile));
  clip_accumulate_fma_kernel<T, kTile><<<grid, 256, 0, st>>>(
      (const T*)L.A, L.lda, L.d, (const T*)L.G, L.ldg, L.p, B, Tn, clip, out, ldo, beta, noise ? noise->amp : -1.f,
      noise ? noise->scale : 1.f, expand_noise_keys(noise ? noise->seed : 0), tensor_id, noise ? noise->step : 0,
      g_step_dev);
  DP_LAUNCH_OK();
  return DP_OK;
}

}  // namespace

dp_status launch_clip_accumulate_fma(const dp_linear_desc& L, dp_dtype dt, int B, int T, const float* clip,
                                     float* out, int64_t ldo, float beta, const GtaNoise* noise,
                                     uint32_t tensor_id, cudaStream_t st) {
  const GtaNoise* fused = noise && L.d % 4 == 0 ? noise : nullptr;
  const bool wide = (long long)ceil_div(L.d, 64) * ceil_div(L.p, 64) >= sm_count();
  dp_status s;
  if (dt == DP_F32)
    s = wide ? clip_fma_t<float, 64>(L, B, T, clip, out, ldo, beta, fused, tensor_id, st)
             : clip_fma_t<float, 32>(L, B, T, clip, out, ldo, beta, fused, tensor_id, st);
  else
    s = wide ? clip_fma_t<__nv_bfloat16, 64>(L, B, T, clip, out, ldo, beta, fused, tensor_id, st)
             : clip_fma_t<__nv_bfloat16, 32>(L, B, T, clip, out, ldo, beta, fused, tensor_id, st);
  if (s != DP_OK || !noise || fused) return s;
  return launch_add_noise(out, L.p, L.d, ldo, false, noise->amp, noise->scale, noise->seed, tensor_id, noise->step,
                          st);
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
                              cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&launch_clip_factors)))
    DP_CUDA_OK(prefer_max_shared(clip_factors_kernel));
  clip_factors_kernel<<<ceil_div(B, 128), 128, 0, st>>>(sq, B, C, clip, norms);
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
