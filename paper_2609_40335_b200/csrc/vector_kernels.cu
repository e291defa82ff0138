// Parameters that act element-wise along the feature axis: biases and LayerNorm gains / shifts.
//
// A bias b in z = W a + b sees the back-propagated signal of every token (Eq. 4 with a constant
// input 1), so its per-example gradient is v_i = sum_t G[i,t,:]; a LayerNorm gain sees
// v_i = sum_t G[i,t,:] * X[i,t,:] with X the normalised input and G the gradient at the
// LayerNorm output (its shift is a bias).  These kernels give
//     norms:        sq[i] += || v_i ||^2                                   (one more block of Eq. 6)
//     clipped sum:  out = beta*out + sum_i R_i v_i  [+ Gaussian noise]      (Eq. 3)
// Both are single streaming passes over G (and X): HBM-bound, 2*T*p (or 4*T*p) bytes per example.  Within one step
// the norms pass writes its v_i down (4*p bytes per example, 1/(T/2) of what it reads) and the clipped sum is a sum
// over examples of those, so G and X are read once.  DistilGPT2 with all its vectors at B = 21, T = 203: clipped sums
// 131 us at the end of the step -> a few beside the GEMM, step 1265 -> 1150 us.
// Summation orders are fixed (warp w takes rows w, w+8, ...; partial sums are combined in
// warp / split order), so results are deterministic.
#include <algorithm>
#include <cstring>

#include "dp_common.cuh"
#include "noise_device.cuh"
#include "vector_kernels.cuh"

namespace dpg {

namespace {

constexpr int kVecCols = 256;        // columns per block (8 per lane)
// 16-byte row loads in flight per lane: eight G rows for a bias, four G and four X rows for a
// LayerNorm gain (kept unconverted: 32 registers), so that four 256-thread blocks
// (<= 64 registers per thread) fit on an SM
constexpr int kVecBatchBias = 8;
constexpr int kVecBatchGain = 4;

struct VecParam {
  const void* G;
  const void* X;          // multiplier or nullptr
  long long ldg, ldx;
  float* out;             // clipped-sum destination (p floats)
  int p;
  int slab_begin;         // first 256-column slab of this parameter in the launch
  int col_begin;          // first column of this parameter in the concatenated partial rows
  uint32_t tensor_id;
};

struct VecParams {
  VecParam prm[kVecMaxParams];
  int n, B, T;
  int total_slabs, total_cols;
};

__device__ __forceinline__ int find_param(const VecParams& P, int slab) {
  int lo = 0, hi = P.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (slab >= P.prm[mid].slab_begin) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// sum over the rows [r0, r1) (stride 8 from warp w) of weight(row) * G[row, cols] * X[row, cols].
// All loads of a batch are issued before any is consumed; rows past r1 re-read row r1-1 with
// weight 0, so the loads are unconditional.  The example of a row (for its clip factor) is
// tracked by stepping, not by a division per row.
template <typename T, bool kWeighted, bool kHasX>
__device__ __forceinline__ void stream_rows_t(const VecParam& q, long long row_base, int r0, int r1,
                                              int c, int nvalid, int Tn, const float* clip,
                                              float (&acc)[8]) {
  // fp32 chunks are twice as large in registers: half the batch
  constexpr int kBatch = (kHasX ? kVecBatchGain : kVecBatchBias) / (sizeof(T) == 2 ? 1 : 2);
  const int w = threadIdx.x >> 5;
  if (r0 + w >= r1) return;
  const T* G = static_cast<const T*>(q.G) + row_base * q.ldg + c;
  const T* X = kHasX ? static_cast<const T*>(q.X) + row_base * q.ldx + c : nullptr;
  const bool gvec = ((reinterpret_cast<uintptr_t>(q.G) & 15) == 0) && ((q.ldg * sizeof(T)) % 16 == 0);
  const bool xvec = kHasX && ((reinterpret_cast<uintptr_t>(q.X) & 15) == 0) && ((q.ldx * sizeof(T)) % 16 == 0);
  // example and token of the first row this warp takes
  long long ex = kWeighted ? (row_base + r0 + w) / Tn : 0;
  int t = kWeighted ? int((row_base + r0 + w) - ex * Tn) : 0;
  for (int rr = r0 + w; rr < r1; rr += 8 * kBatch) {
    Raw8<T> g[kBatch], x[kHasX ? kBatch : 1];
    float wt[kBatch];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int r = rr + 8 * b;
      const int rc = min(r, r1 - 1);
      g[b].load(G + size_t(rc) * q.ldg, nvalid, gvec);
      if (kHasX) x[kHasX ? b : 0].load(X + size_t(rc) * q.ldx, nvalid, xvec);
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      float f = 1.f;
      if (kWeighted) {
        long long eb = ex;
        int tb = t + 8 * b;
        while (tb >= Tn) { tb -= Tn; ++eb; }
        f = (rr + 8 * b < r1) ? __ldg(clip + eb) : 0.f;      // eb < B whenever the row exists
      }
      wt[b] = (rr + 8 * b < r1) ? f : 0.f;
    }
    if (kWeighted) {
      t += 8 * kBatch;
      while (t >= Tn) { t -= Tn; ++ex; }
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      float gv[8], xv[8];
      g[b].unpack(gv);
      if (kHasX) x[kHasX ? b : 0].unpack(xv);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float v = kHasX ? gv[e] * xv[e] : gv[e];
        acc[e] = fmaf(wt[b], v, acc[e]);
      }
    }
  }
}

template <typename T, bool kWeighted>
__device__ __forceinline__ void stream_rows(const VecParam& q, long long row_base, int r0, int r1,
                                            int c, int nvalid, int Tn, const float* clip,
                                            float (&acc)[8]) {
  if (q.X) stream_rows_t<T, kWeighted, true>(q, row_base, r0, r1, c, nvalid, Tn, clip, acc);
  else stream_rows_t<T, kWeighted, false>(q, row_base, r0, r1, c, nvalid, Tn, clip, acc);
}

// 0 * (a column's terms), which is 0 or, where one of them is not finite, not a number
template <typename T>
__device__ __noinline__ float zero_times_terms(const VecParam& q, long long row_base, int rows, int c) {
  float z = 0.f;
  for (int r = 0; r < rows; ++r) {
    const float g = to_f32(static_cast<const T*>(q.G)[(row_base + r) * q.ldg + c]);
    z = fmaf(0.f, q.X ? g * to_f32(static_cast<const T*>(q.X)[(row_base + r) * q.ldx + c]) : g, z);
  }
  return z;
}

// grid = (slabs of all parameters, examples): || sum_t G*X ||^2 restricted to the block's columns
// keep: [B][n_per][256] or nullptr, the block's columns of v_i.  A sum that overflowed is not kept: its example has
// no finite norm, so its factor is 0 and the clipped sum takes 0 times each of its terms, not 0 times infinity.
template <typename T>
__global__ void __launch_bounds__(256, 4)
vector_norm_kernel(const __grid_constant__ VecParams P, float* __restrict__ partials, int n_per,
                   int col0_partial, float* __restrict__ keep) {
  __shared__ float part[8][kVecCols];
  __shared__ float red[32];
  const int slab = blockIdx.x, i = blockIdx.y;
  const VecParam& q = P.prm[find_param(P, slab)];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = (slab - q.slab_begin) * kVecCols + lane * 8;
  const int nvalid = min(8, q.p - c);
  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.f;
  if (nvalid > 0) stream_rows<T, false>(q, (long long)i * P.T, 0, P.T, c, nvalid, P.T, nullptr, acc);
#pragma unroll
  for (int e = 0; e < 8; ++e) part[w][lane * 8 + e] = acc[e];
  __syncthreads();
  float v = 0.f;
#pragma unroll
  for (int ww = 0; ww < 8; ++ww) v += part[ww][threadIdx.x];
  const size_t at = size_t(i) * n_per + col0_partial + slab;
  if (keep) {
    const int cc = (slab - q.slab_begin) * kVecCols + threadIdx.x;
    const bool finite = fabsf(v) <= 3.402823466e38f;
    keep[at * kVecCols + threadIdx.x] = finite ? v : zero_times_terms<T>(q, (long long)i * P.T, P.T, cc);
  }
  const float s = block_sum(v * v, red);
  if (threadIdx.x == 0) partials[at] = s;
}

// grid = (slabs of all parameters, row splits): partial clipped sums of the block's columns
template <typename T>
__global__ void __launch_bounds__(256, 4)
vector_sum_kernel(const __grid_constant__ VecParams P, const float* __restrict__ clip,
                  int rows_per_split, float* __restrict__ partial) {
  __shared__ float part[8][kVecCols];
  const int slab = blockIdx.x, split = blockIdx.y;
  const VecParam& q = P.prm[find_param(P, slab)];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = (slab - q.slab_begin) * kVecCols + lane * 8;
  const int nvalid = min(8, q.p - c);
  const long long rows = (long long)P.B * P.T;
  const long long r0 = (long long)split * rows_per_split;
  const int nrows = (int)max(0LL, min((long long)rows_per_split, rows - r0));
  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.f;
  if (nvalid > 0) stream_rows<T, true>(q, r0, 0, nrows, c, nvalid, P.T, clip, acc);
#pragma unroll
  for (int e = 0; e < 8; ++e) part[w][lane * 8 + e] = acc[e];
  __syncthreads();
  const int cc = (slab - q.slab_begin) * kVecCols + threadIdx.x;
  if (cc < q.p) {
    float v = 0.f;
#pragma unroll
    for (int ww = 0; ww < 8; ++ww) v += part[ww][threadIdx.x];
    partial[size_t(split) * P.total_cols + q.col_begin + cc] = v;
  }
}

// out = beta*out + sum over row splits (in split order), then the Gaussian mechanism of Eq. 3
__global__ void __launch_bounds__(256)
vector_combine_kernel(const __grid_constant__ VecParams P, const float* __restrict__ partial,
                      int nsplit, float beta, int with_noise, float amp, float scale,
                      const __grid_constant__ NoiseKeys keys, uint32_t step,
                      const uint32_t* __restrict__ step_dev) {
  const int slab = blockIdx.x;
  const VecParam& q = P.prm[find_param(P, slab)];
  const int cc = (slab - q.slab_begin) * kVecCols + threadIdx.x;
  if (cc >= q.p) return;
  float v = 0.f;
  for (int s = 0; s < nsplit; ++s) v += partial[size_t(s) * P.total_cols + q.col_begin + cc];
  if (beta != 0.f) v += q.out[cc];
  if (with_noise) {
    float z[4];
    normals4((unsigned long long)(cc >> 2), keys, q.tensor_id, effective_step(step, step_dev), z);
    const int e = cc & 3;
    v = noised(v, e == 0 ? z[0] : e == 1 ? z[1] : e == 2 ? z[2] : z[3], amp, scale);
  }
  q.out[cc] = v;
}

// The same from the v_i that vector_norm_kernel kept.  It runs beside the persistent GEMM, hence 128 threads of 32 registers (see
// embed_kernels.cu); where there is none, the walk over the examples is what counts, so a block has 64 columns, a lane's four are
// one Philox counter, and eight parts of 16 lanes take every eighth row each, four loads in flight (with 256 columns and two parts
// the step of six biases of 768 at B = 96, T = 8 took 38.1 us, 35.5 with the gradients read twice, now 33.1).  A block walks `rows` rows that lie
// `row_step` examples apart, weighted with clip unless that is nullptr.  Large batches take two launches: with `rows_per_part` > 0
// block y sums that many rows and leaves the result in the first of them, which nobody else reads; then one block adds these up.
constexpr int kKeptThreads = 128, kKeptCols = 64, kKeptLanes = kKeptCols / 4, kKeptParts = kKeptThreads / kKeptLanes;
constexpr int kKeptAlone = 448;        // examples that one block walks
constexpr int kKeptRows = 128;         // rows of a part
__global__ void __launch_bounds__(kKeptThreads, 16)
vector_kept_sum_kernel(const __grid_constant__ VecParams P, float* keep, int n_per, int col0, const float* __restrict__ clip,
                       int rows, int row_step, int rows_per_part, float beta, int with_noise, float amp, float scale,
                       const __grid_constant__ NoiseKeys keys, uint32_t step, const uint32_t* __restrict__ step_dev) {
  __shared__ float4 sums[kKeptParts][kKeptLanes];
  const int slab = blockIdx.x / (kVecCols / kKeptCols), col = int(blockIdx.x) % (kVecCols / kKeptCols) * kKeptCols;
  const VecParam& q = P.prm[find_param(P, slab)];
  const int c0 = (slab - q.slab_begin) * kVecCols + col;
  if (c0 >= q.p) return;
  const int lane = threadIdx.x & (kKeptLanes - 1), part = threadIdx.x / kKeptLanes;
  const int r0 = int(blockIdx.y) * rows_per_part, r1 = rows_per_part ? min(rows, r0 + rows_per_part) : rows;
  float4* src = reinterpret_cast<float4*>(keep + size_t(col0 + slab) * kVecCols + col) + lane;
  const size_t pitch = size_t(n_per) * (kVecCols / 4) * row_step;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
  for (int i = r0 + part; i < r1; i += kKeptParts) {
    const float4 v = src[size_t(i) * pitch];
    const float r = clip ? __ldg(clip + i) : 1.f;
    a.x = fmaf(r, v.x, a.x); a.y = fmaf(r, v.y, a.y); a.z = fmaf(r, v.z, a.z); a.w = fmaf(r, v.w, a.w);
  }
  sums[part][lane] = a;
  __syncthreads();
  if (part) return;
#pragma unroll
  for (int k = 1; k < kKeptParts; ++k) {
    const float4 x = sums[k][lane];
    a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
  }
  if (rows_per_part) { src[size_t(r0) * pitch] = a; return; }
  const float v[4] = {a.x, a.y, a.z, a.w};
  const int c = c0 + 4 * lane;
  if (c >= q.p) return;
  float z[4] = {0.f, 0.f, 0.f, 0.f};
  if (with_noise) normals4((unsigned long long)(c >> 2), keys, q.tensor_id, effective_step(step, step_dev), z);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if (c + e >= q.p) break;
    float x = v[e];
    if (beta != 0.f) x += q.out[c + e];
    q.out[c + e] = with_noise ? noised(x, z[e], amp, scale) : x;
  }
}

}  // namespace

namespace {

int fill_params(VecParams& P, const dp_vector_desc* prm, int n0, int n1, float* const* outs,
                const uint32_t* tensor_ids, int B, int T) {
  memset(&P, 0, sizeof(P));
  int slabs = 0, cols = 0;
  for (int k = n0; k < n1; ++k) {
    VecParam& q = P.prm[k - n0];
    q.G = prm[k].G; q.X = prm[k].X; q.ldg = prm[k].ldg; q.ldx = prm[k].ldx; q.p = prm[k].p;
    q.out = outs ? outs[k] : nullptr;
    q.tensor_id = tensor_ids ? tensor_ids[k] : 0u;
    q.slab_begin = slabs; q.col_begin = cols;
    slabs += ceil_div(prm[k].p, kVecCols);
    cols += prm[k].p;
  }
  P.n = n1 - n0; P.B = B; P.T = T; P.total_slabs = slabs; P.total_cols = cols;
  return slabs;
}

}  // namespace

int vector_total_slabs(const dp_vector_desc* prm, int n) {
  int s = 0;
  for (int k = 0; k < n; ++k) s += ceil_div(prm[k].p, kVecCols);
  return s;
}

// row splits of the clipped-sum pass: enough blocks for about eight per SM, >= 64 rows each
int vector_row_splits(const dp_vector_desc* prm, int n, int B, int T, int sms) {
  const long long rows = (long long)B * T;
  const int slabs = std::max(1, vector_total_slabs(prm, std::min(n, kVecMaxParams)));
  long long ns = std::max<long long>(1, (8LL * sms) / slabs);
  ns = std::min<long long>(ns, std::max<long long>(1, rows / 64));
  return (int)ns;
}

dp_status launch_vector_norms(const dp_vector_desc* prm, int n, dp_dtype dt, int B, int T,
                              float* partials, int n_per, cudaStream_t st, float* keep) {
  int col0 = 0;
  for (int n0 = 0; n0 < n; n0 += kVecMaxParams) {
    const int n1 = std::min(n, n0 + kVecMaxParams);
    VecParams P;
    const int slabs = fill_params(P, prm, n0, n1, nullptr, nullptr, B, T);
    dim3 grid(slabs, B);
    if (dt == DP_F32) vector_norm_kernel<float><<<grid, 256, 0, st>>>(P, partials, n_per, col0, keep);
    else vector_norm_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(P, partials, n_per, col0, keep);
    DP_LAUNCH_OK();
    col0 += slabs;
  }
  return DP_OK;
}

dp_status launch_vector_sums(const dp_vector_desc* prm, int n, dp_dtype dt, int B, int T,
                             const float* clip, float* const* outs, float beta, int with_noise,
                             float amp, float scale, uint64_t seed, const uint32_t* tensor_ids,
                             uint32_t step, float* partial_ws, cudaStream_t st) {
  const int sms = sm_count();
  const long long rows = (long long)B * T;
  for (int n0 = 0; n0 < n; n0 += kVecMaxParams) {
    const int n1 = std::min(n, n0 + kVecMaxParams);
    VecParams P;
    const int slabs = fill_params(P, prm, n0, n1, outs, tensor_ids, B, T);
    int nsplit = vector_row_splits(prm + n0, n1 - n0, B, T, sms);
    const int rps = (int)((rows + nsplit - 1) / nsplit);
    nsplit = (int)((rows + rps - 1) / rps);
    dim3 grid(slabs, nsplit);
    if (dt == DP_F32) vector_sum_kernel<float><<<grid, 256, 0, st>>>(P, clip, rps, partial_ws);
    else vector_sum_kernel<__nv_bfloat16><<<grid, 256, 0, st>>>(P, clip, rps, partial_ws);
    DP_LAUNCH_OK();
    vector_combine_kernel<<<slabs, 256, 0, st>>>(P, partial_ws, nsplit, beta, with_noise, amp, scale,
                                                expand_noise_keys(seed), step, g_step_dev);
    DP_LAUNCH_OK();
  }
  return DP_OK;
}

size_t vector_keep_bytes(const dp_vector_desc* prm, int n, int B) {
  return size_t(B) * vector_total_slabs(prm, n) * kVecCols * sizeof(float);
}

dp_status launch_vector_kept_sums(const dp_vector_desc* prm, int n, int B, int T, float* keep, const float* clip,
                                  float* const* outs, float beta, int with_noise, float amp, float scale, uint64_t seed,
                                  const uint32_t* tensor_ids, uint32_t step, cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&vector_kept_sum_kernel)))
    DP_CUDA_OK(prefer_max_shared(vector_kept_sum_kernel));
  const int n_per = vector_total_slabs(prm, n);
  // one block walks all examples as long as that is short; beyond, parts at least as long as there are parts.  Step of six biases of 768
  // at T = 8 and B = 256, 1024, 4096: 72, 167, 478 us with G read twice, 64, 151, 431 now.
  int per_part = 0;
  if (B > kKeptAlone) for (per_part = kKeptRows; (long long)per_part * per_part < B; per_part *= 2) {}
  const int parts = per_part ? ceil_div(B, per_part) : 1;
  int col0 = 0;
  for (int n0 = 0; n0 < n; n0 += kVecMaxParams) {
    VecParams P;
    const int slabs = fill_params(P, prm, n0, std::min(n, n0 + kVecMaxParams), outs, tensor_ids, B, T);
    const int blocks = slabs * (kVecCols / kKeptCols);
    if (per_part) {
      vector_kept_sum_kernel<<<dim3(blocks, parts), kKeptThreads, 0, st>>>(P, keep, n_per, col0, clip, B, 1, per_part, 0.f, 0, 0.f,
                                                                         1.f, expand_noise_keys(seed), step, g_step_dev);
      DP_LAUNCH_OK();
    }
    vector_kept_sum_kernel<<<blocks, kKeptThreads, 0, st>>>(P, keep, n_per, col0, per_part ? nullptr : clip, per_part ? parts : B,
                                                          per_part ? per_part : 1, 0, beta, with_noise, amp, scale,
                                                          expand_noise_keys(seed), step, g_step_dev);
    DP_LAUNCH_OK();
    col0 += slabs;
  }
  return DP_OK;
}

}  // namespace dpg
