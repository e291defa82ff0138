// One DP-SGD step over a few hundred tokens and a few small layers, in two kernels.
//
// Such a step is launches and latency: by itself each of its parts takes 2 to 5 us, of which a few hundred nanoseconds
// are arithmetic.  On two streams, eight kernels and eight event calls took 31 us of host time and a chain of five
// kernels on the GPU.  Here all that needs no clip factor is one launch of blocks with different parts, and all that
// does is a second one:
//   small_norms_kernel  blocks of Gram items (layer, example, pair of 32-token tiles: 32 x 32 entries of A A^T and G G^T, all
//                       columns) and of embedding items (example, 64 columns); one partial sum of ||g_i||^2 each
//   small_sums_kernel   every block first adds up the partial sums of all examples (a few dozen floats) and has the
//                       clip factors; then blocks of 32 x 32 output tiles over all tokens, and of table rows
// Every block brings all its operands in at once (one memory latency, not one per 32 columns or rows).  The second kernel is
// launched while the first runs: it loads operands, finds its tokens, draws its noise and writes the table rows that
// no token touches before it waits for the norms.  No sort: a block of table rows looks through all (at most 512) ids.
// Everything is fp32 and in a fixed order.
//
// Bound by latency: launch, one round trip to memory, and the serial sums of a block.  Step of one 64 x 64 fp32 layer and a 1000-row
// table at B = 4, T = 16: 30 -> 13 us, as a graph 22.6 -> 10.3 (12.4 without the early launch of the second kernel).
#include <algorithm>
#include <cstring>

#include "dp_common.cuh"
#include "fma_kernels.cuh"
#include "noise_device.cuh"
#include "small_step.cuh"

namespace dpg {

namespace {

constexpr int kMaxLayers = 8, kMaxTokens = 512, kMaxT = 64, kMaxB = 64, kMaxCols = 256;
constexpr int kMaxBlocks = 148;          // Gram items, and output tiles: one per SM
constexpr size_t kMostBf16Smem = 150 * 1024;       // bf16 layers: shared memory of the norms' blocks on the busiest SM
constexpr int kThreads = 256;
constexpr int kGramTile = 32;
constexpr int kEmbedCols = 64;         // columns per embedding item
constexpr int kSumTile = 32, kSumRows = 128;      // output tile, token rows per shared-memory stage
constexpr int kTableBlocks = 296, kTableRows = 32;      // blocks and, at most, rows of a block

struct SmallLayer {
  const void *A, *G;
  float* out;
  long long lda, ldg, ldo;
  int d, p, tile_begin, tiles_n;       // output tiles
  uint32_t tensor_id;
};
struct SmallParams {
  SmallLayer layer[kMaxLayers];
  int n_layers, B, T, V, d;            // d: of the table
  int ntp, n_gram, slabs;              // tile pairs per Gram matrix, Gram items, embedding items per example
  int n_per, n_main;                   // partial sums per example: layers' first
  int n_tiles, table_blocks;
  const int* ids;
  const void* G_emb;
  long long ldge;
  float* wte;
  long long ld_wte;
  uint32_t wte_id;
  float* partials;                     // [B][n_per]
  float *sq, *clip, *norms;
  float C, amp;                        // amp < 0: no noise
  NoiseKeys keys;
  uint32_t step;
  const uint32_t* step_dev;
  int* dev_status;
};

// floats between rows in shared memory: 16-byte rows, an odd number of 16-byte words (16 rows' words in 2 wavefronts)
__host__ __device__ __forceinline__ int small_pitch(int cols) { return (((cols + 3) >> 2) | 1) << 2; }

template <typename T> __device__ __forceinline__ float4 load4(const T* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
  const uint2 q = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u), __uint_as_float(q.y << 16),
                     __uint_as_float(q.y & 0xffff0000u));
}

// rows [0, rows) of X, `cols` columns each, into shared memory; rows up to `all` as zeros.  Eight loads in flight.
template <typename T>
__device__ __forceinline__ void bring(float* dst, int pitch, const T* X, long long ld, int rows, int all, int cols) {
  const int words = cols >> 2, n = all * words;
  for (int k0 = threadIdx.x; k0 < n; k0 += 8 * kThreads) {
    float4 v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = k0 + j * kThreads, r = k / words;
      v[j] = k < n && r < rows ? load4(X + r * ld + 4 * (k - r * words)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = k0 + j * kThreads, r = k / words;
      if (k < n) *reinterpret_cast<float4*>(dst + r * pitch + 4 * (k - r * words)) = v[j];
    }
  }
}

// entries (ty, ty + 16) x (tx, tx + 16) of the product of two 32-row tiles; 32 columns by themselves: shorter chains
__device__ __forceinline__ void gram_entries(const float* xi, const float* xj, int pitch, int cols, float (&s)[2][2]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  s[0][0] = s[0][1] = s[1][0] = s[1][1] = 0.f;
  for (int c0 = 0; c0 < cols; c0 += 32) {
    float part[2][2] = {};
    const int c1 = min(cols, c0 + 32);
#pragma unroll 4
    for (int c = c0; c < c1; c += 4) {
      float4 a[2], b[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        a[h] = *reinterpret_cast<const float4*>(xi + (ty + 16 * h) * pitch + c);
        b[h] = *reinterpret_cast<const float4*>(xj + (tx + 16 * h) * pitch + c);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          part[h][g] = fmaf(a[h].x, b[g].x, part[h][g]);
          part[h][g] = fmaf(a[h].y, b[g].y, part[h][g]);
          part[h][g] = fmaf(a[h].z, b[g].z, part[h][g]);
          part[h][g] = fmaf(a[h].w, b[g].w, part[h][g]);
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) s[e >> 1][e & 1] += part[e >> 1][e & 1];
  }
}

template <typename TL, typename TE>
__global__ void __launch_bounds__(kThreads)
small_norms_kernel(const __grid_constant__ SmallParams P) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float red[32];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int T = P.T;
  if (int(blockIdx.x) < P.n_gram) {
    const int tp = blockIdx.x % P.ntp, i = (blockIdx.x / P.ntp) % P.B, l = blockIdx.x / (P.ntp * P.B);
    const SmallLayer& L = P.layer[l];
    const int ri = tp == 2 ? kGramTile : 0, rj = tp == 0 ? 0 : kGramTile;        // tile pairs (0,0), (0,1), (1,1)
    const bool two = ri != rj;
    const TL* A = static_cast<const TL*>(L.A) + size_t(i) * T * L.lda;
    const TL* G = static_cast<const TL*>(L.G) + size_t(i) * T * L.ldg;
    const int pa = small_pitch(L.d), pg = small_pitch(L.p);
    float *ai = sm, *gi = ai + kGramTile * pa, *aj = ai, *gj = gi;
    bring(ai, pa, A + ri * L.lda, L.lda, T - ri, kGramTile, L.d);
    bring(gi, pg, G + ri * L.ldg, L.ldg, T - ri, kGramTile, L.p);
    if (two) {
      aj = gi + kGramTile * pg;
      gj = aj + kGramTile * pa;
      bring(aj, pa, A + rj * L.lda, L.lda, T - rj, kGramTile, L.d);
      bring(gj, pg, G + rj * L.ldg, L.ldg, T - rj, kGramTile, L.p);
    }
    __syncthreads();
    float sa[2][2], sg[2][2], acc = 0.f;
    gram_entries(ai, aj, pa, L.d, sa);
    gram_entries(gi, gj, pg, L.p, sg);
#pragma unroll
    for (int e = 0; e < 4; ++e) acc = fmaf(sa[e >> 1][e & 1], sg[e >> 1][e & 1], acc);
    const float tot = block_sum(acc, red);
    const int slot = i * P.n_per + l * P.ntp + tp;
    if (threadIdx.x == 0 && dp_in_range(slot, P.B * P.n_per, P.dev_status)) P.partials[slot] = two ? 2.f * tot : tot;
    return;
  }
  // embedding: || sum over the tokens of an id ||^2, over the ids of the example
  const int item = int(blockIdx.x) - P.n_gram, slab = item % P.slabs, i = item / P.slabs;
  __shared__ int s_id[kMaxT], s_first[kMaxT];
  __shared__ __align__(16) int s_order[kMaxT];          // where a token's row lies; sign bit = last token of its id
  const int c0 = slab * kEmbedCols, cols = min(kEmbedCols, P.d - c0), pitch = small_pitch(kEmbedCols);
  if (threadIdx.x < kMaxT) {
    int id = -2 - int(threadIdx.x);                      // out of range: by itself, and its row counts as zeros
    if (int(threadIdx.x) < T) {
      const int x = P.ids[i * T + threadIdx.x];
      if (x >= 0 && x < P.V) id = x;
      else if (slab == 0 && P.dev_status) atomicOr(P.dev_status, DP_DEV_BAD_ID);
    }
    s_id[threadIdx.x] = id;
    s_order[threadIdx.x] = 0;
  }
  bring(sm, pitch, static_cast<const TE*>(P.G_emb) + size_t(i) * T * P.ldge + c0, P.ldge, T, T, cols);
  if (threadIdx.x < kEmbedCols) sm[T * pitch + threadIdx.x] = 0.f;
  __syncthreads();
  // a token's place in the order of (first token of the id, position): four threads look at 16 tokens each
  const int t = threadIdx.x >> 2, part = threadIdx.x & 3, id = s_id[t];
  auto add4 = [](int x) { x += __shfl_xor_sync(0xffffffffu, x, 1); return x + __shfl_xor_sync(0xffffffffu, x, 2); };
  int first = t, rank = 0, size = 0;
#pragma unroll
  for (int k = 0; k < kMaxT / 4; ++k) {
    const int s = 4 * k + part;
    const bool same = s_id[s] == id;
    first = same ? min(first, s) : first;
    rank += same && s < t;
    size += same;
  }
  first = min(first, __shfl_xor_sync(0xffffffffu, first, 1));
  first = min(first, __shfl_xor_sync(0xffffffffu, first, 2));
  rank = add4(rank);
  size = add4(size);
  if (part == 0) s_first[t] = first;
  __syncthreads();
  int at = 0;
#pragma unroll
  for (int k = 0; k < kMaxT / 4; ++k) at += s_first[4 * k + part] < first;
  at = add4(at) + rank;                                  // tokens beyond T come last, each by itself
  if (part == 0 && t < T && dp_in_range(at, T, P.dev_status)) s_order[at] = ((id >= 0 ? t : T) * pitch) | (rank + 1 == size ? int(0x80000000u) : 0);
  __syncthreads();
  float tot = 0.f;
  if (int(threadIdx.x) < cols) {
    float run = 0.f;
    for (int r0 = 0; r0 < T; r0 += 16) {
      __align__(16) int o[16];
      float v[16];
#pragma unroll
      for (int k = 0; k < 16; k += 4) *reinterpret_cast<int4*>(o + k) = *reinterpret_cast<const int4*>(s_order + r0 + k);
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = sm[(o[k] & 0x7fffffff) + threadIdx.x];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        if (r0 + k >= T) break;
        run += v[k];
        if (o[k] < 0) { tot = fmaf(run, run, tot); run = 0.f; }
      }
    }
  }
  const float s = block_sum(tot, red);
  const int slot = i * P.n_per + P.n_main + slab;
  if (threadIdx.x == 0 && dp_in_range(slot, P.B * P.n_per, P.dev_status)) P.partials[slot] = s;
}

// clip factors of all examples into shared memory (the norms' kernel is waited for first); block 0 writes the outputs
__device__ __forceinline__ void find_clip(const SmallParams& P, float* s_clip) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (int(threadIdx.x) < P.B) {
    const int i = threadIdx.x;
    const float* p = P.partials + i * P.n_per;
    float part[2] = {0.f, 0.f};
#pragma unroll 8
    for (int k = 0; k < P.n_per; ++k) part[k < P.n_main ? 0 : 1] += __ldcg(p + k);
    const float sq = part[0] + part[1], r = clip_from_sq(sq, P.C);
    s_clip[i] = r;
    if (blockIdx.x == 0) {
      P.sq[i] = sq;
      P.clip[i] = r;
      if (P.norms) P.norms[i] = __fsqrt_rn(sq);
    }
  }
  __syncthreads();
}

__device__ __forceinline__ void store4(float* o, const float (&v)[4], bool vec) {
  if (vec) {
    *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) o[e] = v[e];
  }
}

template <typename TL, typename TE>
__global__ void __launch_bounds__(kThreads)
small_sums_kernel(const __grid_constant__ SmallParams P) {
  __shared__ __align__(16) float buf[2 * kSumRows * (kSumTile + 4)];
  __shared__ float s_clip[kMaxB];
  const bool noisy = P.amp >= 0.f;
  const uint32_t step = noisy ? effective_step(P.step, P.step_dev) : 0u;
  const int n = P.B * P.T;
  if (int(blockIdx.x) < P.n_tiles) {
    // ------------------------------------------------------------- an output tile of a layer
    int l = 0;
    while (l + 1 < P.n_layers && int(blockIdx.x) >= P.layer[l + 1].tile_begin) ++l;
    const SmallLayer& L = P.layer[l];
    const int tile = int(blockIdx.x) - L.tile_begin;
    const int m0 = tile / L.tiles_n * kSumTile, n0 = tile % L.tiles_n * kSumTile;
    constexpr int kPitch = kSumTile + 4;
    float *gs = buf, *as = buf + kSumRows * kPitch;
    // a thread brings four rows of one 16-byte word of each operand per stage
    const int word = threadIdx.x & 7, row = threadIdx.x >> 3;
    const bool in_g = m0 + 4 * word < L.p, in_a = n0 + 4 * word < L.d;
    const TL* G = static_cast<const TL*>(L.G) + m0 + 4 * word;
    const TL* A = static_cast<const TL*>(L.A) + n0 + 4 * word;
    float4 g[4], a[4];
    auto load = [&](int k0) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = k0 + row + 32 * j;
        g[j] = in_g && k < n ? load4(G + k * L.ldg) : make_float4(0.f, 0.f, 0.f, 0.f);
        a[j] = in_a && k < n ? load4(A + k * L.lda) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    };
    load(0);
    const int orow = m0 + (threadIdx.x >> 3), ocol = n0 + 4 * (threadIdx.x & 7);       // the four outputs of this thread
    float z[4];
    if (noisy && orow < L.p && ocol < L.d)
      normals4(((unsigned long long)orow * L.d + ocol) >> 2, P.keys, L.tensor_id, step, z);
    find_clip(P, s_clip);
    // 4 groups of 64 threads take 32 rows of a stage each, a thread 4 x 4 outputs
    const int group = threadIdx.x >> 6, gx = threadIdx.x & 7, gy = (threadIdx.x >> 3) & 7;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < n; k0 += kSumRows) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = row + 32 * j, k = k0 + r;
        const float f = k < n ? s_clip[k / P.T] : 0.f;
        *reinterpret_cast<float4*>(gs + r * kPitch + 4 * word) = make_float4(f * g[j].x, f * g[j].y, f * g[j].z, f * g[j].w);
        *reinterpret_cast<float4*>(as + r * kPitch + 4 * word) = a[j];
      }
      __syncthreads();
      if (k0 + kSumRows < n) load(k0 + kSumRows);
      const int r0 = 32 * group, r1 = min(r0 + 32, n - k0);
#pragma unroll 4
      for (int r = r0; r < r1; ++r) {
        const float4 x = *reinterpret_cast<const float4*>(gs + r * kPitch + 4 * gy);
        const float4 y = *reinterpret_cast<const float4*>(as + r * kPitch + 4 * gx);
        const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(xv[u], yv[v], acc[u][v]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      *reinterpret_cast<float4*>(buf + (group * kSumTile + 4 * gy + u) * kPitch + 4 * gx) =
          make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
    __syncthreads();
    if (orow >= L.p || ocol >= L.d) return;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 x = *reinterpret_cast<const float4*>(buf + (q * kSumTile + orow - m0) * kPitch + ocol - n0);
      v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
    }
    if (noisy)
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = noised(v[e], z[e], P.amp, 1.f);
    float* o = L.out + orow * L.ldo + ocol;
    store4(o, v, (reinterpret_cast<uintptr_t>(o) & 15) == 0);
    return;
  }
  // --------------------------------------------------------------- table rows block, block + blocks, ...
  __shared__ short s_pos[kMaxTokens];
  __shared__ unsigned char s_row[kMaxTokens];
  __shared__ int s_count[kThreads / 32 + 1];
  __shared__ unsigned s_touched;
  const int block = int(blockIdx.x) - P.n_tiles, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int quads = P.d >> 2, parts = kThreads / quads, quad = threadIdx.x % quads, part = threadIdx.x / quads;
  const int rows = (P.V - block + P.table_blocks - 1) / P.table_blocks;
  if (threadIdx.x == 0) s_touched = 0u;
  // this block's tokens, in order: a thread looks at two of the ids
  int row[2] = {-1, -1};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int t = 2 * threadIdx.x + h;
    const int id = t < n ? P.ids[t] : -1;
    if (id >= 0 && id < P.V && id % P.table_blocks == block) row[h] = id / P.table_blocks;
  }
  const int mine = (row[0] >= 0) + (row[1] >= 0);
  int before = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, before, o);
    if (lane >= o) before += y;
  }
  if (lane == 31) s_count[w] = before;
  __syncthreads();
  int entries = 0;
  before -= mine;
#pragma unroll
  for (int k = 0; k < kThreads / 32; ++k) {
    if (k < w) before += s_count[k];
    entries += s_count[k];
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
    if (row[h] >= 0 && dp_in_range(row[h], rows, P.dev_status) && dp_in_range(before, n, P.dev_status)) {
      s_pos[before] = short(2 * threadIdx.x + h);
      s_row[before] = static_cast<unsigned char>(row[h]);
      atomicOr(&s_touched, 1u << row[h]);
      ++before;
    }
  __syncthreads();
  const unsigned touched = s_touched;
  const bool vec = (reinterpret_cast<uintptr_t>(P.wte) & 15) == 0 && (P.ld_wte & 3) == 0;
  // the row's noise (or zeros) plus `sum`
  auto write = [&](int r, const float4& sum) {
    const long long v = block + (long long)r * P.table_blocks;
    if (!dp_in_range(v, P.V, P.dev_status)) return;
    float x[4] = {sum.x, sum.y, sum.z, sum.w};
    if (noisy) {
      float z[4];
      normals4((unsigned long long)(v * quads + quad), P.keys, P.wte_id, step, z);
#pragma unroll
      for (int e = 0; e < 4; ++e) x[e] = noised(0.f, z[e], P.amp, 1.f) + x[e];
    }
    store4(P.wte + v * P.ld_wte + 4 * quad, x, vec);
  };
  if (part < parts)
    for (int r = part; r < rows; r += parts)
      if (!((touched >> r) & 1u)) write(r, make_float4(0.f, 0.f, 0.f, 0.f));
  if (touched == 0u && blockIdx.x != 0) return;          // (the first block writes the norms)
  find_clip(P, s_clip);
  const TE* G = static_cast<const TE*>(P.G_emb) + 4 * quad;
  float4* sums = reinterpret_cast<float4*>(buf);
  for (unsigned left = touched; left; left &= left - 1u) {
    const int r = __ffs(left) - 1;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (part < parts) {
#pragma unroll 4
      for (int k = part; k < entries; k += parts) {
        if (s_row[k] != r) continue;
        const int t = s_pos[k];
        if (!dp_in_range(t, n, P.dev_status)) continue;
        const float f = s_clip[t / P.T];
        const float4 g = load4(G + t * P.ldge);
        acc.x = fmaf(f, g.x, acc.x); acc.y = fmaf(f, g.y, acc.y); acc.z = fmaf(f, g.z, acc.z); acc.w = fmaf(f, g.w, acc.w);
      }
      sums[part * quads + quad] = acc;
    }
    __syncthreads();
    if (part == 0) {
      for (int q = 1; q < parts; ++q) {
        const float4 x = sums[q * quads + quad];
        acc.x += x.x; acc.y += x.y; acc.z += x.z; acc.w += x.w;
      }
      write(r, acc);
    }
    __syncthreads();
  }
}

size_t gram_smem(const dp_step_desc& S) {
  size_t most = size_t(S.T + 1) * small_pitch(kEmbedCols);           // a row of zeros behind the tokens'
  for (int l = 0; l < S.n_layers; ++l)
    most = std::max(most, size_t(S.T > kGramTile ? 2 : 1) * kGramTile *
                              (small_pitch(S.layers[l].d) + small_pitch(S.layers[l].p)));
  return most * sizeof(float);
}
constexpr size_t kMostGramSmem = size_t(2) * kGramTile * 2 * (kMaxCols + 4) * sizeof(float);

template <typename TL, typename TE>
dp_status launch(const SmallParams& P, size_t smem, cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&small_norms_kernel<TL, TE>))) {
    DP_CUDA_OK((allow_shared(small_norms_kernel<TL, TE>, kMostGramSmem)));
    DP_CUDA_OK((prefer_max_shared(small_sums_kernel<TL, TE>)));
  }
  small_norms_kernel<TL, TE><<<P.n_gram + P.B * P.slabs, kThreads, smem, st>>>(P);
  DP_LAUNCH_OK();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(P.n_tiles + P.table_blocks), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  DP_CUDA_OK((cudaLaunchKernelEx(&cfg, small_sums_kernel<TL, TE>, P)));
  ++g_kernel_launches;
  return DP_OK;
}

bool words_aligned(const void* p, int64_t ld, int cols, size_t element) {
  return (reinterpret_cast<uintptr_t>(p) % (4 * element)) == 0 && ld % 4 == 0 && cols % 4 == 0 && cols <= kMaxCols;
}

int partials_per_example(const dp_step_desc& S) {
  const int ntp = S.T > kGramTile ? 3 : 1;
  return S.n_layers * ntp + ceil_div(S.d, kEmbedCols);
}

}  // namespace

// At most 512 tokens in sequences of at most 64, eight layers of at most 256 columns, a table of at most 2^20 values, and at
// most as many Gram items, and output tiles, as there are SMs (the embedding items come on top).  Step of one 256 x 256 layer
// at 512 tokens, call by call and as a graph: fp32 56 and 36 -> 27 and 29 us, bf16 48 and 33 -> 28 and 29; of four, fp32 61 and
// 39 -> 35 and 37, but bf16 50 and 33 -> 36 and 37, hence the line.  bf16 steps, whose Gram products the general path takes on
// the tensor cores, also go there where the norms' blocks fill an SM's shared memory and many are Gram items: two 256 x 256
// layers at B = 64, T = 8 and a table of 256 columns (384 blocks of 66 KiB) 43 and 31 -> 35 and 37, three of 256 x 192 at B =
// 49, T = 10 (343 of 58) 44 and 33 -> 34 and 35, but with 64 table columns (192 of 66) 42 and 33 -> 24 and 27, and with one
// layer (64 Gram items of 320 blocks) 41 and 32 -> 25 and 27; fp32 ones were faster in all of these, both ways.  At the line
// bf16 graphs are even (two 256 x 256 layers at B = 12, T = 42 and B = 16, T = 32: 32.5 and 30.0 -> 32.8 and 30.7) and calls a
// third faster.  Widths in whole words of four values, as everything here is read.
bool small_step_fits(const dp_step_desc& S) {
  if (g_force_fma || S.tied || S.n_vectors || S.pos_ids || S.n_layers > kMaxLayers) return false;
  if (S.T > kMaxT || S.B > kMaxB || (long long)S.B * S.T > kMaxTokens) return false;
  if (S.V > kTableBlocks * kTableRows || (long long)S.V * S.d > (1 << 20)) return false;
  const size_t se = S.embed_dtype == DP_F32 ? 4 : 2, sl = S.layer_dtype == DP_F32 ? 4 : 2;
  if (!words_aligned(S.G_emb, S.ldge, S.d, se)) return false;
  const long long items = (long long)S.n_layers * S.B * (S.T > kGramTile ? 3 : 1);
  long long tiles = 0;
  for (int l = 0; l < S.n_layers; ++l) {
    const dp_linear_desc& L = S.layers[l];
    tiles += (long long)ceil_div(L.d, kSumTile) * ceil_div(L.p, kSumTile);
    if (!words_aligned(L.A, L.lda, L.d, sl) || !words_aligned(L.G, L.ldg, L.p, sl)) return false;
    // AUTO is GHOST here unless the layer is smaller than a Gram matrix
    if (L.mode == DP_NORM_DIRECT || (L.mode == DP_NORM_AUTO && (long long)S.T * S.T > (long long)L.d * L.p)) return false;
  }
  if (items > kMaxBlocks || tiles > kMaxBlocks) return false;
  const long long blocks = items + (long long)S.B * ceil_div(S.d, kEmbedCols);
  if (S.layer_dtype == DP_BF16 && 2 * items > kMaxBlocks &&
      size_t((blocks + kMaxBlocks - 1) / kMaxBlocks) * gram_smem(S) > kMostBf16Smem) return false;
  return S.ws && (reinterpret_cast<uintptr_t>(S.ws) & 3) == 0 && size_t(S.B) * partials_per_example(S) * sizeof(float) <= S.ws_bytes;
}

dp_status launch_small_step(const dp_step_desc& S, cudaStream_t st) {
  SmallParams P;
  memset(&P, 0, sizeof(P));
  P.n_layers = S.n_layers; P.B = S.B; P.T = S.T; P.V = S.V; P.d = S.d;
  P.ntp = S.T > kGramTile ? 3 : 1;
  P.n_gram = S.n_layers * S.B * P.ntp;
  P.slabs = ceil_div(S.d, kEmbedCols);
  P.n_main = S.n_layers * P.ntp; P.n_per = partials_per_example(S);
  for (int l = 0; l < S.n_layers; ++l) {
    dp_linear_desc& D = S.layers[l];
    P.layer[l] = {D.A, D.G, S.outs[l], D.lda, D.ldg, S.ldos[l], D.d, D.p, P.n_tiles, ceil_div(D.d, kSumTile),
                  S.with_noise ? S.tensor_ids[l] : 0u};
    P.n_tiles += ceil_div(D.d, kSumTile) * ceil_div(D.p, kSumTile);
    D.mode_used = DP_NORM_GHOST;
  }
  P.table_blocks = std::min(S.V, kTableBlocks);
  P.ids = S.ids; P.G_emb = S.G_emb; P.ldge = S.ldge;
  P.wte = S.wte; P.ld_wte = S.ld_wte; P.wte_id = S.wte_id;
  P.partials = static_cast<float*>(S.ws);
  P.sq = S.sq; P.clip = S.clip; P.norms = S.norms;
  P.C = S.C; P.amp = S.with_noise ? S.sigma * S.C : -1.f;
  P.keys = expand_noise_keys(S.seed); P.step = S.step; P.step_dev = g_step_dev;
  P.dev_status = S.dev_status;
  const size_t smem = gram_smem(S);
  const bool lf = S.layer_dtype == DP_F32, ef = S.embed_dtype == DP_F32;
  if (lf) return ef ? launch<float, float>(P, smem, st) : launch<float, __nv_bfloat16>(P, smem, st);
  return ef ? launch<__nv_bfloat16, float>(P, smem, st) : launch<__nv_bfloat16, __nv_bfloat16>(P, smem, st);
}

}  // namespace dpg
