// Embedding-table kernels: per-example ghost norm by token-id equality, stable counting sort
// of token positions, and the clipped segmented row sum (scatter-add without atomics).
//
// An embedding is a linear layer whose input is the one-hot row of the token, so Eq. 4 gives
// e_{id_t} g_t^T per token and the per-example gradient has one row per DISTINCT token:
//   || g_i ||_F^2 = sum over distinct v of || sum_{t: id_t = v} g_t ||^2
//                 = sum_{t,s} [id_t == id_s] (g_t . g_s).
#include <algorithm>

#include "dp_common.cuh"
#include "fma_kernels.cuh"

namespace dpg {

namespace {

// ------------------------------------------------------------------ grouping tokens by id
// Block-wide grouping of n tokens by id, in shared memory: first occurrence, stable rank inside the
// group, group size.  Ids meet in a hash table (every id in range finds its slot by linear probing),
// the first occurrence is an atomicMin -- integers, so the outcome does not depend on timing -- and
// the ranks come from one warp that walks the tokens 32 at a time: equal ids of a window are matched
// beforehand by all warps (__match_any_sync), so a window costs the walk two shared-memory accesses.
struct TokenGroups {
  int* id;      // [n]  token id, negative: out of range (a group of its own)
  int* fo;      // [n]  first occurrence
  int* rank;    // [n]  number of earlier tokens of the same group
  int* size;    // [n]  group size, at the first occurrence (0 elsewhere)
};
__host__ __device__ __forceinline__ int group_slots(int n) {       // hash slots: at least 2 n
  int h = 64;
  while (h < 2 * n) h <<= 1;
  return h;
}
__host__ __device__ __forceinline__ size_t group_smem_bytes(int n) {
  return (size_t(3) * ((n + 31) & ~31) + size_t(2) * group_slots(n)) * sizeof(int);
}

// fills g; g.id must hold the n ids already (the function synchronises first and last)
__device__ __forceinline__ void group_tokens(const TokenGroups& g, int* keys, int* first, int slots, int n) {
  if (n <= 32) {                                         // one window: no table (7.3 -> 6.9 us for the norm at B = 1, T = 8, d = 768)
    __syncthreads();
    const int lane = threadIdx.x;
    if (lane < 32) {
      const int id = lane < n ? g.id[lane] : -1;
      const unsigned peers = __match_any_sync(0xffffffffu, id >= 0 ? id : int(0x80000000u | unsigned(lane)));
      if (lane < n) {
        const int fo = __ffs(peers) - 1;
        g.fo[lane] = fo;
        g.rank[lane] = __popc(peers & ((1u << lane) - 1u));
        g.size[lane] = lane == fo ? __popc(peers) : 0;
      }
    }
    __syncthreads();
    return;
  }
  constexpr int kEmpty = int(0x80000000);
  const int shift = __clz(slots) + 1;                    // top log2(slots) bits of the product
  for (int h = threadIdx.x; h < slots; h += blockDim.x) { keys[h] = kEmpty; first[h] = 0x7fffffff; }
  __syncthreads();
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int id = g.id[t];
    int h = -1;
    if (id >= 0) {
      h = int((uint32_t(id) * 0x9E3779B1u) >> shift);
      for (int probe = 0; probe < slots; ++probe) {      // at most half the slots are taken
        const int was = atomicCAS(&keys[h], kEmpty, id);
        if (was == kEmpty || was == id) break;
        h = (h + 1) & (slots - 1);
      }
      atomicMin(&first[h], t);
    }
    g.fo[t] = h;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int n32 = (n + 31) & ~31;
  // first occurrences, and the matches inside every window of 32 tokens: earlier peers, peers
  for (int t = threadIdx.x; t < n32; t += blockDim.x) {
    int fo = t;
    if (t < n && g.fo[t] >= 0) fo = first[g.fo[t]];
    const unsigned peers = __match_any_sync(0xffffffffu, fo);
    if (t < n) {
      g.fo[t] = fo;
      g.rank[t] = __popc(peers & ((1u << lane) - 1u)) | (__popc(peers) << 8);
    }
  }
  __syncthreads();                                       // `first` is read; the table's memory is free
  for (int t = threadIdx.x; t < n; t += blockDim.x) g.size[t] = 0;
  __syncthreads();
  if (threadIdx.x < 32) {
    int fo = lane < n ? g.fo[lane] : 0, info = lane < n ? g.rank[lane] : 0;
    for (int t = lane; t < n32; t += 32) {
      const int next = t + 32;
      const int fo_next = next < n ? g.fo[next] : 0, info_next = next < n ? g.rank[next] : 0;
      const int before = t < n ? g.size[fo] : 0;
      __syncwarp();
      if (t < n) {
        g.rank[t] = before + (info & 255);
        if ((info & 255) == 0) g.size[fo] = before + (info >> 8);
      }
      __syncwarp();
      fo = fo_next;
      info = info_next;
    }
  }
  __syncthreads();
}

// exclusive prefix sum of the n values a[] into out[] over the whole block (a and out may not alias)
__device__ __forceinline__ void block_exclusive_scan(const int* a, int* out, int n, int* warp_sums /* [33] */) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int per = (n + blockDim.x - 1) / blockDim.x, lo = threadIdx.x * per, hi = min(n, lo + per);
  int s = 0;
  for (int k = lo; k < hi; ++k) s += a[k];
  int inc = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_sums[w] = inc;
  __syncthreads();
  if (w == 0) {
    const int x = lane < nw ? warp_sums[lane] : 0;
    int t = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    warp_sums[lane] = t - x;
  }
  __syncthreads();
  int run = warp_sums[w] + inc - s;
  for (int k = lo; k < hi; ++k) { out[k] = run; run += a[k]; }
  __syncthreads();
}

// ------------------------------------------------------------------ norm kernel
// One block (8 warps) per (example, 256-column slab, part of the rows).  The tokens are ordered by
// (first occurrence, position); the ordered rows are cut into 8 * parts contiguous ranges, one per
// warp, a group belonging to the range that holds its first row.  A lane owns 8 columns and folds a
// batch of rows (16-byte loads, all in flight together) into running group sums.  Groups of more
// than kEmbedLong rows (a frequent token) are summed by all eight warps, row w, w+8, ... each, and
// added in warp order.  Every row of G is read once.  Bound by latency: ordering the tokens, then one
// or two batches of loads; parts exist so that few examples still fill the chip, and three blocks per
// SM with 8 rows in flight per lane beat two with 16 (B = 64, T = 256: 19.8 against 26.2 us).
// Comparing every pair of tokens instead of hashing took (norm and its reduce, d = 768) 138 us at
// B = 6, T = 1024 against 24.6, 33.2 against 19.8 at B = 64, T = 256, 16.5 against 13.1 at B = 32, T = 128.
constexpr int kEmbedNormThreads = 256;
constexpr int kEmbedLong = 48;

template <typename T>
__global__ void __launch_bounds__(kEmbedNormThreads, 3)
embed_norm_kernel(const int* __restrict__ ids, const T* __restrict__ G, long long ldg, int Tn, int d,
                  int V, int slabs, int parts, float* __restrict__ partials, int* __restrict__ first_occ,
                  int* __restrict__ dev_status) {
  extern __shared__ __align__(16) int sm_i[];
  __shared__ float red[32];
  __shared__ int wsum[33];
  __shared__ int s_long[kEmbedMaxT / kEmbedLong + 1], s_nlong;
  __shared__ float s_part[8][kEmbedColsPerBlock];
  constexpr int kBatch = sizeof(T) == 2 ? 8 : 4, kLongBatch = kBatch;
  constexpr int kWarps = kEmbedNormThreads / 32;
  const int part = blockIdx.x % parts, slab = (blockIdx.x / parts) % slabs, i = blockIdx.x / (parts * slabs);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n32 = (Tn + 31) & ~31, slots = group_slots(Tn);
  int* keys = sm_i + 3 * n32;
  int* first = keys + slots;
  const TokenGroups g{sm_i, sm_i + n32, sm_i + 2 * n32, keys};
  int* s_start = keys + n32;             // group start in the order, at the first occurrence
  int* s_ord = first;                    // rows in order; sign bit = group end

  for (int t = threadIdx.x; t < Tn; t += blockDim.x) {
    int id = ids[size_t(i) * Tn + t];
    if (id < 0 || id >= V) {
      id = -1;
      if (dev_status) atomicOr(dev_status, DP_DEV_BAD_ID);
    }
    g.id[t] = id;
  }
  group_tokens(g, keys, first, slots, Tn);
  block_exclusive_scan(g.size, s_start, Tn, wsum);
  for (int t = threadIdx.x; t < Tn; t += blockDim.x) {
    const int fo = g.fo[t], r = s_start[fo] + g.rank[t];
    const bool end = g.rank[t] + 1 == g.size[fo];
    if (dp_in_range(r, Tn, dev_status)) s_ord[r] = t | (end ? int(0x80000000u) : 0);
    if (slab == 0 && part == 0 && first_occ) first_occ[size_t(i) * Tn + t] = fo;
  }
  // this block's ordered rows; the long groups among them, in order
  const int per = (Tn + kWarps * parts - 1) / (kWarps * parts);
  const int blo = min(Tn, part * kWarps * per), bhi = min(Tn, (part + 1) * kWarps * per);
  if (warp == 0) {
    int cnt = 0;
    for (int t0 = 0; t0 < Tn; t0 += 32) {
      const int t = t0 + lane;
      const bool is = t < Tn && g.size[t] > kEmbedLong && s_start[t] >= blo && s_start[t] < bhi;
      const unsigned m = __ballot_sync(0xffffffffu, is);
      if (is) s_long[cnt + __popc(m & ((1u << lane) - 1u))] = t;
      cnt += __popc(m);
    }
    if (lane == 0) s_nlong = cnt;
  }
  __syncthreads();

  const int c = slab * kEmbedColsPerBlock + 8 * lane;
  const int nvalid = min(8, d - c);
  const bool vec = ((reinterpret_cast<uintptr_t>(G) & 15) == 0) && ((ldg * sizeof(T)) % 16 == 0);
  const T* Gi = G + size_t(i) * Tn * ldg + c;
  // first group start at or after row r
  auto snap = [&](int r) {
    while (r > 0 && r < Tn && s_ord[r - 1] >= 0) {         // the previous row does not end a group
      const int fo = g.fo[s_ord[r - 1]];
      r = s_start[fo] + g.size[fo];
    }
    return min(r, Tn);
  };
  float tot = 0.f;
  if (nvalid > 0) {
    const int lo = snap(min(Tn, blo + warp * per)), hi = snap(min(Tn, blo + (warp + 1) * per));
    float run[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) run[e] = 0.f;
    int r0 = lo;
    while (r0 < hi) {
      const int t0 = s_ord[r0] & 0x7fffffff, fo0 = g.fo[t0];
      if (s_start[fo0] == r0 && g.size[fo0] > kEmbedLong) { r0 += g.size[fo0]; continue; }
      Raw8<T> v[kBatch];
      int o[kBatch];
      int nb = 0;                                          // rows of this batch
      bool stop = false;
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        const int r = r0 + b;
        o[b] = 0;
        if (!stop && r < hi) {
          o[b] = s_ord[r];
          const int t = o[b] & 0x7fffffff, fo = g.fo[t];
          if (b > 0 && g.size[fo] > kEmbedLong) {          // a long group starts: the batch ends here
            stop = true;
          } else {
            nb = b + 1;
            if (dp_in_range(t, Tn, dev_status) && g.id[t] >= 0) v[b].load(Gi + size_t(t) * ldg, nvalid, vec);
            else v[b].zero();
          }
        }
      }
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        if (b < nb) {
          float x[8];
          v[b].unpack(x);
#pragma unroll
          for (int e = 0; e < 8; ++e) run[e] += x[e];
          if (o[b] < 0) {
#pragma unroll
            for (int e = 0; e < 8; ++e) { tot = fmaf(run[e], run[e], tot); run[e] = 0.f; }
          }
        }
      }
      r0 += nb;
    }
  }
  const int n_long = s_nlong;
  for (int k = 0; k < n_long; ++k) {                       // uniform over the block
    const int fo = s_long[k], a = s_start[fo], b = a + g.size[fo];
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    if (nvalid > 0) {
      for (int r0 = a + warp; r0 < b; r0 += kWarps * kLongBatch) {
        Raw8<T> v[kLongBatch];
#pragma unroll
        for (int j = 0; j < kLongBatch; ++j) {
          const int r = r0 + kWarps * j;
          if (r < b) v[j].load(Gi + size_t(s_ord[r] & 0x7fffffff) * ldg, nvalid, vec);
          else v[j].zero();
        }
#pragma unroll
        for (int j = 0; j < kLongBatch; ++j) {
          float x[8];
          v[j].unpack(x);
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[e] += x[e];
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) s_part[warp][8 * lane + e] = acc[e];
    __syncthreads();
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) sum += s_part[w][threadIdx.x];
    tot = fmaf(sum, sum, tot);
    __syncthreads();
  }
  const float s = block_sum(tot, red);
  if (threadIdx.x == 0) partials[(size_t(i) * slabs + slab) * parts + part] = s;
}

// ------------------------------------------------------------------ side-stream kernels
// The kernels from here on run on a second stream beside the persistent tensor-core kernels, whose CTAs
// leave 4096 registers per SM (gemm_gta_big_kernel also 33 KiB of shared memory): blocks of 128
// threads with 32 registers (one warp per quarter of an SM, whose register file they share out) fit
// beside one; larger ones, such as the 256 and 1024 threads that these kernels had, wait until it has
// ended.  The step, sustained: GPT-2 small B = 64, T = 256 with positions 5442 -> 5349 us, DistilGPT2 with all
// its vectors B = 21, T = 203 1447 -> 1383, untied B = 32, T = 128 983 -> 937 (with the persistent kernels asking
// for the carve-out, see allow_shared).
constexpr int kSideThreads = 128;

// zeros; a memset's own kernel does not fit beside a persistent one
__global__ void __launch_bounds__(kSideThreads, 16) clear_kernel(uint4* __restrict__ p, size_t n16) {
  const size_t stride = size_t(gridDim.x) * kSideThreads;
#pragma unroll 4
  for (size_t k = size_t(blockIdx.x) * kSideThreads + threadIdx.x; k < n16; k += stride) p[k] = make_uint4(0, 0, 0, 0);
}

// ------------------------------------------------------------------ sort kernels
// Stable counting sort of the token ids: perm lists the positions by (id, position), seg[v] = number
// of positions with id < v.
//   few tokens and ids (sort_in_one_block): one kernel of one block (grouping, counts into seg, scan over V, placing);
//   more: the tokens are cut into chunks, one block each --
//     sort_rank_kernel   groups a chunk: rank of every token inside its chunk, counts[chunk][id],
//                        the total of every id and of every 1024 ids (integer atomics)
//     sort_scan_kernel   exclusive scan of the totals -> seg
//     sort_place_kernel  perm[seg[id] + counts of the chunks before + rank] = position
//   with more than kSortWalk chunks sort_prefix_kernel first turns counts[chunk][id] into those of the chunks
//   before, so that placing a token stays one read.
// Latency again: four short dependent launches.  Against histogram, prefix over the chunks, scan and a
// placing kernel that compared a token with all earlier ones of its chunk (V = 50257, Zipf ids, replayed as a graph): 9.5 ->
// 7.9 us at n = 8, 24.7 -> 18.6 at 4096, 33 -> 21 at 16384, 115 -> 34 at 131072, 6.1 -> 0.67 ms at 4 194 304.
constexpr int kSortThreads = 1024;
constexpr int kSortBlocksShared = 256;     // blocks of 1024 ids that a chunk counts in shared memory

__device__ __forceinline__ void load_ids(const int* ids, int n, int V, int* out, int* dev_status) {
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    int id = ids[t];
    if (id < 0 || id >= V) {
      id = -1;
      if (dev_status) atomicOr(dev_status, DP_DEV_BAD_ID);
    }
    out[t] = id;
  }
}

__global__ void __launch_bounds__(kSortThreads)
sort_one_block_kernel(const int* __restrict__ ids, int n, int V, int* __restrict__ seg,
                      int* __restrict__ perm, int* __restrict__ dev_status) {
  extern __shared__ __align__(16) int sm_i[];
  __shared__ int wsum[33];
  const int n32 = (n + 31) & ~31, slots = group_slots(n);
  int* keys = sm_i + 3 * n32;
  const TokenGroups g{sm_i, sm_i + n32, sm_i + 2 * n32, keys};
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int v = threadIdx.x; v <= V; v += kSortThreads) seg[v] = 0;
  load_ids(ids, n, V, g.id, dev_status);
  group_tokens(g, keys, keys + slots, slots, n);
  for (int t = threadIdx.x; t < n; t += kSortThreads)
    if (g.size[t] > 0 && g.id[t] >= 0) seg[g.id[t]] = g.size[t];
  __syncthreads();
  // exclusive scan over V, 8 entries per thread and step
  int carry = 0;
  for (int v0 = 0; v0 <= V; v0 += 8 * kSortThreads) {
    const int lo = v0 + 8 * threadIdx.x;
    int x[8], s = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) { x[e] = lo + e < V ? seg[lo + e] : 0; s += x[e]; }
    int inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    int before = carry, all = 0;
    for (int k = 0; k < kSortThreads / 32; ++k) {
      const int y = wsum[k];
      if (k < w) before += y;
      all += y;
    }
    int run = before + inc - s;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (lo + e <= V) seg[lo + e] = run;
      run += x[e];
    }
    carry += all;
    __syncthreads();
  }
  for (int t = threadIdx.x; t < n; t += kSortThreads) {
    const int id = g.id[t];
    if (id < 0) continue;
    const int dst = seg[id] + g.rank[t];
    if (dp_in_range(dst, n, dev_status)) perm[dst] = t;
  }
}

template <int kThreads>
__global__ void __launch_bounds__(kThreads, 2048 / kThreads)
sort_rank_kernel(const int* __restrict__ ids, int n, int V, int chunk_len, int* __restrict__ counts,
                 int* __restrict__ totals, int* __restrict__ blocks, int* __restrict__ rank,
                 int* __restrict__ dev_status) {
  extern __shared__ __align__(16) int sm_i[];
  const int chunk = blockIdx.x, j0 = chunk * chunk_len, m = min(chunk_len, n - j0);
  const int n32 = (m + 31) & ~31, slots = group_slots(m);
  int* keys = sm_i + 3 * n32;
  const TokenGroups g{sm_i, sm_i + n32, sm_i + 2 * n32, keys};
  load_ids(ids + j0, m, V, g.id, dev_status);
  group_tokens(g, keys, keys + slots, slots, m);
  // tokens per 1024 ids, added up for the chunk first (ids below 1024 are the most frequent)
  __shared__ int s_blocks[kSortBlocksShared];
  const int n_blocks = (V + 1023) >> 10;
  const bool shared = n_blocks <= kSortBlocksShared;
  if (shared) {
    for (int b = threadIdx.x; b < n_blocks; b += kThreads) s_blocks[b] = 0;
    __syncthreads();
  }
  for (int t = threadIdx.x; t < m; t += kThreads) {
    rank[j0 + t] = g.rank[t];
    const int id = g.id[t];
    if (id >= 0 && g.size[t] > 0) {
      counts[size_t(chunk) * V + id] = g.size[t];
      atomicAdd(&totals[id], g.size[t]);
      atomicAdd(shared ? &s_blocks[id >> 10] : &blocks[id >> 10], g.size[t]);
    }
  }
  if (shared) {
    __syncthreads();
    for (int b = threadIdx.x; b < n_blocks; b += kThreads)
      if (s_blocks[b]) atomicAdd(&blocks[b], s_blocks[b]);
  }
}

// counts[chunk][id] -> tokens of the id in earlier chunks
__global__ void __launch_bounds__(kSideThreads, 16)
sort_prefix_kernel(int* __restrict__ counts, int chunks, int V) {
  const int v = blockIdx.x * kSideThreads + threadIdx.x;
  if (v >= V) return;
  int run = 0;
  for (int c0 = 0; c0 < chunks; c0 += 8) {             // eight reads in flight
    int x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = c0 + k < chunks ? counts[size_t(c0 + k) * V + v] : 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (c0 + k < chunks) counts[size_t(c0 + k) * V + v] = run;
      run += x[k];
    }
  }
}

// exclusive scan of the totals: block b adds up those of the blocks before its 1024 entries.  (Reading all totals
// before them instead was a chain of loads of 10 us at V = 50257.)
__global__ void __launch_bounds__(kSideThreads, 16)
sort_scan_kernel(const int* __restrict__ totals, const int* __restrict__ blocks, int V, int* __restrict__ seg) {
  constexpr int kWarps = kSideThreads / 32;
  static_assert(kSideThreads * 8 == 1024, "eight entries per thread");
  __shared__ int wsum[kWarps], wbase[kWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int base = 0;
  for (int b = threadIdx.x; b < int(blockIdx.x); b += kSideThreads) base += blocks[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) base += __shfl_xor_sync(0xffffffffu, base, o);
  const int v0 = blockIdx.x * 1024 + 8 * threadIdx.x;
  int x[8], s = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) { x[e] = v0 + e < V ? totals[v0 + e] : 0; s += x[e]; }
  int inc = s;                                         // inclusive scan inside the warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) { wsum[w] = inc; wbase[w] = base; }
  __syncthreads();
  int run = inc - s;
#pragma unroll
  for (int k = 0; k < kWarps; ++k) run += wbase[k] + (k < w ? wsum[k] : 0);
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (v0 + e <= V) seg[v0 + e] = run;                // entry V: all tokens
    run += x[e];
  }
}

__global__ void __launch_bounds__(kSideThreads, 16)
sort_place_kernel(const int* __restrict__ ids, int n, int V, int chunk_len, const int* __restrict__ counts,
                  const int* __restrict__ rank, const int* __restrict__ seg, int* __restrict__ perm,
                  int prefixed, int* __restrict__ dev_status) {
  const int j = blockIdx.x * kSideThreads + threadIdx.x;
  if (j >= n) return;
  const int id = ids[j];
  if (id < 0 || id >= V) return;
  int dst = seg[id] + rank[j];
  const int chunk = j / chunk_len;
  if (prefixed) {
    dst += counts[size_t(chunk) * V + id];
  } else {
#pragma unroll 8
    for (int c = 0; c < chunk; ++c) dst += counts[size_t(c) * V + id];
  }
  if (dp_in_range(dst, n, dev_status)) perm[dst] = j;
}

// ------------------------------------------------------------------ segmented row sum
// The sorted order is cut into 32-position chunks; grid = (chunks, 128-column slabs).
//   pass 1 (embed_scatter_kernel): a block finds the segments (runs of one token id) that meet
//     its chunk.  Short segments (<= 32 rows) are summed by the warp in whose quarter of the chunk
//     they start, in sorted order, and written to the table.  Rows of LONG segments (a frequent
//     token) are summed per chunk by the whole block -- warp w takes rows w, w+4, ... and the four
//     warp sums are added in warp order -- into a partial buffer [chunk][slot][column]; slot 0 is the
//     segment that continues from the previous chunk, slot 1 the one that starts in this chunk
//     (a 32-position chunk can meet at most one of each).
//   pass 2 (embed_scatter_combine_kernel): the block whose chunk holds a long segment's head
//     adds that segment's partials in chunk order and writes the table row.
// Every order is fixed, so the result does not depend on timing (no floating-point atomics),
// and a very frequent token is spread over as many blocks as it has chunks.
constexpr int kScatChunk = 32;     // sorted positions per block
constexpr int kScatShort = 32;     // longest segment handled by a single warp
constexpr int kScatCols = 128;     // columns per block, four per lane
constexpr int kScatWarps = kSideThreads / 32;

// four consecutive values of one row
template <typename T> struct Raw4;
template <> struct Raw4<__nv_bfloat16> {
  uint2 q;
  __device__ __forceinline__ void load(const __nv_bfloat16* p, int nvalid, bool vec) {
    if (vec && nvalid >= 4) {
      q = *reinterpret_cast<const uint2*>(p);
    } else {
      uint32_t w[2] = {0u, 0u};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (e < nvalid) w[e >> 1] |= uint32_t(__bfloat16_as_ushort(p[e])) << (16 * (e & 1));
      q = make_uint2(w[0], w[1]);
    }
  }
  __device__ __forceinline__ float4 unpack() const {
    return make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u),
                       __uint_as_float(q.y << 16), __uint_as_float(q.y & 0xffff0000u));
  }
};
template <> struct Raw4<float> {
  float4 q;
  __device__ __forceinline__ void load(const float* p, int nvalid, bool vec) {
    if (vec && nvalid >= 4) q = *reinterpret_cast<const float4*>(p);
    else q = make_float4(p[0], nvalid > 1 ? p[1] : 0.f, nvalid > 2 ? p[2] : 0.f, nvalid > 3 ? p[3] : 0.f);
  }
  __device__ __forceinline__ float4 unpack() const { return q; }
};
__device__ __forceinline__ void fma4(float4& a, float r, const float4& x) {
  a.x = fmaf(r, x.x, a.x); a.y = fmaf(r, x.y, a.y); a.z = fmaf(r, x.z, a.z); a.w = fmaf(r, x.w, a.w);
}

template <typename T>
__global__ void __launch_bounds__(kSideThreads, 16)
embed_scatter_kernel(const int* __restrict__ ids, const T* __restrict__ G, long long ldg, int Tn,
                     int d, const float* __restrict__ clip, const int* __restrict__ perm,
                     const int* __restrict__ seg, int V, float* __restrict__ out, long long ldo,
                     float beta, float scale, float* __restrict__ long_part, int n_rows,
                     int* __restrict__ dev_status) {
  constexpr int kBatch = sizeof(T) == 2 ? 4 : 2;         // row loads in flight per lane
  static_assert(kScatChunk + kScatShort <= kSideThreads, "one staged row per thread");
  __shared__ float4 part[kScatWarps][kScatCols / 4];
  __shared__ int s_pos[kScatChunk + kScatShort], s_end[kScatChunk + kScatShort], s_n[kScatChunk];
  __shared__ float s_r[kScatChunk + kScatShort];
  __shared__ unsigned s_short, s_long0, s_long1;
  const int n_valid = seg[V];
  const int kc = blockIdx.x * kScatChunk;
  if (kc >= n_valid) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;

  // ---- stage positions and clip factors of the chunk and of the kScatShort rows after it, and
  //      classify the chunk's positions (warp 0)
  {
    const int k = kc + threadIdx.x;
    int pos = 0, v = -1;
    const bool staged = threadIdx.x < kScatChunk + kScatShort;
    if (staged && k < n_valid) {
      pos = perm[k];
      if (!dp_in_range(pos, n_rows, dev_status)) pos = 0;   // checked build: flagged, row 0 stands in
      if (w == 0) v = ids[pos];                             // on its way while the factor is waited for
      s_pos[threadIdx.x] = pos;
      s_r[threadIdx.x] = clip[pos / Tn];
    }
    if (staged) s_end[threadIdx.x] = -1;
    if (w == 0) {
      int n = 0, s0 = 0;
      if (k < n_valid && dp_in_range(v, V, dev_status)) {
        s0 = seg[v];
        n = seg[v + 1] - s0;
      }
      const bool head = n > 0 && s0 == k, is_long = n > kScatShort;
      const unsigned sh = __ballot_sync(0xffffffffu, head && !is_long);
      const unsigned l0 = __ballot_sync(0xffffffffu, is_long && s0 < kc);     // continues from before
      const unsigned l1 = __ballot_sync(0xffffffffu, is_long && s0 >= kc);    // starts in this chunk
      if (lane == 0) { s_short = sh; s_long0 = l0; s_long1 = l1; }
      s_n[lane] = n;
      __syncwarp();
    }
    __syncthreads();
    if (w == 0 && ((s_short >> lane) & 1u)) s_end[lane + s_n[lane] - 1] = v;   // id at a segment's last row
  }
  __syncthreads();

  const int c = blockIdx.y * kScatCols + lane * 4;
  const int nvalid = min(4, d - c);
  const bool vec = (reinterpret_cast<uintptr_t>(G) % (4 * sizeof(T)) == 0) && ((ldg & 3) == 0);
  const bool ovec = ((reinterpret_cast<uintptr_t>(out) & 15) == 0) && ((ldo & 3) == 0) && nvalid == 4;

  // ---- short segments: a warp takes those that start in its part of the chunk.  Their rows lie one after
  //      the other (a long segment can only be the chunk's last), so batches of loads run across them.
  constexpr int kPerWarp = kScatChunk / kScatWarps;
  const unsigned mine = s_short & (((1u << kPerWarp) - 1u) << (kPerWarp * w));
  if (mine != 0u && nvalid > 0) {
    const int last = 31 - __clz(mine), end = last + s_n[last];
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int o0 = __ffs(mine) - 1; o0 < end; o0 += kBatch) {
      Raw4<T> g[kBatch];
#pragma unroll
      for (int b = 0; b < kBatch; ++b)
        if (o0 + b < end) g[b].load(G + size_t(s_pos[o0 + b]) * ldg + c, nvalid, vec);
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        if (o0 + b >= end) break;
        fma4(acc, s_r[o0 + b], g[b].unpack());
        const int v = s_end[o0 + b];
        if (v >= 0) {
          float* o = out + size_t(v) * ldo + c;
          if (ovec) {
            float4 p = make_float4(acc.x * scale, acc.y * scale, acc.z * scale, acc.w * scale);
            if (beta != 0.f) {
              const float4 q = *reinterpret_cast<const float4*>(o);
              p.x += q.x; p.y += q.y; p.z += q.z; p.w += q.w;
            }
            *reinterpret_cast<float4*>(o) = p;
          } else {
            const float a[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) if (e < nvalid) o[e] = (beta != 0.f ? o[e] : 0.f) + a[e] * scale;
          }
          acc = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
  }

  // ---- rows of long segments inside this chunk: per-chunk partial sums
#pragma unroll 1
  for (int slot = 0; slot < 2; ++slot) {
    const unsigned m = slot == 0 ? s_long0 : s_long1;
    if (m == 0u) continue;                               // uniform over the block
    const int a = __ffs(m) - 1, b = 32 - __clz(m);       // the rows form one run [a, b)
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (nvalid > 0) {
      for (int k0 = a + w; k0 < b; k0 += kScatWarps * kBatch) {
        Raw4<T> g[kBatch];
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
          if (k0 + kScatWarps * j < b) g[j].load(G + size_t(s_pos[k0 + kScatWarps * j]) * ldg + c, nvalid, vec);
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
          if (k0 + kScatWarps * j < b) fma4(acc, s_r[k0 + kScatWarps * j], g[j].unpack());
      }
    }
    part[w][lane] = acc;
    __syncthreads();
    const int cc = blockIdx.y * kScatCols + threadIdx.x;
    if (cc < d) {
      float sum = 0.f;
#pragma unroll
      for (int ww = 0; ww < kScatWarps; ++ww) sum += reinterpret_cast<const float*>(part[ww])[threadIdx.x];
      long_part[(size_t(blockIdx.x) * 2 + slot) * d + cc] = sum;
    }
    __syncthreads();
  }
}

// pass 2: table row of every long segment = beta*row + scale * (its partials in chunk order)
__global__ void __launch_bounds__(kSideThreads, 16)
embed_scatter_combine_kernel(const int* __restrict__ ids, const int* __restrict__ perm,
                             const int* __restrict__ seg, int V, int d,
                             const float* __restrict__ long_part, float* __restrict__ out,
                             long long ldo, float beta, float scale, int n_rows,
                             int* __restrict__ dev_status) {
  __shared__ int s_v, s_k0, s_n;
  const int n_valid = seg[V];
  const int kc = blockIdx.x * kScatChunk;
  if (kc >= n_valid) return;
  if (threadIdx.x < 32) {                                // at most one long head per chunk
    const int k = kc + threadIdx.x;
    int v = -1, n = 0;
    bool long_head = false;
    if (k < n_valid) {
      const int pos = perm[k];
      if (dp_in_range(pos, n_rows, dev_status)) v = ids[pos];
      if (dp_in_range(v, V, dev_status)) {
        const int s0 = seg[v];
        n = seg[v + 1] - s0;
        long_head = (s0 == k) && (n > kScatShort);
      }
    }
    if (threadIdx.x == 0) s_n = 0;
    __syncwarp();
    if (long_head) { s_v = v; s_k0 = k; s_n = n; }
  }
  __syncthreads();
  const int n = s_n;
  if (n == 0) return;
  const int cc = blockIdx.y * kSideThreads + threadIdx.x;
  if (cc >= d) return;
  const int c0 = blockIdx.x, c1 = (s_k0 + n - 1) / kScatChunk;
  float sum = long_part[(size_t(c0) * 2 + 1) * d + cc];            // starts in its own chunk
#pragma unroll 8
  for (int cch = c0 + 1; cch <= c1; ++cch) sum += long_part[(size_t(cch) * 2 + 0) * d + cc];
  float* o = out + size_t(s_v) * ldo + cc;
  sum *= scale;
  *o = (beta != 0.f) ? (*o + sum) : sum;
}

}  // namespace

// Row parts per (example, slab): enough blocks for two per SM, at least 64 rows (8 per warp) each.
// A function of the sizes alone, since the partial sums it implies are part of the workspace size.
int embed_norm_parts(int B, int T, int d) {
  const long long blocks = (long long)B * ceil_div(d, kEmbedColsPerBlock);
  return (int)std::max(1LL, std::min((long long)ceil_div(T, 64), (296 + blocks - 1) / blocks));
}

dp_status launch_embed_norms(const int* ids, const void* G, int64_t ldg, dp_dtype dt, int B, int T,
                             int d, int V, int parts, float* partials, int* first_occ, int* dev_status,
                             cudaStream_t st) {
  const int slabs = ceil_div(d, kEmbedColsPerBlock);
  const size_t smem = group_smem_bytes(T);
  if (first_use_on_this_device(reinterpret_cast<const void*>(&launch_embed_norms))) {
    DP_CUDA_OK(cudaFuncSetAttribute(embed_norm_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)group_smem_bytes(kEmbedMaxT)));
    DP_CUDA_OK(cudaFuncSetAttribute(embed_norm_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)group_smem_bytes(kEmbedMaxT)));
    DP_CUDA_OK(prefer_max_shared(embed_norm_kernel<float>));
    DP_CUDA_OK(prefer_max_shared(embed_norm_kernel<__nv_bfloat16>));
  }
  const int grid = B * slabs * parts;
  if (dt == DP_F32)
    embed_norm_kernel<float><<<grid, kEmbedNormThreads, smem, st>>>(
        ids, (const float*)G, ldg, T, d, V, slabs, parts, partials, first_occ, dev_status);
  else
    embed_norm_kernel<__nv_bfloat16><<<grid, kEmbedNormThreads, smem, st>>>(
        ids, (const __nv_bfloat16*)G, ldg, T, d, V, slabs, parts, partials, first_occ, dev_status);
  DP_LAUNCH_OK();
  return DP_OK;
}

dp_status launch_clear(void* p, size_t bytes, cudaStream_t st) {
  if ((reinterpret_cast<uintptr_t>(p) & 15) != 0) {
    DP_CUDA_OK(cudaMemsetAsync(p, 0, bytes, st));
    return DP_OK;
  }
  const size_t n16 = bytes / 16;
  if (n16) {
    if (first_use_on_this_device(reinterpret_cast<const void*>(&launch_clear)))
      DP_CUDA_OK(prefer_max_shared(clear_kernel));
    const size_t blocks = std::min((n16 + kSideThreads - 1) / kSideThreads, size_t(sm_count()) * 16);
    clear_kernel<<<(unsigned)blocks, kSideThreads, 0, st>>>(static_cast<uint4*>(p), n16);
    DP_LAUNCH_OK();
  }
  if (bytes & 15) DP_CUDA_OK(cudaMemsetAsync(static_cast<char*>(p) + n16 * 16, 0, bytes & 15, st));
  return DP_OK;
}

dp_status launch_embed_sort(const int* ids, int n, int V, const EmbedSortWs& ws, int* dev_status,
                            cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&launch_embed_sort))) {
    DP_CUDA_OK(cudaFuncSetAttribute(sort_one_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)group_smem_bytes(kSortOneBlock)));
    DP_CUDA_OK(allow_shared(sort_rank_kernel<kSideThreads>, group_smem_bytes(kSortChunk)));
    DP_CUDA_OK(allow_shared(sort_rank_kernel<4 * kSideThreads>, group_smem_bytes(4 * kSortChunk)));
    DP_CUDA_OK(prefer_max_shared(sort_one_block_kernel));
    DP_CUDA_OK(prefer_max_shared(sort_scan_kernel));
    DP_CUDA_OK(prefer_max_shared(sort_prefix_kernel));
    DP_CUDA_OK(prefer_max_shared(sort_place_kernel));
  }
  if (sort_in_one_block(n, V)) {
    sort_one_block_kernel<<<1, kSortThreads, group_smem_bytes(n), st>>>(ids, n, V, ws.seg, ws.perm, dev_status);
    DP_LAUNCH_OK();
    return DP_OK;
  }
  // short chunks keep a block's walk over its tokens short; with many tokens longer ones keep the
  // counts of the chunks before a token few
  const int chunk_len = n <= 32 * kSortChunk ? kSortChunk : 4 * kSortChunk;
  const int chunks = ceil_div(n, chunk_len);
  const int blocks = ceil_div(V, 1024);
  int* block_totals = ws.totals + V;
  int* counts = block_totals + blocks;
  dp_status s = launch_clear(ws.totals, align_up((size_t(V) + blocks + size_t(chunks) * V) * sizeof(int), 16), st);
  if (s != DP_OK) return s;
  if (chunk_len == kSortChunk)
    sort_rank_kernel<kSideThreads><<<chunks, kSideThreads, group_smem_bytes(chunk_len), st>>>(
        ids, n, V, chunk_len, counts, ws.totals, block_totals, ws.rank, dev_status);
  else
    sort_rank_kernel<4 * kSideThreads><<<chunks, 4 * kSideThreads, group_smem_bytes(chunk_len), st>>>(
        ids, n, V, chunk_len, counts, ws.totals, block_totals, ws.rank, dev_status);
  DP_LAUNCH_OK();
  const bool prefix = chunks > kSortWalk;
  if (prefix) {
    sort_prefix_kernel<<<ceil_div(V, kSideThreads), kSideThreads, 0, st>>>(counts, chunks, V);
    DP_LAUNCH_OK();
  }
  sort_scan_kernel<<<ceil_div(V + 1, 1024), kSideThreads, 0, st>>>(ws.totals, block_totals, V, ws.seg);
  DP_LAUNCH_OK();
  sort_place_kernel<<<ceil_div(n, kSideThreads), kSideThreads, 0, st>>>(ids, n, V, chunk_len, counts, ws.rank,
                                                                       ws.seg, ws.perm, prefix ? 1 : 0, dev_status);
  DP_LAUNCH_OK();
  return DP_OK;
}

// Test hook of the checked build: one thread runs the range test on (idx, n) and touches no
// memory -- shows that an index outside its array is reported (and only in the checked build).
__global__ void bounds_probe_kernel(long long idx, long long n, int* dev_status) {
  (void)dp_in_range(idx, n, dev_status);
}
dp_status launch_bounds_probe(long long idx, long long n, int* dev_status, cudaStream_t st) {
  bounds_probe_kernel<<<1, 1, 0, st>>>(idx, n, dev_status);
  DP_LAUNCH_OK();
  return DP_OK;
}

size_t embed_scatter_partial_bytes(long long n, int d) {
  return align_up(size_t((n + kScatChunk - 1) / kScatChunk) * 2 * size_t(d) * sizeof(float), 256);
}

dp_status launch_embed_scatter(const int* ids, const void* G, int64_t ldg, dp_dtype dt, int n,
                               int T, int d, int V, const float* clip, const int* perm,
                               const int* seg, float* out, int64_t ldo, float beta, float scale,
                               bool clear, float* long_part, cudaStream_t st, int* dev_status) {
  // beta == 0: the table is cleared once (unless the caller already filled it, e.g. with
  // noise), then every touched row receives table + scale*sum
  if (beta == 0.f && clear) {
    DP_CUDA_OK(cudaMemset2DAsync(out, size_t(ldo) * sizeof(float), 0, size_t(d) * sizeof(float),
                                 size_t(V), st));
  }
  if (first_use_on_this_device(reinterpret_cast<const void*>(&launch_embed_scatter))) {
    DP_CUDA_OK(prefer_max_shared(embed_scatter_kernel<float>));
    DP_CUDA_OK(prefer_max_shared(embed_scatter_kernel<__nv_bfloat16>));
    DP_CUDA_OK(prefer_max_shared(embed_scatter_combine_kernel));
  }
  static_assert(kScatCols == kSideThreads, "both passes take 128 columns per block");
  const dim3 grid(ceil_div(n, kScatChunk), ceil_div(d, kScatCols));
  if (dt == DP_F32)
    embed_scatter_kernel<float><<<grid, kSideThreads, 0, st>>>(ids, (const float*)G, ldg, T, d, clip, perm,
                                                     seg, V, out, ldo, 1.f, scale, long_part, n,
                                                     dev_status);
  else
    embed_scatter_kernel<__nv_bfloat16><<<grid, kSideThreads, 0, st>>>(ids, (const __nv_bfloat16*)G, ldg, T,
                                                             d, clip, perm, seg, V, out, ldo, 1.f,
                                                             scale, long_part, n, dev_status);
  DP_LAUNCH_OK();
  if (n <= kScatShort) return DP_OK;                     // no segment is long
  embed_scatter_combine_kernel<<<grid, kSideThreads, 0, st>>>(ids, perm, seg, V, d, long_part, out, ldo, 1.f,
                                                     scale, n, dev_status);
  DP_LAUNCH_OK();
  return DP_OK;
}

}  // namespace dpg
