// Ghost norm of linear layers on tcgen05 tensor cores (bf16 in, fp32 accumulate).
//
// For example i and a linear layer with input A_i (T x d) and output gradient G_i (T x p),
// the squared Frobenius norm of the per-example weight gradient G_i^T A_i equals
// <A_i A_i^T, G_i G_i^T>_F (Eq. 4 - Eq. 5 extended from one token to T tokens).  A work item
// is one 128 x 128 tile pair (ti <= tj) of the two T x T Gram matrices of one (layer,
// example): both tiles are accumulated in tensor memory, multiplied element by element and
// summed by the epilogue warps; off-diagonal tile pairs count twice (symmetry).
//
// The Frobenius product is linear in each Gram matrix, so a very wide operand (the LM head's
// V = 50257 columns) is split into column chunks handled by different CTAs; each chunk CTA
// recomputes the full Gram tile of the narrow operand.
//
// Roles per CTA (192 threads): warp 0 = TMA producer, warp 1 = MMA issuer (one thread),
// warps 2..5 = epilogue.  Two TMEM accumulator sets let the epilogue of one item overlap the
// MMAs of the next.  Partial sums go to a workspace and are added in a fixed order by a
// second kernel, so results are deterministic.
#include <cuda.h>
#include <cuda_bf16.h>

#include "dp_common.cuh"
#include "ghost_plan.cuh"
#include "ptx_sm100.cuh"
#include "tma_host.cuh"

namespace dpg {

namespace {

constexpr int kTile = 128;                       // Gram tile edge (rows of A_i / G_i)
constexpr int kKStep = 64;                       // bf16 columns per stage row (128 bytes)
constexpr int kTileBytes = kTile * kKStep * 2;   // 16 KiB
// A stage holds row tile ti and, for off-diagonal tile pairs, row tile tj.  When T <= 128 every
// pair is diagonal, so stages shrink to one tile and twice as many are kept in flight (the
// kernel is HBM-bound there: bytes in flight are what counts).  Split operands (fp32 inputs) bring
// two tiles, high and low terms, for each.
// Up to 64 tokens tiles are as tall as their examples, rounded up to 16 rows (kShort), and where that is less than half
// of one a stage holds two or four of them, 64 columns each (kBoxes): a stage's hand-offs take 550 cycles whatever it
// carries.  Where there is work enough a tile holds several examples (kPacked): the rows of a batch lie one after the
// other, so 128 / T of them fill it, its Gram matrix has theirs on the diagonal, and the epilogue multiplies only those
// blocks.  An example by itself has the plainer epilogue (a GPT-2-small block at B = 1, 2 and 4, T = 64 10.0, 10.8 and
// 10.8 us with the other, 9.7, 10.3 and 10.3 with its own).  97 layers of d = 128 at B = 95, T = 17 115 -> 50 us, 49 at
// B = 91, T = 39 70 -> 50; never so many examples that fewer than two items per SM remain (5 fp32 layers at B = 2, T =
// 54: 7.7 -> 10.2 with both in one tile).  Above 64 tokens short tiles and sizes known at run time cost more than they
// save (115 -> 122 us at B = 32, T = 128): there tiles are full and everything is constant.
constexpr int kRingBytes = 12 * kTileBytes;
constexpr int kMaxStages = 32;
constexpr size_t kSmemBytes = kRingBytes + 1024 /*alignment slack*/ + 1024 /*barriers*/ + 4 * kTile * sizeof(float) /*row sums*/;
constexpr int kThreads = 192;
constexpr int kTmemCols = 512;                   // 2 buffers x (S_A 128 + S_G 128) columns; split: hi hi, small products

// rows of a tile: a tile of one example's; one short example's; several short examples'
enum Rows { kFullTile, kShortTile, kPackedTile };

struct __align__(64) GhostParams {
  CUtensorMap tmA[kGhostMaxLayers];
  CUtensorMap tmG[kGhostMaxLayers];
  GhostLayerPlan layer[kGhostMaxLayers];
  int n_layers;
  int B, T, nt, ntp;
  int rows, stages;          // short: rows of a tile, stages of the ring
  int pack;                  // packed: examples per tile
  int low_plane;             // split operands: first plane of low terms
  int total_items;
  int n_per;                 // partial sums per example in the workspace
  float* partials;           // [B][n_per]
  int* dev_status;
  long long wait_limit;      // cycles a barrier wait may take before the CTA gives up
};

struct Item {
  int layer, example, ti, tj, a0, a1, g0, g1, pidx;      // packed: which tile of examples; its place in an example's sums
};

// `l` is the caller's running layer index: a role's items ascend, so the search goes on from the layer
// of its previous item instead of walking the list (a constant-memory line per layer) every time.
template <bool kPacked>
__device__ __forceinline__ Item decode_item(const GhostParams& P, int item, int& l) {
  Item it;
  while (l + 1 < P.n_layers && item >= P.layer[l + 1].item_begin) ++l;
  const GhostLayerPlan& L = P.layer[l];
  const int local = item - L.item_begin;
  const int s = local % L.nsplit;
  const int tp = (local / L.nsplit) % P.ntp;
  it.example = local / (L.nsplit * P.ntp);
  it.layer = l;
  int ti = 0, rem = tp;                   // tile pairs enumerated row by row, tj >= ti
  while (rem >= P.nt - ti) { rem -= P.nt - ti; ++ti; }
  it.ti = ti;
  it.tj = ti + rem;
  const int c0 = s * L.chunk_steps;
  if (L.split_on_g) {
    it.a0 = 0; it.a1 = L.a_steps;
    it.g0 = c0; it.g1 = min(c0 + L.chunk_steps, L.g_steps);
  } else {
    it.g0 = 0; it.g1 = L.g_steps;
    it.a0 = c0; it.a1 = min(c0 + L.chunk_steps, L.a_steps);
  }
  it.pidx = (kPacked ? 0 : it.example * P.n_per) + L.col_begin + tp * L.nsplit + s;
  return it;
}

__device__ __forceinline__ uint32_t add_f32(uint32_t a, uint32_t b) {
  return __float_as_uint(__uint_as_float(a) + __uint_as_float(b));
}

// kSplit: fp32 operands stored as bf16 planes of high and low terms (see split_kernels.cu).  Every Gram
// tile is then S = hi hi^T + hi lo^T + lo hi^T, three MMAs per K step on tiles loaded once.  An MMA rounds its sum
// towards zero, by as much as the sum is large, and the diagonal of S is a sum of positive terms: the two small
// products have an accumulator of their own, the second buffer's, which leaves a third of the roundings.
// 25 layers of DistilGPT2's shapes at B = 64, T = 256, error against 64 bits: 2.2e-5 with all three in one, now
// 1.4e-5.  The epilogue no longer overlaps the next item's MMAs; fewer chunks of wide operands make up for it (the fp32
// step of DistilGPT2 at B = 8, T = 128: no difference beyond 0.5 %).
template <bool kDiagOnly, bool kSplit, Rows kRows, int kBoxes>
__global__ void __launch_bounds__(kThreads, 1)
ghost_norm_tc_kernel(const __grid_constant__ GhostParams P) {
  constexpr bool kShort = kRows != kFullTile, kPacked = kRows == kPackedTile;
  static_assert(kDiagOnly || !kShort, "short tiles: diagonal pairs only");
  static_assert(kShort || kBoxes == 1, "several column tiles per stage: short tiles only");
  // an MMA reads 128 rows of its first operand whatever `rows` is: rows beyond it come from the next
  // stages (the ring ends a whole tile after its last tile begins) and fill accumulator rows nobody reads
  const int rows = kShort ? P.rows : kTile;
  const uint32_t tile_bytes = uint32_t(rows) * (kKStep * 2);
  const uint32_t term_bytes = (kSplit ? 2 : 1) * tile_bytes;             // one row tile, all its terms
  const uint32_t stage_bytes = (kDiagOnly ? kBoxes : 2) * term_bytes;
  const int n_stages = kShort ? P.stages : kRingBytes / int((kDiagOnly ? 1 : 2) * (kSplit ? 2 : 1) * kTileBytes);
  extern __shared__ uint8_t smem_raw[];
  // 128-byte swizzled tiles need 1024-byte alignment
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + kRingBytes);
  uint64_t* full = bars;                   // [n_stages] TMA -> MMA
  uint64_t* empty = bars + kMaxStages;     // [n_stages] MMA -> TMA
  uint64_t* acc_full = bars + 2 * kMaxStages; // [2]     MMA -> epilogue
  uint64_t* acc_empty = acc_full + 2;      // [2]        epilogue -> MMA
  uint64_t* mma_done = acc_empty + 2;      // only used when the MMA issuer gives up
  uint64_t* red_bar = mma_done + 1;        // [4]        epilogue warps -> epilogue warp 0
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(red_bar + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* epi_red = reinterpret_cast<float*>(tmem_slot + 2);   // [4][4]; packed: [4][kTile], a sum for each row

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < n_stages; ++s) { ptx::mbar_init(&full[s], 1); ptx::mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { ptx::mbar_init(&acc_full[b], 1); ptx::mbar_init(&acc_empty[b], 4); }
    ptx::mbar_init(mma_done, 1);
    for (int b = 0; b < 4; ++b) ptx::mbar_init(&red_bar[b], 4);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) {                    // one warp owns the TMEM allocation
    ptx::tmem_alloc(tmem_slot, kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tiles_a = ptx::smem_u32(tiles), full_a = ptx::smem_u32(full), empty_a = ptx::smem_u32(empty);

  if (warp == 0) {
    // ------------------------------------------------------------- TMA producer
    // producer and issuer: the whole warp runs the loop, an elected lane issues (see ptx::warp_ok)
    uint32_t stage = 0, phase = 0, issued = 0;
    int lay = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < P.total_items && ok; item += gridDim.x) {
      const Item it = decode_item<kPacked>(P, item, lay);
      const bool diag = kDiagOnly || (it.ti == it.tj);
      const uint32_t bytes = diag ? term_bytes : stage_bytes;
      const int ex = kPacked ? 0 : it.example, low = ex + P.low_plane;       // planes (split: high and low terms)
      const int row_i = kPacked ? it.example * P.pack * P.T : it.ti * kTile;
      for (int pass = 0; pass < 2 && ok; ++pass) {
        const uint64_t tm = reinterpret_cast<uint64_t>(pass == 0 ? &P.tmA[it.layer] : &P.tmG[it.layer]);
        const int k0 = pass == 0 ? it.a0 : it.g0, k1 = pass == 0 ? it.a1 : it.g1;
        for (int k = k0; k < k1; k += kBoxes) {
          ok = ptx::warp_ok(ptx::mbar_wait_a(empty_a + 8 * stage, phase ^ 1, abort_flag, P.wait_limit));
          if (!ok) break;
          const uint32_t dst = tiles_a + stage * stage_bytes, bar = full_a + 8 * stage;
          const int nb = kShort ? min(kBoxes, k1 - k) : 1;
          if (ptx::elect_one()) {
            ptx::mbar_arrive_expect_tx_a(bar, kShort ? nb * term_bytes : bytes);
#pragma unroll
            for (int b = 0; b < kBoxes; ++b) {
              if (b >= nb) break;
              ptx::tma_load_3d_a(dst + b * term_bytes, tm, bar, (k + b) * kKStep, row_i, ex);
              if (kSplit)
                ptx::tma_load_3d_a(dst + b * term_bytes + tile_bytes, tm, bar, (k + b) * kKStep, row_i, low);
            }
            if (!diag) {
              ptx::tma_load_3d_a(dst + term_bytes, tm, bar, k * kKStep, it.tj * kTile, ex);
              if (kSplit)
                ptx::tma_load_3d_a(dst + term_bytes + tile_bytes, tm, bar, k * kKStep, it.tj * kTile, low);
            }
          }
          __syncwarp();
          ++issued;
          if (++stage == uint32_t(n_stages)) { stage = 0; phase ^= 1; }
        }
      }
    }
    if (!ok && ptx::elect_one()) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
      ptx::drain_issued_copies(full, n_stages, issued);   // copies in flight land before exit
    }
  } else if (warp == 1) {
    // --------------------------------------------------------------- MMA issuer
    const uint32_t idesc = ptx::idesc_bf16_f32(kTile, rows, 0, 0);
    // K-major operand, 128-byte swizzle: 8-row groups are 1024 bytes apart; 16 bf16 = 32 bytes
    // further along K inside the swizzle atom
    constexpr uint64_t dbase = ptx::smem_desc_base(16, 1024, ptx::SWIZZLE_128B);
    constexpr uint32_t desc_hi = uint32_t(dbase >> 32);
    const uint32_t desc_lo0 = uint32_t(dbase) | ((tiles_a >> 4) & 0x3FFF);
    uint32_t stage = 0, phase = 0, n_item = 0;
    int lay = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < P.total_items && ok; item += gridDim.x, ++n_item) {
      const Item it = decode_item<kPacked>(P, item, lay);
      const bool diag = kDiagOnly || (it.ti == it.tj);
      const uint32_t buf = kSplit ? 0 : n_item & 1, acc_phase = (kSplit ? n_item : n_item >> 1) & 1;
      ok = ptx::warp_ok(ptx::mbar_wait(&acc_empty[buf], acc_phase ^ 1, abort_flag, P.wait_limit));
      if (!ok) break;
      ptx::tc_fence_after();
      for (int pass = 0; pass < 2 && ok; ++pass) {
        const uint32_t d_tmem = tmem_base + buf * 256 + pass * 128;
        const int nsteps = pass == 0 ? it.a1 - it.a0 : it.g1 - it.g0;
        for (int k = 0; k < nsteps; k += kBoxes) {
          ok = ptx::warp_ok(ptx::mbar_wait_a(full_a + 8 * stage, phase, abort_flag, P.wait_limit));
          if (!ok) break;
          ptx::tc_fence_after();
          const int nb = kShort ? min(kBoxes, nsteps - k) : 1;
          if (ptx::elect_one()) {
#pragma unroll
            for (int b = 0; b < kBoxes; ++b) {
              if (b >= nb) break;
              const uint32_t sa = desc_lo0 + ((stage * stage_bytes + b * term_bytes) >> 4);
              const uint32_t sb = diag ? sa : sa + (term_bytes >> 4);
#pragma unroll
              for (int kk = 0; kk < kKStep / 16; ++kk) {
                const uint32_t ah = sa + kk * 2, bh = sb + kk * 2, low = tile_bytes >> 4;
                ptx::mma_bf16_ss_lh(d_tmem, ah, bh, desc_hi, idesc, (k + b > 0 || kk > 0) ? 1u : 0u);
                if (kSplit) {
                  ptx::mma_bf16_ss_lh(d_tmem + 256, ah, bh + low, desc_hi, idesc, (k + b > 0 || kk > 0) ? 1u : 0u);
                  ptx::mma_bf16_ss_lh(d_tmem + 256, ah + low, bh, desc_hi, idesc, 1u);
                }
              }
            }
            ptx::mma_commit_a(empty_a + 8 * stage);      // stage reusable once these MMAs retire
            if (pass == 1 && k + nb >= nsteps) ptx::mma_commit(&acc_full[buf]);     // both Gram tiles complete
          }
          __syncwarp();
          if (++stage == uint32_t(n_stages)) { stage = 0; phase ^= 1; }
        }
      }
    }
    if (!ok && ptx::elect_one()) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
      ptx::drain_issued_mmas(mma_done, false);
    }
  } else {
    // ----------------------------------------------------------------- epilogue
    const int q = warp & 3;                          // TMEM lane quarter this warp may read
    const int ew = warp - 2;
    uint32_t n_item = 0;
    int lay = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < P.total_items && ok; item += gridDim.x, ++n_item) {
      const Item it = decode_item<kPacked>(P, item, lay);
      const uint32_t buf = kSplit ? 0 : n_item & 1, acc_phase = (kSplit ? n_item : n_item >> 1) & 1;
      if (!ptx::mbar_wait_relaxed(&acc_full[buf], acc_phase, abort_flag, P.wait_limit)) { ok = false; break; }
      ptx::tc_fence_after();
      const uint32_t t0 = tmem_base + (uint32_t(q * 32) << 16) + buf * 256;
      float acc = 0.f;
      // packed: this row's example and the columns of its tokens; the warp's rows have those of [c_lo, c_hi)
      const int row = q * 32 + lane, own = kPacked ? row / P.T * P.T : 0;
      const int c_lo = kPacked ? (q * 32 / P.T * P.T) & ~15 : 0;
      const int c_hi = kPacked ? min(rows, (q * 32 + 31) / P.T * P.T + P.T) : 0;
      auto add32 = [&](int c) {
        uint32_t ra[32], rg[32];
        ptx::tmem_ld_32x32b_x32(t0 + c, ra);
        ptx::tmem_ld_32x32b_x32(t0 + 128 + c, rg);
        if (kSplit) {
          uint32_t sa[32], sg[32];
          ptx::tmem_ld_32x32b_x32(t0 + 256 + c, sa);
          ptx::tmem_ld_32x32b_x32(t0 + 384 + c, sg);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) { ra[j] = add_f32(ra[j], sa[j]); rg[j] = add_f32(rg[j], sg[j]); }
        } else {
          ptx::tmem_ld_wait();
        }
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (!kPacked || unsigned(c + j - own) < unsigned(P.T))
            acc = fmaf(__uint_as_float(ra[j]), __uint_as_float(rg[j]), acc);
      };
      auto add16 = [&](int c) {                          // the last 16 columns
        uint32_t ra[16], rg[16];
        ptx::tmem_ld_32x32b_x16(t0 + c, ra);
        ptx::tmem_ld_32x32b_x16(t0 + 128 + c, rg);
        if (kSplit) {
          uint32_t sa[16], sg[16];
          ptx::tmem_ld_32x32b_x16(t0 + 256 + c, sa);
          ptx::tmem_ld_32x32b_x16(t0 + 384 + c, sg);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j) { ra[j] = add_f32(ra[j], sa[j]); rg[j] = add_f32(rg[j], sg[j]); }
        } else {
          ptx::tmem_ld_wait();
        }
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (!kPacked || unsigned(c + j - own) < unsigned(P.T))
            acc = fmaf(__uint_as_float(ra[j]), __uint_as_float(rg[j]), acc);
      };
      if (kPacked) {
#pragma unroll 1
        for (int c = c_lo; c < c_hi; c += 32)
          if (c + 32 <= rows) add32(c);
          else add16(c);
      } else {
#pragma unroll 1
        for (int c = 0; c + 32 <= rows; c += 32) add32(c);
        if (kShort && (rows & 16)) add16(rows - 16);
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&acc_empty[buf]);   // accumulators may be overwritten
      // The four warps' sums meet through an mbarrier, not a blocking named barrier: a warp that
      // gave up above never arrives, and warp 0's wait for the others is bounded like every other.
      // Four slots: the other warps can run at most two items ahead of a waiting warp 0 (they
      // need its acc_empty arrivals), so a slot is never rewritten before it has been read.
      const uint32_t slot = n_item & 3, red_phase = (n_item >> 2) & 1;
      if (kPacked) {
        epi_red[slot * kTile + row] = acc;
        __syncwarp();
      } else {
        if (kShort && row >= P.T) acc = 0.f;         // a row beyond the tile: whatever lay there
        acc = warp_sum(acc);
        if (lane == 0) epi_red[slot * 4 + ew] = acc;
      }
      if (lane == 0) ptx::mbar_arrive(&red_bar[slot]);
      if (ew == 0) {
        if (!ptx::mbar_wait_relaxed(&red_bar[slot], red_phase, abort_flag, P.wait_limit)) { ok = false; break; }
        if (kPacked) {
          for (int e = lane; e < P.pack; e += 32) {      // a lane adds up the rows of an example
            const int example = it.example * P.pack + e;
            const long long at = (long long)example * P.n_per + it.pidx;
            if (example >= P.B || !dp_in_range(at, (long long)P.B * P.n_per, P.dev_status)) break;
            const float* of = epi_red + slot * kTile + e * P.T;
            float s = 0.f;
#pragma unroll 8
            for (int k = 0; k < P.T; ++k) s += of[k];
            P.partials[at] = s;
          }
        } else if (lane == 0 && dp_in_range(it.pidx, (long long)P.B * P.n_per, P.dev_status)) {
          const float s = (epi_red[slot * 4 + 0] + epi_red[slot * 4 + 1]) +
                          (epi_red[slot * 4 + 2] + epi_red[slot * 4 + 3]);
          P.partials[it.pidx] = (it.ti == it.tj) ? s : 2.f * s;
        }
      }
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
}

__global__ void reduce_partials_kernel(const float* __restrict__ partials, int n_per, int B,
                                       float* __restrict__ sq, float factor,
                                       float* __restrict__ plain_out, int overwrite) {
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= B) return;
  float s = 0.f;
  for (int j = lane; j < n_per; j += 32) s += partials[size_t(i) * n_per + j];
  s = warp_sum(s);
  if (lane == 0) {
    if (plain_out) plain_out[i] = s;
    if (sq) sq[i] = (overwrite ? 0.f : sq[i]) + factor * s;
  }
}

}  // namespace

dp_status launch_reduce_partials(const float* partials, int n_per, int B, float* sq,
                                 float factor, float* plain_out, cudaStream_t st, bool overwrite) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&launch_reduce_partials)))
    DP_CUDA_OK(prefer_max_shared(reduce_partials_kernel));
  const int warps = 4;
  reduce_partials_kernel<<<ceil_div(B, warps), warps * 32, 0, st>>>(partials, n_per, B, sq,
                                                                  factor, plain_out, overwrite ? 1 : 0);
  DP_LAUNCH_OK();
  return DP_OK;
}

namespace {

template <bool kDiagOnly, bool kSplit, Rows kRows, int kBoxes>
dp_status launch_variant(const GhostParams& P, cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&ghost_norm_tc_kernel<kDiagOnly, kSplit, kRows, kBoxes>)))
    DP_CUDA_OK((allow_shared(ghost_norm_tc_kernel<kDiagOnly, kSplit, kRows, kBoxes>, kSmemBytes)));
  const int grid = std::min(P.total_items, sm_count());
  ghost_norm_tc_kernel<kDiagOnly, kSplit, kRows, kBoxes><<<grid, kThreads, kSmemBytes, st>>>(P);
  DP_LAUNCH_OK();
  return DP_OK;
}

}  // namespace

// Enqueue the tensor-core ghost norm for the planned layers; partial sums land in
// plan.partials layout inside `partials` (the caller reduces them afterwards).
dp_status launch_ghost_norm_tc(const dp_linear_desc* layers, const GhostPlan& plan, int B, int T,
                               float* partials, int* dev_status, cudaStream_t st, bool split) {
  const int nt = ceil_div(T, kTile);
  const Rows kind = T > 64 ? kFullTile : plan.pack == 1 ? kShortTile : kPackedTile;
  const bool packed = kind == kPackedTile;                     // the rows of the batch as one dimension
  const int rows = kind == kFullTile ? kTile : (plan.pack * T + 15) / 16 * 16, tile_bytes = rows * kKStep * 2;
  const int map_rows = packed ? B * T : T, examples = packed ? 1 : B, planes = (split ? 2 : 1) * examples;
  const int boxes = kind == kFullTile || rows > 64 ? 1 : rows > 32 || split ? 2 : 4;
  const int stages = std::min(kMaxStages, (kRingBytes - (kTileBytes - tile_bytes)) / (boxes * (split ? 2 : 1) * tile_bytes));
  const int groups = packed ? ceil_div(B, plan.pack) : B;
  // layers are processed in groups that fit one parameter block
  for (size_t g0 = 0; g0 < plan.ghost_layers.size(); g0 += kGhostMaxLayers) {
    const size_t g1 = std::min(plan.ghost_layers.size(), g0 + kGhostMaxLayers);
    GhostParams P;
    memset(&P, 0, sizeof(P));
    int items = 0;
    for (size_t g = g0; g < g1; ++g) {
      const int li = plan.ghost_layers[g];
      const dp_linear_desc& L = layers[li];
      dp_status s = make_tmap_bf16_3d(&P.tmA[g - g0], L.A, L.lda, L.d, map_rows, planes, kKStep, rows);
      if (s != DP_OK) return s;
      s = make_tmap_bf16_3d(&P.tmG[g - g0], L.G, L.ldg, L.p, map_rows, planes, kKStep, rows);
      if (s != DP_OK) return s;
      GhostLayerPlan lp = plan.layer[li];
      lp.item_begin = items;
      items += groups * plan.ntp * lp.nsplit;
      P.layer[g - g0] = lp;
    }
    P.n_layers = int(g1 - g0);
    P.B = B; P.T = T; P.nt = nt; P.ntp = plan.ntp;
    P.rows = rows; P.stages = stages; P.pack = plan.pack; P.low_plane = examples;
    P.total_items = items;
    P.n_per = plan.n_per;
    P.partials = partials;
    P.dev_status = dev_status;
    P.wait_limit = g_wait_limit;
    dp_status s;
    if (split)
      s = nt > 1              ? launch_variant<false, true, kFullTile, 1>(P, st)
          : kind == kFullTile ? launch_variant<true, true, kFullTile, 1>(P, st)
          : !packed           ? launch_variant<true, true, kShortTile, 2>(P, st)
          : boxes == 1        ? launch_variant<true, true, kPackedTile, 1>(P, st)
                              : launch_variant<true, true, kPackedTile, 2>(P, st);
    else
      s = nt > 1              ? launch_variant<false, false, kFullTile, 1>(P, st)
          : kind == kFullTile ? launch_variant<true, false, kFullTile, 1>(P, st)
          : !packed           ? (boxes == 2 ? launch_variant<true, false, kShortTile, 2>(P, st)
                                            : launch_variant<true, false, kShortTile, 4>(P, st))
          : boxes == 1        ? launch_variant<true, false, kPackedTile, 1>(P, st)
          : boxes == 2        ? launch_variant<true, false, kPackedTile, 2>(P, st)
                              : launch_variant<true, false, kPackedTile, 4>(P, st);
    if (s != DP_OK) return s;
  }
  return DP_OK;
}

}  // namespace dpg
