// Ghost norm of linear layers for sequences longer than 128 tokens, on CTA pairs.
//
// Same quantity as ghost_norm_tc.cu -- <A_i A_i^T, G_i G_i^T>_F per example and layer (Eq. 4 -
// Eq. 5 extended from one token to T tokens) -- but a work item is one 256 x 256 tile pair
// (I <= J) of the two T x T Gram matrices, computed by two CTAs with cta_group::2 MMAs: each CTA
// loads 128 rows of row block I and 128 rows of row block J per 64-column K step (32 KiB for
// 2 x 128 x 256 x 64 multiply-adds), half the shared-memory fill per flop of a 128 x 128 tile.
// With T > 128 the single-CTA kernel is bound by the L2 -> SM fill rate, not by the tensor pipe;
// the larger tile trades 20 - 33 % more flops (the diagonal 256 x 256 tiles are computed in full)
// for half the operand traffic.
//
// Tensor memory holds S_A in columns 0..255 and S_G in columns 256..511 of each CTA (its 128 rows
// of the tile).  There is no room for a second pair of accumulators, so the overlap is in time:
// the epilogue warps copy S_A into registers while the MMAs of S_G run, which frees S_A for the
// next item before S_G is complete, and they multiply S_G against those registers while the next
// item's S_A is being accumulated.
//
// Row blocks are as tall as the sequence needs: ceil(T / 256) blocks of equal height, in steps of 32 rows (kHalf
// rows from each CTA; the N of an MMA is the block's height, its M stays 256, the rows beyond are nobody's).
// With blocks of 256 rows the last one was multiplied, and its zeros written to shared memory, as if it were full.
// Where all of T is one block every tile pair is a diagonal one (kDiag) and a stage holds two column steps of it.
// DistilGPT2 at B = 21, T = 203 (blocks of 224 rows): step 1297 -> 1276 us; T a multiple of 256: no difference.
//
// Roles per CTA (640 threads): warp 0 TMA producer, warp 1 MMA issuer (rank 0 only), warp 2 tells
// rank 0 that this CTA's half of a stage has landed, warp 3 idle, warps 4..19 epilogue (four per
// TMEM lane quarter, 64 columns each).  Every wait is bounded.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "dp_common.cuh"
#include "ghost_plan.cuh"
#include "ptx_sm100.cuh"
#include "tma_host.cuh"

namespace dpg {

namespace {

constexpr int kMmaRows = 128;                     // rows that an MMA reads of each CTA's first operand
constexpr int kTile2 = 2 * kMmaRows;              // largest block height; columns of one accumulator
constexpr int kKStep = 64;                        // bf16 columns per stage row (128 bytes)
constexpr int kRingBytes = 7 * 32 * 1024;
constexpr size_t kSmemBytes = kRingBytes + 1024 /*alignment slack*/ + 1024;

// kHalf: rows of a block that one CTA supplies, a multiple of 16
template <int kHalf>
struct Geo {
  static constexpr int kBlock = 2 * kHalf;                 // rows of a block, edge of a Gram tile
  static constexpr int kTileBytes = kHalf * kKStep * 2;
  static constexpr int kStageBytes = 2 * kTileBytes;       // rows of block I and of block J, or two column steps of one
  // the MMAs of the last tile read kMmaRows rows as well
  static constexpr int kStages = (kRingBytes - (kMmaRows - kHalf) * kKStep * 2) / kStageBytes;
};
constexpr int kEpiWarp0 = 4, kEpiWarps = 16;
constexpr int kThreads = (kEpiWarp0 + kEpiWarps) * 32;
constexpr int kTmemCols = 512;

struct __align__(64) PairParams {
  CUtensorMap tmA[kGhostMaxLayers];
  CUtensorMap tmG[kGhostMaxLayers];
  GhostLayerPlan layer[kGhostMaxLayers];
  int n_layers;
  int B, T, nt, ntp;         // nt row blocks, ntp = nt (nt + 1) / 2 tile pairs
  int total_items;
  int n_per;
  float* partials;           // [B][n_per]; an item owns two consecutive slots (one per CTA)
  int* dev_status;
  long long wait_limit;
};
static_assert(sizeof(PairParams) <= 32764, "kernel parameter block too large");

struct Item {
  int layer, example, ti, tj, a0, a1, g0, g1, pidx;
};

// `l` is the caller's running layer index: a role's items ascend, so the search goes on from the layer
// of its previous item instead of walking the list (a constant-memory line per layer) every time.
__device__ __forceinline__ Item decode_item(const PairParams& P, int item, int& l) {
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
  it.pidx = it.example * P.n_per + L.col_begin + (tp * L.nsplit + s) * 2;
  return it;
}

template <int kHalf, bool kDiag>
__global__ void __launch_bounds__(kThreads, 1)
ghost_norm_pair_kernel(const __grid_constant__ PairParams P) {
  using G = Geo<kHalf>;
  constexpr int kStages = G::kStages, kStageBytes = G::kStageBytes, kTileBytes = G::kTileBytes;
  constexpr int kSteps = kDiag ? 2 : 1;            // column steps per stage
  const uint32_t rank = ptx::cluster_ctarank();
  const int first_item = int(blockIdx.x >> 1);
  const int item_stride = int(gridDim.x >> 1);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + kRingBytes);
  uint64_t* full = bars;                       // [kStages] this CTA's TMA landed
  uint64_t* ready = bars + kStages;            // [kStages] both CTAs' tiles landed (rank 0's copy)
  uint64_t* empty = bars + 2 * kStages;        // [kStages] MMAs retired
  uint64_t* sa_full = bars + 3 * kStages;      // S_A complete
  uint64_t* sg_full = sa_full + 1;             // S_G complete
  uint64_t* sa_empty = sa_full + 2;            // S_A copied to registers in both CTAs (rank 0's copy)
  uint64_t* sg_empty = sa_full + 3;            // S_G consumed in both CTAs (rank 0's copy)
  uint64_t* mma_done = sa_full + 4;
  uint64_t* red_bar = mma_done + 1;            // [4] this CTA's epilogue warps -> its epilogue warp 0
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(red_bar + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* epi_red = reinterpret_cast<float*>(tmem_slot + 2);   // [4][kEpiWarps]
  uint32_t* sink = reinterpret_cast<uint32_t*>(epi_red + 4 * kEpiWarps);   // [kStages] written by st.async, never read

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&ready[s], 1);             // rank 0's relay arrives and announces 4 bytes, rank 1's sends them
      ptx::mbar_init(&empty[s], 1);
    }
    ptx::mbar_init(sa_full, 1);
    ptx::mbar_init(sg_full, 1);
    ptx::mbar_init(sa_empty, kEpiWarps * 2);
    ptx::mbar_init(sg_empty, kEpiWarps * 2);
    ptx::mbar_init(mma_done, 1);
    for (int b = 0; b < 4; ++b) ptx::mbar_init(&red_bar[b], kEpiWarps);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) { ptx::tmem_alloc_pair(tmem_slot, kTmemCols); ptx::tmem_relinquish_pair(); }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync_all();        // the partner's barriers exist before anyone arrives on them
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tiles_a = ptx::smem_u32(tiles), full_a = ptx::smem_u32(full), empty_a = ptx::smem_u32(empty);

  if (warp == 0) {
    // ------------------------------------------------------------- TMA producer
    // producer, issuer and relay: the whole warp runs the loop, an elected lane issues (see ptx::warp_ok)
    uint32_t stage = 0, phase = 0, issued = 0;
    int lay = 0;
    bool ok = true;
    for (int item = first_item; item < P.total_items && ok; item += item_stride) {
      const Item it = decode_item(P, item, lay);
      const bool diag = kDiag || it.ti == it.tj;
      const int row_i = it.ti * G::kBlock + int(rank) * kHalf;  // this CTA's rows of block I
      const int row_j = it.tj * G::kBlock + int(rank) * kHalf;  // and of block J
      for (int pass = 0; pass < 2 && ok; ++pass) {
        const uint64_t tm = reinterpret_cast<uint64_t>(pass == 0 ? &P.tmA[it.layer] : &P.tmG[it.layer]);
        const int k0 = pass == 0 ? it.a0 : it.g0, k1 = pass == 0 ? it.a1 : it.g1;
        for (int k = k0; k < k1; k += kSteps) {
          ok = ptx::warp_ok(ptx::mbar_wait_a(empty_a + 8 * stage, phase ^ 1, abort_flag, P.wait_limit));
          if (!ok) break;
          const uint32_t dst = tiles_a + stage * kStageBytes, bar = full_a + 8 * stage;
          const bool second = kDiag ? k + 1 < k1 : !diag;
          if (ptx::elect_one()) {
            ptx::mbar_arrive_expect_tx_a(bar, second ? kStageBytes : kTileBytes);
            ptx::tma_load_3d_a(dst, tm, bar, k * kKStep, row_i, it.example);
            if (second)
              ptx::tma_load_3d_a(dst + kTileBytes, tm, bar, (kDiag ? k + 1 : k) * kKStep, kDiag ? row_i : row_j, it.example);
          }
          __syncwarp();
          ++issued;
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
      }
    }
    if (!ok && ptx::elect_one()) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
      ptx::drain_issued_copies(full, kStages, issued);
    }
  } else if (warp == 1) {
    // --------------------------------------------------------------- MMA issuer
    if (rank == 0) {
      constexpr uint32_t idesc = ptx::idesc_bf16_f32(kTile2, G::kBlock, 0, 0);
      constexpr uint64_t dbase = ptx::smem_desc_base(16, 1024, ptx::SWIZZLE_128B);   // K-major
      constexpr uint32_t desc_hi = uint32_t(dbase >> 32);
      const uint32_t desc_lo0 = uint32_t(dbase) | ((tiles_a >> 4) & 0x3FFF);
      const uint32_t ready_a = ptx::smem_u32(ready);
      uint32_t stage = 0, phase = 0, n_item = 0;
      int lay = 0;
      bool ok = true;
      for (int item = first_item; item < P.total_items && ok; item += item_stride, ++n_item) {
        const Item it = decode_item(P, item, lay);
        const bool diag = kDiag || it.ti == it.tj;
        const uint32_t ph = n_item & 1;
        for (int pass = 0; pass < 2 && ok; ++pass) {
          // the accumulator of this pass must have been read out for the previous item
          uint64_t* freed = pass == 0 ? sa_empty : sg_empty;
          ok = ptx::warp_ok(ptx::mbar_wait_cluster(freed, ph ^ 1, abort_flag, P.wait_limit));
          if (!ok) break;
          ptx::tc_fence_after();
          const uint32_t d_tmem = tmem_base + pass * kTile2;
          const int nsteps = pass == 0 ? it.a1 - it.a0 : it.g1 - it.g0;
          for (int k = 0; k < nsteps; k += kSteps) {
            ok = ptx::warp_ok(ptx::mbar_wait_cluster_a(ready_a + 8 * stage, phase, abort_flag, P.wait_limit));
            if (!ok) break;
            ptx::tc_fence_after();
            const uint32_t sa = desc_lo0 + stage * (kStageBytes >> 4);
            const uint32_t sb = diag ? sa : sa + (kTileBytes >> 4);
            if (ptx::elect_one()) {
#pragma unroll
              for (int kk = 0; kk < kKStep / 16; ++kk)
                ptx::mma_bf16_ss_pair_lh(d_tmem, sa + kk * 2, sb + kk * 2, desc_hi, idesc, (k > 0 || kk > 0) ? 1u : 0u);
              if (kDiag && k + 1 < nsteps) {
                const uint32_t s1 = sa + (kTileBytes >> 4);
#pragma unroll
                for (int kk = 0; kk < kKStep / 16; ++kk)
                  ptx::mma_bf16_ss_pair_lh(d_tmem, s1 + kk * 2, s1 + kk * 2, desc_hi, idesc, 1u);
              }
              ptx::mma_commit_pair_a(empty_a + 8 * stage, 3);
              if (k + kSteps >= nsteps) ptx::mma_commit_pair(pass == 0 ? sa_full : sg_full, 3);
            }
            __syncwarp();
            if (++stage == kStages) { stage = 0; phase ^= 1; }
          }
        }
      }
      if (!ok && ptx::elect_one()) {
        *abort_flag = 1;
        if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
        ptx::drain_issued_mmas(mma_done, true);
      }
    }
  } else if (warp == 2) {
    // -------------------------------------------------------------------- relay
    // Tells rank 0's MMA issuer that this CTA's half of a stage has landed.  Rank 0's relay
    // arrives on its own `ready` barrier and announces 4 more bytes; rank 1's relay, which has
    // acquired its `full` barrier (so the TMA data are visible to it), delivers those 4 bytes with
    // an asynchronous store into rank 0's shared memory whose completion on the barrier is a
    // release at cluster scope.
    const uint32_t ready_a = ptx::smem_u32(ready), sink_a = ptx::smem_u32(sink);
    const uint32_t ready_remote = ptx::mapa_u32(ready_a, 0), sink_remote = ptx::mapa_u32(sink_a, 0);
    uint32_t stage = 0, phase = 0;
    int lay = 0;
    bool ok = true;
    for (int item = first_item; item < P.total_items && ok; item += item_stride) {
      const Item it = decode_item(P, item, lay);
      const int stages = (it.a1 - it.a0 + kSteps - 1) / kSteps + (it.g1 - it.g0 + kSteps - 1) / kSteps;
      for (int k = 0; k < stages; ++k) {
        ok = ptx::warp_ok(ptx::mbar_wait_a(full_a + 8 * stage, phase, abort_flag, P.wait_limit));
        if (!ok) break;
        if (ptx::elect_one()) {
          if (rank == 0) ptx::mbar_arrive_expect_tx_a(ready_a + 8 * stage, 4);
          else ptx::st_async_signal_a(ready_remote + 8 * stage, sink_remote + 4 * stage);
        }
        __syncwarp();
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    }
    if (!ok && ptx::elect_one()) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
    }
  } else if (warp >= kEpiWarp0) {
    // ----------------------------------------------------------------- epilogue
    const int q = warp & 3;                          // TMEM lane quarter this warp may read
    const int ew = warp - kEpiWarp0;
    const int cg = ew >> 2;                          // which quarter of the columns
    constexpr int kCols = G::kBlock / (kEpiWarps / 4), kChunks = kCols / 8;      // of a warp; in chunks of eight
    const uint32_t t_sa = tmem_base + (uint32_t(q * 32) << 16) + cg * kCols;
    const bool mine = q * 32 + lane < kHalf;         // a row of the block
    const uint32_t t_sg = t_sa + kTile2;
    uint32_t n_item = 0;
    int lay = 0;
    bool ok = true;
    for (int item = first_item; item < P.total_items && ok; item += item_stride, ++n_item) {
      const Item it = decode_item(P, item, lay);
      const uint32_t ph = n_item & 1;
      // S_A -> registers, then the accumulator is free for the next item
      if (!ptx::mbar_wait_relaxed(sa_full, ph, abort_flag, P.wait_limit)) { ok = false; break; }
      ptx::tc_fence_after();
      uint32_t sa[kCols];
#pragma unroll
      for (int c = 0; c < kChunks; ++c) ptx::tmem_ld_32x32b_x8(t_sa + c * 8, sa + c * 8);
      ptx::tmem_ld_wait();
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive_cluster(sa_empty, 0);
      // S_G against the registers
      if (!ptx::mbar_wait_relaxed(sg_full, ph, abort_flag, P.wait_limit)) { ok = false; break; }
      ptx::tc_fence_after();
      float acc = 0.f;
#pragma unroll
      for (int c = 0; c < kChunks; c += 2) {
        uint32_t g[16];
        ptx::tmem_ld_32x32b_x8(t_sg + c * 8, g);
        if (c + 1 < kChunks) ptx::tmem_ld_32x32b_x8(t_sg + c * 8 + 8, g + 8);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < (c + 1 < kChunks ? 16 : 8); ++j)
          acc = fmaf(__uint_as_float(sa[c * 8 + j]), __uint_as_float(g[j]), acc);
      }
      if (kHalf < kMmaRows && !mine) acc = 0.f;      // whatever lay in the rows beyond
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive_cluster(sg_empty, 0);
      // the warps' sums meet through an mbarrier with a bounded wait (no blocking named barrier:
      // a warp that gave up never arrives); four slots, since the other warps can run at most one
      // item ahead of a waiting warp 0 (they need its sa_empty arrival)
      acc = warp_sum(acc);
      const uint32_t slot = n_item & 3, red_phase = (n_item >> 2) & 1;
      if (lane == 0) { epi_red[slot * kEpiWarps + ew] = acc; ptx::mbar_arrive(&red_bar[slot]); }
      if (ew == 0) {
        if (!ptx::mbar_wait_relaxed(&red_bar[slot], red_phase, abort_flag, P.wait_limit)) { ok = false; break; }
        if (lane == 0 && dp_in_range(it.pidx + int(rank), (long long)P.B * P.n_per, P.dev_status)) {
          float s = 0.f;
#pragma unroll
          for (int e = 0; e < kEpiWarps; ++e) s += epi_red[slot * kEpiWarps + e];
          P.partials[it.pidx + int(rank)] = (it.ti == it.tj) ? s : 2.f * s;
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
  ptx::cluster_sync_all();        // neither CTA leaves while the partner may still use its memory
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

template <int kHalf, bool kDiag>
dp_status launch_variant(const PairParams& P, cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&ghost_norm_pair_kernel<kHalf, kDiag>)))
    DP_CUDA_OK((allow_shared(ghost_norm_pair_kernel<kHalf, kDiag>, kSmemBytes)));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * std::min(P.total_items, sm_count() / 2), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  DP_CUDA_OK(cudaLaunchKernelEx(&cfg, ghost_norm_pair_kernel<kHalf, kDiag>, P));
  ++g_kernel_launches;
  return DP_OK;
}

template <int kHalf>
dp_status launch_half(const PairParams& P, cudaStream_t st) {
  return P.nt == 1 ? launch_variant<kHalf, true>(P, st) : launch_variant<kHalf, false>(P, st);
}

}  // namespace

dp_status launch_ghost_norm_pair(const dp_linear_desc* layers, const GhostPlan& plan, int B, int T,
                                 float* partials, int* dev_status, cudaStream_t st) {
  const int nt = ceil_div(T, kTile2);
  const int half = ceil_div(ceil_div(T, nt), 32) * 16;         // T > 128: 80, 96, 112 or 128
  for (size_t g0 = 0; g0 < plan.ghost_layers.size(); g0 += kGhostMaxLayers) {
    const size_t g1 = std::min(plan.ghost_layers.size(), g0 + kGhostMaxLayers);
    PairParams P;
    memset(&P, 0, sizeof(P));
    int items = 0;
    for (size_t g = g0; g < g1; ++g) {
      const int li = plan.ghost_layers[g];
      const dp_linear_desc& L = layers[li];
      dp_status s = make_tmap_bf16_3d(&P.tmA[g - g0], L.A, L.lda, L.d, T, B, kKStep, half);
      if (s != DP_OK) return s;
      s = make_tmap_bf16_3d(&P.tmG[g - g0], L.G, L.ldg, L.p, T, B, kKStep, half);
      if (s != DP_OK) return s;
      GhostLayerPlan lp = plan.layer[li];
      lp.item_begin = items;
      items += B * plan.ntp * lp.nsplit;
      P.layer[g - g0] = lp;
    }
    P.n_layers = int(g1 - g0);
    P.B = B; P.T = T; P.nt = nt; P.ntp = plan.ntp;
    P.total_items = items;
    P.n_per = plan.n_per;
    P.partials = partials;
    P.dev_status = dev_status;
    P.wait_limit = g_wait_limit;
    const dp_status s = half <= 80 ? launch_half<80>(P, st) : half == 96 ? launch_half<96>(P, st)
                        : half == 112 ? launch_half<112>(P, st) : launch_half<128>(P, st);
    if (s != DP_OK) return s;
  }
  return DP_OK;
}

}  // namespace dpg
