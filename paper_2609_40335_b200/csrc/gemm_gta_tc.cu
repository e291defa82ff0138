// G^T A on tcgen05 tensor cores: the contraction over tokens shared by
//   (a) the clipped gradient sum  out = beta*out + sum_i R_i G_i^T A_i   (inner sum of Eq. 3,
//       R_i of Eq. 7), one GEMM with M = p, N = d, K = B*T whose K rows carry R_i, and
//   (b) the DIRECT per-example norm  || G_i^T A_i ||_F^2  (Eq. 4 summed over tokens), where
//       each 128 x 256 tile of the p x d gradient lives only in tensor memory and the
//       epilogue sums its squares.
//
// Both operands are contiguous along M / N (token rows are the K dimension), so shared
// memory holds MN-major tiles: every TMA box is 64 token rows x 64 columns (128-byte rows,
// 128-byte swizzle).  In (a) the K steps run over the rows of the whole batch (see GtaRows), in (b)
// over one example's (tensor map column, token, example; its token tail is zero-filled).  A "scaler" warp
// multiplies the rows of a G tile by their R_i in shared memory (packed bf16 FMAs with R_i split into two
// bf16 parts) between the TMA-full and MMA-ready barriers; four such warps work on four consecutive stages
// at once.
//
// Roles per CTA (736 threads): warps 0 and 2 TMA producers (G and A), warp 1 MMA issuer, warps 3-6 scalers,
// warps 7-22 epilogue (four per TMEM lane quarter, two 32-column chunks each; they also draw
// the fused Gaussian noise, which is latency-bound per warp -- hence so many); two TMEM
// accumulators overlap the epilogue with the next tile.
//
// Clipped sums run on CTA PAIRS (cta_group::2, cluster of 2; here those with few output tiles, the others
// in gemm_gta_big.cu): a 256 x 256 output tile per pair,
// each CTA loading its own 128 G rows and half of the A tile's columns, rank 0 issuing the MMAs
// for both, stage-free and accumulator-ready signals multicast to both CTAs by tcgen05.commit,
// scaler and epilogue warps of rank 1 signalling rank 0's barriers by asynchronous stores.  The DIRECT-norm variant
// stays on single CTAs.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "dp_common.cuh"
#include "gemm_gta.cuh"
#include "noise_device.cuh"
#include "ptx_sm100.cuh"
#include "tma_host.cuh"

namespace dpg {

namespace {

constexpr int kBM = 128, kBN = 256, kBK = 64;
constexpr int kBoxBytes = kBK * 128;                // kBK token rows x 128 bytes
constexpr int kGBytes = (kBM / 64) * kBoxBytes;     // 16 KiB: this CTA's 128 rows of the G tile

// Tile geometry.  Single CTA: 128 x 256 output tile, the CTA loads all 256 columns of the A
// tile (48 KiB per stage, 4 stages).  CTA pair (cta_group::2): 256 x 256 output tile per pair;
// each CTA loads its own 128 G rows and HALF of the A tile's columns (32 KiB per stage, 7
// stages: all the shared memory there is -- the ring is latency-bound, 7 stages measured 973
// TFLOP/s where 6 gave 895; 32- and 128-row K steps were both slower), the pair's MMA reads
// both halves -- a third less operand traffic per flop.
template <bool kPair>
struct Geo {
  static constexpr int kAColsPerCta = kPair ? kBN / 2 : kBN;
  static constexpr int kABytes = (kAColsPerCta / 64) * kBoxBytes;
  static constexpr int kStageBytes = kGBytes + kABytes;
  static constexpr int kStages = kPair ? 7 : 4;
  static constexpr int kTileM = kPair ? 2 * kBM : kBM;       // output rows per work item
  static constexpr size_t kSmemBytes = size_t(kStages) * kStageBytes + 1024 + 1024;
};
constexpr int kProducerAWarp = 2;                    // warp 0 loads G, warp 2 loads A, warp 1 issues MMAs
constexpr int kScalerWarp0 = 3;
constexpr int kScalerWarps = 4;
constexpr int kEpiWarp0 = kScalerWarp0 + kScalerWarps;   // first epilogue warp
constexpr int kEpiWarps = 16;         // kEpiWarps/4 per TMEM lane quarter (column groups)
constexpr int kThreads = (kEpiWarp0 + kEpiWarps) * 32;
constexpr int kTmemCols = 512;                      // 2 accumulators x 256 columns

struct __align__(64) GtaParams {
  CUtensorMap tmG[kGtaMaxLayers];
  CUtensorMap tmA[kGtaMaxLayers];
  GtaLayer layer[kGtaMaxLayers];
  int n_layers;
  int B, T, tsteps;          // planes along K and rows of each; tsteps = terms * ceil(T / 64) K steps per plane
  int low_plane;             // split operands: first plane of low terms
  int example_rows, rows, example_steps;     // scaling: tokens per example; all rows, or 0 and the steps of an example
  int nsplit, ksteps_per_split;   // K splits, the same for all layers of a call; multiples of `terms` steps
  float beta;
  int total_items;
  const float* clip;         // [B] R_i (scale mode)
  NoiseKeys noise_keys;      // Gaussian stream of the fused noise (per-layer id)
  uint32_t noise_step;
  const uint32_t* step_dev;  // optional device counter added to noise_step
  float noise_scale;
  float* sq_partials;        // [B][n_per] (square-sum mode)
  int n_per;
  int* dev_status;
  long long wait_limit;      // cycles a barrier wait may take before the CTA gives up
};
static_assert(sizeof(GtaParams) <= 32764, "kernel parameter block too large");

struct Item {
  int layer, tm, tn, k0, k1, split, example;
};

// `l` is the caller's running layer index: a role's items ascend, so the search goes on from the layer
// of its previous item.  (From layer 0 it was a chain of up to 97 dependent constant loads, a line
// each, in every role and for every tile.)
template <bool kSqsum, int kTileM>
__device__ __forceinline__ Item decode_item(const GtaParams& P, int item, int& l) {
  Item it;
  while (l + 1 < P.n_layers && item >= P.layer[l + 1].item_begin) ++l;
  const GtaLayer& L = P.layer[l];
  int local = item - L.item_begin;
  it.layer = l;
  const int tiles_n = (L.N + kBN - 1) / kBN, tiles_m = (L.M + kTileM - 1) / kTileM;
  it.tn = local % tiles_n; local /= tiles_n;
  it.tm = local % tiles_m; local /= tiles_m;
  if (kSqsum) {
    it.example = local; it.split = 0;
    it.k0 = local * P.tsteps; it.k1 = it.k0 + P.tsteps;
  } else {
    it.example = -1; it.split = local;
    it.k0 = local * P.ksteps_per_split;
    it.k1 = min(it.k0 + P.ksteps_per_split, P.B * P.tsteps);
  }
  return it;
}

template <bool kScale, bool kSqsum, bool kPair, bool kSplit, bool kByRow>
__global__ void __launch_bounds__(kThreads, 1)
gemm_gta_kernel(const __grid_constant__ GtaParams P) {
  static_assert(kScale || !kPair, "CTA pairs need the scaler warps' cross-CTA stage hand-off");
  constexpr int kStages = Geo<kPair>::kStages;
  constexpr int kStageBytes = Geo<kPair>::kStageBytes;
  constexpr int kTileM = Geo<kPair>::kTileM;
  // pair: rank 0 issues the MMAs; both CTAs walk the same list of work items
  const uint32_t rank = kPair ? ptx::cluster_ctarank() : 0u;
  const int first_item = kPair ? int(blockIdx.x >> 1) : int(blockIdx.x);
  const int item_stride = kPair ? int(gridDim.x >> 1) : int(gridDim.x);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + size_t(kStages) * kStageBytes);
  uint64_t* full = bars;                      // both producers' TMA loads landed
  uint64_t* ready = bars + kStages;           // G tile scaled in both CTAs (scale mode; rank 0's copy)
  uint64_t* empty = bars + 2 * kStages;       // MMAs retired
  uint64_t* acc_full = bars + 3 * kStages;    // [2]
  uint64_t* acc_empty = acc_full + 2;         // [2]
  uint64_t* mma_done = acc_empty + 2;         // only used when the MMA issuer gives up
  uint64_t* red_bar = mma_done + 1;           // [4] epilogue warps -> epilogue warp 0 (square-sum mode)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(red_bar + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* epi_red = reinterpret_cast<float*>(tmem_slot + 2);   // [4][kEpiWarps]
  uint32_t* sink = reinterpret_cast<uint32_t*>(epi_red + 4 * kEpiWarps);   // [kStages] written by st.async, never read

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t tiles_a = ptx::smem_u32(tiles);
  const uint32_t full_a = ptx::smem_u32(full), ready_a = ptx::smem_u32(ready), empty_a = ptx::smem_u32(empty);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(&full[s], 2);             // the G producer and the A producer
      // pair: rank 0's scaler warp arrives (and announces 4 bytes), rank 1's sends those 4 bytes
      ptx::mbar_init(&ready[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(&acc_full[b], 1);
      ptx::mbar_init(&acc_empty[b], kEpiWarps);    // this CTA's epilogue warps (pair: + 4 bytes from each of rank 1's)
    }
    ptx::mbar_init(mma_done, 1);
    for (int b = 0; b < 4; ++b) ptx::mbar_init(&red_bar[b], kEpiWarps);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) {
    if (kPair) { ptx::tmem_alloc_pair(tmem_slot, kTmemCols); ptx::tmem_relinquish_pair(); }
    else { ptx::tmem_alloc(tmem_slot, kTmemCols); ptx::tmem_relinquish(); }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (kPair) ptx::cluster_sync_all();     // the partner's barriers exist before anyone arrives on them
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0 || warp == kProducerAWarp) {
    // ------------------------------------------------------------- TMA producers
    // Two threads in two warps: one loads this CTA's G rows, the other its A columns.  The time
    // a producer needs per stage is part of every stage's round trip, so the work is halved and
    // the loop is kept to a few instructions (32-bit shared addresses, running example / token
    // counters instead of a division).
    if (lane == 0) {
      const bool is_a = (warp != 0);
      constexpr int kBoxes = kBM / 64;
      constexpr int kBoxesA = Geo<kPair>::kAColsPerCta / 64;
      const uint32_t my_bytes = is_a ? uint32_t(Geo<kPair>::kABytes) : uint32_t(kGBytes);
      const int nbox = is_a ? kBoxesA : kBoxes;
      uint32_t stage = 0, phase = 0, issued = 0;
      int lay = 0;
      bool ok = true;
      for (int item = first_item; item < P.total_items && ok; item += item_stride) {
        const Item it = decode_item<kSqsum, kTileM>(P, item, lay);
        const uint64_t tm = reinterpret_cast<uint64_t>(is_a ? &P.tmA[it.layer] : &P.tmG[it.layer]);
        // first column of this CTA's part of the tile: its G rows, or its share of the A columns
        const int c0 = is_a ? it.tn * kBN + int(rank) * Geo<kPair>::kAColsPerCta
                            : it.tm * kTileM + int(rank) * kBM;
        constexpr int kTerms = kSplit ? 3 : 1;
        GtaWalk<kSplit> at(0, it.k0 / kTerms, it.k1 / kTerms, P.tsteps / kTerms);
        for (int ks = it.k0; ks < it.k1; ++ks) {
          if (!ptx::mbar_wait_a(empty_a + 8 * stage, phase ^ 1, abort_flag, P.wait_limit)) { ok = false; break; }
          const uint32_t bar = full_a + 8 * stage;
          const uint32_t dst = tiles_a + stage * kStageBytes + (is_a ? kGBytes : 0);
          ptx::mbar_arrive_expect_tx_a(bar, my_bytes);
          for (int j = 0; j < nbox; ++j)
            ptx::tma_load_3d_a(dst + j * kBoxBytes, tm, bar, c0 + j * 64, at.ts * kBK, at.plane(is_a, P.low_plane));
          ++issued;
          at.next();
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
      }
      if (!ok) {
        *abort_flag = 1;
        if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
        ptx::drain_issued_copies(full, kStages, issued);   // copies in flight land before exit
      }
    }
  } else if (warp == 1) {
    // --------------------------------------------------------------- MMA issuer
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = ptx::idesc_bf16_f32(kTileM, kBN, 1, 1);
      // MN-major, 128-byte swizzle: 64-column chunks are one box (8 KiB) apart, groups of
      // 8 token rows are 1 KiB apart.  Only the 14-bit start address in the low word changes.
      constexpr uint64_t dbase = ptx::smem_desc_base(kBoxBytes, 1024, ptx::SWIZZLE_128B);
      constexpr uint32_t desc_hi = uint32_t(dbase >> 32);
      const uint32_t desc_lo0 = uint32_t(dbase) | ((tiles_a >> 4) & 0x3FFF);
      const uint32_t go_a = kScale ? ready_a : full_a;
      uint32_t stage = 0, phase = 0, n_item = 0;
      int lay = 0;
      bool ok = true;
      for (int item = first_item; item < P.total_items && ok; item += item_stride, ++n_item) {
        const Item it = decode_item<kSqsum, kTileM>(P, item, lay);
        const uint32_t buf = n_item & 1, acc_phase = (n_item >> 1) & 1;
        if (!(kPair ? ptx::mbar_wait_cluster(&acc_empty[buf], acc_phase ^ 1, abort_flag, P.wait_limit)
                    : ptx::mbar_wait(&acc_empty[buf], acc_phase ^ 1, abort_flag, P.wait_limit))) { ok = false; break; }
        ptx::tc_fence_after();
        const uint32_t d_tmem = tmem_base + buf * kBN;
        uint32_t accum = 0;
        for (int ks = it.k0; ks < it.k1; ++ks) {
          if (!(kPair ? ptx::mbar_wait_cluster_a(go_a + 8 * stage, phase, abort_flag, P.wait_limit)
                      : ptx::mbar_wait_a(go_a + 8 * stage, phase, abort_flag, P.wait_limit))) { ok = false; break; }
          ptx::tc_fence_after();
          const uint32_t lo_g = desc_lo0 + stage * (kStageBytes >> 4);
          const uint32_t lo_a = lo_g + (kGBytes >> 4);
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
            // 16 token rows further = two 1 KiB row groups
            if (kPair) ptx::mma_bf16_ss_pair_lh(d_tmem, lo_g + kk * 128, lo_a + kk * 128, desc_hi, idesc, accum);
            else ptx::mma_bf16_ss_lh(d_tmem, lo_g + kk * 128, lo_a + kk * 128, desc_hi, idesc, accum);
            accum = 1;
          }
          // stage reusable in both CTAs once these MMAs retire
          if (kPair) ptx::mma_commit_pair_a(empty_a + 8 * stage, 3);
          else ptx::mma_commit_a(empty_a + 8 * stage);
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
        if (ok) {
          if (kPair) ptx::mma_commit_pair(&acc_full[buf], 3);
          else ptx::mma_commit(&acc_full[buf]);
        }
      }
      if (!ok) {
        *abort_flag = 1;
        if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
        ptx::drain_issued_mmas(mma_done, kPair);
      }
    }
  } else if (warp < kEpiWarp0) {
    // ------------------------------------------------------------------ scalers
    if (kScale) {
      // Each scaler warp owns every kScalerWarps-th K step, so kScalerWarps stages are scaled
      // concurrently: the per-stage latency (shared-memory round trip, proxy fence, barrier
      // hand-off) is overlapped instead of serialised.
      //
      // Hand-off to the MMA issuer (rank 0).  Rank 0's warp arrives on its own `ready` barrier
      // and announces 4 more bytes; rank 1's warp delivers those 4 bytes with an asynchronous
      // store into rank 0's shared memory whose completion on the barrier is a release at
      // cluster scope: the scaled tile it wrote (made visible to the tensor core's proxy by the
      // fence before) is ordered before the MMAs that rank 0 issues after its acquire.
      const int sw = warp - kScalerWarp0;
      const uint32_t ready_remote = kPair ? ptx::mapa_u32(ready_a, 0) : 0u;
      const uint32_t sink_remote = kPair ? ptx::mapa_u32(ptx::smem_u32(sink), 0) : 0u;
      uint32_t cnt = 0;
      int lay = 0;
      bool ok = true;
      for (int item = first_item; item < P.total_items && ok; item += item_stride) {
        const Item it = decode_item<kSqsum, kTileM>(P, item, lay);
        const bool scale_here = P.clip && !P.layer[it.layer].prescaled;
        // first K step of this item that belongs to this warp
        int ks = it.k0 + int((uint32_t(sw) + kScalerWarps - cnt % kScalerWarps) % kScalerWarps);
        uint32_t c = cnt + uint32_t(ks - it.k0);
        // no scaling here when the operand arrives scaled: clip == NULL (the split fp32 path) or a
        // layer whose narrow operand was multiplied by R_i in a pass of its own (see prescale)
        RowFactors r_next{1.f, 1.f, true};
        if (scale_here && ks < it.k1) r_next = row_factors<kByRow>(P.clip, ks, lane, P.example_rows, P.rows, P.example_steps);
        for (; ks < it.k1; ks += kScalerWarps, c += kScalerWarps) {
          const RowFactors r = r_next;
          // the factors of this warp's next K step are fetched before the waits, off the stage's path
          if (scale_here && ks + kScalerWarps < it.k1)
            r_next = row_factors<kByRow>(P.clip, ks + kScalerWarps, lane, P.example_rows, P.rows, P.example_steps);
          const uint32_t stage = c % kStages, fill = c / kStages, phase = fill & 1u;
          // A warp hops between stages, so it has not seen the previous fill of this one, and the
          // parity of `full` alone cannot tell "fill n landed" from "fill n-1 still in flight".
          // Waiting first until the MMAs have retired fill n-1 (the same condition the producers
          // wait for before they issue fill n, so no time is lost) leaves only "fill n pending"
          // or "fill n landed".
          if (fill > 0 && !ptx::mbar_wait_a(empty_a + 8 * stage, phase ^ 1, abort_flag, P.wait_limit)) { ok = false; break; }
          if (!ptx::mbar_wait_a(full_a + 8 * stage, phase, abort_flag, P.wait_limit)) { ok = false; break; }
          uint4* part = reinterpret_cast<uint4*>(tiles + size_t(stage) * kStageBytes);
          if (kByRow && !r.one) scale_rows(part, r.lo, r.hi, lane);
          else if (r.lo != 1.0f) scale_part(part, r.lo, lane);
          if (scale_here) ptx::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (!kPair) ptx::mbar_arrive(&ready[stage]);
            else if (rank == 0) ptx::mbar_arrive_expect_tx_a(ready_a + 8 * stage, 4);
            else ptx::st_async_signal_a(ready_remote + 8 * stage, sink_remote + 4 * stage);
          }
        }
        cnt += uint32_t(it.k1 - it.k0);
      }
      if (!ok && lane == 0) {
        *abort_flag = 1;
        if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
      }
    }
  } else {
    // ----------------------------------------------------------------- epilogue
    const int q = warp & 3;                          // TMEM lane quarter this warp may read
    const int ew = warp - kEpiWarp0;
    // this warp's 32-column chunks: the 8 chunks are dealt to the kEpiWarps/4 column groups
    constexpr int kGroups = kEpiWarps / 4;
    const int c_lo = ((ew >> 2) * (kBN / 32)) / kGroups, c_hi = (((ew >> 2) + 1) * (kBN / 32)) / kGroups;
    // Frees an accumulator once this warp has read its part of it.  Across the pair it signals like
    // the scaler warps do, not with mbarrier.arrive.release.cluster: that arrive waits until every
    // store the warp has issued is acknowledged by the L2, thousands of cycles when all SMs write.
    const uint32_t acc_empty_a = ptx::smem_u32(acc_empty);
    const uint32_t acc_empty_remote = kPair ? ptx::mapa_u32(acc_empty_a, 0) : 0u;
    const uint32_t sink_remote = kPair ? ptx::mapa_u32(ptx::smem_u32(sink), 0) : 0u;
    auto free_acc = [&](uint32_t buf) {
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (!kPair) ptx::mbar_arrive(&acc_empty[buf]);
        else if (rank == 0) ptx::mbar_arrive_expect_tx_a(acc_empty_a + 8 * buf, 4);
        else ptx::st_async_signal_a(acc_empty_remote + 8 * buf, sink_remote);
      }
    };
    uint32_t n_item = 0;
    int lay = 0;
    bool ok = true;
    for (int item = first_item; item < P.total_items && ok; item += item_stride, ++n_item) {
      const Item it = decode_item<kSqsum, kTileM>(P, item, lay);
      const GtaLayer& L = P.layer[it.layer];
      const uint32_t buf = n_item & 1, acc_phase = (n_item >> 1) & 1;
      if (!ptx::mbar_wait_relaxed(&acc_full[buf], acc_phase, abort_flag, P.wait_limit)) { ok = false; break; }
      ptx::tc_fence_after();
      const uint32_t t0 = tmem_base + (uint32_t(q * 32) << 16) + buf * kBN;
      const int row = it.tm * kTileM + int(rank) * kBM + q * 32 + lane;
      if (kSqsum) {
        float acc = 0.f;
#pragma unroll 1
        for (int c = c_lo; c < c_hi; ++c) {
          uint32_t r[32];
          ptx::tmem_ld_32x32b_x32(t0 + c * 32, r);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) { const float v = __uint_as_float(r[j]); acc = fmaf(v, v, acc); }
        }
        free_acc(buf);
        // the warps' sums meet through an mbarrier with a bounded wait (no blocking named
        // barrier: a warp that gave up never arrives); four slots, since the other warps can run
        // at most two items ahead of a waiting warp 0 (they need its acc_empty arrivals)
        acc = warp_sum(acc);
        const uint32_t slot = n_item & 3, red_phase = (n_item >> 2) & 1;
        if (lane == 0) { epi_red[slot * kEpiWarps + ew] = acc; ptx::mbar_arrive(&red_bar[slot]); }
        if (ew == 0) {
          if (!ptx::mbar_wait_relaxed(&red_bar[slot], red_phase, abort_flag, P.wait_limit)) { ok = false; break; }
          const int tiles_n = (L.N + kBN - 1) / kBN;
          const long long slot_idx = (long long)it.example * P.n_per + L.col_begin + it.tm * tiles_n + it.tn;
          if (lane == 0 && dp_in_range(slot_idx, (long long)P.B * P.n_per, P.dev_status)) {
            float s = 0.f;
#pragma unroll
            for (int e = 0; e < kEpiWarps; ++e) s += epi_red[slot * kEpiWarps + e];
            P.sq_partials[slot_idx] = s;
          }
        }
      } else {
        // destination: the layer's output (no K split) or this split's partial plane
        float* dst;
        long long ld;
        float beta;
        if (P.nsplit == 1) { dst = L.out; ld = L.ldo; beta = P.beta; }
        else { dst = L.partial + size_t(it.split) * size_t(L.M) * L.N; ld = L.N; beta = 0.f; }
        // 32-byte (8 columns) or 16-byte accesses where the pitch and the base allow them
        const bool vec8 = ((ld & 7) == 0) && ((reinterpret_cast<uintptr_t>(dst) & 31) == 0);
        const bool vec4 = ((ld & 3) == 0) && ((reinterpret_cast<uintptr_t>(dst) & 15) == 0);
        // fused Gaussian mechanism (Eq. 3): only on the final destination, never on a K-split plane
        const bool noisy = (L.noise_amp >= 0.f) && (P.nsplit == 1);
        const float amp = L.noise_amp;
        const uint32_t tensor_id = L.tensor_id, step = effective_step(P.noise_step, P.step_dev);
#pragma unroll 1
        for (int c = c_lo; c < c_hi; ++c) {
          uint32_t r[32];
          ptx::tmem_ld_32x32b_x32(t0 + c * 32, r);
          ptx::tmem_ld_wait();
          // the accumulator is free as soon as its last part is in registers: the next tile's MMAs
          // do not wait for this warp's noise and stores
          if (c + 1 == c_hi) free_acc(buf);
          const int col0 = it.tn * kBN + c * 32;
          if (row < L.M) {
            // One row per lane, eight columns at a time: two Philox counters (N is a multiple of 4
            // where noise is fused, so a counter never straddles rows) and one 32-byte store, a whole
            // sector, per lane -- no in-register transpose (48 shuffles and 96 selects per chunk).
            // Together with the early release and the running layer search: 49 GPT-2-small layers at
            // B = 3, T = 77 (six K steps per tile) 480 -> 301 us with noise, 276 -> 215 us without;
            // 72 GPT-2-medium layers at B = 16, T = 128: 1161 -> 973 us; B = 64, T = 256: 1.19 -> 1.13 ms.
            float* o = dst + size_t(row) * ld + col0;
            const unsigned long long q0 = ((unsigned long long)row * L.N + col0) >> 2;   // first counter
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              const int left = L.N - col0 - 8 * g;             // columns of this row from here on
              if (left > 0) {
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[8 * g + e]);
                float* og = o + 8 * g;
                if (beta != 0.f) {
                  if (vec4 && left >= 8) {
                    const float4 a = *reinterpret_cast<const float4*>(og), b = *reinterpret_cast<const float4*>(og + 4);
                    v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
                    v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
                  } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e) if (e < left) v[e] += og[e];
                  }
                }
                if (noisy) {
#pragma unroll
                  for (int h = 0; h < 2; ++h) {
                    float z[4];
                    normals4(q0 + 2 * g + h, P.noise_keys, tensor_id, step, z);
#pragma unroll
                    for (int e = 0; e < 4; ++e) v[4 * h + e] = noised(v[4 * h + e], z[e], amp, P.noise_scale);
                  }
                }
                if (vec8 && left >= 8) {
                  ptx::st_global_v8(og, v);
                } else if (vec4 && left >= 8) {
                  __stcs(reinterpret_cast<float4*>(og), make_float4(v[0], v[1], v[2], v[3]));
                  __stcs(reinterpret_cast<float4*>(og + 4), make_float4(v[4], v[5], v[6], v[7]));
                } else {
#pragma unroll
                  for (int e = 0; e < 8; ++e) if (e < left) og[e] = v[e];
                }
              }
            }
          }
          __syncwarp();                                        // the TMEM load is a warp operation
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
  // pair: neither CTA may leave while the partner can still read its shared memory or arrive on
  // its barriers (every wait above is bounded, so both always get here)
  if (kPair) ptx::cluster_sync_all();
  if (warp == 1) {
    ptx::tc_fence_after();
    if (kPair) ptx::tmem_dealloc_pair(tmem_base, kTmemCols);
    else ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
}

// out = beta*out + sum over K splits of the partial planes, in split order, then the Gaussian
// mechanism of Eq. 3 -- for all layers of the launch in one kernel (a reduce and a noise pass per
// layer were two launches each).  A thread owns one Philox counter: four consecutive elements of
// the row-major output.
struct ReduceLayer {
  float* out;
  const float* partial;
  long long ldo;
  int M, N, block_begin;
  uint32_t tensor_id;
};
struct ReduceParams {
  ReduceLayer layer[kGtaMaxLayers];
  int n_layers, nsplit, with_noise;
  float beta, amp, scale;
  NoiseKeys keys;
  uint32_t step;
  const uint32_t* step_dev;
};
// Two quads per thread of 256-thread blocks, four planes in flight each; where that leaves SMs idle one quad per thread of 64,
// eight planes in flight: with its GEMM, one 64 x 64 layer of 148 planes (bf16, B = 16, T = 512) 18.4 -> 13.5 us, fp32 38 -> 19; one of
// 768 x 768 and 16 planes would go from 16.2 to 17.7 in that form.
template <int kThreads, int kPerThread, int kPlanes>
__global__ void __launch_bounds__(kThreads)
splitk_reduce_kernel(const __grid_constant__ ReduceParams P) {
  int lo = 0, hi = P.n_layers - 1;                   // the layer this block belongs to
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (int(blockIdx.x) >= P.layer[mid].block_begin) lo = mid; else hi = mid - 1;
  }
  const ReduceLayer& L = P.layer[lo];
  const size_t total = size_t(L.M) * L.N;
  const bool vec = (total & 3) == 0 && (reinterpret_cast<uintptr_t>(L.partial) & 15) == 0;
  const bool ovec = (L.N & 3) == 0 && (L.ldo & 3) == 0 && (reinterpret_cast<uintptr_t>(L.out) & 15) == 0;
  const uint32_t step = effective_step(P.step, P.step_dev);
#pragma unroll
  for (int k = 0; k < kPerThread; ++k) {
    const size_t q = (size_t(int(blockIdx.x) - L.block_begin) * kPerThread + k) * kThreads + threadIdx.x;
    const size_t e0 = 4 * q;
    if (e0 >= total) break;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (vec) {
      const float* src = L.partial + e0;
#pragma unroll kPlanes
      for (int s = 0; s < P.nsplit; ++s) {
        const float4 x = __ldcs(reinterpret_cast<const float4*>(src + size_t(s) * total));
        v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
      }
    } else {
      for (int s = 0; s < P.nsplit; ++s)
#pragma unroll
        for (int e = 0; e < 4; ++e) if (e0 + e < total) v[e] += L.partial[size_t(s) * total + e0 + e];
    }
    float z[4];
    if (P.with_noise) normals4(q, P.keys, L.tensor_id, step, z);
    const size_t r = e0 / L.N, c = e0 - r * L.N;
    float* o = L.out + r * L.ldo + c;
    if (ovec) {
      if (P.beta != 0.f) {
        const float4 x = *reinterpret_cast<const float4*>(o);
        v[0] = x.x + v[0]; v[1] = x.y + v[1]; v[2] = x.z + v[2]; v[3] = x.w + v[3];
      }
      if (P.with_noise)
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = noised(v[e], z[e], P.amp, P.scale);
      *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (e0 + e < total) {
          const size_t re = (e0 + e) / L.N;
          float* oe = L.out + re * L.ldo + (e0 + e - re * L.N);
          float x = (P.beta != 0.f) ? (*oe + v[e]) : v[e];
          if (P.with_noise) x = noised(x, z[e], P.amp, P.scale);
          *oe = x;
        }
      }
    }
  }
}

// out[r, :] = bf16(R_{r / T} * src[r, :]) for the B*T token rows of a narrow operand
__global__ void __launch_bounds__(256)
prescale_rows_kernel(const __nv_bfloat16* __restrict__ src, long long lds, __nv_bfloat16* __restrict__ dst,
                     int cp, long long rows, int T, int c, const float* __restrict__ clip) {
  const int per_row = cp >> 3;                      // 16-byte chunks per output row
  const long long total = rows * per_row;
  const bool vec = ((reinterpret_cast<uintptr_t>(src) & 15) == 0) && ((lds & 7) == 0);
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long r = e / per_row;
    const int c0 = int(e - r * per_row) << 3;
    float v[8];
    load8<__nv_bfloat16>(src + r * lds + c0, c - c0, vec, v);   // columns >= c read as zero
    const float f = clip[r / T];
    uint4 o;
    __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
    for (int k = 0; k < 4; ++k) o2[k] = __floats2bfloat162_rn(v[2 * k] * f, v[2 * k + 1] * f);
    *reinterpret_cast<uint4*>(dst + r * cp + c0) = o;
  }
}

// A layer whose narrow operand is at most a twentieth of its input bytes (the LM head: d = 768
// against p = 50257) gets that operand multiplied by R_i in a pass of its own -- a few
// microseconds -- and then runs through the GEMM unscaled: the in-pipeline scaling costs
// shared-memory bandwidth on EVERY K step of every tile of the wide operand, the copy does not.
inline bool prescale_layer(const dp_linear_desc& L) {
  return 20LL * std::min(L.d, L.p) <= (long long)L.d + L.p;
}
inline size_t prescale_bytes(const dp_linear_desc& L, int B, int T) {
  const int cp = (std::min(L.d, L.p) + 7) / 8 * 8;
  return align_up(size_t(B) * T * cp * 2, 256);
}

// The clipped sum always runs with kScale = true: on CTA pairs the scaler warps are also what
// tells rank 0's MMA issuer that BOTH CTAs' halves of a stage have landed.  (kScale = false is
// for the single-CTA DIRECT-norm kernel only; a pair kernel without the scalers' hand-off would
// let the issuer run ahead of the partner's loads and re-arm a stage barrier in mid-phase.)
constexpr bool kClipScale = true;

constexpr bool kUsePair = true;

// Launch on `units` persistent CTAs (single) or CTA pairs (cluster of 2).
template <bool kScale, bool kSqsum, bool kPair, bool kSplit, bool kByRow>
dp_status launch_gta(const GtaParams& P, int units, cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&gemm_gta_kernel<kScale, kSqsum, kPair, kSplit, kByRow>)))
    DP_CUDA_OK(allow_shared(gemm_gta_kernel<kScale, kSqsum, kPair, kSplit, kByRow>, Geo<kPair>::kSmemBytes));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kPair ? 2 * units : units, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = Geo<kPair>::kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kPair ? 2 : 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  DP_CUDA_OK(cudaLaunchKernelEx(&cfg, gemm_gta_kernel<kScale, kSqsum, kPair, kSplit, kByRow>, P));
  ++g_kernel_launches;
  return DP_OK;
}

}  // namespace

// K-split factor shared by all layers of one grouped call: 1 when the output tiles alone give
// every SM at least two items, otherwise enough splits to get there (>= 4 K steps per split).
long long gta_tiles(const dp_linear_desc& L) {
  return (long long)ceil_div(L.p, Geo<kUsePair>::kTileM) * ceil_div(L.d, kBN);
}

static long long gta_tiles(const dp_linear_desc* layers, int n_layers) {
  long long tiles = 0;
  for (int l = 0; l < n_layers; ++l) tiles += gta_tiles(layers[l]);
  return tiles;
}

bool gta_prescales(const dp_linear_desc& L) { return prescale_layer(L); }

static int choose_nsplit(long long tiles, int ksteps, int sms) {
  const int units = kUsePair ? sms / 2 : sms;          // persistent CTAs or CTA pairs
  if (tiles >= 2LL * units) return 1;
  long long ns = std::max<long long>(1, (2LL * units) / std::max<long long>(tiles, 1));
  ns = std::min<long long>(ns, std::max(1, ksteps / 4));
  return (int)std::max<long long>(1, ns);
}

// Two splits of one 64-token block each, three K steps, are no gain: 6 steps stay whole (fp32 at B = 1, T = 128: 4 GPT-2-small
// layers of d = 256 14.7 us, 17.6 in two).
int gta_choose_nsplit(long long tiles, int B, int T, int terms, int sms) {
  const GtaRows K = gta_rows(B, T, terms);
  return choose_nsplit(tiles, K.B * terms * ceil_div(K.T, kBK), sms);
}


size_t gta_partial_bytes(const dp_linear_desc* layers, int n_layers, int B, int T, int terms, int sms, bool ample) {
  const long long tiles = gta_tiles(layers, n_layers);
  const int ns = ample ? choose_nsplit(tiles, B * terms * ceil_div(T, kBK), sms) : gta_choose_nsplit(tiles, B, T, terms, sms);
  size_t n = 0;
  for (int l = 0; l < n_layers; ++l) {
    if (ns > 1) n += align_up(size_t(ns) * size_t(layers[l].p) * size_t(layers[l].d) * sizeof(float), 256);
    if (terms == 1 && prescale_layer(layers[l])) n += prescale_bytes(layers[l], B, T);
  }
  return n;
}

dp_status launch_clip_accumulate_tc(const dp_linear_desc* layers, int n_layers, int B, int T, int terms,
                                    const float* clip, float* const* outs, const int64_t* ldos,
                                    float beta, const GtaNoise* noise, float* partial_ws,
                                    int* dev_status, cudaStream_t st) {
  dp_status s = DP_OK;
  const int sms = sm_count();
  const GtaRows K = gta_rows(B, T, terms);
  const int tsteps = terms * ceil_div(K.T, kBK), planes = terms > 1 ? 2 * K.B : K.B;
  const int ksteps = K.B * tsteps;
  int nsplit = gta_choose_nsplit(gta_tiles(layers, n_layers), B, T, terms, sms);
  const int kps = terms * ceil_div(ksteps / terms, nsplit);   // whole 64-token blocks
  nsplit = ceil_div(ksteps, kps);                       // drop empty trailing splits
  // Two tiles per item need the tiles for it: at least two per CTA pair (the bound below which K is split;
  // with fewer, one-tile items spread over more SMs).
  const bool use_big = gta_tiles(layers, n_layers) >= 2LL * (sms / 2);
  char* pw = reinterpret_cast<char*>(partial_ws);
  char* pre = pw;                                       // pre-scaled copies sit behind the K-split planes
  if (pw && nsplit > 1)
    for (int l = 0; l < n_layers; ++l)
      pre += align_up(size_t(nsplit) * size_t(layers[l].p) * size_t(layers[l].d) * sizeof(float), 256);
  for (int g0 = 0; g0 < n_layers; g0 += kGtaMaxLayers) {
    const int g1 = std::min(n_layers, g0 + kGtaMaxLayers);
    GtaParams P;
    memset(&P, 0, sizeof(P));
    std::vector<GtaBigJob> big;
    int items = 0;
    for (int g = g0; g < g1; ++g) {
      dp_linear_desc D = layers[g];
      GtaLayer& L = P.layer[g - g0];
      L.prescaled = 0;
      if (clip && pw && prescale_layer(D)) {
        // R_i onto the narrow operand, into the workspace; the GEMM then reads the copy
        const bool narrow_a = D.d <= D.p;
        const int c = narrow_a ? D.d : D.p, cp = (c + 7) / 8 * 8;
        __nv_bfloat16* copy = reinterpret_cast<__nv_bfloat16*>(pre);
        pre += prescale_bytes(D, B, T);
        const long long rows = (long long)B * T;
        const int blocks = (int)std::min<long long>((rows * (cp >> 3) + 255) / 256, (long long)sms * 16);
        if (first_use_on_this_device(reinterpret_cast<const void*>(&prescale_rows_kernel)))
          DP_CUDA_OK(prefer_max_shared(prescale_rows_kernel));
        prescale_rows_kernel<<<blocks, 256, 0, st>>>(
            static_cast<const __nv_bfloat16*>(narrow_a ? D.A : D.G), narrow_a ? D.lda : D.ldg, copy, cp,
            rows, T, c, clip);
        DP_LAUNCH_OK();
        if (narrow_a) { D.A = copy; D.lda = cp; } else { D.G = copy; D.ldg = cp; }
        L.prescaled = 1;
      }
      if (!use_big) {
        s = make_tmap_bf16_3d(&P.tmG[g - g0], D.G, D.ldg, D.p, K.T, planes, 64, kBK);
        if (s != DP_OK) return s;
        s = make_tmap_bf16_3d(&P.tmA[g - g0], D.A, D.lda, D.d, K.T, planes, 64, kBK);
        if (s != DP_OK) return s;
      }
      L.out = outs[g]; L.ldo = ldos[g];
      L.M = D.p; L.N = D.d;
      L.partial = nullptr;
      if (nsplit > 1) {
        L.partial = reinterpret_cast<float*>(pw);
        pw += align_up(size_t(nsplit) * size_t(D.p) * size_t(D.d) * sizeof(float), 256);
      }
      L.item_begin = items; L.col_begin = 0;
      // noise is drawn in the epilogue when the layer is not K-split and its width is a
      // multiple of 4; otherwise a stand-alone pass follows (negative amp: no fused noise)
      const bool fuse = noise && nsplit == 1 && (D.d % 4 == 0);
      L.noise_amp = fuse ? noise->amp : -1.f;
      L.tensor_id = noise ? noise->tensor_ids[g] : 0u;
      if (use_big)
        big.push_back({D.A, D.lda, D.G, D.ldg, D.d, D.p, L.out, L.ldo, L.prescaled, L.noise_amp, L.tensor_id});
      items += ceil_div(D.p, Geo<kUsePair>::kTileM) * ceil_div(D.d, kBN) * nsplit;
    }
    if (noise) {
      P.noise_keys = expand_noise_keys(noise->seed);
      P.noise_step = noise->step; P.noise_scale = noise->scale;
      P.step_dev = g_step_dev;
    }
    P.n_layers = g1 - g0; P.B = K.B; P.T = K.T; P.tsteps = tsteps; P.low_plane = K.B;
    P.example_rows = T; P.rows = K.scaled_rows; P.example_steps = K.scaled_steps;
    P.total_items = items;
    P.nsplit = nsplit; P.ksteps_per_split = kps; P.beta = beta;
    P.clip = clip;
    P.dev_status = dev_status;
    P.wait_limit = g_wait_limit;
    const int units = std::min(items, kUsePair ? sms / 2 : sms);
    s = use_big ? launch_gta_big(big.data(), (int)big.size(), B, T, terms, clip, beta, noise, dev_status, st)
        : terms > 1     ? launch_gta<kClipScale, false, kUsePair, true, false>(P, units, st)
        : K.scaled_rows ? launch_gta<kClipScale, false, kUsePair, false, true>(P, units, st)
                        : launch_gta<kClipScale, false, kUsePair, false, false>(P, units, st);
    if (s != DP_OK) return s;
    if (nsplit > 1) {
      ReduceParams R;
      R.n_layers = P.n_layers; R.nsplit = nsplit; R.with_noise = noise ? 1 : 0; R.beta = beta;
      R.amp = noise ? noise->amp : 0.f; R.scale = noise ? noise->scale : 1.f;
      R.keys = expand_noise_keys(noise ? noise->seed : 0);
      R.step = noise ? noise->step : 0; R.step_dev = noise ? g_step_dev : nullptr;
      long long quads = 0, blocks = 0;
      for (int k = 0; k < P.n_layers; ++k) quads += ((long long)P.layer[k].M * P.layer[k].N + 3) / 4;
      const bool few = quads < (long long)sms * 512;
      const int per_block = few ? 64 : 512;
      for (int k = 0; k < P.n_layers; ++k) {
        const GtaLayer& L = P.layer[k];
        R.layer[k] = {L.out, L.partial, L.ldo, L.M, L.N, int(blocks), L.tensor_id};
        blocks += ((long long)L.M * L.N + 4LL * per_block - 1) / (4LL * per_block);
      }
      if (few) splitk_reduce_kernel<64, 1, 8><<<(unsigned)blocks, 64, 0, st>>>(R);
      else splitk_reduce_kernel<256, 2, 4><<<(unsigned)blocks, 256, 0, st>>>(R);
      DP_LAUNCH_OK();
      continue;
    }
    for (int g = g0; g < g1; ++g) {
      const GtaLayer& L = P.layer[g - g0];
      if (noise && L.noise_amp < 0.f) {        // not fused for this layer: stand-alone pass
        const dp_status ns = launch_add_noise(L.out, L.M, L.N, L.ldo, false, noise->amp,
                                              noise->scale, noise->seed, noise->tensor_ids[g],
                                              noise->step, st);
        if (ns != DP_OK) return ns;
      }
    }
  }
  return DP_OK;
}


dp_status launch_direct_norm_tc(const dp_linear_desc* layers, const GhostPlan& plan, int B, int T, int terms,
                                float* partials, int* dev_status, cudaStream_t st) {
  dp_status s = DP_OK;
  const int sms = sm_count(), planes = terms > 1 ? 2 * B : B;
  for (size_t g0 = 0; g0 < plan.direct_layers.size(); g0 += kGtaMaxLayers) {
    const size_t g1 = std::min(plan.direct_layers.size(), g0 + kGtaMaxLayers);
    GtaParams P;
    memset(&P, 0, sizeof(P));
    int items = 0;
    for (size_t g = g0; g < g1; ++g) {
      const int li = plan.direct_layers[g];
      const dp_linear_desc& D = layers[li];
      s = make_tmap_bf16_3d(&P.tmG[g - g0], D.G, D.ldg, D.p, T, planes, 64, kBK);
      if (s != DP_OK) return s;
      s = make_tmap_bf16_3d(&P.tmA[g - g0], D.A, D.lda, D.d, T, planes, 64, kBK);
      if (s != DP_OK) return s;
      GtaLayer& L = P.layer[g - g0];
      L.M = D.p; L.N = D.d;
      L.col_begin = plan.direct[li].col_begin;
      L.item_begin = items;
      items += B * plan.direct[li].tiles_m * plan.direct[li].tiles_n;
    }
    P.n_layers = int(g1 - g0);
    P.B = B; P.T = T; P.tsteps = terms * ceil_div(T, kBK); P.low_plane = B;
    P.total_items = items;
    P.nsplit = 1;
    P.sq_partials = partials; P.n_per = plan.n_per;
    P.dev_status = dev_status;
    P.wait_limit = g_wait_limit;
    s = terms > 1 ? launch_gta<false, true, false, true, false>(P, std::min(items, sms), st)
                  : launch_gta<false, true, false, false, false>(P, std::min(items, sms), st);
    if (s != DP_OK) return s;
  }
  return DP_OK;
}

}  // namespace dpg
