// Clipped sums out_l = beta*out_l + sum_i R_i G_i^T A_i (inner sum of Eq. 3) where there are tiles enough for
// every SM: the CTA-pair GEMM of gemm_gta_tc.cu with work items of two 256 x 256 output tiles that
// share an operand.
//
// What bounds the clipped sums at full size is energy: the chip sits at its power limit and the SM
// clock gives way (1.0 - 1.1 GHz).  Moving operand tiles from L2 to shared memory is about 30 % of it
// (leaving out the A loads of the one-tile kernel: + 19 % sustained throughput, both: + 42 %), and
// rewriting every G tile in shared memory to apply R_i another 8 %.  An item here keeps both
// accumulators of tensor memory busy -- two sub-tiles stacked along p ("tall") or side by side
// along d ("wide") -- and loads the shared operand X once for both: 48 KiB per 64 tokens instead of
// 64, and the clip factor goes onto X alone, half the shared-memory traffic per product.
//
// With both accumulators in one item nothing is double-buffered, so the sub-tiles are staggered: the
// first `skew` K steps of an item feed sub-tile 0 only, the steps up to the last feed both, and sub-tile
// 1 makes up for the steps it missed at the end.  While one sub-tile's accumulator is read -- and its
// Gaussian noise drawn, which takes thousands of cycles -- the tensor cores work on the other.  The
// price is loading X of `skew` steps twice and running those steps at half the products per stage (with
// few K steps it is not paid: skew 0).
// (Drawing the noise beside the item's MMAs and parking it, or the sums, in the output cost 8 % of the
// kernel in output traffic.)
//
// Sustained time of a call, one-tile kernel -> this one, same box: 48 GPT-2-medium layers at B = 16,
// T = 512: 2440 -> 2252 us (2410 -> 2159 without noise); 24 GPT-2-small layers at B = 64, T = 256: 1325 ->
// 1286; 72 medium layers at B = 8, T = 128: 762 -> 726, at B = 3, T = 77: 550 -> 537.  K steps of 32 tokens
// in nine stages instead of 64 in four: 2445 against 2290.
//
// Leftover rows or columns of tiles, and as many items as would fill only part of a last wave, run as
// single tiles in the same kernel (they alternate between the two accumulators).
//
// Roles per CTA (768 threads): warps 0, 2 and 3 TMA producers, warp 1 MMA issuer (rank 0), warps 4 - 7
// scalers, warps 8 - 23 epilogue.  Hand-offs across the pair as in gemm_gta_tc.cu; every wait is bounded.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "dp_common.cuh"
#include "gemm_gta.cuh"
#include "noise_device.cuh"
#include "ptx_sm100.cuh"
#include "tma_host.cuh"

namespace dpg {

namespace {

constexpr int kTile = 256;                           // sub-tile edge (both CTAs)
constexpr int kHalf = 128;                           // the part of it that one CTA loads
constexpr int kBK = 64;                              // tokens per K step
constexpr int kBoxBytes = kBK * 128;                 // 64 tokens x 64 columns
constexpr int kPartBytes = (kHalf / 64) * kBoxBytes; // 16 KiB: 128 columns of one operand
constexpr int kStageBytes = 3 * kPartBytes;          // X, Y of sub-tile 0, Y of sub-tile 1
constexpr int kStages = 4;
constexpr size_t kSmemBytes = size_t(kStages) * kStageBytes + 1024 + 1024;
// warp 0 loads Y of sub-tile 0, warp 2 X, warp 3 Y of sub-tile 1; warp 1 issues MMAs
constexpr int kProducerXWarp = 2, kProducerY1Warp = 3;
constexpr int kScalerWarp0 = 4, kScalerWarps = 4;
constexpr int kEpiWarp0 = kScalerWarp0 + kScalerWarps, kEpiWarps = 16;
constexpr int kColsPerWarp = kTile / (kEpiWarps / 4), kChunks = kColsPerWarp / 32;   // columns a warp reads, in chunks of 32
constexpr int kThreads = (kEpiWarp0 + kEpiWarps) * 32;
constexpr int kTmemCols = 512;

struct BigLayer {
  float* out;
  long long ldo;
  int M, N;                  // p, d
  int big_begin;             // first two-tile item of this layer
  int n_main;                // its items in the layer's own orientation; the rest lie along the leftover line
  int single_begin;          // leftover tiles of the layers before (one layer has at most one)
  int wide;                  // 1: the two sub-tiles lie side by side along N, 0: stacked along M
  int prescaled;             // 1: the clip factors were applied to this layer's narrow operand beforehand
  float noise_amp;           // sigma*C of the fused noise, negative = none
  uint32_t tensor_id;
};

struct __align__(64) BigParams {
  CUtensorMap tmG[kGtaMaxLayers];
  CUtensorMap tmA[kGtaMaxLayers];
  BigLayer layer[kGtaMaxLayers];
  int n_layers;
  int tsteps, ksteps;        // K steps per plane (split fp32: three per 64 tokens), K steps in all
  int low_plane;             // split operands: first plane of low terms
  int example_rows, rows, example_steps;     // scaling: tokens per example; all rows, or 0 and the steps of an example
  int skew;                  // K steps that sub-tile 1 of an item lags behind
  int n_big, n_big_total;    // two-tile items run as such, and in all (the rest as two singles each)
  int total_items;
  float beta;
  const float* clip;         // [B] R_i, NULL: operands arrive scaled
  NoiseKeys noise_keys;
  uint32_t noise_step;
  const uint32_t* step_dev;
  float noise_scale;
  int* dev_status;
  long long wait_limit;
};
static_assert(sizeof(BigParams) <= 32764, "kernel parameter block too large");

struct Item {
  int layer, wide, m0, n0;   // sub-tile indices of the first sub-tile
  int nsub;
};

// position and orientation of one two-tile item of layer L
__device__ __forceinline__ void big_tile(const BigLayer& L, int local, Item& it) {
  const int nt = (L.N + kTile - 1) / kTile, mt = (L.M + kTile - 1) / kTile;
  if (local < L.n_main) {
    it.wide = L.wide;
    if (L.wide) { const int pn = nt >> 1; it.n0 = 2 * (local % pn); it.m0 = local / pn; }
    else { it.n0 = local % nt; it.m0 = 2 * (local / nt); }
  } else {                                         // along the leftover column (wide) or row (tall)
    const int along = 2 * (local - L.n_main);
    it.wide = !L.wide;
    if (L.wide) { it.m0 = along; it.n0 = nt - 1; }
    else { it.n0 = along; it.m0 = mt - 1; }
  }
}

// `l` is the caller's running layer index (items of one kind ascend through the layers)
__device__ __forceinline__ Item decode_item(const BigParams& P, int item, int& l) {
  Item it;
  const int converted = 2 * (P.n_big_total - P.n_big);
  const int s = item - P.n_big;                    // index among the single tiles
  if (s < converted) {
    const int big = s < 0 ? item : P.n_big + (s >> 1);
    if (big < P.layer[l].big_begin) l = 0;
    while (l + 1 < P.n_layers && big >= P.layer[l + 1].big_begin) ++l;
    const BigLayer& L = P.layer[l];
    big_tile(L, big - L.big_begin, it);
    it.nsub = s < 0 ? 2 : 1;
    if (s >= 0) { if (it.wide) it.n0 += s & 1; else it.m0 += s & 1; }
  } else {
    const int k = s - converted;
    if (k < P.layer[l].single_begin) l = 0;
    while (l + 1 < P.n_layers && k >= P.layer[l + 1].single_begin) ++l;
    const BigLayer& L = P.layer[l];                // a layer's last corner
    it.m0 = (L.M + kTile - 1) / kTile - 1;
    it.n0 = (L.N + kTile - 1) / kTile - 1;
    it.wide = 0;
    it.nsub = 1;
  }
  it.layer = l;
  return it;
}

// Which accumulators an item uses, and how often each was used before: the same sequence in every role.
struct Slots {
  uint32_t uses0 = 0, uses1 = 0, toggle = 0;
  __device__ __forceinline__ uint32_t first(int nsub) const { return nsub == 2 ? 0u : toggle; }
  __device__ __forceinline__ uint32_t uses(uint32_t slot) const { return slot ? uses1 : uses0; }
  __device__ __forceinline__ void advance(int nsub) {
    if (nsub == 2) { ++uses0; ++uses1; }
    else { if (toggle) ++uses1; else ++uses0; toggle ^= 1u; }
  }
};

// What the epilogue writes.  kPlain: sums without noise.  kStraight: noise at scale 1 onto outputs that are written whole, 32 bytes
// at a time, has straight code of its own, and what little else there is calls the generator: with one path for all the epilogue took 180
// instructions per counter, 137 of them the generator's, and where few tokens meet many parameters its rate is the step's (the call for
// 48 GPT-2-small layers at B = 3, T = 77 202 -> 183 us, for 96 of GPT-2 medium at B = 16, T = 128 1310 -> 1255).
// kGeneral: everything else, the generator in line (called from there, 48 GPT-2-small layers at B = 3, T = 77 with scale 1/B took
// 276 us instead of 206, with beta = 1 401 instead of 294).
enum Epilogue { kPlain, kStraight, kGeneral };

static __device__ __noinline__ float4 normals4_call(unsigned long long q, const NoiseKeys& K, uint32_t id, uint32_t step) {
  float z[4];
  normals4(q, K, id, step, z);
  return make_float4(z[0], z[1], z[2], z[3]);
}

template <bool kSplit, bool kByRow, Epilogue kEpilogue>
__global__ void __launch_bounds__(kThreads, 1)
gemm_gta_big_kernel(const __grid_constant__ BigParams P) {
  const uint32_t rank = ptx::cluster_ctarank();
  const int first_item = int(blockIdx.x >> 1), item_stride = int(gridDim.x >> 1);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + size_t(kStages) * kStageBytes);
  uint64_t* full = bars;                      // the producers' TMA loads landed
  uint64_t* ready = bars + kStages;           // X scaled and all loaded in both CTAs (rank 0's copy)
  uint64_t* empty = bars + 2 * kStages;       // MMAs retired
  uint64_t* acc_full = bars + 3 * kStages;    // [2]
  uint64_t* acc_empty = acc_full + 2;         // [2]
  uint64_t* mma_done = acc_empty + 2;         // only used when the MMA issuer gives up
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint32_t* sink = tmem_slot + 2;             // [kStages + 1] written by st.async, never read

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t tiles_a = ptx::smem_u32(tiles);
  const uint32_t full_a = ptx::smem_u32(full), ready_a = ptx::smem_u32(ready), empty_a = ptx::smem_u32(empty);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(&full[s], 3);            // the three producers
      ptx::mbar_init(&ready[s], 1);           // rank 0's scaler warp announces the 4 bytes rank 1's sends
      ptx::mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(&acc_full[b], 1);
      ptx::mbar_init(&acc_empty[b], kEpiWarps);   // + 4 bytes from each epilogue warp of rank 1
    }
    ptx::mbar_init(mma_done, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) { ptx::tmem_alloc_pair(tmem_slot, kTmemCols); ptx::tmem_relinquish_pair(); }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync_all();                    // the partner's barriers exist before anyone arrives on them
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0 || warp == kProducerXWarp || warp == kProducerY1Warp) {
    // ------------------------------------------------------------- TMA producers
    // the whole warp runs the loop, an elected lane issues (see ptx::warp_ok)
    const bool is_x = warp == kProducerXWarp;
    const int sub = warp == kProducerY1Warp ? 1 : 0;         // the Y part this warp loads
    uint32_t stage = 0, phase = 0, issued = 0;
    int lay = 0;
    bool ok = true;
    for (int item = first_item; item < P.total_items && ok; item += item_stride) {
      const Item it = decode_item(P, item, lay);
      // tall: X = A, Y = G; wide: X = G, Y = A
      const bool is_g = is_x == (it.wide != 0);
      const uint64_t tm = reinterpret_cast<uint64_t>(is_g ? &P.tmG[it.layer] : &P.tmA[it.layer]);
      const int c0 = ((is_g ? it.m0 : it.n0) + sub) * kTile + int(rank) * kHalf;
      const bool loads = sub < it.nsub;
      const uint32_t dst0 = tiles_a + (is_x ? 0 : (1 + sub) * kPartBytes);
      const int skew = it.nsub == 2 ? P.skew : 0, steps = P.ksteps + skew;
      // the steps in which this warp's part takes part
      const int from = sub ? skew : 0, to = is_x || sub ? steps : P.ksteps;
      constexpr int kTerms = kSplit ? 3 : 1;
      GtaWalk<kSplit> at(0, 0, P.ksteps / kTerms, P.tsteps / kTerms);
      for (int j = 0; j < steps; ++j) {
        if (j == P.ksteps) at = GtaWalk<kSplit>(0, 0, P.ksteps / kTerms, P.tsteps / kTerms);
        ok = ptx::warp_ok(ptx::mbar_wait_a(empty_a + 8 * stage, phase ^ 1, abort_flag, P.wait_limit));
        if (!ok) break;
        const uint32_t bar = full_a + 8 * stage;
        const uint32_t dst = dst0 + stage * kStageBytes;
        const bool go = loads && j >= from && j < to;
        if (ptx::elect_one()) {
          ptx::mbar_arrive_expect_tx_a(bar, go ? uint32_t(kPartBytes) : 0u);
          if (go)
#pragma unroll
            for (int b = 0; b < kHalf / 64; ++b)
              ptx::tma_load_3d_a(dst + b * kBoxBytes, tm, bar, c0 + b * 64, at.ts * kBK, at.plane(!is_g, P.low_plane));
        }
        __syncwarp();
        ++issued;
        at.next();
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    }
    if (!ok && ptx::elect_one()) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
      ptx::drain_issued_copies(full, kStages, issued);   // copies in flight land before exit
    }
  } else if (warp == 1) {
    // --------------------------------------------------------------- MMA issuer
    // the whole warp runs the loop, an elected lane issues (see ptx::warp_ok)
    if (rank == 0) {
      constexpr uint32_t idesc = ptx::idesc_bf16_f32(kTile, kTile, 1, 1);
      // MN-major, 128-byte swizzle: 64-column boxes are kBoxBytes apart, groups of 8 tokens 1 KiB
      constexpr uint64_t dbase = ptx::smem_desc_base(kBoxBytes, 1024, ptx::SWIZZLE_128B);
      constexpr uint32_t desc_hi = uint32_t(dbase >> 32);
      const uint32_t desc_lo0 = uint32_t(dbase) | ((tiles_a >> 4) & 0x3FFF);
      uint32_t stage = 0, phase = 0;
      int lay = 0;
      bool ok = true;
      Slots slots;
      for (int item = first_item; item < P.total_items && ok; item += item_stride) {
        const Item it = decode_item(P, item, lay);
        const uint32_t slot0 = slots.first(it.nsub);
        constexpr uint32_t part = kPartBytes >> 4;
        const uint32_t off_g = it.wide ? 0u : part, off_a = it.wide ? part : 0u;       // first sub-tile's Y
        const uint32_t step_g = off_g, step_a = off_a;                                 // to the second one's
        const int skew = it.nsub == 2 ? P.skew : P.ksteps, steps = it.nsub == 2 ? P.ksteps + skew : P.ksteps;
        for (int j = 0; j < steps; ++j) {
          ok = ptx::warp_ok(ptx::mbar_wait_cluster_a(ready_a + 8 * stage, phase, abort_flag, P.wait_limit));
          // an accumulator's first use in this item: it has been read for the item before
          if (ok && j == 0)
            ok = ptx::warp_ok(ptx::mbar_wait_cluster(&acc_empty[slot0], (slots.uses(slot0) & 1) ^ 1, abort_flag, P.wait_limit));
          if (ok && j == skew)
            ok = ptx::warp_ok(ptx::mbar_wait_cluster(&acc_empty[1], (slots.uses1 & 1) ^ 1, abort_flag, P.wait_limit));
          if (!ok) break;
          ptx::tc_fence_after();
          const uint32_t lo = desc_lo0 + stage * (kStageBytes >> 4);
          const uint32_t lo_g = lo + off_g, lo_a = lo + off_a;
          if (j < P.ksteps && ptx::elect_one()) {
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              ptx::mma_bf16_ss_pair_lh(tmem_base + slot0 * kTile, lo_g + kk * 128, lo_a + kk * 128, desc_hi, idesc,
                                       (j > 0 || kk > 0) ? 1u : 0u);
            if (j + 1 == P.ksteps) ptx::mma_commit_pair(&acc_full[slot0], 3);
          }
          __syncwarp();
          if (j >= skew && ptx::elect_one()) {
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              ptx::mma_bf16_ss_pair_lh(tmem_base + kTile, lo_g + step_g + kk * 128, lo_a + step_a + kk * 128, desc_hi,
                                       idesc, (j > skew || kk > 0) ? 1u : 0u);
            if (j + 1 == steps) ptx::mma_commit_pair(&acc_full[1], 3);
          }
          __syncwarp();
          if (ptx::elect_one()) ptx::mma_commit_pair_a(empty_a + 8 * stage, 3);   // stage reusable in both CTAs
          __syncwarp();
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
        slots.advance(it.nsub);
      }
      if (!ok && ptx::elect_one()) {
        *abort_flag = 1;
        if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
        ptx::drain_issued_mmas(mma_done, true);
      }
    }
  } else if (warp < kEpiWarp0) {
    // ------------------------------------------------------------------ scalers
    // Every scaler warp owns every fourth K step: it waits for the stage, multiplies X's rows by their
    // examples' clip factors where that has not been done yet, and tells rank 0's issuer (see gemm_gta_tc.cu for the
    // barriers' reasoning: the wait on `empty` makes the parity of `full` exact).
    const int sw = warp - kScalerWarp0;
    const uint32_t ready_remote = ptx::mapa_u32(ready_a, 0);
    const uint32_t sink_remote = ptx::mapa_u32(ptx::smem_u32(sink), 0);
    uint32_t cnt = 0;
    int lay = 0;
    bool ok = true;
    for (int item = first_item; item < P.total_items && ok; item += item_stride) {
      const Item it = decode_item(P, item, lay);
      const bool scale_here = P.clip && !P.layer[it.layer].prescaled;
      const int steps = P.ksteps + (it.nsub == 2 ? P.skew : 0);
      auto factors = [&](int j) {              // of step j (the last `skew` steps are the first again)
        if (!scale_here || j >= steps) return RowFactors{1.f, 1.f, true};
        return row_factors<kByRow>(P.clip, j < P.ksteps ? j : j - P.ksteps, lane, P.example_rows, P.rows, P.example_steps);
      };
      int j = int((uint32_t(sw) + kScalerWarps - cnt % kScalerWarps) % kScalerWarps);
      uint32_t c = cnt + uint32_t(j);
      RowFactors r_next = factors(j);
      for (; j < steps; j += kScalerWarps, c += kScalerWarps) {
        const RowFactors r = r_next;
        r_next = factors(j + kScalerWarps);
        const uint32_t stage = c % kStages, fill = c / kStages, phase = fill & 1u;
        if (fill > 0 && !ptx::mbar_wait_a(empty_a + 8 * stage, phase ^ 1, abort_flag, P.wait_limit)) { ok = false; break; }
        if (!ptx::mbar_wait_a(full_a + 8 * stage, phase, abort_flag, P.wait_limit)) { ok = false; break; }
        uint4* part = reinterpret_cast<uint4*>(tiles + size_t(stage) * kStageBytes);
        if (kByRow && !r.one) scale_rows(part, r.lo, r.hi, lane);
        else if (r.lo != 1.0f) scale_part(part, r.lo, lane);
        if (scale_here) ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (rank == 0) ptx::mbar_arrive_expect_tx_a(ready_a + 8 * stage, 4);
          else ptx::st_async_signal_a(ready_remote + 8 * stage, sink_remote + 4 * stage);
        }
      }
      cnt += uint32_t(steps);
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
    }
  } else {
    // ----------------------------------------------------------------- epilogue
    const int q = warp & 3;                          // TMEM lane quarter this warp may read
    const int cg = (warp - kEpiWarp0) >> 2;          // which kColsPerWarp of the 256 columns
    const uint32_t acc_empty_a = ptx::smem_u32(acc_empty);
    const uint32_t acc_empty_remote = ptx::mapa_u32(acc_empty_a, 0);
    const uint32_t sink_remote = ptx::mapa_u32(ptx::smem_u32(sink + kStages), 0);
    auto free_acc = [&](uint32_t slot) {
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0) ptx::mbar_arrive_expect_tx_a(acc_empty_a + 8 * slot, 4);
        else ptx::st_async_signal_a(acc_empty_remote + 8 * slot, sink_remote);
      }
    };
    const uint32_t step = effective_step(P.noise_step, P.step_dev);
    int lay = 0;
    bool ok = true;
    Slots slots;
    for (int item = first_item; item < P.total_items && ok; item += item_stride) {
      const Item it = decode_item(P, item, lay);
      const BigLayer& L = P.layer[it.layer];
      const long long ld = L.ldo;
      const bool vec8 = ((ld & 7) == 0) && ((reinterpret_cast<uintptr_t>(L.out) & 31) == 0);
      const bool vec4 = ((ld & 3) == 0) && ((reinterpret_cast<uintptr_t>(L.out) & 15) == 0);
      const bool noisy = kEpilogue != kPlain && L.noise_amp >= 0.f;
      const float amp = L.noise_amp;
      const uint32_t tensor_id = L.tensor_id;
      const bool straight = kEpilogue == kStraight && noisy && vec8;
      for (int h = 0; h < it.nsub; ++h) {
        const uint32_t slot = slots.first(it.nsub) + h;
        if (!ptx::mbar_wait_relaxed(&acc_full[slot], slots.uses(slot) & 1, abort_flag, P.wait_limit)) { ok = false; break; }
        ptx::tc_fence_after();
        const int row = (it.m0 + (it.wide ? 0 : h)) * kTile + int(rank) * kHalf + q * 32 + lane;
        const int colh = (it.n0 + (it.wide ? h : 0)) * kTile + cg * kColsPerWarp;
        const uint32_t t0 = tmem_base + (uint32_t(q * 32) << 16) + slot * kTile + cg * kColsPerWarp;
#pragma unroll 1
        for (int c = 0; c < kChunks; ++c) {
          const int col0 = colh + c * 32;
          float* o = L.out + size_t(row) * ld + col0;
          uint32_t r[32];
          ptx::tmem_ld_32x32b_x32(t0 + c * 32, r);
          ptx::tmem_ld_wait();
          // free as soon as the last part is in registers, before its noise is drawn
          if (c + 1 == kChunks) free_acc(slot);
          if (straight && row < L.M && col0 + 32 <= L.N) {
            const unsigned long long q0 = ((unsigned long long)row * L.N + col0) >> 2;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              float v[8];
#pragma unroll
              for (int k = 0; k < 2; ++k) {
                float z[4];
                normals4(q0 + 2 * g + k, P.noise_keys, tensor_id, step, z);
#pragma unroll
                for (int e = 0; e < 4; ++e) v[4 * k + e] = noised(__uint_as_float(r[8 * g + 4 * k + e]), z[e], amp, 1.f);
              }
              ptx::st_global_v8(o + 8 * g, v);
            }
          } else if (row < L.M) {
            // eight columns at a time: two Philox counters (N is a multiple of 4 where noise is fused, so
            // a counter never straddles rows) and one 32-byte store, a whole sector, per lane
            const unsigned long long q0 = ((unsigned long long)row * L.N + col0) >> 2;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              const int left = L.N - col0 - 8 * g;           // columns of this row from here on
              if (left > 0) {
                float v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[8 * g + e]);
                float* og = o + 8 * g;
                if (P.beta != 0.f) {
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
                  for (int k = 0; k < 2; ++k) {
                    float z[4];
                    if (kEpilogue == kGeneral) {
                      normals4(q0 + 2 * g + k, P.noise_keys, tensor_id, step, z);
                    } else {
                      const float4 f = normals4_call(q0 + 2 * g + k, P.noise_keys, tensor_id, step);
                      z[0] = f.x; z[1] = f.y; z[2] = f.z; z[3] = f.w;
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) v[4 * k + e] = noised(v[4 * k + e], z[e], amp, P.noise_scale);
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
          __syncwarp();
        }
      }
      slots.advance(it.nsub);
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

}  // namespace

template <bool kSplit, bool kByRow, Epilogue kEpilogue>
static dp_status launch_big(const BigParams& P, int units, cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&gemm_gta_big_kernel<kSplit, kByRow, kEpilogue>)))
    DP_CUDA_OK((allow_shared(gemm_gta_big_kernel<kSplit, kByRow, kEpilogue>, kSmemBytes)));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * units, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  DP_CUDA_OK((cudaLaunchKernelEx(&cfg, gemm_gta_big_kernel<kSplit, kByRow, kEpilogue>, P)));
  ++g_kernel_launches;
  return DP_OK;
}

// The straight epilogue runs beside the scalers that know factors per row, used or not: without that code the scalers are ready
// sooner and poll more beside warps that are bound by their instructions (24 GPT-2-small layers at B = 32, T = 128 with noise 373 us, 377
// without; sums alone 368 and 367).
template <bool kSplit, bool kByRow>
static dp_status launch_big(const BigParams& P, Epilogue epilogue, int units, cudaStream_t st) {
  return epilogue == kPlain      ? launch_big<kSplit, kByRow, kPlain>(P, units, st)
         : epilogue == kStraight ? launch_big<kSplit, !kSplit, kStraight>(P, units, st)
                                 : launch_big<kSplit, kByRow, kGeneral>(P, units, st);
}

// One launch over at most kGtaMaxLayers layers without a K split.
dp_status launch_gta_big(const GtaBigJob* jobs, int n, int B, int T, int terms, const float* clip, float beta,
                         const GtaNoise* noise, int* dev_status, cudaStream_t st) {
  BigParams P;
  memset(&P, 0, sizeof(P));
  const GtaRows K = gta_rows(B, T, terms);
  const int planes = terms > 1 ? 2 * K.B : K.B;
  int bigs = 0, singles = 0;
  long long outputs = 0, odd = 0;               // with noise; of these, not in a full chunk of 32 columns on a 32-byte boundary
  for (int k = 0; k < n; ++k) {
    const GtaBigJob& J = jobs[k];
    if (J.noise_amp >= 0.f) {
      outputs += (long long)J.p * J.d;
      odd += (long long)J.p * (reinterpret_cast<uintptr_t>(J.out) % 32 == 0 && J.ldo % 8 == 0 ? J.d % 32 : J.d);
    }
    dp_status s = make_tmap_bf16_3d(&P.tmG[k], J.G, J.ldg, J.p, K.T, planes, 64, kBK);
    if (s != DP_OK) return s;
    s = make_tmap_bf16_3d(&P.tmA[k], J.A, J.lda, J.d, K.T, planes, 64, kBK);
    if (s != DP_OK) return s;
    BigLayer& L = P.layer[k];
    L.out = J.out; L.ldo = J.ldo; L.M = J.p; L.N = J.d;
    L.prescaled = J.prescaled; L.noise_amp = J.noise_amp; L.tensor_id = J.tensor_id;
    // the orientation that leaves the shorter line of tiles; that line is paired along its length
    const int mt = ceil_div(J.p, kTile), nt = ceil_div(J.d, kTile);
    const int left_tall = (mt & 1) * nt, left_wide = (nt & 1) * mt;
    L.wide = left_wide < left_tall ? 1 : 0;
    const int line = std::min(left_tall, left_wide);
    L.n_main = L.wide ? mt * (nt / 2) : (mt / 2) * nt;
    L.big_begin = bigs; L.single_begin = singles;
    bigs += L.n_main + line / 2;
    singles += line & 1;
  }
  const int pairs = sm_count() / 2;
  // items that would fill only part of a wave of two-tile items: as singles if that ends sooner
  const int rest = bigs % pairs;
  const int keep = 2 + ceil_div(singles, pairs), convert = ceil_div(2 * rest + singles, pairs);
  P.n_big_total = bigs;
  P.n_big = (rest && convert < keep) ? bigs - rest : bigs;
  P.total_items = P.n_big + 2 * (bigs - P.n_big) + singles;
  P.n_layers = n;
  P.tsteps = terms * ceil_div(K.T, kBK); P.ksteps = K.B * P.tsteps; P.low_plane = K.B;
  P.example_rows = T; P.rows = K.scaled_rows; P.example_steps = K.scaled_steps;
  // Long enough to read one accumulator, and to draw its noise, while the other is fed: with noise 4, 6, 8,
  // 10, 12, 24 and 40 steps gave 2341, 2278, 2252, 2265, 2283, 2407 and 2513 us (B = 16, T = 512).  The same
  // without noise, which would do with 2 or none, so that a sum does not depend on whether noise is fused.
  // With few K steps the epilogue is all there is and the staggered steps only cost loads: no skew below 16.
  // Sustained, with noise: 215.0 -> 204.6 us at 6 steps (B = 3, T = 77, 48 GPT-2-small layers), 243.5 -> 232.6 at 8
  // (B = 4, T = 128), but 298.6 -> 305.9 at 16 and 772 -> 790 at 32.  (Without noise
  // 258.7 -> 241.6 at 16 as well.)
  P.skew = P.ksteps < 16 ? 0 : 8;
  P.beta = beta; P.clip = clip;
  if (noise) {
    P.noise_keys = expand_noise_keys(noise->seed);
    P.noise_step = noise->step; P.noise_scale = noise->scale; P.step_dev = g_step_dev;
  }
  P.dev_status = dev_status;
  P.wait_limit = g_wait_limit;
  const int units = std::min(P.total_items, pairs);
  // A called generator costs a third of an output's time, the straight code saves a twelfth: one output in eight may be odd.
  const Epilogue epilogue = !noise ? kPlain : beta == 0.f && noise->scale == 1.f && 8 * odd <= outputs ? kStraight : kGeneral;
  return terms > 1       ? launch_big<true, false>(P, epilogue, units, st)
         : K.scaled_rows ? launch_big<false, true>(P, epilogue, units, st)
                         : launch_big<false, false>(P, epilogue, units, st);
}

}  // namespace dpg
