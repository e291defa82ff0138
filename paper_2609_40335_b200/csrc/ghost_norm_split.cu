// Ghost norm of fp32 layers of at most 128 tokens, and their split into two bf16 terms, in one pass over the operands.
//
// The Gram products are those of ghost_norm_tc.cu on split operands (S = hi hi^T + hi lo^T + lo hi^T, the two small
// products in an accumulator of their own); the terms are those of split_kernels.cu.  There the split read 4 bytes per value and
// wrote 4, and the Gram kernel read 4 again.  Here the tiles arrive in fp32 and eight converter warps make both terms on the way, into
// shared memory, in the swizzled layout that the MMAs read; and, where clipped sums follow that can use them, into the planes where
// these look for them.  That is the wider operand of a layer: the narrower one is split again, scaled, for the sums.  Each column of the
// operand that is cut into chunks is some item's own; the other, which every chunk of a layer multiplies, is written by the first.
//
// Bound by HBM (4 bytes in, and 4 out for the values that are kept) and by its last wave (156 steps on the busiest SM, 119 on average).
// Norms alone of DistilGPT2's 25 layers at B = 8, T = 128: 275 us split first, 227 with every plane stored, 145 with none; the step
// 850 -> 801.
//
// A tile holds the rows of as many whole examples as fit into 128 (one above 64 tokens; see ghost_norm_tc.cu), rounded up to
// 16 rows.  Roles per CTA (448 threads): warp 0 TMA producer, warp 1 MMA issuer, warps 2 - 5 epilogue, warps 6 - 13
// converters (16 rows each).  Two rings of 32 KiB stages: fp32 tiles, and pairs of bf16 tiles.  Every wait is bounded.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "dp_common.cuh"
#include "ghost_plan.cuh"
#include "ptx_sm100.cuh"
#include "split_kernels.cuh"
#include "tma_host.cuh"

namespace dpg {

namespace {

constexpr int kTile = 128;                         // most rows of a tile
constexpr int kKStep = 64;                         // columns per stage
constexpr int kHalfBytes = kTile * 128;            // 32 fp32 or 64 bf16 columns of 128 rows
constexpr int kStageBytes = 2 * kHalfBytes;        // fp32: columns 0 - 31 and 32 - 63; bf16: high and low terms
constexpr int kStagesIn = 3, kStages = 3;
constexpr int kEpiWarp0 = 2, kConvWarp0 = 6, kConvWarps = 8;
constexpr int kThreads = (kConvWarp0 + kConvWarps) * 32;
constexpr int kTmemCols = 512;                     // S_A, S_G of hi hi^T; the same of the small products
constexpr int kMaxLayers = 96;
constexpr size_t kRingBytes = size_t(kStagesIn + kStages) * kStageBytes;
constexpr size_t kSmemBytes = kRingBytes + 1024 /*alignment slack*/ + 1024 /*barriers*/ + 4 * kTile * sizeof(float);

struct SplitPlanes {
  __nv_bfloat16* hi;                               // nullptr: not kept
  __nv_bfloat16* lo;
  int cols;                                        // pitch, a multiple of 8
};
struct __align__(64) SplitGramParams {
  CUtensorMap tmA[kMaxLayers];                     // fp32, the rows of the batch as one dimension
  CUtensorMap tmG[kMaxLayers];
  GhostLayerPlan layer[kMaxLayers];
  SplitPlanes A[kMaxLayers], G[kMaxLayers];
  int n_layers;
  int B, T, pack, rows;                            // examples per tile and its rows
  int total_items, n_per;
  float* partials;                                 // [B][n_per]
  int* dev_status;
  long long wait_limit;
};
static_assert(sizeof(SplitGramParams) <= 32764, "kernel parameter block too large");

struct Item {
  int layer, tile, a0, a1, g0, g1, col;
  bool write_a, write_g;
};
__device__ __forceinline__ Item decode_item(const SplitGramParams& P, int item, int& l) {
  Item it;
  while (l + 1 < P.n_layers && item >= P.layer[l + 1].item_begin) ++l;
  const GhostLayerPlan& L = P.layer[l];
  const int local = item - L.item_begin, s = local % L.nsplit, c0 = s * L.chunk_steps;
  it.tile = local / L.nsplit;
  it.layer = l;
  it.a0 = L.split_on_g ? 0 : c0;
  it.a1 = L.split_on_g ? L.a_steps : min(c0 + L.chunk_steps, L.a_steps);
  it.g0 = L.split_on_g ? c0 : 0;
  it.g1 = L.split_on_g ? min(c0 + L.chunk_steps, L.g_steps) : L.g_steps;
  it.write_a = !L.split_on_g || s == 0;
  it.write_g = L.split_on_g || s == 0;
  it.col = L.col_begin + s;
  return it;
}

__global__ void __launch_bounds__(kThreads, 1)
ghost_norm_split_kernel(const __grid_constant__ SplitGramParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* in = tiles + size_t(kStages) * kStageBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles + kRingBytes);     // [kStages]   converters -> MMA
  uint64_t* empty = full + kStages;                // [kStages]   MMA -> converters
  uint64_t* in_full = empty + kStages;             // [kStagesIn] TMA -> converters
  uint64_t* in_empty = in_full + kStagesIn;        // [kStagesIn] converters -> TMA
  uint64_t* acc_full = in_empty + kStagesIn;       //             MMA -> epilogue
  uint64_t* acc_empty = acc_full + 1;              //             epilogue -> MMA
  uint64_t* mma_done = acc_empty + 1;              // only used when the MMA issuer gives up
  uint64_t* red_bar = mma_done + 1;                // [4]         epilogue warps -> epilogue warp 0
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(red_bar + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* row_sum = reinterpret_cast<float*>(tmem_slot + 2);             // [4][kTile]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { ptx::mbar_init(&full[s], kConvWarps); ptx::mbar_init(&empty[s], 1); }
    for (int s = 0; s < kStagesIn; ++s) { ptx::mbar_init(&in_full[s], 1); ptx::mbar_init(&in_empty[s], kConvWarps); }
    ptx::mbar_init(acc_full, 1);
    ptx::mbar_init(acc_empty, 4);
    ptx::mbar_init(mma_done, 1);
    for (int b = 0; b < 4; ++b) ptx::mbar_init(&red_bar[b], 4);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 1) { ptx::tmem_alloc(tmem_slot, kTmemCols); ptx::tmem_relinquish(); }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tiles_a = ptx::smem_u32(tiles), in_a = ptx::smem_u32(in);
  const uint32_t full_a = ptx::smem_u32(full), empty_a = ptx::smem_u32(empty);
  const uint32_t in_full_a = ptx::smem_u32(in_full), in_empty_a = ptx::smem_u32(in_empty);

  if (warp == 0) {
    // ------------------------------------------------------------- TMA producer
    // producer and issuer: the whole warp runs the loop, an elected lane issues (see ptx::warp_ok)
    uint32_t stage = 0, phase = 0, issued = 0;
    int lay = 0;
    bool ok = true;
    const uint32_t bytes = uint32_t(P.rows) * 256u;
    for (int item = blockIdx.x; item < P.total_items && ok; item += gridDim.x) {
      const Item it = decode_item(P, item, lay);
      const int row = it.tile * P.pack * P.T;
      for (int pass = 0; pass < 2 && ok; ++pass) {
        const uint64_t tm = reinterpret_cast<uint64_t>(pass == 0 ? &P.tmA[it.layer] : &P.tmG[it.layer]);
        const int k0 = pass == 0 ? it.a0 : it.g0, k1 = pass == 0 ? it.a1 : it.g1;
        for (int k = k0; k < k1; ++k) {
          ok = ptx::warp_ok(ptx::mbar_wait_a(in_empty_a + 8 * stage, phase ^ 1, abort_flag, P.wait_limit));
          if (!ok) break;
          const uint32_t dst = in_a + stage * kStageBytes, bar = in_full_a + 8 * stage;
          if (ptx::elect_one()) {
            ptx::mbar_arrive_expect_tx_a(bar, bytes);
            ptx::tma_load_3d_a(dst, tm, bar, k * kKStep, row, 0);
            ptx::tma_load_3d_a(dst + kHalfBytes, tm, bar, k * kKStep + 32, row, 0);
          }
          __syncwarp();
          ++issued;
          if (++stage == kStagesIn) { stage = 0; phase ^= 1; }
        }
      }
    }
    if (!ok && ptx::elect_one()) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
      ptx::drain_issued_copies(in_full, kStagesIn, issued);
    }
  } else if (warp == 1) {
    // --------------------------------------------------------------- MMA issuer
    const uint32_t idesc = ptx::idesc_bf16_f32(kTile, P.rows, 0, 0);
    constexpr uint64_t dbase = ptx::smem_desc_base(16, 1024, ptx::SWIZZLE_128B);          // K-major
    constexpr uint32_t desc_hi = uint32_t(dbase >> 32), low = kHalfBytes >> 4;
    const uint32_t desc_lo0 = uint32_t(dbase) | ((tiles_a >> 4) & 0x3FFF);
    uint32_t stage = 0, phase = 0, n_item = 0;
    int lay = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < P.total_items && ok; item += gridDim.x, ++n_item) {
      const Item it = decode_item(P, item, lay);
      ok = ptx::warp_ok(ptx::mbar_wait(acc_empty, (n_item & 1) ^ 1, abort_flag, P.wait_limit));
      if (!ok) break;
      ptx::tc_fence_after();
      for (int pass = 0; pass < 2 && ok; ++pass) {
        const uint32_t d_tmem = tmem_base + pass * kTile;
        const int nsteps = pass == 0 ? it.a1 - it.a0 : it.g1 - it.g0;
        for (int k = 0; k < nsteps; ++k) {
          ok = ptx::warp_ok(ptx::mbar_wait_a(full_a + 8 * stage, phase, abort_flag, P.wait_limit));
          if (!ok) break;
          ptx::tc_fence_after();
          if (ptx::elect_one()) {
            const uint32_t hi = desc_lo0 + ((stage * kStageBytes) >> 4);
#pragma unroll
            for (int kk = 0; kk < kKStep / 16; ++kk) {
              const uint32_t h = hi + kk * 2, acc = (k > 0 || kk > 0) ? 1u : 0u;
              ptx::mma_bf16_ss_lh(d_tmem, h, h, desc_hi, idesc, acc);
              ptx::mma_bf16_ss_lh(d_tmem + 256, h, h + low, desc_hi, idesc, acc);
              ptx::mma_bf16_ss_lh(d_tmem + 256, h + low, h, desc_hi, idesc, 1u);
            }
            ptx::mma_commit_a(empty_a + 8 * stage);
            if (pass == 1 && k + 1 == nsteps) ptx::mma_commit(acc_full);
          }
          __syncwarp();
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
      }
    }
    if (!ok && ptx::elect_one()) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
      ptx::drain_issued_mmas(mma_done, false);
    }
  } else if (warp >= kConvWarp0) {
    // --------------------------------------------------------------- converters
    // Eight lanes a row, eight columns a lane.  Lanes 4 - 7 of a row find theirs in the second half's tile, in the banks
    // of lanes 0 - 3, and read their two 16-byte words in the other order.
    const int cw = warp - kConvWarp0, c8 = lane & 7, other = (c8 >> 2) & 1;
    const long long batch_rows = (long long)P.B * P.T;
    uint32_t s_in = 0, ph_in = 0, stage = 0, phase = 0;
    int lay = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < P.total_items && ok; item += gridDim.x) {
      const Item it = decode_item(P, item, lay);
      const long long row0 = (long long)it.tile * P.pack * P.T;
      const int own = (int)min((long long)P.pack * P.T, batch_rows - row0);        // rows of this tile's examples
      for (int pass = 0; pass < 2 && ok; ++pass) {
        const SplitPlanes& D = pass == 0 ? P.A[it.layer] : P.G[it.layer];
        const bool write = D.hi && (pass == 0 ? it.write_a : it.write_g);
        const int k0 = pass == 0 ? it.a0 : it.g0, k1 = pass == 0 ? it.a1 : it.g1;
        for (int k = k0; k < k1; ++k) {
          ok = ptx::mbar_wait_a(in_full_a + 8 * s_in, ph_in, abort_flag, P.wait_limit) &&
               ptx::mbar_wait_a(empty_a + 8 * stage, phase ^ 1, abort_flag, P.wait_limit);
          ok = ptx::warp_ok(ok);
          if (!ok) break;
          const uint8_t* src = in + size_t(s_in) * kStageBytes + size_t(other) * kHalfBytes + (c8 & 3) * 32;
          uint8_t* dst = tiles + size_t(stage) * kStageBytes;
          const int col = k * kKStep + 8 * c8;
          if (16 * cw < P.rows) {
            float4 v[4][2];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int r = 16 * cw + 4 * j + (lane >> 3);
              v[j][0] = *reinterpret_cast<const float4*>(src + r * 128 + 16 * other);
              v[j][1] = *reinterpret_cast<const float4*>(src + r * 128 + 16 * (other ^ 1));
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int r = 16 * cw + 4 * j + (lane >> 3);
              const float4 x = other ? v[j][1] : v[j][0], y = other ? v[j][0] : v[j][1];
              const float f[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
              uint4 h, l;
              __nv_bfloat162* h2 = reinterpret_cast<__nv_bfloat162*>(&h);
              __nv_bfloat162* l2 = reinterpret_cast<__nv_bfloat162*>(&l);
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                h2[e] = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
                const float2 b = __bfloat1622float2(h2[e]);
                l2[e] = __floats2bfloat162_rn(f[2 * e] - b.x, f[2 * e + 1] - b.y);
              }
              uint8_t* at = dst + r * 128 + ((c8 ^ (r & 7)) << 4);
              *reinterpret_cast<uint4*>(at) = h;
              *reinterpret_cast<uint4*>(at + kHalfBytes) = l;
              if (write && r < own && col < D.cols) {
                const size_t o = size_t(row0 + r) * D.cols + col;
                *reinterpret_cast<uint4*>(D.hi + o) = h;
                *reinterpret_cast<uint4*>(D.lo + o) = l;
              }
            }
            ptx::fence_proxy_async_smem();           // the MMAs read these tiles
          }
          __syncwarp();
          if (lane == 0) { ptx::mbar_arrive(&full[stage]); ptx::mbar_arrive(&in_empty[s_in]); }
          if (++s_in == kStagesIn) { s_in = 0; ph_in ^= 1; }
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
      }
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      if (P.dev_status) atomicOr(P.dev_status, DP_DEV_TIMEOUT);
    }
  } else {
    // ----------------------------------------------------------------- epilogue
    const int q = warp & 3, ew = warp - kEpiWarp0;
    const int row = q * 32 + lane, own = row / P.T * P.T;       // this row's example begins there, and its columns
    const int c_lo = (q * 32 / P.T * P.T) & ~15, c_hi = min(P.rows, (q * 32 + 31) / P.T * P.T + P.T);
    const uint32_t t0 = tmem_base + (uint32_t(q * 32) << 16);
    uint32_t n_item = 0;
    int lay = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < P.total_items && ok; item += gridDim.x, ++n_item) {
      const Item it = decode_item(P, item, lay);
      if (!ptx::mbar_wait_relaxed(acc_full, n_item & 1, abort_flag, P.wait_limit)) { ok = false; break; }
      ptx::tc_fence_after();
      float acc = 0.f;
#pragma unroll 1
      for (int c = c_lo; c < c_hi; c += 16) {
        uint32_t a[16], g[16], sa[16], sg[16];
        ptx::tmem_ld_32x32b_x16(t0 + c, a);
        ptx::tmem_ld_32x32b_x16(t0 + kTile + c, g);
        ptx::tmem_ld_32x32b_x16(t0 + 256 + c, sa);
        ptx::tmem_ld_32x32b_x16(t0 + 256 + kTile + c, sg);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (unsigned(c + j - own) < unsigned(P.T))
            acc = fmaf(__uint_as_float(a[j]) + __uint_as_float(sa[j]), __uint_as_float(g[j]) + __uint_as_float(sg[j]), acc);
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(acc_empty);
      // the rows' sums meet as in ghost_norm_tc.cu: four slots, a bounded wait
      const uint32_t slot = n_item & 3, red_phase = (n_item >> 2) & 1;
      row_sum[slot * kTile + row] = acc;
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&red_bar[slot]);
      if (ew == 0) {
        if (!ptx::mbar_wait_relaxed(&red_bar[slot], red_phase, abort_flag, P.wait_limit)) { ok = false; break; }
        if (P.pack == 1) {                            // one example: all lanes
          float s = 0.f;
          for (int k = lane; k < P.T; k += 32) s += row_sum[slot * kTile + k];
          s = warp_sum(s);
          const long long at = (long long)it.tile * P.n_per + it.col;
          if (lane == 0 && dp_in_range(at, (long long)P.B * P.n_per, P.dev_status)) P.partials[at] = s;
        } else if (lane < P.pack) {                   // at most four, of 32 tokens or more: a lane each
          const int example = it.tile * P.pack + lane;
          const long long at = (long long)example * P.n_per + it.col;
          if (example < P.B && dp_in_range(at, (long long)P.B * P.n_per, P.dev_status)) {
            float s = 0.f;
#pragma unroll 8
            for (int k = 0; k < P.T; ++k) s += row_sum[slot * kTile + lane * P.T + k];
            P.partials[at] = s;
          }
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

}  // namespace

// Whether TMA can read the fp32 operands as they are, and a tile holds whole examples.
bool ghost_norm_splits(const dp_linear_desc& L, int B, int T) {
  return T >= 32 && T <= kTile && (long long)B * T <= 0x7fffffffLL - kTile && aligned16(L.A) && aligned16(L.G) &&
         L.lda % 4 == 0 && L.ldg % 4 == 0;
}

// Whether one pass over the layers in `index` takes less time than the split and the Gram kernel after it.  A K step takes 0.6 us here
// whatever its rows, and more on the busiest SM than on average; there 12 bytes per value go through memory, 0.014 us per row and
// step of the average SM, here 4, or with stores 7.  The lines, in steps of the busiest SM over the average: rows / 42, with stores rows / 55.
// Norms alone, split first -> in one pass: 24 GPT-2-small layers at T = 128, B = 1, 2, 8 (2.05, 1.03, 1.03 against 3.0) 29, 44, 165 -> 27, 28,
// 104 us, at T = 64, B = 1, 2, 8 (the same against 1.5) 21.5, 26, 92 -> 22, 22, 69, at T = 32 (against 0.8) 19, 20, 63 -> 21, 21, 61; one
// of them, T = 128, B = 1 and 8 (48 and 6) 21 and 23 -> 25 and 26.  Steps, with stores: 24 layers at T = 64, B = 2, 8 (1.03 against 1.16) 97, 226
// -> 91, 214, 4 of d = 576 at T = 64, B = 16 (1.54) 82 -> 92, at T = 128, B = 8 (1.54 against 2.3) 89 -> 85, one layer at T = 128, B = 1 38 -> 45.
// Norms alone of a dozen steps at most are launches only: 4 layers of d = 256, B = 1, T = 32 and 64 12.7 and 13.1 -> 12.2 and 12.6, beyond 80 rows
// longer (15 -> 16).
bool ghost_norm_split_pays(const std::vector<int>& index, const GhostPlan& plan, int B, int T, bool keep, int sms) {
  const int rows = (plan.pack * T + 15) / 16 * 16, groups = ceil_div(B, plan.pack);
  long long total = 0, busiest = 0, items = 0, next = 0;       // the first SM has the longest item of every wave
  for (int l : index) {
    const GhostLayerPlan& L = plan.layer[size_t(l)];
    const int narrow = std::min(L.a_steps, L.g_steps), wide = std::max(L.a_steps, L.g_steps);
    items += (long long)groups * L.nsplit;
    total += (long long)groups * (L.nsplit * narrow + wide);
    for (; next < items; next += sms) busiest += narrow + L.chunk_steps;
  }
  if (!keep && busiest <= 12 && rows <= 80) return true;
  return busiest * sms * (keep ? 55 : 42) <= total * rows;
}

// index: layers of the plan, with the fp32 operands in `layers`; jobs: their split, A and G of layer k at 2k and 2k + 1;
// keep: the wider operand's is stored
dp_status launch_ghost_norm_split(const dp_linear_desc* layers, const SplitJob* jobs, const std::vector<int>& index,
                                  const GhostPlan& plan, int B, int T, bool keep, float* partials, int* dev_status, cudaStream_t st) {
  if (first_use_on_this_device(reinterpret_cast<const void*>(&ghost_norm_split_kernel)))
    DP_CUDA_OK(allow_shared(ghost_norm_split_kernel, kSmemBytes));
  const int rows = (plan.pack * T + 15) / 16 * 16, groups = ceil_div(B, plan.pack);
  for (size_t g0 = 0; g0 < index.size(); g0 += kMaxLayers) {
    const size_t g1 = std::min(index.size(), g0 + kMaxLayers);
    SplitGramParams P;
    memset(&P, 0, sizeof(P));
    int items = 0;
    for (size_t g = g0; g < g1; ++g) {
      const int li = index[g];
      const size_t k = g - g0;
      const dp_linear_desc& L = layers[li];
      dp_status s = make_tmap_f32_3d(&P.tmA[k], L.A, L.lda, L.d, B * T, 1, 32, rows);
      if (s != DP_OK) return s;
      s = make_tmap_f32_3d(&P.tmG[k], L.G, L.ldg, L.p, B * T, 1, 32, rows);
      if (s != DP_OK) return s;
      auto planes = [&](const SplitJob& J) {
        __nv_bfloat16* hi = static_cast<__nv_bfloat16*>(J.dst);
        return SplitPlanes{hi, hi + size_t(B) * T * split_padded(J.c), split_padded(J.c)};
      };
      if (keep) (a_is_scaled(L) ? P.G[k] : P.A[k]) = planes(jobs[a_is_scaled(L) ? 2 * li + 1 : 2 * li]);
      P.layer[k] = plan.layer[li];
      P.layer[k].item_begin = items;
      items += groups * plan.layer[li].nsplit;
    }
    P.n_layers = int(g1 - g0);
    P.B = B; P.T = T; P.pack = plan.pack; P.rows = rows;
    P.total_items = items; P.n_per = plan.n_per;
    P.partials = partials; P.dev_status = dev_status; P.wait_limit = g_wait_limit;
    ghost_norm_split_kernel<<<std::min(items, sm_count()), kThreads, kSmemBytes, st>>>(P);
    DP_LAUNCH_OK();
  }
  return DP_OK;
}

}  // namespace dpg
