// extern "C" entry points: argument checks, work planning, workspace carving, launches.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <set>
#include <utility>

#include "cross_term.cuh"
#include "dp_common.cuh"
#include "fma_kernels.cuh"
#include "gemm_gta.cuh"
#include "ghost_plan.cuh"
#include "small_step.cuh"
#include "split_kernels.cuh"
#include "tma_host.cuh"
#include "vector_kernels.cuh"

namespace dpg {

int g_last_cuda_error = 0;
int g_force_fma = 0;
long long g_kernel_launches = 0;
long long g_wait_limit = 1500000000LL;
const uint32_t* g_step_dev = nullptr;
int g_ghost_single = 0;
int g_reserved_sms = 0;

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_device_mutex;
}

static int device_sm_count() {
  static int n[kMaxDevices] = {};
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 148;
  if (n[dev] == 0) {
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
      n[dev] = v;
    else
      return 148;          // B200; not cached so a later call can still query the device
  }
  return n[dev];
}

// SMs the persistent kernels size their grids for: all of the device's, less the ones the caller
// set aside (dp_set_reserved_sms), kept even (CTA pairs) and never below two.
int sm_count() {
  const int n = device_sm_count() - g_reserved_sms;
  return std::max(2, n & ~1);
}

bool first_use_on_this_device(const void* key) {
  static std::set<std::pair<const void*, int>> seen;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return true;     // set up again rather than never
  std::lock_guard<std::mutex> lock(g_device_mutex);
  return seen.insert(std::make_pair(key, dev)).second;
}

// ---- planning of dp_ghost_norms ------------------------------------------------------------
GhostPlan plan_ghost_norms(const dp_linear_desc* layers, int n_layers, int B, int T, int sms, bool split) {
  GhostPlan plan;
  plan.pair = !split && T > 128 && !g_ghost_single;
  const int nt = ceil_div(T, plan.pair ? 256 : 128);
  const int slots = plan.pair ? 2 : 1;           // partial sums per work item
  const int units = plan.pair ? sms / 2 : sms;   // persistent CTAs or CTA pairs
  plan.ntp = nt * (nt + 1) / 2;
  plan.layer.resize(n_layers);
  plan.direct.resize(n_layers);
  plan.mode_used.resize(n_layers);
  for (int l = 0; l < n_layers; ++l) {
    int mode = layers[l].mode;
    if (mode == DP_NORM_AUTO)
      mode = ((long long)T * T > (long long)layers[l].d * layers[l].p) ? DP_NORM_DIRECT : DP_NORM_GHOST;
    plan.mode_used[l] = mode;
    (mode == DP_NORM_GHOST ? plan.ghost_layers : plan.direct_layers).push_back(l);
  }
  // as many examples per tile as fit, while two items per SM remain; the rows of the batch are counted in 32 bits
  if (T <= 64 && (long long)B * T <= 0x7fffffffLL - 128) {
    const long long most = (long long)B * (long long)plan.ghost_layers.size() / (2LL * units);
    plan.pack = (int)std::max(1LL, std::min(most, (long long)std::min(B, 128 / T)));
  }
  const int groups = ceil_div(B, plan.pack);
  // Column chunking of wide operands.  The per-item step budget shrinks until there are at
  // least two items per SM (or the budget bottoms out).  Split operands have sums no longer than those of layers
  // planned one by one on widened operands (24 steps at d = 768, with 2.4 times the error per step): see
  // ghost_norm_tc_kernel.
  int budget = split ? 48 : 64;
  for (;;) {
    long long items = 0;
    for (int l : plan.ghost_layers) {
      GhostLayerPlan& L = plan.layer[l];
      L.a_steps = ceil_div(layers[l].d, 64);
      L.g_steps = ceil_div(layers[l].p, 64);
      const int small = std::min(L.a_steps, L.g_steps), large = std::max(L.a_steps, L.g_steps);
      L.split_on_g = L.g_steps >= L.a_steps;
      int chunk = std::max(std::max(budget - small, small), 8);
      if (small + large <= budget + budget / 2) chunk = large;
      L.nsplit = ceil_div(large, chunk);
      L.chunk_steps = ceil_div(large, L.nsplit);
      L.nsplit = ceil_div(large, L.chunk_steps);
      items += (long long)groups * plan.ntp * L.nsplit;
    }
    if (items >= 2LL * units || budget <= 8 || plan.ghost_layers.empty()) break;
    budget /= 2;
  }
  // longest items first: with a static round-robin split the last, partly filled wave then
  // holds the cheapest items
  std::stable_sort(plan.ghost_layers.begin(), plan.ghost_layers.end(), [&](int a, int b) {
    auto cost = [&](int l) {
      const GhostLayerPlan& L = plan.layer[l];
      return std::min(L.a_steps, L.g_steps) + L.chunk_steps;
    };
    return cost(a) > cost(b);
  });
  int col = 0;
  for (int l = 0; l < n_layers; ++l) {
    if (plan.mode_used[l] == DP_NORM_GHOST) {
      plan.layer[l].col_begin = col;
      plan.layer[l].item_begin = 0;
      col += plan.ntp * plan.layer[l].nsplit * slots;
    } else {
      plan.direct[l].tiles_m = ceil_div(layers[l].p, 128);
      plan.direct[l].tiles_n = ceil_div(layers[l].d, 256);
      plan.direct[l].col_begin = col;
      col += plan.direct[l].tiles_m * plan.direct[l].tiles_n;
    }
  }
  plan.n_per = col;
  return plan;
}

static bool finite_pos(float x) { return std::isfinite(x) && x > 0.f; }

static dp_status check_linear(const dp_linear_desc& L, dp_dtype dt, bool tc) {
  if (!L.A || !L.G || L.d <= 0 || L.p <= 0 || L.lda < L.d || L.ldg < L.p) return DP_ERR_INVALID_ARG;
  if (L.mode != DP_NORM_AUTO && L.mode != DP_NORM_GHOST && L.mode != DP_NORM_DIRECT)
    return DP_ERR_INVALID_ARG;
  if (tc && (!aligned16(L.A) || !aligned16(L.G) || (L.lda % 8) || (L.ldg % 8))) return DP_ERR_ALIGNMENT;
  (void)dt;
  return DP_OK;
}

// ---- fp32 inputs on the tensor cores (operands split into two bf16 terms, see split_kernels.cu)
// Taken for layers that are large enough for a tensor-core tile to pay; tiny layers (and the test
// hook dp_debug_force_fma) stay on the plain fp32 kernels.
static bool f32_on_tensor_cores(const dp_linear_desc& L, int T) {
  return !g_force_fma && T >= 32 && L.d >= 64 && L.p >= 64;
}

static int resolve_mode(const dp_linear_desc& L, int T) {
  if (L.mode != DP_NORM_AUTO) return L.mode;
  return ((long long)T * T > (long long)L.d * L.p) ? DP_NORM_DIRECT : DP_NORM_GHOST;
}

// Layers whose split operands share the workspace and run through the kernels together.  How many
// there are follows from the workspace at hand: it holds the largest layer with room to spare (the
// *_ws_bytes functions see to that), and so several ordinary layers beside a head-sized one.
struct SplitGroup {
  std::vector<int> index;               // into the caller's layers
  std::vector<dp_linear_desc> source;   // the layers
  std::vector<dp_linear_desc> desc;     // the same on their split operands
  std::vector<SplitJob> jobs;
  size_t bytes = 0;                     // workspace taken by the split operands
  size_t bound = 0;                     // norms: by all of it, at most

  // scale: the narrower operand is to be multiplied by the clip factors
  void add(const dp_linear_desc& L, int l, int B, int T, bool scale, char* base) {
    dp_linear_desc D = L;
    const long long rows = (long long)B * T;
    D.mode = resolve_mode(L, T);
    D.A = base + bytes; D.lda = split_padded(L.d);
    jobs.push_back({static_cast<const float*>(L.A), L.lda, L.d, scale && a_is_scaled(L), base + bytes});
    bytes += split_bytes(rows, L.d);
    D.G = base + bytes; D.ldg = split_padded(L.p);
    jobs.push_back({static_cast<const float*>(L.G), L.ldg, L.p, scale && !a_is_scaled(L), base + bytes});
    bytes += split_bytes(rows, L.p);
    index.push_back(l);
    source.push_back(L);
    desc.push_back(D);
  }
};

static size_t split_layer_bytes(const dp_linear_desc& L, int B, int T) {
  return split_bytes((long long)B * T, L.d) + split_bytes((long long)B * T, L.p);
}

// What a layer takes of the workspace for its norm.  Planned alone it is cut into at least as many
// chunks (partial sums) as in company, so the sums of these bound a group's needs.
static size_t f32_norm_bytes(const dp_linear_desc& L, int B, int T, int sms) {
  dp_linear_desc one = L;
  one.mode = resolve_mode(L, T);
  const GhostPlan plan = plan_ghost_norms(&one, 1, B, T, sms, true);
  return split_layer_bytes(L, B, T) + align_up(size_t(B) * plan.n_per * sizeof(float), 256);
}

// norms of a group of fp32 layers: split, Gram or gradient-tile kernels, one reduction (or, with `left`,
// the place of the partial sums).  keep: split operands that clipped sums can use are in place afterwards
static dp_status f32_norm_group(const SplitGroup& g, int B, int T, float* sq, char* ws, int* dev_status,
                                cudaStream_t st, bool overwrite, NormSource* left, bool keep) {
  GhostPlan plan = plan_ghost_norms(g.desc.data(), (int)g.desc.size(), B, T, sm_count(), true);
  float* partials = reinterpret_cast<float*>(ws + g.bytes);
  // ghost norms that split their operands on the way, and what is split beforehand
  std::vector<int> fused;
  std::vector<SplitJob> before;
  std::vector<char> is_fused(g.desc.size(), 0);
  for (int l : plan.ghost_layers)
    if (ghost_norm_splits(g.source[size_t(l)], B, T)) fused.push_back(l);
  if (!ghost_norm_split_pays(fused, plan, B, T, keep, sm_count())) fused.clear();
  for (int l : fused) is_fused[size_t(l)] = 1;
  for (size_t l = 0; l < g.desc.size(); ++l)
    if (!is_fused[l]) { before.push_back(g.jobs[2 * l]); before.push_back(g.jobs[2 * l + 1]); }
  dp_status s = launch_split(before.data(), (int)before.size(), B, T, nullptr, st);
  if (s != DP_OK) return s;
  if (!fused.empty()) {
    s = launch_ghost_norm_split(g.source.data(), g.jobs.data(), fused, plan, B, T, keep, partials, dev_status, st);
    if (s != DP_OK) return s;
  }
  plan.ghost_layers.erase(std::remove_if(plan.ghost_layers.begin(), plan.ghost_layers.end(),
                                         [&](int l) { return is_fused[size_t(l)] != 0; }), plan.ghost_layers.end());
  if (!plan.ghost_layers.empty()) {
    s = launch_ghost_norm_tc(g.desc.data(), plan, B, T, partials, dev_status, st, true);
    if (s != DP_OK) return s;
  }
  if (!plan.direct_layers.empty()) {
    s = launch_direct_norm_tc(g.desc.data(), plan, B, T, 3, partials, dev_status, st);
    if (s != DP_OK) return s;
  }
  if (left) { *left = NormSource{partials, plan.n_per, 1.f, nullptr}; return DP_OK; }
  return launch_reduce_partials(partials, plan.n_per, B, sq, 1.f, nullptr, st, overwrite);
}

}  // namespace dpg

using namespace dpg;

// Clip factors of a clip-accumulate call.  With sq given they are computed (Eq. 7) into the
// workspace and copied to `clip` if the caller wants them; with sq == NULL the caller has them
// already (dp_clip_factors / dp_clip_factors_sum) and `clip` is the input.
static dp_status resolve_clip(const float* sq, int B, float C, float* clip, float** clip_ws,
                              cudaStream_t st) {
  if (!sq) { *clip_ws = clip; return DP_OK; }
  const dp_status s = launch_clip_factors(sq, B, C, *clip_ws, nullptr, st);
  if (s != DP_OK) return s;
  if (clip) DP_CUDA_OK(cudaMemcpyAsync(clip, *clip_ws, size_t(B) * sizeof(float),
                                       cudaMemcpyDeviceToDevice, st));
  return DP_OK;
}

extern "C" {

const char* dp_status_string(dp_status s) {
  switch (s) {
    case DP_OK: return "ok";
    case DP_ERR_INVALID_ARG: return "invalid argument";
    case DP_ERR_UNSUPPORTED: return "size not supported by the built kernels";
    case DP_ERR_ALIGNMENT: return "pointer or leading dimension not aligned for TMA";
    case DP_ERR_WORKSPACE: return "workspace missing or too small";
    case DP_ERR_CUDA: return "CUDA error (see dp_last_cuda_error)";
    case DP_ERR_SCRATCH_LIMIT:
      return "problem needs more scratch than the library's built-in array holds "
             "(B * ceil(d/256) > DP_STATIC_SCRATCH_FLOATS); use dp_embed_norms with a workspace";
  }
  return "unknown status";
}

int32_t dp_last_cuda_error(void) { return g_last_cuda_error; }
const char* dp_version(void) { return "dp_ghost 0.1.0 (sm_100a)"; }
int64_t dp_kernel_launches(void) { return g_kernel_launches; }

int32_t dp_set_reserved_sms(int32_t n) {
  const int prev = g_reserved_sms;
  g_reserved_sms = std::max(0, std::min(n, device_sm_count() - 2));
  return prev;
}
int32_t dp_debug_ghost_single(int32_t on) {
  const int prev = g_ghost_single;
  g_ghost_single = on ? 1 : 0;
  return prev;
}
int64_t dp_debug_set_wait_limit(int64_t cycles) {
  const long long prev = g_wait_limit;
  g_wait_limit = cycles < 0 ? 1500000000LL : cycles;
  return prev;
}
dp_status dp_debug_noise_error_scan(float t_max, double* out3, void* stream) {
  if (!out3) return DP_ERR_INVALID_ARG;
  return launch_noise_error_scan(t_max, out3, (cudaStream_t)stream);
}
int32_t dp_debug_bounds_checked(void) { return kBoundsChecked; }
dp_status dp_debug_bounds_probe(int64_t idx, int64_t n, int32_t* dev_status, void* stream) {
  if (!dev_status) return DP_ERR_INVALID_ARG;
  return launch_bounds_probe(idx, n, dev_status, (cudaStream_t)stream);
}
int64_t dp_debug_tensor_map_encodes(void) { return tmap_encode_count(); }
int32_t dp_debug_force_fma(int32_t on) {
  const int prev = g_force_fma;
  g_force_fma = on ? 1 : 0;
  return prev;
}

// ---------------------------------------------------------------------------- ghost norms
static bool on_tensor_cores(const dp_linear_desc& L, dp_dtype dt, int T) {
  return dt == DP_F32 ? f32_on_tensor_cores(L, T) : !g_force_fma;
}

// split operands of the largest layer three times over (what runs together follows from the room), and ...
static size_t f32_norms_bytes(const dp_linear_desc* layers, int n_layers, dp_dtype dt, int B, int T) {
  size_t need = 0;
  for (int l = 0; l < n_layers; ++l)
    if (dt == DP_F32 && f32_on_tensor_cores(layers[l], T))
      need = std::max(need, f32_norm_bytes(layers[l], B, T, sm_count()) + 2 * split_layer_bytes(layers[l], B, T));
  return need;
}

// ... where there is room for them, the partial sums of the ghost norms on the fp32 kernels
static int fma_norms_partials(const dp_linear_desc* layers, int n_layers, dp_dtype dt, int T) {
  int n = 0;
  for (int l = 0; l < n_layers; ++l)
    if (!on_tensor_cores(layers[l], dt, T) && resolve_mode(layers[l], T) == DP_NORM_GHOST)
      n += gram_fma_partials(layers[l], T);
  return n;
}
static size_t fma_norms_bytes(const dp_linear_desc* layers, int n_layers, dp_dtype dt, int B, int T) {
  return align_up(size_t(B) * fma_norms_partials(layers, n_layers, dt, T) * sizeof(float), 256);
}

size_t dp_ghost_norms_ws_bytes(const dp_linear_desc* layers, int32_t n_layers, dp_dtype dt,
                               int32_t B, int32_t T) {
  if (!layers || n_layers <= 0 || B <= 0 || T <= 0) return 0;
  if (dt == DP_F32 || g_force_fma) return f32_norms_bytes(layers, n_layers, dt, B, T);
  const GhostPlan plan = plan_ghost_norms(layers, n_layers, B, T, sm_count());
  return align_up(size_t(B) * plan.n_per * sizeof(float), 256);
}

// all that can be wrong with a call, before anything is enqueued; and its plan
static dp_status ghost_norms_check(const dp_linear_desc* layers, int32_t n_layers, dp_dtype dt, int32_t B, int32_t T,
                                   const float* sq, const void* ws, size_t ws_bytes, GhostPlan* plan) {
  if (!layers || n_layers <= 0 || B <= 0 || T <= 0 || !sq) return DP_ERR_INVALID_ARG;
  if (dt != DP_F32 && dt != DP_BF16) return DP_ERR_INVALID_ARG;
  const bool tc = (dt == DP_BF16) && !g_force_fma;
  bool split = false;
  for (int l = 0; l < n_layers; ++l) {
    const dp_status s = check_linear(layers[l], dt, tc);
    if (s != DP_OK) return s;
    split = split || (dt == DP_F32 && f32_on_tensor_cores(layers[l], T));
  }
  *plan = plan_ghost_norms(layers, n_layers, B, T, sm_count());
  const size_t need = tc ? align_up(size_t(B) * plan->n_per * sizeof(float), 256) : f32_norms_bytes(layers, n_layers, dt, B, T);
  if (ws_bytes < need || ((tc || split) && !ws) || (split && !aligned16(ws))) return DP_ERR_WORKSPACE;
  return DP_OK;
}

// overwrite: sq is written instead of added to (its first contribution of a step); the call has been checked
static dp_status ghost_norms_impl(const GhostPlan& plan, dp_linear_desc* layers, int32_t n_layers, dp_dtype dt, int32_t B,
                                  int32_t T, float* sq, void* ws, size_t ws_bytes, int32_t* dev_status,
                                  void* stream, bool overwrite, NormSource* left = nullptr,
                                  SplitGroup* kept = nullptr) {
  // left: the last reduction is not done; *left says where its partial sums are (or sq itself)
  // kept: the split operands of fp32 layers, where they stay in ws all together; empty if they do not
  cudaStream_t st = (cudaStream_t)stream;
  const bool tc = (dt == DP_BF16) && !g_force_fma;
  if (!tc) {
    const size_t split_need = f32_norms_bytes(layers, n_layers, dt, B, T);
    SplitGroup group;
    char* base = static_cast<char*>(ws);
    if (left) *left = NormSource{sq, 1, 1.f, nullptr};
    // ghost norms on the fp32 kernels: all layers in one launch, their partial sums at the workspace's end
    // (at its start if nothing else needs it); without room for them a launch per layer
    std::vector<int> fma;
    for (int l = 0; l < n_layers; ++l)
      if (!on_tensor_cores(layers[l], dt, T) && plan.mode_used[l] == DP_NORM_GHOST) fma.push_back(l);
    const size_t fma_need = fma_norms_bytes(layers, n_layers, dt, B, T);
    const bool together = !fma.empty() && ws && aligned16(ws) && split_need + fma_need <= ws_bytes &&
                          !(fma.size() == 1 && gram_alone_fma(layers[fma[0]], T));
    if (together) {
      char* at = base;
      if (split_need) {
        ws_bytes = (ws_bytes - fma_need) & ~size_t(255);
        at += ws_bytes;
      }
      float* partials = reinterpret_cast<float*>(at);
      const int n_per = fma_norms_partials(layers, n_layers, dt, T);
      dp_status s = launch_gram_norms_fma(layers, fma.data(), (int)fma.size(), dt, B, T, partials, n_per, st);
      if (s != DP_OK) return s;
      for (int l : fma) layers[l].mode_used = plan.mode_used[l];
      if (left && (int)fma.size() == n_layers) {
        *left = NormSource{partials, n_per, 1.f, nullptr};
        return DP_OK;
      }
      s = launch_reduce_partials(partials, n_per, B, sq, 1.f, nullptr, st, overwrite);
      if (s != DP_OK) return s;
      overwrite = false;
    }
    bool one_group = true;               // so far
    auto flush = [&](bool last) {
      if (group.index.empty()) return DP_OK;
      const bool all = (int)group.index.size() == n_layers, keep = kept && last && one_group;
      const dp_status s = f32_norm_group(group, B, T, sq, base, dev_status, st, overwrite, all ? left : nullptr, keep);
      overwrite = one_group = false;
      if (keep) *kept = std::move(group);
      group = SplitGroup();
      return s;
    };
    for (int l = 0; l < n_layers; ++l) {
      dp_status s = DP_OK;
      if (together && !on_tensor_cores(layers[l], dt, T) && plan.mode_used[l] == DP_NORM_GHOST) continue;
      if (dt == DP_F32 && f32_on_tensor_cores(layers[l], T)) {
        const size_t more = f32_norm_bytes(layers[l], B, T, sm_count());
        if (group.bound + more > ws_bytes) s = flush(false);
        if (s != DP_OK) return s;
        group.bound += more;
        group.add(layers[l], l, B, T, false, base);
      } else {
        s = launch_norms_fma(layers[l], dt, plan.mode_used[l], B, T, sq, st, overwrite);
        overwrite = false;
      }
      if (s != DP_OK) return s;
      layers[l].mode_used = plan.mode_used[l];
    }
    return flush(true);
  }
  float* partials = static_cast<float*>(ws);
  dp_status s = DP_OK;
  if (!plan.ghost_layers.empty()) {
    s = plan.pair ? launch_ghost_norm_pair(layers, plan, B, T, partials, dev_status, st)
                  : launch_ghost_norm_tc(layers, plan, B, T, partials, dev_status, st);
    if (s != DP_OK) return s;
  }
  if (!plan.direct_layers.empty()) {
    s = launch_direct_norm_tc(layers, plan, B, T, 1, partials, dev_status, st);
    if (s != DP_OK) return s;
  }
  if (left) *left = NormSource{partials, plan.n_per, 1.f, nullptr};
  else s = launch_reduce_partials(partials, plan.n_per, B, sq, 1.f, nullptr, st, overwrite);
  if (s != DP_OK) return s;
  for (int l = 0; l < n_layers; ++l) layers[l].mode_used = plan.mode_used[l];
  return DP_OK;
}

dp_status dp_ghost_norms(dp_linear_desc* layers, int32_t n_layers, dp_dtype dt, int32_t B,
                         int32_t T, float* sq, void* ws, size_t ws_bytes, int32_t* dev_status,
                         void* stream) {
  GhostPlan plan;
  const dp_status s = ghost_norms_check(layers, n_layers, dt, B, T, sq, ws, ws_bytes, &plan);
  return s != DP_OK ? s : ghost_norms_impl(plan, layers, n_layers, dt, B, T, sq, ws, ws_bytes, dev_status, stream, false);
}

// ------------------------------------------------------------------------ embedding norms
size_t dp_embed_norms_ws_bytes(int32_t B, int32_t T, int32_t d) {
  if (B <= 0 || T <= 0 || d <= 0) return 0;
  return align_up(size_t(B) * ceil_div(d, kEmbedColsPerBlock) * embed_norm_parts(B, T, d) * sizeof(float), 256);
}

static dp_status embed_norms_impl(const int32_t* ids, const void* G, int64_t ldg, dp_dtype dt, int32_t B,
                                  int32_t T, int32_t d, int32_t V, float* sq, int32_t* first_occ, void* ws,
                                  size_t ws_bytes, int32_t* dev_status, void* stream, bool overwrite,
                                  NormSource* left = nullptr) {
  if (!ids || !G || !sq || B <= 0 || T <= 0 || d <= 0 || V <= 0 || ldg < d) return DP_ERR_INVALID_ARG;
  if (dt != DP_F32 && dt != DP_BF16) return DP_ERR_INVALID_ARG;
  if (T > kEmbedMaxT) return DP_ERR_UNSUPPORTED;
  if (!ws || ws_bytes < dp_embed_norms_ws_bytes(B, T, d)) return DP_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  float* partials = static_cast<float*>(ws);
  const int parts = embed_norm_parts(B, T, d);
  dp_status s = launch_embed_norms(ids, G, ldg, dt, B, T, d, V, parts, partials, first_occ, dev_status, st);
  if (s != DP_OK) return s;
  const int n_per = ceil_div(d, kEmbedColsPerBlock) * parts;
  if (left) { *left = NormSource{partials, n_per, 1.f, nullptr}; return DP_OK; }
  return launch_reduce_partials(partials, n_per, B, sq, 1.f, nullptr, st, overwrite);
}

dp_status dp_embed_norms(const int32_t* ids, const void* G, int64_t ldg, dp_dtype dt, int32_t B,
                         int32_t T, int32_t d, int32_t V, float* sq, int32_t* first_occ, void* ws,
                         size_t ws_bytes, int32_t* dev_status, void* stream) {
  return embed_norms_impl(ids, G, ldg, dt, B, T, d, V, sq, first_occ, ws, ws_bytes, dev_status, stream, false);
}

// ------------------------------------------------------------------------ tied cross term
size_t dp_tied_cross_term_ws_bytes(int32_t B, int32_t T, int32_t d, int32_t V) {
  (void)d; (void)V;
  if (B <= 0 || T <= 0) return 0;
  // enough for either kernel: one partial per 16-token slab (fp32 path) or per tile
  const int per = std::max(ceil_div(T, 16), cross_term_tc_partials_per_example(T));
  return align_up(size_t(B) * per * sizeof(float), 256);
}

static dp_status cross_term_check(const int32_t* ids, const void* G_emb, int64_t ldge, const void* A_lm, int64_t ldal,
                                  const void* G_lm, int64_t ldgl, dp_dtype dt, int32_t B, int32_t T, int32_t d, int32_t V,
                                  const void* ws, size_t ws_bytes) {
  if (!ids || !G_emb || !A_lm || !G_lm || B <= 0 || T <= 0 || d <= 0 || V <= 0)
    return DP_ERR_INVALID_ARG;
  if (ldge < d || ldal < d || ldgl < V) return DP_ERR_INVALID_ARG;
  if (dt != DP_F32 && dt != DP_BF16) return DP_ERR_INVALID_ARG;
  const bool tc = (dt == DP_BF16) && !g_force_fma;
  if (tc && (!aligned16(G_emb) || !aligned16(A_lm) || (ldge % 8) || (ldal % 8))) return DP_ERR_ALIGNMENT;
  return !ws || ws_bytes < dp_tied_cross_term_ws_bytes(B, T, d, V) ? DP_ERR_WORKSPACE : DP_OK;
}

static dp_status cross_term_impl(const int32_t* ids, const void* G_emb, int64_t ldge, const void* A_lm,
                                 int64_t ldal, const void* G_lm, int64_t ldgl, dp_dtype dt, int32_t B,
                                 int32_t T, int32_t d, int32_t V, float* sq, float* cross, void* ws,
                                 size_t ws_bytes, int32_t* dev_status, void* stream, NormSource* left) {
  if (!sq && !cross) return DP_ERR_INVALID_ARG;
  dp_status s = cross_term_check(ids, G_emb, ldge, A_lm, ldal, G_lm, ldgl, dt, B, T, d, V, ws, ws_bytes);
  if (s != DP_OK) return s;
  const bool tc = (dt == DP_BF16) && !g_force_fma;
  cudaStream_t st = (cudaStream_t)stream;
  float* partials = static_cast<float*>(ws);
  int per;
  if (tc) {
    s = launch_cross_term_tc(ids, G_emb, ldge, A_lm, ldal, G_lm, ldgl, B, T, d, V, partials,
                             dev_status, st);
    per = cross_term_tc_partials_per_example(T);
  } else {
    s = launch_cross_term_fma(ids, G_emb, ldge, A_lm, ldal, G_lm, ldgl, dt, B, T, d, V, partials,
                              dev_status, st);
    per = ceil_div(T, 16);
  }
  if (s != DP_OK) return s;
  if (left) { *left = NormSource{partials, per, 2.f, cross}; return DP_OK; }
  return launch_reduce_partials(partials, per, B, sq, 2.f, cross, st);
}

dp_status dp_tied_cross_term(const int32_t* ids, const void* G_emb, int64_t ldge, const void* A_lm,
                             int64_t ldal, const void* G_lm, int64_t ldgl, dp_dtype dt, int32_t B,
                             int32_t T, int32_t d, int32_t V, float* sq, float* cross, void* ws,
                             size_t ws_bytes, int32_t* dev_status, void* stream) {
  return cross_term_impl(ids, G_emb, ldge, A_lm, ldal, G_lm, ldgl, dt, B, T, d, V, sq, cross, ws, ws_bytes,
                         dev_status, stream, nullptr);
}

// ------------------------------------------------------- bias / LayerNorm parameters
static dp_status check_vectors(const dp_vector_desc* prm, int32_t n, int32_t B, int32_t T) {
  if (!prm || n <= 0 || B <= 0 || T <= 0) return DP_ERR_INVALID_ARG;
  for (int k = 0; k < n; ++k) {
    if (!prm[k].G || prm[k].p <= 0 || prm[k].ldg < prm[k].p) return DP_ERR_INVALID_ARG;
    if (prm[k].X && prm[k].ldx < prm[k].p) return DP_ERR_INVALID_ARG;
  }
  return DP_OK;
}

size_t dp_vector_norms_ws_bytes(const dp_vector_desc* prm, int32_t n, int32_t B, int32_t T) {
  if (check_vectors(prm, n, B, T) != DP_OK) return 0;
  return align_up(size_t(B) * vector_total_slabs(prm, n) * sizeof(float), 256);
}

static dp_status vector_norms_impl(const dp_vector_desc* prm, int32_t n, dp_dtype dt, int32_t B, int32_t T,
                                   float* sq, void* ws, size_t ws_bytes, void* stream, NormSource* left,
                                   float* keep = nullptr) {
  const dp_status c = check_vectors(prm, n, B, T);
  if (c != DP_OK) return c;
  if (!sq || (dt != DP_F32 && dt != DP_BF16)) return DP_ERR_INVALID_ARG;
  if (!ws || ws_bytes < dp_vector_norms_ws_bytes(prm, n, B, T)) return DP_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  float* partials = static_cast<float*>(ws);
  const int n_per = vector_total_slabs(prm, n);
  dp_status s = launch_vector_norms(prm, n, dt, B, T, partials, n_per, st, keep);
  if (s != DP_OK) return s;
  if (left) { *left = NormSource{partials, n_per, 1.f, nullptr}; return DP_OK; }
  return launch_reduce_partials(partials, n_per, B, sq, 1.f, nullptr, st);
}

dp_status dp_vector_norms(const dp_vector_desc* prm, int32_t n, dp_dtype dt, int32_t B, int32_t T,
                          float* sq, void* ws, size_t ws_bytes, void* stream) {
  return vector_norms_impl(prm, n, dt, B, T, sq, ws, ws_bytes, stream, nullptr);
}

static size_t vector_partial_bytes(const dp_vector_desc* prm, int32_t n, int32_t B, int32_t T) {
  size_t worst = 0;
  for (int n0 = 0; n0 < n; n0 += kVecMaxParams) {
    const int n1 = std::min(n, n0 + kVecMaxParams);
    size_t cols = 0;
    for (int k = n0; k < n1; ++k) cols += size_t(prm[k].p);
    worst = std::max(worst, cols * vector_row_splits(prm + n0, n1 - n0, B, T, sm_count()));
  }
  return align_up(worst * sizeof(float), 256);
}

size_t dp_clip_accumulate_vectors_ws_bytes(const dp_vector_desc* prm, int32_t n, int32_t B,
                                           int32_t T) {
  if (check_vectors(prm, n, B, T) != DP_OK) return 0;
  return align_up(size_t(B) * sizeof(float), 256) + vector_partial_bytes(prm, n, B, T);
}

dp_status dp_clip_accumulate_vectors(const dp_vector_desc* prm, int32_t n, dp_dtype dt, int32_t B,
                                     int32_t T, const float* sq, float C, float* clip,
                                     float* const* outs, float beta, int32_t with_noise, float sigma,
                                     float scale, uint64_t seed, const uint32_t* tensor_ids,
                                     uint32_t step, void* ws, size_t ws_bytes, void* stream) {
  const dp_status c = check_vectors(prm, n, B, T);
  if (c != DP_OK) return c;
  if ((!sq && !clip) || !outs || (dt != DP_F32 && dt != DP_BF16)) return DP_ERR_INVALID_ARG;
  if (!(beta == 0.f || beta == 1.f) || !finite_pos(C)) return DP_ERR_INVALID_ARG;
  for (int k = 0; k < n; ++k) if (!outs[k]) return DP_ERR_INVALID_ARG;
  if (with_noise && (!tensor_ids || !std::isfinite(sigma) || sigma < 0.f || !std::isfinite(scale)))
    return DP_ERR_INVALID_ARG;
  if (!ws || ws_bytes < dp_clip_accumulate_vectors_ws_bytes(prm, n, B, T)) return DP_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  float* clip_ws = static_cast<float*>(ws);
  dp_status s = resolve_clip(sq, B, C, clip, &clip_ws, st);
  if (s != DP_OK) return s;
  float* partial = reinterpret_cast<float*>(static_cast<char*>(ws) +
                                            align_up(size_t(B) * sizeof(float), 256));
  return launch_vector_sums(prm, n, dt, B, T, clip_ws, outs, beta, with_noise ? 1 : 0, sigma * C,
                            with_noise ? scale : 1.f, seed, tensor_ids, step, partial, st);
}

// --------------------------------------------------------------------------- clip factors
dp_status dp_clip_factors_sum(float* sq, const float* sq_extra, int32_t B, float C, float* clip,
                              float* norms, void* stream) {
  if (!sq || !sq_extra || B <= 0 || !finite_pos(C)) return DP_ERR_INVALID_ARG;
  return launch_clip_factors(sq, B, C, clip, norms, (cudaStream_t)stream, sq_extra, sq);
}

dp_status dp_clip_factors(const float* sq, int32_t B, float C, float* clip, float* norms,
                          void* stream) {
  if (!sq || B <= 0 || (!clip && !norms) || !finite_pos(C)) return DP_ERR_INVALID_ARG;
  return launch_clip_factors(sq, B, C, clip, norms, (cudaStream_t)stream);
}

// ------------------------------------------------------------------------ clip accumulate
size_t dp_clip_accumulate_grouped_ws_bytes(const dp_linear_desc* layers, int32_t n_layers,
                                           dp_dtype dt, int32_t B, int32_t T) {
  if (!layers || n_layers <= 0 || B <= 0 || T <= 0) return 0;
  size_t n = align_up(size_t(B) * sizeof(float), 256);          // clip factors
  if (dt == DP_BF16 && !g_force_fma) n += gta_partial_bytes(layers, n_layers, B, T, 1, sm_count());
  if (dt == DP_F32) {            // split operands of the largest layer, half as much again, and its K-split planes or more
    size_t need = 0;
    for (int l = 0; l < n_layers; ++l)
      if (f32_on_tensor_cores(layers[l], T))
        need = std::max(need, split_layer_bytes(layers[l], B, T) * 3 / 2 +
                                  gta_partial_bytes(layers + l, 1, B, T, 3, sm_count(), true));
    n += need;
  }
  return n;
}

static dp_status clip_accumulate_check(const dp_linear_desc* layers, int32_t n_layers, dp_dtype dt, int32_t B, int32_t T,
                                       float* const* outs, const int64_t* ldos, float beta, float C, const void* ws,
                                       size_t ws_bytes) {
  if (!layers || n_layers <= 0 || !outs || !ldos || B <= 0 || T <= 0) return DP_ERR_INVALID_ARG;
  if (dt != DP_F32 && dt != DP_BF16) return DP_ERR_INVALID_ARG;
  if (!(beta == 0.f || beta == 1.f) || !finite_pos(C)) return DP_ERR_INVALID_ARG;
  const bool tc = (dt == DP_BF16) && !g_force_fma;
  for (int l = 0; l < n_layers; ++l) {
    dp_linear_desc one = layers[l];
    one.mode = DP_NORM_AUTO;
    const dp_status s = check_linear(one, dt, tc);
    if (s != DP_OK) return s;
    if (!outs[l] || ldos[l] < layers[l].d) return DP_ERR_INVALID_ARG;
  }
  if (!ws || ws_bytes < dp_clip_accumulate_grouped_ws_bytes(layers, n_layers, dt, B, T))
    return DP_ERR_WORKSPACE;
  for (int l = 0; l < n_layers && !aligned16(ws); ++l)     // operands that TMA reads from there
    if (tc ? gta_prescales(layers[l]) : dt == DP_F32 && f32_on_tensor_cores(layers[l], T)) return DP_ERR_ALIGNMENT;
  return DP_OK;
}

// the call has been checked
static dp_status clip_accumulate_impl(const dp_linear_desc* layers, int32_t n_layers, dp_dtype dt,
                                      int32_t B, int32_t T, const float* sq, float C, float* clip,
                                      float* const* outs, const int64_t* ldos, float beta,
                                      const GtaNoise* noise, void* ws, size_t ws_bytes,
                                      int32_t* dev_status, void* stream, const SplitGroup* kept = nullptr) {
  const bool tc = (dt == DP_BF16) && !g_force_fma;
  cudaStream_t st = (cudaStream_t)stream;
  float* clip_ws = static_cast<float*>(ws);
  dp_status s = resolve_clip(sq, B, C, clip, &clip_ws, st);
  if (s != DP_OK) return s;
  if (!tc) {
    const size_t head = align_up(size_t(B) * sizeof(float), 256);
    char* base = static_cast<char*>(ws) + head;
    SplitGroup group;
    auto flush = [&]() {
      if (group.index.empty()) return DP_OK;
      // R_i multiplies the narrower operand in fp32 before the split, so the GEMM runs unscaled (clip = NULL)
      dp_status s = launch_split(group.jobs.data(), (int)group.jobs.size(), B, T, clip_ws, st);
      if (s != DP_OK) return s;
      std::vector<float*> out;
      std::vector<int64_t> ldo;
      std::vector<uint32_t> ids;
      for (int l : group.index) {
        out.push_back(outs[l]); ldo.push_back(ldos[l]);
        if (noise) ids.push_back(noise->tensor_ids[l]);
      }
      GtaNoise nz;
      if (noise) { nz = *noise; nz.tensor_ids = ids.data(); }
      s = launch_clip_accumulate_tc(group.desc.data(), (int)group.desc.size(), B, T, 3, nullptr, out.data(),
                                    ldo.data(), beta, noise ? &nz : nullptr,
                                    reinterpret_cast<float*>(base + group.bytes), dev_status, st);
      group = SplitGroup();
      return s;
    };
    // The layers that go together from layer l on, up to the one returned: as many as fit with the K split, and so the planes of
    // partial sums, that all their tiles give (fewer layers are split more, so a part of them may not fit where all do).
    auto group_end = [&](int first) {
      size_t bytes = head, out_bytes = 0;
      long long tiles = 0;
      int end = first + 1;
      for (int l = first; l < n_layers; ++l) {
        if (!f32_on_tensor_cores(layers[l], T)) continue;
        bytes += split_layer_bytes(layers[l], B, T);
        if (l > first && bytes > ws_bytes) break;
        tiles += gta_tiles(layers[l]);
        out_bytes += align_up(size_t(layers[l].p) * size_t(layers[l].d) * sizeof(float), 256);
        const int ns = gta_choose_nsplit(tiles, B, T, 3, sm_count());
        if (bytes + (ns > 1 ? size_t(ns) * out_bytes : 0) <= ws_bytes) end = l + 1;
      }
      return end;
    };
    int end = 0;
    std::vector<int> fma;                // layers on the fp32 kernels: one launch for all of them
    if (kept && !kept->index.empty() && !sq &&
        kept->bytes + gta_partial_bytes(kept->desc.data(), (int)kept->desc.size(), B, T, 3, sm_count()) <= ws_bytes) {
      // the norms' split operands are still there, but for the narrower one of each layer, which is split (again), scaled
      group = *kept;
      base = static_cast<char*>(ws);
      group.jobs.clear();
      for (size_t k = 0; k < kept->index.size(); ++k) {
        SplitJob J = kept->jobs[2 * k + (a_is_scaled(layers[kept->index[k]]) ? 0 : 1)];
        J.scaled = true;
        group.jobs.push_back(J);
      }
      s = flush();
      if (s != DP_OK) return s;
    } else {
      kept = nullptr;
    }
    for (int l = 0; l < n_layers; ++l) {
      if (dt == DP_F32 && f32_on_tensor_cores(layers[l], T)) {
        if (kept) continue;
        if (l >= end) {
          s = flush();
          if (s != DP_OK) return s;
          end = group_end(l);
        }
        group.add(layers[l], l, B, T, true, base);
        continue;
      }
      fma.push_back(l);
    }
    s = flush();
    if (s != DP_OK || fma.empty()) return s;
    return launch_clip_accumulate_fma(layers, fma.data(), (int)fma.size(), dt, B, T, clip_ws, outs, ldos, beta, noise,
                                      st);
  }
  float* partial = reinterpret_cast<float*>(static_cast<char*>(ws) +
                                            align_up(size_t(B) * sizeof(float), 256));
  return launch_clip_accumulate_tc(layers, n_layers, B, T, 1, clip_ws, outs, ldos, beta, noise, partial,
                                   dev_status, st);
}

dp_status dp_clip_accumulate_grouped(const dp_linear_desc* layers, int32_t n_layers, dp_dtype dt,
                                     int32_t B, int32_t T, const float* sq, float C, float* clip,
                                     float* const* outs, const int64_t* ldos, float beta, void* ws,
                                     size_t ws_bytes, int32_t* dev_status, void* stream) {
  if (!sq && !clip) return DP_ERR_INVALID_ARG;
  const dp_status s = clip_accumulate_check(layers, n_layers, dt, B, T, outs, ldos, beta, C, ws, ws_bytes);
  return s != DP_OK ? s : clip_accumulate_impl(layers, n_layers, dt, B, T, sq, C, clip, outs, ldos, beta, nullptr, ws,
                                               ws_bytes, dev_status, stream);
}

static bool noise_args_ok(float sigma, float C, float scale) {
  return std::isfinite(sigma) && sigma >= 0.f && finite_pos(C) && std::isfinite(scale);
}

dp_status dp_clip_accumulate_noise_grouped(const dp_linear_desc* layers, int32_t n_layers,
                                           dp_dtype dt, int32_t B, int32_t T, const float* sq,
                                           float C, float* clip, float* const* outs,
                                           const int64_t* ldos, float beta, float sigma, float scale,
                                           uint64_t seed, const uint32_t* tensor_ids, uint32_t step,
                                           void* ws, size_t ws_bytes, int32_t* dev_status,
                                           void* stream) {
  if (!tensor_ids || !noise_args_ok(sigma, C, scale) || (!sq && !clip)) return DP_ERR_INVALID_ARG;
  const dp_status s = clip_accumulate_check(layers, n_layers, dt, B, T, outs, ldos, beta, C, ws, ws_bytes);
  if (s != DP_OK) return s;
  const GtaNoise noise{sigma * C, scale, seed, step, tensor_ids};
  return clip_accumulate_impl(layers, n_layers, dt, B, T, sq, C, clip, outs, ldos, beta, &noise, ws,
                              ws_bytes, dev_status, stream);
}

static dp_linear_desc one_layer(const void* A, int64_t lda, const void* G, int64_t ldg, int32_t d,
                                int32_t p) {
  dp_linear_desc L;
  L.A = A; L.lda = lda; L.d = d; L.G = G; L.ldg = ldg; L.p = p;
  L.mode = DP_NORM_AUTO; L.mode_used = 0;
  return L;
}

size_t dp_clip_accumulate_ws_bytes(dp_dtype dt, int32_t B, int32_t T, int32_t d, int32_t p) {
  if (B <= 0 || T <= 0 || d <= 0 || p <= 0) return 0;
  const dp_linear_desc L = one_layer(nullptr, d, nullptr, p, d, p);
  return dp_clip_accumulate_grouped_ws_bytes(&L, 1, dt, B, T);
}

dp_status dp_clip_accumulate(const void* A, int64_t lda, const void* G, int64_t ldg, dp_dtype dt,
                             int32_t B, int32_t T, int32_t d, int32_t p, const float* sq, float C,
                             float* clip, float* out, int64_t ldo, float beta, void* ws,
                             size_t ws_bytes, int32_t* dev_status, void* stream) {
  if (!A || !G || !out || d <= 0 || p <= 0) return DP_ERR_INVALID_ARG;
  const dp_linear_desc L = one_layer(A, lda, G, ldg, d, p);
  float* outs[1] = {out};
  const int64_t ldos[1] = {ldo};
  return dp_clip_accumulate_grouped(&L, 1, dt, B, T, sq, C, clip, outs, ldos, beta, ws, ws_bytes,
                                    dev_status, stream);
}

// ------------------------------------------------------------------ clip accumulate, embedding
// scratch of the sort: counts per id, per 1024 ids, and per chunk and id
static size_t sort_totals_bytes(size_t n, int V) {
  const size_t chunks = (n + kSortChunk - 1) / kSortChunk;
  return align_up(((chunks + 1) * V + ceil_div(V, 1024)) * sizeof(int), 256);
}

static void embed_ws_layout(int B, int T, int d, int V, size_t* off_clip, size_t* off_totals,
                            size_t* off_seg, size_t* off_perm, size_t* off_rank, size_t* off_part,
                            size_t* total) {
  const size_t n = size_t(B) * T;
  size_t o = 0;
  *off_clip = o;   o += align_up(size_t(B) * sizeof(float), 256);
  *off_totals = o; o += sort_totals_bytes(n, V);
  *off_seg = o;    o += align_up(size_t(V + 1) * sizeof(int), 256);
  *off_perm = o;   o += align_up(n * sizeof(int), 256);
  *off_rank = o;   o += align_up(n * sizeof(int), 256);
  *off_part = o;   o += embed_scatter_partial_bytes((long long)n, d);
  *total = o;
}

size_t dp_clip_accumulate_embed_ws_bytes(int32_t B, int32_t T, int32_t d, int32_t V) {
  if (B <= 0 || T <= 0 || V <= 0 || d <= 0) return 0;
  size_t a, b, c, e, f, g, total;
  embed_ws_layout(B, T, d, V, &a, &b, &c, &e, &f, &g, &total);
  return total;
}

struct EmbedNoise { float amp, scale; uint64_t seed; uint32_t tensor_id, step; };

static dp_status clip_accumulate_embed_impl(const int32_t* ids, const void* G, int64_t ldg,
                                            dp_dtype dt, int32_t B, int32_t T, int32_t d, int32_t V,
                                            const float* sq, float C, float* clip, float* out,
                                            int64_t ldo, float beta, const EmbedNoise* noise,
                                            int32_t* perm, int32_t* seg, void* ws, size_t ws_bytes,
                                            int32_t* dev_status, void* stream,
                                            const int32_t* perm_in = nullptr,
                                            const int32_t* seg_in = nullptr) {
  if (!ids || !G || (!sq && !clip) || !out || B <= 0 || T <= 0 || d <= 0 || V <= 0) return DP_ERR_INVALID_ARG;
  if ((perm_in == nullptr) != (seg_in == nullptr)) return DP_ERR_INVALID_ARG;
  if (ldg < d || ldo < d) return DP_ERR_INVALID_ARG;
  if (dt != DP_F32 && dt != DP_BF16) return DP_ERR_INVALID_ARG;
  if (!(beta == 0.f || beta == 1.f) || !finite_pos(C)) return DP_ERR_INVALID_ARG;
  if ((long long)B * T > 0x7fffffffLL) return DP_ERR_UNSUPPORTED;
  size_t o_clip, o_totals, o_seg, o_perm, o_rank, o_part, total;
  embed_ws_layout(B, T, d, V, &o_clip, &o_totals, &o_seg, &o_perm, &o_rank, &o_part, &total);
  if (!ws || ws_bytes < total) return DP_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  char* w = static_cast<char*>(ws);
  float* clip_ws = reinterpret_cast<float*>(w + o_clip);
  EmbedSortWs sw;
  sw.totals = reinterpret_cast<int*>(w + o_totals);
  sw.seg = reinterpret_cast<int*>(w + o_seg);
  sw.perm = reinterpret_cast<int*>(w + o_perm);
  sw.rank = reinterpret_cast<int*>(w + o_rank);
  const int n = B * T;
  dp_status s = resolve_clip(sq, B, C, clip, &clip_ws, st);
  if (s != DP_OK) return s;
  if (perm_in) {                         // sorted earlier by dp_embed_sort
    sw.perm = const_cast<int*>(perm_in);
    sw.seg = const_cast<int*>(seg_in);
  } else {
    s = launch_embed_sort(ids, n, V, sw, dev_status, st);
    if (s != DP_OK) return s;
  }
  if (perm) DP_CUDA_OK(cudaMemcpyAsync(perm, sw.perm, size_t(n) * sizeof(int),
                                       cudaMemcpyDeviceToDevice, st));
  if (seg) DP_CUDA_OK(cudaMemcpyAsync(seg, sw.seg, size_t(V + 1) * sizeof(int),
                                      cudaMemcpyDeviceToDevice, st));
  // With noise and beta == 0 the table is filled with scale*sigma*C*z (write only) in place of
  // the zero fill; with beta == 1 the noise was already drawn by whoever wrote the table first.
  bool clear = true;
  float scale = 1.f;
  if (noise) {
    scale = noise->scale;
    if (beta == 0.f) {
      s = launch_add_noise(out, V, d, ldo, true, noise->amp, noise->scale, noise->seed,
                           noise->tensor_id, noise->step, st);
      if (s != DP_OK) return s;
      clear = false;
    }
  }
  return launch_embed_scatter(ids, G, ldg, dt, n, T, d, V, clip_ws, sw.perm, sw.seg, out, ldo, beta,
                              scale, clear, reinterpret_cast<float*>(w + o_part), st, dev_status);
}

dp_status dp_clip_accumulate_embed(const int32_t* ids, const void* G, int64_t ldg, dp_dtype dt,
                                   int32_t B, int32_t T, int32_t d, int32_t V, const float* sq,
                                   float C, float* clip, float* out, int64_t ldo, float beta,
                                   int32_t* perm, int32_t* seg, void* ws, size_t ws_bytes,
                                   int32_t* dev_status, void* stream) {
  return clip_accumulate_embed_impl(ids, G, ldg, dt, B, T, d, V, sq, C, clip, out, ldo, beta, nullptr,
                                    perm, seg, ws, ws_bytes, dev_status, stream);
}

size_t dp_embed_sort_ws_bytes(int32_t B, int32_t T, int32_t V) {
  if (B <= 0 || T <= 0 || V <= 0) return 0;
  const size_t n = size_t(B) * T;
  return sort_totals_bytes(n, V) + align_up(n * sizeof(int), 256);
}

dp_status dp_embed_sort(const int32_t* ids, int32_t B, int32_t T, int32_t V, int32_t* perm,
                        int32_t* seg, void* ws, size_t ws_bytes, int32_t* dev_status, void* stream) {
  if (!ids || !perm || !seg || B <= 0 || T <= 0 || V <= 0) return DP_ERR_INVALID_ARG;
  if ((long long)B * T > 0x7fffffffLL) return DP_ERR_UNSUPPORTED;
  if (!ws || ws_bytes < dp_embed_sort_ws_bytes(B, T, V)) return DP_ERR_WORKSPACE;
  const int n = B * T;
  EmbedSortWs sw;
  sw.totals = static_cast<int*>(ws);
  sw.rank = reinterpret_cast<int*>(static_cast<char*>(ws) + sort_totals_bytes(size_t(n), V));
  sw.seg = seg;
  sw.perm = perm;
  return launch_embed_sort(ids, n, V, sw, dev_status, (cudaStream_t)stream);
}

dp_status dp_clip_accumulate_embed_sorted(const int32_t* ids, const void* G, int64_t ldg, dp_dtype dt,
                                          int32_t B, int32_t T, int32_t d, int32_t V, const float* sq,
                                          float C, float* clip, float* out, int64_t ldo, float beta,
                                          const int32_t* perm, const int32_t* seg, void* ws,
                                          size_t ws_bytes, int32_t* dev_status, void* stream) {
  if (!perm || !seg) return DP_ERR_INVALID_ARG;
  return clip_accumulate_embed_impl(ids, G, ldg, dt, B, T, d, V, sq, C, clip, out, ldo, beta, nullptr,
                                    nullptr, nullptr, ws, ws_bytes, dev_status, stream, perm, seg);
}

dp_status dp_clip_accumulate_embed_noise(const int32_t* ids, const void* G, int64_t ldg, dp_dtype dt,
                                         int32_t B, int32_t T, int32_t d, int32_t V, const float* sq,
                                         float C, float* clip, float* out, int64_t ldo, float beta,
                                         float sigma, float scale, uint64_t seed, uint32_t tensor_id,
                                         uint32_t step, int32_t* perm, int32_t* seg, void* ws,
                                         size_t ws_bytes, int32_t* dev_status, void* stream) {
  if (!noise_args_ok(sigma, C, scale)) return DP_ERR_INVALID_ARG;
  const EmbedNoise noise{sigma * C, scale, seed, tensor_id, step};
  return clip_accumulate_embed_impl(ids, G, ldg, dt, B, T, d, V, sq, C, clip, out, ldo, beta, &noise,
                                    perm, seg, ws, ws_bytes, dev_status, stream);
}

// ----------------------------------------------------------------------------------- noise
dp_status dp_add_noise(float* out, int64_t n, float sigma, float C, float scale, uint64_t seed,
                       uint32_t tensor_id, uint32_t step, void* stream) {
  if (!out || n < 0) return DP_ERR_INVALID_ARG;
  if (!std::isfinite(sigma) || sigma < 0.f || !finite_pos(C) || !std::isfinite(scale))
    return DP_ERR_INVALID_ARG;
  if (!aligned16(out)) return DP_ERR_ALIGNMENT;
  // a flat buffer is the (n, 1) tensor with pitch 1
  return launch_add_noise(out, n, 1, 1, false, sigma * C, scale, seed, tensor_id, step,
                          (cudaStream_t)stream);
}

dp_status dp_add_noise_slice(float* out, int64_t n, int64_t first_element, float sigma, float C,
                             float scale, uint64_t seed, uint32_t tensor_id, uint32_t step,
                             void* stream) {
  if (!out || n < 0 || first_element < 0) return DP_ERR_INVALID_ARG;
  if (!noise_args_ok(sigma, C, scale)) return DP_ERR_INVALID_ARG;
  if (!aligned16(out) || (first_element & 3)) return DP_ERR_ALIGNMENT;   // whole Philox counters
  return launch_add_noise(out, n, 1, 1, false, sigma * C, scale, seed, tensor_id, step,
                          (cudaStream_t)stream, first_element >> 2);
}

dp_status dp_noise_step_device(const uint32_t* dev_counter) {
  g_step_dev = dev_counter;
  return DP_OK;
}

dp_status dp_fill_noise(float* out, int64_t n, float sigma, float C, float scale, uint64_t seed,
                        uint32_t tensor_id, uint32_t step, void* stream) {
  if (!out || n < 0) return DP_ERR_INVALID_ARG;
  if (!noise_args_ok(sigma, C, scale)) return DP_ERR_INVALID_ARG;
  if (!aligned16(out)) return DP_ERR_ALIGNMENT;
  return launch_add_noise(out, n, 1, 1, true, sigma * C, scale, seed, tensor_id, step,
                          (cudaStream_t)stream);
}

// ------------------------------------------------------------------------------ whole step
// Workspace with which fp32 layers are split once per step: the group of all of them, the norms' partial
// sums, the K-split planes.  Beyond 16 GiB the layers go through less in groups.  With the partial sums
// of layers on the fp32 kernels, whose norms then take one launch.
size_t dp_step_ws_bytes(const dp_linear_desc* layers, int32_t n_layers, dp_dtype dt, int32_t B, int32_t T) {
  if (!layers || n_layers <= 0 || B <= 0 || T <= 0 || dt != DP_F32) return 0;
  std::vector<dp_linear_desc> on;
  size_t need = 0;
  for (int l = 0; l < n_layers; ++l)
    if (f32_on_tensor_cores(layers[l], T)) {
      need += f32_norm_bytes(layers[l], B, T, sm_count());
      on.push_back(layers[l]);
    }
  if (!on.empty()) need += gta_partial_bytes(on.data(), (int)on.size(), B, T, 3, sm_count(), true);
  if (need > (size_t(16) << 30)) need = f32_norms_bytes(layers, n_layers, dt, B, T);
  return need + fma_norms_bytes(layers, n_layers, dt, B, T);
}

// Row sums of the vectors' examples, from the norms of a step to its clipped sums.  Reading G again costs 2T or 4T bytes
// per column and example, these 8; below eight tokens there is nothing to gain.
size_t dp_step_vectors_ws_bytes(const dp_vector_desc* vectors, int32_t n, int32_t B, int32_t T) {
  if (check_vectors(vectors, n, B, T) != DP_OK || T < 8) return 0;
  return align_up(vector_keep_bytes(vectors, n, B), 256);
}

// All that can be wrong with a step, before anything is enqueued: an error found halfway would leave work on two
// streams.  Workspaces as the requested phases use them; plan: of the layers' norms, if those are among them.
static dp_status check_step(const dp_step_desc* S, int32_t phases, GhostPlan* plan) {
  if (!S || S->B <= 0 || S->T <= 0 || S->V <= 0 || S->d <= 0 || S->n_layers < 0 || S->n_vectors < 0)
    return DP_ERR_INVALID_ARG;
  if (!S->ids || !S->G_emb || !S->wte || !S->sq || !S->clip || !S->side_sq || !S->perm || !S->seg)
    return DP_ERR_INVALID_ARG;
  if (S->n_layers && (!S->layers || !S->outs || !S->ldos || (S->with_noise && !S->tensor_ids)))
    return DP_ERR_INVALID_ARG;
  if (S->tied && S->n_layers == 0) return DP_ERR_INVALID_ARG;
  auto dtype_ok = [](int32_t t) { return t == DP_F32 || t == DP_BF16; };
  if (!dtype_ok(S->layer_dtype) || !dtype_ok(S->vector_dtype) || !dtype_ok(S->embed_dtype)) return DP_ERR_INVALID_ARG;
  if (S->tied && S->embed_dtype != S->layer_dtype) return DP_ERR_INVALID_ARG;      // one type in the cross term
  if (S->pos_ids && (!S->wpe || !S->pos_perm || !S->pos_seg || S->pos_rows <= 0)) return DP_ERR_INVALID_ARG;
  for (int k = 0; k < 4; ++k) if (!S->events[k]) return DP_ERR_INVALID_ARG;
  if (!finite_pos(S->C) || (S->with_noise && !noise_args_ok(S->sigma, S->C, 1.f))) return DP_ERR_INVALID_ARG;
  if (S->ldge < S->d || S->ld_wte < S->d || (S->pos_ids && S->ld_wpe < S->d)) return DP_ERR_INVALID_ARG;
  const int B = S->B, T = S->T, d = S->d;
  if (S->n_vectors) {
    const dp_status s = check_vectors(S->vectors, S->n_vectors, B, T);
    if (s != DP_OK) return s;
    if (!S->vector_outs || (S->with_noise && !S->vector_ids)) return DP_ERR_INVALID_ARG;
    for (int k = 0; k < S->n_vectors; ++k) if (!S->vector_outs[k]) return DP_ERR_INVALID_ARG;
  }
  if (T > kEmbedMaxT || (long long)B * T > 0x7fffffffLL) return DP_ERR_UNSUPPORTED;
  const int32_t rows[2] = {S->V, S->pos_ids ? S->pos_rows : 0};              // of the tables
  size_t ws = 0, side = 0;
  if (phases & DP_STEP_NORMS) {
    if (S->n_layers) {
      const dp_status s = ghost_norms_check(S->layers, S->n_layers, (dp_dtype)S->layer_dtype, B, T, S->sq, S->ws, S->ws_bytes, plan);
      if (s != DP_OK) return s;
    }
    if (S->n_vectors) ws = std::max(ws, dp_vector_norms_ws_bytes(S->vectors, S->n_vectors, B, T));
    if (S->tied) {
      const dp_linear_desc& lm = S->layers[S->n_layers - 1];
      const dp_status s = cross_term_check(S->ids, S->G_emb, S->ldge, lm.A, lm.lda, lm.G, lm.ldg, (dp_dtype)S->embed_dtype, B, T,
                                           d, S->V, S->ws, S->ws_bytes);
      if (s != DP_OK) return s;
    }
    side = dp_embed_norms_ws_bytes(B, T, d);
    for (int32_t r : rows) side = std::max(side, dp_embed_sort_ws_bytes(B, T, r));
  }
  if ((phases & DP_STEP_GEMM) && S->n_layers) {
    const dp_status s = clip_accumulate_check(S->layers, S->n_layers, (dp_dtype)S->layer_dtype, B, T, S->outs, S->ldos, 0.f, S->C,
                                              S->ws, S->ws_bytes);
    if (s != DP_OK) return s;
  }
  if (phases & DP_STEP_REST) {
    for (int k = 0; k < 2; ++k) {
      size_t& w = k == 0 && S->tied ? ws : side;
      w = std::max(w, dp_clip_accumulate_embed_ws_bytes(B, T, d, rows[k]));
    }
    if (S->n_vectors) ws = std::max(ws, dp_clip_accumulate_vectors_ws_bytes(S->vectors, S->n_vectors, B, T));
  }
  if (S->ws_bytes < ws || (ws && !S->ws) || S->side_ws_bytes < side || (side && !S->side_ws)) return DP_ERR_WORKSPACE;
  return DP_OK;
}

// A table that no GEMM writes starts as its noise (or as zeros), so that the row sums can be added.
static dp_status start_table(const dp_step_desc* S, float* table, int64_t ld, int64_t rows, uint32_t tid,
                             cudaStream_t st) {
  if (S->with_noise)
    return launch_add_noise(table, rows, S->d, ld, true, S->sigma * S->C, 1.f, S->seed, tid, S->step, st);
  if (ld == S->d) return launch_clear(table, size_t(rows) * size_t(ld) * sizeof(float), st);
  DP_CUDA_OK(cudaMemset2DAsync(table, size_t(ld) * sizeof(float), 0, size_t(S->d) * sizeof(float),
                               size_t(rows), st));
  return DP_OK;
}

// events: [0] the step began, [1] embedding norms done, [2] row sums done, [3] clip factors exist (as the clipped sums
// take them)
static dp_status step_norms(const dp_step_desc* S, const GhostPlan& plan, SplitGroup* kept, float* row_sums) {
  cudaStream_t main = (cudaStream_t)S->stream, side = (cudaStream_t)S->side_stream;
  const dp_dtype embed_dt = (dp_dtype)S->embed_dtype;
  const int B = S->B, T = S->T;
  dp_status s;
  NormSources N;                 // partial sums that the last kernel of this phase adds up
  N.n = 0;
  size_t held = 0;               // bytes at the head of ws that hold such sums
  char* ws = static_cast<char*>(S->ws);
  DP_CUDA_OK(cudaEventRecord((cudaEvent_t)S->events[0], main));
  if (S->n_layers) {
    s = ghost_norms_impl(plan, S->layers, S->n_layers, (dp_dtype)S->layer_dtype, B, T, S->sq, S->ws, S->ws_bytes,
                         S->dev_status, main, true, &N.src[0], kept);
    if (s != DP_OK) return s;
    N.n = 1;
    if (N.src[0].partials != S->sq)
      held = size_t(reinterpret_cast<const char*>(N.src[0].partials) - ws) +
             align_up(size_t(B) * N.src[0].n_per * sizeof(float), 256);
    if (kept) held = std::max(held, kept->bytes);
  }
  // Side stream: all that needs neither the big norm kernel nor the clip factors.  It is enqueued
  // after that kernel: what is already resident keeps the kernel's CTAs out until it ends, what
  // arrives second shares the SMs with them.
  DP_CUDA_OK(cudaStreamWaitEvent(side, (cudaEvent_t)S->events[0], 0));     // earlier readers are done
  // The embedding norms' partial sums stay at the end of side_ws, out of the sorts' way, where it has room.
  const size_t each = dp_embed_norms_ws_bytes(B, T, S->d), tables = S->pos_ids ? 2 : 1;
  const size_t sorts = std::max(dp_embed_sort_ws_bytes(B, T, S->V),
                                S->pos_ids ? dp_embed_sort_ws_bytes(B, T, S->pos_rows) : size_t(0));
  char* side_ws = static_cast<char*>(S->side_ws);
  size_t side_bytes = S->side_ws_bytes & ~size_t(255);
  const bool keep = side_bytes >= sorts + tables * each;
  NormSource embed[2];
  for (size_t k = 0; k < tables; ++k) {
    char* w = side_ws;
    if (keep) { side_bytes -= each; w += side_bytes; }
    s = embed_norms_impl(k ? S->pos_ids : S->ids, S->G_emb, S->ldge, embed_dt, B, T, S->d, k ? S->pos_rows : S->V, S->side_sq,
                         nullptr, w, keep ? each : S->side_ws_bytes, S->dev_status, side, k == 0, keep ? &embed[k] : nullptr);
    if (s != DP_OK) return s;
  }
  if (!keep) embed[0] = NormSource{S->side_sq, 1, 1.f, nullptr};
  DP_CUDA_OK(cudaEventRecord((cudaEvent_t)S->events[1], side));
  s = dp_embed_sort(S->ids, B, T, S->V, S->perm, S->seg, side_ws, side_bytes, S->dev_status, side);
  if (s != DP_OK) return s;
  if (S->pos_ids) {
    s = dp_embed_sort(S->pos_ids, B, T, S->pos_rows, S->pos_perm, S->pos_seg, side_ws, side_bytes, S->dev_status,
                      side);
    if (s != DP_OK) return s;
    s = start_table(S, S->wpe, S->ld_wpe, S->pos_rows, S->wpe_id, side);
    if (s != DP_OK) return s;
  }
  if (!S->tied) {
    s = start_table(S, S->wte, S->ld_wte, S->V, S->wte_id, side);
    if (s != DP_OK) return s;
  }
  // main stream again.  Where ws has no room behind the sums it holds, they are added up first.
  auto room = [&](size_t need) {
    if (held + need <= S->ws_bytes) return DP_OK;
    if (kept) *kept = SplitGroup();
    for (int k = 0; k < N.n; ++k) {
      if (N.src[k].partials == S->sq) continue;
      const dp_status r = launch_reduce_partials(N.src[k].partials, N.src[k].n_per, B, S->sq, N.src[k].factor,
                                                 N.src[k].plain_out, main, k == 0);
      if (r != DP_OK) return r;
    }
    if (N.n) { N.src[0] = NormSource{S->sq, 1, 1.f, nullptr}; N.n = 1; }
    held = 0;
    return DP_OK;
  };
  if (S->n_vectors) {
    const size_t need = dp_vector_norms_ws_bytes(S->vectors, S->n_vectors, B, T);
    s = room(need);
    if (s != DP_OK) return s;
    s = vector_norms_impl(S->vectors, S->n_vectors, (dp_dtype)S->vector_dtype, B, T, S->sq, ws + held, S->ws_bytes - held,
                          main, &N.src[N.n], row_sums);
    if (s != DP_OK) return s;
    ++N.n;
    held += need;
  }
  if (S->tied) {
    const dp_linear_desc& lm = S->layers[S->n_layers - 1];
    s = room(dp_tied_cross_term_ws_bytes(B, T, S->d, S->V));
    if (s != DP_OK) return s;
    s = cross_term_impl(S->ids, S->G_emb, S->ldge, lm.A, lm.lda, lm.G, lm.ldg, embed_dt, B, T, S->d, S->V, S->sq,
                        S->cross, ws + held, S->ws_bytes - held, S->dev_status, main, &N.src[N.n]);
    if (s != DP_OK) return s;
    ++N.n;
  }
  N.n_main = N.n;
  N.src[N.n++] = embed[0];
  if (keep && tables == 2) N.src[N.n++] = embed[1];
  DP_CUDA_OK(cudaStreamWaitEvent(main, (cudaEvent_t)S->events[1], 0));
  s = launch_finish_norms(N, B, S->C, S->sq, S->clip, S->norms, main);
  if (s != DP_OK) return s;
  DP_CUDA_OK(cudaEventRecord((cudaEvent_t)S->events[3], main));
  return DP_OK;
}

static dp_status step_gemm(const dp_step_desc* S, const SplitGroup* kept) {
  if (!S->n_layers) return DP_OK;
  const GtaNoise noise{S->sigma * S->C, 1.f, S->seed, S->step, S->tensor_ids};
  return clip_accumulate_impl(S->layers, S->n_layers, (dp_dtype)S->layer_dtype, S->B, S->T, nullptr, S->C, S->clip,
                              S->outs, S->ldos, 0.f, S->with_noise ? &noise : nullptr, S->ws, S->ws_bytes, S->dev_status,
                              S->stream, kept);
}

static dp_status step_rest(const dp_step_desc* S, float* row_sums) {
  cudaStream_t main = (cudaStream_t)S->stream, side = (cudaStream_t)S->side_stream;
  const dp_dtype dt = (dp_dtype)S->embed_dtype;
  dp_status s;
  // Row sums of tables that no GEMM writes need the clip factors only: on the side stream they run
  // where the GEMM's last wave leaves SMs idle.
  DP_CUDA_OK(cudaStreamWaitEvent(side, (cudaEvent_t)S->events[3], 0));
  if (row_sums) {
    s = launch_vector_kept_sums(S->vectors, S->n_vectors, S->B, S->T, row_sums, S->clip, S->vector_outs, 0.f, S->with_noise,
                                S->sigma * S->C, 1.f, S->seed, S->vector_ids, S->step, side);
    if (s != DP_OK) return s;
  }
  if (!S->tied) {
    s = dp_clip_accumulate_embed_sorted(S->ids, S->G_emb, S->ldge, dt, S->B, S->T, S->d, S->V, nullptr, S->C,
                                        S->clip, S->wte, S->ld_wte, 1.f, S->perm, S->seg, S->side_ws,
                                        S->side_ws_bytes, S->dev_status, side);
    if (s != DP_OK) return s;
  }
  if (S->pos_ids) {
    s = dp_clip_accumulate_embed_sorted(S->pos_ids, S->G_emb, S->ldge, dt, S->B, S->T, S->d, S->pos_rows, nullptr,
                                        S->C, S->clip, S->wpe, S->ld_wpe, 1.f, S->pos_perm, S->pos_seg,
                                        S->side_ws, S->side_ws_bytes, S->dev_status, side);
    if (s != DP_OK) return s;
  }
  DP_CUDA_OK(cudaEventRecord((cudaEvent_t)S->events[2], side));
  DP_CUDA_OK(cudaStreamWaitEvent(main, (cudaEvent_t)S->events[2], 0));
  if (S->tied) {                       // onto the head's sum and noise
    s = dp_clip_accumulate_embed_sorted(S->ids, S->G_emb, S->ldge, dt, S->B, S->T, S->d, S->V, nullptr, S->C,
                                        S->clip, S->wte, S->ld_wte, 1.f, S->perm, S->seg, S->ws,
                                        S->ws_bytes, S->dev_status, main);
    if (s != DP_OK) return s;
  }
  if (S->n_vectors && !row_sums)
    return dp_clip_accumulate_vectors(S->vectors, S->n_vectors, (dp_dtype)S->vector_dtype, S->B, S->T, nullptr, S->C, S->clip,
                                      S->vector_outs, 0.f, S->with_noise, S->sigma, 1.f, S->seed,
                                      S->vector_ids, S->step, S->ws, S->ws_bytes, main);
  return DP_OK;
}

// A step short of work uses `stream` alone.  What `side_stream` still has to do, an earlier fill of a table say, comes
// before it, and what is put there later comes after it, as when the step used both; inside a capture `side_stream`
// joins first and is joined again.
static dp_status small_step(const dp_step_desc* S) {
  cudaStream_t main = (cudaStream_t)S->stream, side = (cudaStream_t)S->side_stream;
  cudaStreamCaptureStatus capture;
  DP_CUDA_OK(cudaStreamIsCapturing(main, &capture));
  auto after = [](cudaStream_t later, cudaStream_t earlier, void* event) {
    DP_CUDA_OK(cudaEventRecord((cudaEvent_t)event, earlier));
    DP_CUDA_OK(cudaStreamWaitEvent(later, (cudaEvent_t)event, 0));
    return DP_OK;
  };
  dp_status s = DP_OK;
  if (capture != cudaStreamCaptureStatusNone) s = after(side, main, S->events[0]);
  if (s == DP_OK) s = after(main, side, S->events[2]);
  if (s == DP_OK) s = launch_small_step(*S, main);
  if (s == DP_OK) s = after(side, main, S->events[0]);
  if (s == DP_OK && capture != cudaStreamCaptureStatusNone) s = after(main, side, S->events[2]);
  return s;
}

dp_status dp_step_enqueue(const dp_step_desc* step, int32_t phases) {
  GhostPlan plan;
  dp_status s = DP_ERR_WORKSPACE;
  dp_step_desc desc;
  const dp_step_desc* S = step;
  // The vectors' row sums lie at the end of ws, where it has room for them beside all else.
  float* row_sums = nullptr;
  if (step && phases == DP_STEP_ALL && step->n_vectors > 0 && step->vectors && step->ws && aligned16(step->ws)) {
    const size_t all = step->ws_bytes & ~size_t(255);
    const size_t rows = dp_step_vectors_ws_bytes(step->vectors, step->n_vectors, step->B, step->T);
    // (room that split fp32 layers can use comes first)
    const size_t layers = dp_step_ws_bytes(step->layers, step->n_layers, (dp_dtype)step->layer_dtype, step->B, step->T);
    if (rows && all >= rows + layers) {
      desc = *step;
      desc.ws_bytes = all - rows;
      s = check_step(&desc, phases, &plan);
      if (s == DP_OK) {
        S = &desc;
        row_sums = reinterpret_cast<float*>(static_cast<char*>(step->ws) + desc.ws_bytes);
      }
    }
  }
  if (s == DP_ERR_WORKSPACE) s = check_step(step, phases, &plan);
  if (s != DP_OK) return s;
  if (phases == DP_STEP_ALL && small_step_fits(*S)) return small_step(S);
  // fp32 layers: within one call the sums can use the norms' split operands
  SplitGroup split;
  SplitGroup* kept = phases == DP_STEP_ALL && S->layer_dtype == DP_F32 ? &split : nullptr;
  if (phases & DP_STEP_NORMS) s = step_norms(S, plan, kept, row_sums);
  // a call of its own: what `stream` did in between (other clip factors, say) comes before the row sums as well
  if ((phases & (DP_STEP_NORMS | DP_STEP_GEMM)) == DP_STEP_GEMM)
    DP_CUDA_OK(cudaEventRecord((cudaEvent_t)S->events[3], (cudaStream_t)S->stream));
  if (s == DP_OK && (phases & DP_STEP_GEMM)) s = step_gemm(S, kept);
  if (s == DP_OK && (phases & DP_STEP_REST)) s = step_rest(S, row_sums);
  if (s != DP_OK) {
    // a launch failed: whatever the side stream still does to the caller's tensors, `stream` waits for it
    const int error = g_last_cuda_error;
    if (cudaEventRecord((cudaEvent_t)S->events[2], (cudaStream_t)S->side_stream) == cudaSuccess)
      (void)cudaStreamWaitEvent((cudaStream_t)S->stream, (cudaEvent_t)S->events[2], 0);
    (void)cudaGetLastError();
    g_last_cuda_error = error;
  }
  return s;
}

}  // extern "C"
