// C ABI of the VSA2 library: argument checks, workspace layout, kernel sequencing.
#include <cuda.h>
#include <math.h>
#include <string.h>

#include <atomic>

#include "pooled_inputs.cuh"

using namespace vsa2;

namespace {

cudaEvent_t g_prof_start[VSA2_KERNEL_COUNT];
cudaEvent_t g_prof_stop[VSA2_KERNEL_COUNT];
std::atomic<long long> g_launches{0};

struct RouteLayout {
  size_t status, qr, kr, lse_r, pr, hist, state, row_tau, row_eq_take, row_cnt, row_gt, row_eq, bitmap, bitmap_t, total;
  int words;
};
struct BwdLayout {
  size_t status, delta, absmax, ds_exp, full, d_oc_hat, dqc, dkc, dvc, pooled, total;
};

struct Carver {
  size_t off = 0;
  size_t take(size_t bytes) {
    size_t o = off;
    off = align_up(off + bytes, 256);
    return o;
  }
};

int fill_geo(const vsa2_params* p, Geo* g) {
  if (p == nullptr) return VSA2_ERR_INVALID_ARG;
  if (p->batch <= 0 || p->heads_q <= 0 || p->heads_kv <= 0 || p->grid_t <= 0 || p->grid_h <= 0 || p->grid_w <= 0 ||
      p->cube_t <= 0 || p->cube_h <= 0 || p->cube_w <= 0 || p->rpool_t <= 0 || p->rpool_h <= 0 || p->rpool_w <= 0)
    return VSA2_ERR_INVALID_ARG;
  if (p->heads_q % p->heads_kv) return VSA2_ERR_INVALID_ARG;
  if (p->select_mode < VSA2_PER_SEQUENCE || p->select_mode > VSA2_PER_QUERY_BUDGET) return VSA2_ERR_INVALID_ARG;
  if (p->out_dtype != VSA2_BF16 && p->out_dtype != VSA2_F32) return VSA2_ERR_INVALID_ARG;
  if (p->topk < 0 || p->nnz_cap < 0 || !(p->softmax_scale >= 0.f) || p->text_len < 0) return VSA2_ERR_INVALID_ARG;
  if (p->cube_t % p->rpool_t || p->cube_h % p->rpool_h || p->cube_w % p->rpool_w) return VSA2_ERR_INVALID_ARG;
  if (p->head_dim != 64 && p->head_dim != 128) return VSA2_ERR_UNSUPPORTED;
  // 64-token cubes, or 128-token cubes that split along w into two 64-token halves the router pooling respects
  const long long cube_tokens = (long long)p->cube_t * p->cube_h * p->cube_w;
  const bool wide = cube_tokens == 2 * kBlockTokens;
  if (cube_tokens != kBlockTokens && !wide) return VSA2_ERR_UNSUPPORTED;
  if (wide && (p->cube_w % 2 || (p->cube_w / 2) % p->rpool_w)) return VSA2_ERR_UNSUPPORTED;
  if (p->batch > 65535 || p->heads_q > 65535 || p->heads_q / p->heads_kv > 16) return VSA2_ERR_UNSUPPORTED;
  g->batch = p->batch; g->Hq = p->heads_q; g->Hkv = p->heads_kv; g->rep = p->heads_q / p->heads_kv; g->D = p->head_dim;
  g->T = p->grid_t; g->H = p->grid_h; g->W = p->grid_w;
  long long L = (long long)g->T * g->H * g->W;
  if (L + p->text_len > 0x7fffffffLL / 128) return VSA2_ERR_UNSUPPORTED;
  g->L = (int)L;
  g->Lt = p->text_len;
  g->S = (int)L + p->text_len;
  g->Bt = p->cube_t; g->Bh = p->cube_h; g->Bw = p->cube_w;
  g->Nt = (g->T + g->Bt - 1) / g->Bt; g->Nh = (g->H + g->Bh - 1) / g->Bh; g->Nw = (g->W + g->Bw - 1) / g->Bw;
  g->N = g->Nt * g->Nh * g->Nw;
  geo_set_magics(*g);
  g->Nvid = g->N;
  g->Rt = p->rpool_t; g->Rh = p->rpool_h; g->Rw = p->rpool_w;
  g->Gt = g->Bt / g->Rt; g->Gh = g->Bh / g->Rh; g->Gw = g->Bw / g->Rw;
  g->G = g->Gt * g->Gh * g->Gw;
  if (128 % (wide ? g->G / 2 : g->G)) return VSA2_ERR_UNSUPPORTED;
  int K = p->topk;
  if (K == 0) {
    if (!(p->keep_fraction > 0.f) || p->keep_fraction > 1.f) {
      if (p->select_mode != VSA2_PER_QUERY_BUDGET) return VSA2_ERR_INVALID_ARG;
      K = 1;
    } else {
      K = (int)lroundf(p->keep_fraction * (float)g->N);
      if (K < 1) K = 1;
    }
  }
  if (K > g->N) K = g->N;
  g->K = K;
  g->mode = p->select_mode;
  g->out_f32 = p->out_dtype == VSA2_F32;
  g->flags = p->flags;
  g->scale = p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf((float)g->D);
  if (p->nnz_cap > 0) g->nnz_cap = p->nnz_cap;
  else if (p->select_mode == VSA2_PER_QUERY_BUDGET) return VSA2_ERR_INVALID_ARG;
  else g->nnz_cap = (long long)g->N * K;
  return VSA2_OK;
}

// Block problem of the fine kernels with text tokens: the N video cubes followed by ceil(Lt / 64) text blocks; its maps
// are the video maps with the text blocks appended to every row and one dense row per text block.
int text_blocks(const Geo& g) { return (g.Lt + kBlockTokens - 1) / kBlockTokens; }
Geo text_geo(const Geo& g) {
  Geo x = g;
  const int tb = text_blocks(g);
  x.N = g.Nvid + tb;
  x.nnz_cap = g.nnz_cap + (long long)g.Nvid * tb + (long long)tb * x.N;
  return x;
}
struct TextMapLayout {
  size_t ptr, idx, cptr, ridx, total;     // offsets behind the call's other workspace regions
};
TextMapLayout text_map_layout(const Geo& g, bool with_csc) {
  TextMapLayout r = {};
  if (g.Lt == 0) return r;
  const Geo x = text_geo(wide_cube(g) ? narrow_geo(g) : g);      // (128-token cubes: the block problem of the half-cubes)
  Carver c;
  const size_t BHq = (size_t)g.batch * g.Hq;
  r.ptr = c.take(BHq * (x.N + 1) * sizeof(int));
  r.idx = c.take(BHq * (size_t)x.nnz_cap * sizeof(int));
  if (with_csc) {
    r.cptr = c.take(BHq * (x.N + 1) * sizeof(int));
    r.ridx = c.take(BHq * (size_t)x.nnz_cap * sizeof(int));
  }
  r.total = c.off;
  return r;
}

// `folded`: g is a half-cube problem whose scores the router folds itself (its own block scores and selection never exist)
RouteLayout route_layout(const Geo& g, bool folded = false) {
  RouteLayout r;
  Carver c;
  const size_t BHq = (size_t)g.batch * g.Hq, BHk = (size_t)g.batch * g.Hkv, NG = (size_t)g.N * g.G;
  r.words = (g.N + 31) / 32;
  r.status = c.take(sizeof(StatusBlock));
  r.qr = c.take(BHq * NG * g.D * sizeof(bf16));
  r.kr = c.take(BHk * NG * g.D * sizeof(bf16));
  r.lse_r = c.take(router_tc_supported(g) ? 0 : BHq * NG * sizeof(float));      // (the tensor-core router keeps them on chip)
  r.pr = c.take(folded ? 0 : BHq * (size_t)g.N * g.N * sizeof(float));
  r.hist = c.take(BHq * 3 * 2048 * sizeof(unsigned));
  r.state = c.take(BHq * 8 * sizeof(unsigned));
  r.row_tau = c.take(BHq * g.N * sizeof(float));
  r.row_eq_take = c.take(BHq * g.N * sizeof(int));
  r.row_cnt = c.take(BHq * g.N * sizeof(int));
  r.row_gt = c.take(BHq * g.N * sizeof(int));
  r.row_eq = c.take(BHq * g.N * sizeof(int));
  r.bitmap = c.take(BHq * (size_t)g.N * r.words * sizeof(unsigned));
  r.bitmap_t = c.take(BHq * (size_t)g.N * r.words * sizeof(unsigned));
  r.total = c.off;
  return r;
}

// `of_wide`: a level of a 128-token-cube problem, where dO_c_hat goes through memory in fp32 (else the preprocess leaves it in the pooled region)
BwdLayout bwd_layout(const Geo& g, bool of_wide) {
  BwdLayout r;
  Carver c;
  const size_t BHq = (size_t)g.batch * g.Hq;
  r.status = c.take(sizeof(StatusBlock));
  r.delta = c.take(BHq * g.S * sizeof(float));
  r.absmax = c.take(BHq * (g.N + text_blocks(g)) * sizeof(float2));
  r.ds_exp = c.take((size_t)g.batch * g.Hkv * sizeof(int));
  r.full = c.take(packed_cubes(g, nullptr).shift > 0 ? BHq * (g.N + text_blocks(g)) * sizeof(int) : 0);
  r.d_oc_hat = c.take(of_wide ? BHq * g.N * g.D * sizeof(float) : 0);
  r.dqc = c.take(BHq * g.N * g.D * sizeof(float));
  r.dkc = c.take(BHq * g.N * g.D * sizeof(float));
  r.dvc = c.take(BHq * g.N * g.D * sizeof(float));
  r.pooled = c.take(pooled_layout(g, true).total);
  r.total = c.off;
  return r;
}

// [StatusBlock + rescue list of the fine forward][scratch of the coarse branch on the pooled grid]
size_t fwd_pooled_offset() { return align_up(fine_fwd_tc_workspace_bytes(), 256); }

// 128-token cubes whose halves have eight sub-cubes: the router folds the scores itself
bool router_folds(const Geo& g) { return wide_cube(g) && narrow_geo(g).G == 8; }

// 128-token cubes: the regions above are laid out for the half-cube problem (`n` = narrow_geo), followed by what
// links the two levels: cube-level router scores, half-cube copies of the coarse tensors and of the block map.
struct WideRouteLayout {
  RouteLayout narrow;      // status, qr, kr, lse_r, pr (half-cube scores, unless folded); its selection scratch is unused
  RouteLayout cube;        // selection scratch and pr at cube level, offsets relative to `cube_base`
  size_t cube_base, total;
};
WideRouteLayout wide_route_layout(const Geo& g) {
  WideRouteLayout r;
  r.narrow = route_layout(narrow_geo(g), router_folds(g));
  r.cube = route_layout(g);
  r.cube_base = align_up(r.narrow.hist, 256);     // everything from the half-cube histograms on is not needed
  r.total = r.cube_base + r.cube.total;
  return r;
}
struct WideFwdLayout {
  size_t pooled, x64, oc_hat64, ptr64, idx64, total;
};
WideFwdLayout wide_fwd_layout(const Geo& g) {
  const Geo n = narrow_geo(g);
  WideFwdLayout r;
  Carver c;
  const size_t BHq = (size_t)g.batch * g.Hq;
  c.take(fine_fwd_tc_workspace_bytes());
  r.pooled = c.take(pooled_layout(g, false).total);
  r.x64 = c.take(BHq * n.N * n.D * sizeof(float));
  r.oc_hat64 = c.take(BHq * n.N * n.D * sizeof(float));
  r.ptr64 = c.take(BHq * (n.N + 1) * sizeof(int));
  r.idx64 = c.take(BHq * (size_t)n.nnz_cap * sizeof(int));
  r.total = c.off;
  return r;
}
struct WideBwdLayout {
  BwdLayout narrow;        // status, delta, absmax, ds_exp, d_oc_hat, dqc, dkc, dvc at half-cube level (pooled unused)
  BwdLayout cube;          // d_oc_hat, dqc, dkc, dvc, pooled at cube level, offsets relative to `cube_base`
  size_t cube_base, oc_hat64, ptr64, idx64, cptr64, ridx64, total;
};
WideBwdLayout wide_bwd_layout(const Geo& g) {
  const Geo n = narrow_geo(g);
  WideBwdLayout r;
  r.narrow = bwd_layout(n, true);
  r.cube = bwd_layout(g, true);
  r.cube_base = align_up(r.narrow.pooled, 256);
  Carver c;
  c.off = r.cube_base + r.cube.total;
  const size_t BHq = (size_t)g.batch * g.Hq;
  r.oc_hat64 = c.take(BHq * n.N * n.D * sizeof(float));
  r.ptr64 = c.take(BHq * (n.N + 1) * sizeof(int));
  r.idx64 = c.take(BHq * (size_t)n.nnz_cap * sizeof(int));
  r.cptr64 = c.take(BHq * (n.N + 1) * sizeof(int));
  r.ridx64 = c.take(BHq * (size_t)n.nnz_cap * sizeof(int));
  r.total = c.off;
  return r;
}

// One-pass router (router_tc.cu): half-cubes, or 64-token cubes, of eight sub-cubes.  Asked for from kRouterOneTiles key tiles on.  Below, the launches that settle the map (4 per query, 11 per sequence) cost more than the exponentials:
// whole route call, two-pass / one-pass, us: 7,056 tiles (336 cubes, 16 heads of 64 channels) 189 / 208; 7,776 tiles (288 cubes, 24
// heads) 203 / 223; 18,252 tiles (624 cubes, 12 heads) 322 / 273; 81,000 tiles (1440 cubes, 10 heads) 1145 / 873.
constexpr long long kRouterOneTiles = 12000;
constexpr int kSettlePairs = 1 << 17;      // pairs next to a threshold: about one in 10^5 of a problem's
bool router_one_supported(const Geo& g) { return wide_cube(g) ? router_folds(g) && router_one_runs(narrow_geo(g)) : router_one_runs(g); }
struct RouteOneLayout {
  size_t park, lse2, pairs, rows, total;
};
RouteOneLayout route_one_layout(const Geo& g) {
  const Geo r = wide_cube(g) ? narrow_geo(g) : g;
  RouteOneLayout l;
  Carver c;
  l.park = c.take(router_one_park_bytes(r, router_folds(g)));
  l.lse2 = c.take((size_t)g.batch * g.Hq * r.N * r.G * sizeof(float));
  l.pairs = c.take((size_t)kSettlePairs * sizeof(int2));
  l.rows = c.take((size_t)g.batch * g.Hq * g.N * sizeof(int));
  l.total = c.off;
  return l;
}

size_t route_workspace_bytes(const Geo& g) { return wide_cube(g) ? wide_route_layout(g).total : route_layout(g).total; }
size_t fwd_base_bytes(const Geo& g) {
  return wide_cube(g) ? wide_fwd_layout(g).total : align_up(fwd_pooled_offset() + pooled_layout(g, false).total, 256);
}
size_t bwd_base_bytes(const Geo& g) { return wide_cube(g) ? wide_bwd_layout(g).total : align_up(bwd_layout(g, false).total, 256); }
size_t fwd_workspace_bytes(const Geo& g) { return fwd_base_bytes(g) + text_map_layout(g, false).total; }
// fp16 copies of Q and K for the dQ pass (behind the other regions of the backward's workspace)
bool dq_pass_f16(const Geo& g) { return fine_bwd_dq_uses_f16(g); }
size_t bwd_f16_offset(const Geo& g) { return align_up(bwd_base_bytes(g) + text_map_layout(g, true).total, 256); }
size_t bwd_q16_bytes(const Geo& g) { return align_up((size_t)g.batch * g.Hq * g.S * g.D * sizeof(bf16), 256); }
size_t bwd_k16_bytes(const Geo& g) { return align_up((size_t)g.batch * g.Hkv * g.S * g.D * sizeof(bf16), 256); }
// GQA groups: fp16 copies of V and dO as well, for the all-fp16 dK/dV pass (behind the copies of Q and K)
bool dkv_pass_gqa_f16(const Geo& g) { return dq_pass_f16(g) && fine_bwd_dkv_gqa_uses_f16(g); }
size_t bwd_workspace_bytes(const Geo& g) {
  if (!dq_pass_f16(g)) return bwd_base_bytes(g) + text_map_layout(g, true).total;
  size_t n = bwd_f16_offset(g) + bwd_q16_bytes(g) + bwd_k16_bytes(g);
  if (dkv_pass_gqa_f16(g)) n += bwd_k16_bytes(g) + bwd_q16_bytes(g);      // V like K, dO like Q
  return n;
}

// dS tiles that the dK/dV pass leaves for the dQ pass (fine_bwd_dq_ds_tc.cu), in a scratch region of the caller's (offsets are
// relative to it): 8 KB per kept pair of 64-token blocks, for as many KV groups at a time as fit.  Without room for one group
// the dQ pass recomputes dS.  The preferred size stops at kStoredDsBytes of tiles (9 heads of 720p top-64, one group of the
// 16..256-cube budget with four heads a group): a launch over fewer blocks loses more on its last, unevenly filled items
// (one head of 720p at a time: 10 blocks per SM), more scratch gains nothing.
constexpr size_t kStoredDsBytes = (size_t)7 << 30;
// 128-token cubes keep dS where both passes run on 128 x 128 tiles: a tile of 32 KB per pair of cubes, places and orders of the
// cube map.  219,600 tokens, 10 heads, top-64, backward: 33.8 ms without, 31.9 with a head (4 GB) at a time, 31.8 with four
constexpr size_t kStoredDsBytesWide = (size_t)8 << 30;      // two such heads
bool wide_stored_ds(const Geo& g) { return g.Lt == 0 && g.rep == 1 && !fine_bwd_dkv_wants_pair(g) && fine_bwd128_supported(narrow_geo(g)); }
struct DsLayout {
  size_t counters, pos, order, tiles, total;
  int groups;          // KV groups per chunk, 0: no stored dS
};
DsLayout ds_layout(const Geo& g, size_t avail, bool preferred) {
  DsLayout r{};
  const bool wide = wide_cube(g);
  if (!dq_pass_f16(g) || (wide && !wide_stored_ds(g))) return r;
  const Geo x = g.Lt > 0 ? text_geo(g) : g;
  const size_t tokens = wide ? 2 * kBlockTokens : kBlockTokens;
  const size_t all = (size_t)g.batch * g.Hkv, group = (size_t)x.rep * x.nnz_cap * tokens * tokens * sizeof(bf16);
  if (group == 0) return r;
  Carver c;
  r.counters = c.take(2 * all * sizeof(int));
  r.pos = c.take((size_t)g.batch * g.Hq * x.nnz_cap * sizeof(int));
  r.order = c.take(all * x.N * sizeof(int));
  r.tiles = c.off;
  const size_t room = preferred ? (wide ? kStoredDsBytesWide : kStoredDsBytes) : avail > r.tiles ? avail - r.tiles : 0;
  // (the dK/dV pass counts the tiles of a chunk in an int)
  const size_t most = 0x7fffffffULL / ((size_t)x.rep * x.nnz_cap);
  size_t fit = room / group < all ? room / group : all;
  if (fit > most) fit = most;
  if (fit == 0) return r;
  const size_t chunks = (all + fit - 1) / fit;
  r.groups = (int)((all + chunks - 1) / chunks);
  r.total = r.tiles + r.groups * group;
  return r;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
bool aligned256(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 255u) == 0; }

// The kernels are built for sm_100a only.  (A device's answer does not change: it is asked once.)
int check_device() {
  static std::atomic<int> known[kMaxDevices];      // compute capability major
  int dev = 0, major = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return VSA2_ERR_CUDA;
  if (dev < kMaxDevices) major = known[dev].load(std::memory_order_relaxed);
  if (major == 0) {
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return VSA2_ERR_CUDA;
    if (dev < kMaxDevices) known[dev].store(major, std::memory_order_relaxed);
  }
  return major == 10 ? VSA2_OK : VSA2_ERR_UNSUPPORTED;
}

template <typename T>
T* at(void* ws, size_t off) { return reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(ws) + off); }

cudaError_t g_last_cuda_error = cudaSuccess;

#define VSA2_CUDA(call)                              \
  do {                                               \
    cudaError_t e_ = (call);                         \
    if (e_ != cudaSuccess) {                         \
      g_last_cuda_error = e_;                        \
      return VSA2_ERR_CUDA;                          \
    }                                                \
  } while (0)

}  // namespace

namespace vsa2 {
cudaError_t sm_count(int* sms) {
  static std::atomic<int> known[kMaxDevices];
  int dev = 0, n = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev < kMaxDevices) n = known[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if ((e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (dev < kMaxDevices) known[dev].store(n, std::memory_order_relaxed);
  }
  *sms = n;
  return cudaSuccess;
}

// the driver's number of the current context, never given twice in a process; 0 if there is none yet (or it cannot be had)
static unsigned long long context_id() {
  typedef CUresult (*GetId)(CUcontext, unsigned long long*);
  static const GetId get_id = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult found;
    const bool ok = cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &found) == cudaSuccess && found == cudaDriverEntryPointSuccess;
    return ok ? reinterpret_cast<GetId>(p) : nullptr;
  }();
  unsigned long long id = 0;
  return get_id != nullptr && get_id(nullptr, &id) == CUDA_SUCCESS && id < 1ull << 44 ? id : 0;
}

cudaError_t prepare_kernel(const void* kernel, KernelAttr& attr, size_t smem, int threads, int least_registers) {
  int dev = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  const unsigned long long ctx = dev < kMaxDevices ? context_id() : 0;      // 0: not known, ask the driver every time
  auto allowed = [&] {
    const unsigned long long k = attr.known[dev].load(std::memory_order_acquire);
    return ctx != 0 && k >> 20 == ctx && (k & 0xfffffu) >= smem;
  };
  if (ctx != 0 && allowed()) return cudaSuccess;
  std::lock_guard<std::mutex> lock(attr.lock);        // (the limit only grows: two threads must not lower it for each other)
  if (ctx != 0 && allowed()) return cudaSuccess;
  if (least_registers > 0) {
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, kernel)) != cudaSuccess) return e;
    if (fa.numRegs * threads < least_registers) return cudaErrorLaunchOutOfResources;
  }
  if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  if (ctx != 0) attr.known[dev].store(ctx << 20 | smem, std::memory_order_release);
  return cudaSuccess;
}

cudaError_t cluster_room(const void* kernel, ClusterRoom& room, int ctas, int threads, size_t smem, bool* fits) {
  int dev = 0, clusters = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  const unsigned long long ctx = dev < kMaxDevices ? context_id() : 0;
  if (ctx != 0) {
    const unsigned long long k = room.known[dev].load(std::memory_order_relaxed);
    if (k >> 1 == ctx) {
      *fits = k & 1;
      return cudaSuccess;
    }
  }
  if ((e = prepare_kernel(kernel, room.attr, smem)) != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = ctas;
  cfg.blockDim = threads;
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {(unsigned)ctas, 1, 1};
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) {      // (as good as no room; the error is not left behind)
    clusters = 0;
    cudaGetLastError();
  }
  *fits = clusters > 0;
  if (ctx != 0) room.known[dev].store(ctx << 1 | (unsigned long long)*fits, std::memory_order_relaxed);
  return cudaSuccess;
}

void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

ProfScope::ProfScope(int kernel_id, cudaStream_t stream) : id(kernel_id), st(stream) {
  if (g_prof_start[id] != nullptr) cudaEventRecord(g_prof_start[id], st);
}
ProfScope::~ProfScope() {
  if (g_prof_stop[id] != nullptr) cudaEventRecord(g_prof_stop[id], st);
}
}  // namespace vsa2

extern "C" {

int vsa2_profile_events(int32_t kernel_id, void* start_event, void* stop_event) {
  if (kernel_id < 0 || kernel_id >= VSA2_KERNEL_COUNT) return VSA2_ERR_INVALID_ARG;
  g_prof_start[kernel_id] = reinterpret_cast<cudaEvent_t>(start_event);
  g_prof_stop[kernel_id] = reinterpret_cast<cudaEvent_t>(stop_event);
  return VSA2_OK;
}

int64_t vsa2_launch_count(void) { return g_launches.load(); }

int32_t vsa2_debug_rescue_capacity(int32_t capacity) {
  set_fwd_rescue_capacity(capacity);
  return fwd_rescue_capacity();
}

const char* vsa2_last_cuda_error(void) { return cudaGetErrorString(g_last_cuda_error); }

int vsa2_query_sizes(const vsa2_params* p, vsa2_sizes* out) {
  if (out == nullptr) return VSA2_ERR_INVALID_ARG;
  Geo g;
  int rc = fill_geo(p, &g);
  if (rc != VSA2_OK) return rc;
  memset(out, 0, sizeof(*out));
  out->n_cubes = g.N;
  out->n_subcubes = g.G;
  out->block_tokens = g.Bt * g.Bh * g.Bw;
  out->topk_eff = g.K;
  out->seq_len = g.L;
  out->nnz_cap = g.nnz_cap;
  const long long BHq = (long long)g.batch * g.Hq, BHk = (long long)g.batch * g.Hkv;
  out->ptr_elems = BHq * (g.N + 1);
  out->idx_elems = BHq * g.nnz_cap;
  out->pooled_q_elems = BHq * g.N * g.D;
  out->pooled_kv_elems = BHk * g.N * g.D;
  out->lse_c_elems = BHq * g.N;
  out->o_res_elems = g.out_f32 ? 0 : BHq * (long long)g.S * g.D;
  out->tokens_per_head = g.S;
  out->text_blocks = text_blocks(g);
  out->route_workspace_bytes = route_workspace_bytes(g);
  out->fwd_workspace_bytes = fwd_workspace_bytes(g);
  out->bwd_workspace_bytes = bwd_workspace_bytes(g);
  return VSA2_OK;
}

size_t vsa2_attn_bwd_scratch_bytes(const vsa2_params* p) {
  Geo g;
  return fill_geo(p, &g) == VSA2_OK ? ds_layout(g, 0, true).total : 0;
}

size_t vsa2_attn_bwd_preferred_workspace_bytes(const vsa2_params* p) {
  Geo g;
  if (fill_geo(p, &g) != VSA2_OK) return 0;
  const size_t least = bwd_workspace_bytes(g), scratch = ds_layout(g, 0, true).total;
  return scratch > 0 ? align_up(least, 256) + scratch : least;
}

int vsa2_route(const vsa2_params* p, const void* q, const void* k, const int32_t* budgets, const vsa2_map* map,
               void* workspace, size_t workspace_bytes, void* cuda_stream) {
  return vsa2_route_scratch(p, q, k, budgets, map, workspace, workspace_bytes, nullptr, 0, cuda_stream);
}

size_t vsa2_route_scratch_bytes(const vsa2_params* p) {
  Geo g;
  if (fill_geo(p, &g) != VSA2_OK || !router_one_supported(g)) return 0;
  const Geo r = wide_cube(g) ? narrow_geo(g) : g;
  const long long tiles = ((long long)r.N * r.G + 127) / 128;
  return g.batch * g.Hq * tiles * tiles >= kRouterOneTiles ? route_one_layout(g).total : 0;
}

int vsa2_route_scratch(const vsa2_params* p, const void* q, const void* k, const int32_t* budgets, const vsa2_map* map,
                       void* workspace, size_t workspace_bytes, void* scratch, size_t scratch_bytes, void* cuda_stream) {
  Geo g;
  int rc = fill_geo(p, &g);
  if (rc != VSA2_OK) return rc;
  if (!q || !k || !map || !workspace || !map->row_ptr || !map->col_idx || !map->col_ptr || !map->row_idx)
    return VSA2_ERR_INVALID_ARG;
  if (g.mode == VSA2_PER_QUERY_BUDGET && budgets == nullptr) return VSA2_ERR_INVALID_ARG;
  if (g.mode == VSA2_PER_QUERY_BUDGET && (g.flags & VSA2_FLAG_GROUP_ROUTING)) return VSA2_ERR_UNSUPPORTED;
  if (!aligned16(q) || !aligned16(k) || !aligned256(workspace) || !aligned256(scratch)) return VSA2_ERR_MISALIGNED;
  if (workspace_bytes < route_workspace_bytes(g)) return VSA2_ERR_WORKSPACE_TOO_SMALL;
  if ((rc = check_device()) != VSA2_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  // 128-token cubes: sub-cube means and router scores at half-cube level (`r`), folded to cube scores; the
  // selection then runs on the cube-level matrix
  const bool wide = wide_cube(g);
  const Geo r = wide ? narrow_geo(g) : g;
  const bool folded = router_folds(g);
  const RouteLayout rl = route_layout(r, folded);
  RouteLayout lay = rl;
  unsigned char* sel_base = reinterpret_cast<unsigned char*>(workspace);
  if (wide) {
    const WideRouteLayout wl = wide_route_layout(g);
    lay = wl.cube;
    sel_base += wl.cube_base;
  }
  StatusBlock* status = at<StatusBlock>(workspace, rl.status);
  bf16* qr = at<bf16>(workspace, rl.qr);
  bf16* kr = at<bf16>(workspace, rl.kr);
  {
    ProfScope ps(VSA2_KERNEL_POOL_ROUTER, st);
    VSA2_CUDA(launch_pool_router(r, reinterpret_cast<const bf16*>(q), reinterpret_cast<const bf16*>(k), qr, kr, status, st));
  }
  float* pr = folded ? at<float>(sel_base, lay.pr) : at<float>(workspace, rl.pr);
  const bool group_sum = (g.flags & VSA2_FLAG_GROUP_ROUTING) && g.rep > 1;
  const RouteOneLayout ol = router_one_supported(g) ? route_one_layout(g) : RouteOneLayout{};
  const bool one = router_one_supported(g) && scratch != nullptr && scratch_bytes >= ol.total;
  int* redo = one ? &status->pad[0] : nullptr;      // (the status block is cleared by the pooling)
  float* lse2 = one ? at<float>(scratch, ol.lse2) : nullptr;
  if (router_tc_supported(r)) {
    { ProfScope lse(VSA2_KERNEL_ROUTER_LSE, st); }      // (both passes are timed as the second)
    ProfScope ps(VSA2_KERNEL_ROUTER_POOL, st);
    if (one) VSA2_CUDA(launch_router_one(r, folded, qr, kr, pr, at<unsigned char>(scratch, ol.park), lse2, redo, status, st));
    else VSA2_CUDA(launch_router_scores_tc(r, folded, qr, kr, pr, nullptr, status, st));
  } else   // sub-cube counts the tensor-core kernel has no layout for (G = 1 is the VSA router of Sec. 2.1)
    VSA2_CUDA(launch_router_scores(r, qr, kr, at<float>(workspace, rl.lse_r), pr, st));
  if (wide && !folded) {
    float* pr_cube = at<float>(sel_base, lay.pr);
    VSA2_CUDA(launch_fold_scores(r, pr, pr_cube, st));
    pr = pr_cube;
  }
  if (group_sum) VSA2_CUDA(launch_group_sum_scores(g, pr, nullptr, st));
  workspace = sel_base;
  SelectScratch s;
  s.hist = at<unsigned>(workspace, lay.hist);
  s.state = at<unsigned>(workspace, lay.state);
  s.row_tau = at<float>(workspace, lay.row_tau);
  s.row_eq_take = at<int>(workspace, lay.row_eq_take);
  s.row_cnt = at<int>(workspace, lay.row_cnt);
  s.row_gt = at<int>(workspace, lay.row_gt);
  s.row_eq = at<int>(workspace, lay.row_eq);
  s.bitmap = at<unsigned>(workspace, lay.bitmap);
  s.bitmap_t = at<unsigned>(workspace, lay.bitmap_t);
  s.words = lay.words;
  {
    ProfScope ps(VSA2_KERNEL_SELECT, st);
    if (one) {
      const Settle se{redo, &status->pad[1], at<int2>(scratch, ol.pairs), kSettlePairs, &status->pad[2], at<int>(scratch, ol.rows)};
      VSA2_CUDA(launch_select_band(g, pr, budgets, s, se, st));
      VSA2_CUDA(launch_router_exact(r, folded, qr, kr, lse2, se.pairs, se.count, se.cap, group_sum ? g.rep : 1, redo, pr, status, st));
      VSA2_CUDA(launch_select_settle(g, pr, budgets, s, se, st));
      // (these and the thresholds of launch_select return at once unless the flag is up)
      VSA2_CUDA(launch_router_scores_tc(r, folded, qr, kr, pr, redo, status, st));
      if (group_sum) VSA2_CUDA(launch_group_sum_scores(g, pr, redo, st));
    }
    VSA2_CUDA(launch_select(g, pr, budgets, s, redo, map->row_ptr, map->col_idx, map->col_ptr, map->row_idx, status, st));
  }
  return VSA2_OK;
}

const float* vsa2_route_scores(const vsa2_params* p, const void* workspace) {
  Geo g;
  if (workspace == nullptr || fill_geo(p, &g) != VSA2_OK) return nullptr;
  size_t off = route_layout(g).pr;
  if (wide_cube(g)) {
    const WideRouteLayout wl = wide_route_layout(g);
    off = wl.cube_base + wl.cube.pr;
  }
  return reinterpret_cast<const float*>(reinterpret_cast<const unsigned char*>(workspace) + off);
}

int vsa2_attn_fwd(const vsa2_params* p, const void* q, const void* k, const void* v, const float* gate,
                  const vsa2_map* map, void* o, float* lse, const vsa2_saved* saved, void* workspace,
                  size_t workspace_bytes, void* cuda_stream) {
  Geo g;
  int rc = fill_geo(p, &g);
  if (rc != VSA2_OK) return rc;
  if (!q || !k || !v || !map || !o || !lse || !workspace || !map->row_ptr || !map->col_idx) return VSA2_ERR_INVALID_ARG;
  const bool coarse = !(g.flags & VSA2_FLAG_NO_COARSE);
  if (coarse && (!saved || !saved->qc || !saved->kc || !saved->vc || !saved->oc_hat || !saved->lse_c))
    return VSA2_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned256(workspace))
    return VSA2_ERR_MISALIGNED;
  if (saved != nullptr && !g.out_f32 && saved->o_res != nullptr && !aligned16(saved->o_res)) return VSA2_ERR_MISALIGNED;
  if (workspace_bytes < fwd_workspace_bytes(g)) return VSA2_ERR_WORKSPACE_TOO_SMALL;
  if ((rc = check_device()) != VSA2_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  StatusBlock* status = reinterpret_cast<StatusBlock*>(workspace);      // cleared by the first launch
  if (!coarse) VSA2_CUDA(cudaMemsetAsync(status, 0, sizeof(StatusBlock), st));
  const bf16* qb = reinterpret_cast<const bf16*>(q);
  const bf16* kb = reinterpret_cast<const bf16*>(k);
  const bf16* vb = reinterpret_cast<const bf16*>(v);
  // 128-token cubes: the fine kernels run on the half-cube problem `n` with the expanded map; the coarse branch
  // runs at cube level from folded half-cube means
  const bool wide = wide_cube(g);
  const Geo n = wide ? narrow_geo(g) : g;
  const WideFwdLayout wl = wide ? wide_fwd_layout(g) : WideFwdLayout();
  const size_t pooled_off = wide ? wl.pooled : fwd_pooled_offset();
  const int* row_ptr = map->row_ptr;
  const int* col_idx = map->col_idx;
  const float* oc_hat = coarse ? saved->oc_hat : nullptr;
  if (coarse) {
    {
      ProfScope ps(VSA2_KERNEL_POOL, st);
      if (!wide) {
        VSA2_CUDA(launch_pool_coarse(g, qb, kb, vb, saved->qc, saved->kc, saved->vc, status, st));
      } else {
        float* x64 = at<float>(workspace, wl.x64);
        VSA2_CUDA(launch_pool(n, qb, n.Hq, nullptr, x64, status, st));
        VSA2_CUDA(launch_fold_mean(n, n.Hq, x64, saved->qc, st));
        VSA2_CUDA(launch_pool(n, kb, n.Hkv, nullptr, x64, nullptr, st));
        VSA2_CUDA(launch_fold_mean(n, n.Hkv, x64, saved->kc, st));
        VSA2_CUDA(launch_pool(n, vb, n.Hkv, nullptr, x64, nullptr, st));
        VSA2_CUDA(launch_fold_mean(n, n.Hkv, x64, saved->vc, st));
      }
    }
    {
      ProfScope ps(VSA2_KERNEL_COARSE_FWD, st);
      if (!(g.flags & VSA2_FLAG_BF16_COARSE_FWD))
        VSA2_CUDA(launch_coarse_fwd_mma(g, saved->qc, saved->kc, saved->vc, saved->oc_hat, saved->lse_c, st));
      else
        VSA2_CUDA(launch_coarse_fwd_pooled(g, saved->qc, saved->kc, saved->vc, saved->oc_hat, saved->lse_c,
                                           at<unsigned char>(workspace, pooled_off),
                                           reinterpret_cast<StatusBlock*>(workspace), st));
      if (wide) {
        VSA2_CUDA(launch_expand_rows(n, n.Hq, false, saved->oc_hat, at<float>(workspace, wl.oc_hat64), st));
        oc_hat = at<float>(workspace, wl.oc_hat64);
      }
    }
  }
  if (wide) {
    VSA2_CUDA(launch_expand_map(n, map->row_ptr, map->col_idx, at<int>(workspace, wl.ptr64), at<int>(workspace, wl.idx64), st));
    row_ptr = at<int>(workspace, wl.ptr64);
    col_idx = at<int>(workspace, wl.idx64);
  }
  bf16* o_res = (saved != nullptr && !g.out_f32) ? reinterpret_cast<bf16*>(saved->o_res) : nullptr;
  Geo fx = n;                                   // geometry of the fine kernels' block problem
  if (g.Lt > 0) {
    // text tokens: append the text blocks to the map (in the workspace) and run the kernels on the block problem
    // (with 128-token cubes the half-cube map built above is what gets extended, and the 64-token kernels run)
    const TextMapLayout tl = text_map_layout(g, false);
    unsigned char* tbase = at<unsigned char>(workspace, fwd_base_bytes(g));
    fx = text_geo(n);
    if (!fine_fwd_rows_supported(fx)) return VSA2_ERR_UNSUPPORTED;
    VSA2_CUDA(launch_extend_map(n, text_blocks(g), row_ptr, col_idx, at<int>(tbase, tl.ptr), at<int>(tbase, tl.idx),
                                fx.nnz_cap, st));
    row_ptr = at<int>(tbase, tl.ptr);
    col_idx = at<int>(tbase, tl.idx);
  }
  {
    ProfScope ps(VSA2_KERNEL_FINE_FWD, st);
    if (g.flags & VSA2_FLAG_EXACT_MAX_FWD)
      VSA2_CUDA(launch_fine_fwd(fx, qb, kb, vb, coarse ? gate : nullptr, row_ptr, col_idx, oc_hat, o, o_res, lse, st));
    else if ((wide || (g.flags & VSA2_FLAG_GROUP_ROUTING)) && fine_fwd_rows2_supported(n, !wide))
      // 128 query rows per tile: the halves of a 128-token cube, or two heads of a group that share their map
      VSA2_CUDA(launch_fine_fwd_rows2_tc(n, !wide, qb, kb, vb, coarse ? gate : nullptr, row_ptr, col_idx, oc_hat, o, o_res, lse,
                                         reinterpret_cast<StatusBlock*>(workspace), st));
    else if (fine_fwd_rows_supported(fx))
      VSA2_CUDA(launch_fine_fwd_rows_tc(fx, qb, kb, vb, coarse ? gate : nullptr, row_ptr, col_idx, oc_hat, o, o_res, lse,
                                        reinterpret_cast<StatusBlock*>(workspace), st));
    else
      VSA2_CUDA(launch_fine_fwd_tc(n, qb, kb, vb, coarse ? gate : nullptr, row_ptr, col_idx, oc_hat, o, o_res, lse,
                                   reinterpret_cast<StatusBlock*>(workspace), st));
  }
  return VSA2_OK;
}

int vsa2_attn_bwd(const vsa2_params* p, const void* q, const void* k, const void* v, const float* gate,
                  const vsa2_map* map, const void* o, const float* lse, const vsa2_saved* saved, const void* d_o,
                  void* dq, void* dk, void* dv, float* dgate, void* workspace, size_t workspace_bytes,
                  void* cuda_stream) {
  Geo g;
  int rc = fill_geo(p, &g);
  if (rc != VSA2_OK) return rc;
  // (what the workspace holds beyond the least serves as the scratch; the checks of the call come first)
  const size_t least = align_up(bwd_workspace_bytes(g), 256);
  const bool more = workspace != nullptr && workspace_bytes > least;
  return vsa2_attn_bwd_scratch(p, q, k, v, gate, map, o, lse, saved, d_o, dq, dk, dv, dgate, workspace, workspace_bytes,
                               more ? at<unsigned char>(workspace, least) : nullptr, more ? workspace_bytes - least : 0, cuda_stream);
}

int vsa2_attn_bwd_scratch(const vsa2_params* p, const void* q, const void* k, const void* v, const float* gate,
                          const vsa2_map* map, const void* o, const float* lse, const vsa2_saved* saved, const void* d_o,
                          void* dq, void* dk, void* dv, float* dgate, void* workspace, size_t workspace_bytes, void* scratch,
                          size_t scratch_bytes, void* cuda_stream) {
  Geo g;
  int rc = fill_geo(p, &g);
  if (rc != VSA2_OK) return rc;
  if (!q || !k || !v || !map || !o || !lse || !d_o || !dq || !dk || !dv || !workspace || !map->row_ptr ||
      !map->col_idx || !map->col_ptr || !map->row_idx)
    return VSA2_ERR_INVALID_ARG;
  const bool coarse = !(g.flags & VSA2_FLAG_NO_COARSE) && gate != nullptr;
  if (coarse && (!saved || !saved->qc || !saved->kc || !saved->vc || !saved->oc_hat || !saved->lse_c))
    return VSA2_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned16(d_o) || !aligned16(dq) ||
      !aligned16(dk) || !aligned16(dv) || !aligned256(workspace) || !aligned256(scratch))
    return VSA2_ERR_MISALIGNED;
  if (workspace_bytes < bwd_workspace_bytes(g)) return VSA2_ERR_WORKSPACE_TOO_SMALL;
  if ((rc = check_device()) != VSA2_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  // (the status block is cleared by the preprocess: the first kernel that could write it comes after)
  // 128-token cubes: preprocess and the fine passes run on the half-cube problem `n` (regions `lay`), the coarse
  // backward at cube level (regions `cl` behind `cube_ws`); folds and expansions link the two
  const bool wide = wide_cube(g);
  const Geo n = wide ? narrow_geo(g) : g;
  const WideBwdLayout wl = wide ? wide_bwd_layout(g) : WideBwdLayout();
  const BwdLayout lay = wide ? wl.narrow : bwd_layout(g, false);
  const BwdLayout cl = wide ? wl.cube : lay;
  void* cube_ws = wide ? at<unsigned char>(workspace, wl.cube_base) : workspace;
  const bf16* qb = reinterpret_cast<const bf16*>(q);
  const bf16* kb = reinterpret_cast<const bf16*>(k);
  const bf16* vb = reinterpret_cast<const bf16*>(v);
  const bf16* dob = reinterpret_cast<const bf16*>(d_o);
  float* delta = at<float>(workspace, lay.delta);
  float* d_oc_hat = at<float>(workspace, lay.d_oc_hat);      // (128-token cubes)
  float* dqc = at<float>(workspace, lay.dqc);
  float* dkc = at<float>(workspace, lay.dkc);
  float* dvc = at<float>(workspace, lay.dvc);
  float* d_oc_hat_cube = at<float>(cube_ws, cl.d_oc_hat);
  float* dqc_cube = at<float>(cube_ws, cl.dqc);
  float* dkc_cube = at<float>(cube_ws, cl.dkc);
  float* dvc_cube = at<float>(cube_ws, cl.dvc);
  const int* row_ptr = map->row_ptr;
  const int* col_idx = map->col_idx;
  const int* col_ptr = map->col_ptr;
  const int* row_idx = map->row_idx;
  const float* oc_hat = coarse ? saved->oc_hat : nullptr;
  if (wide) {
    VSA2_CUDA(launch_expand_map(n, map->row_ptr, map->col_idx, at<int>(workspace, wl.ptr64), at<int>(workspace, wl.idx64), st));
    VSA2_CUDA(launch_expand_map(n, map->col_ptr, map->row_idx, at<int>(workspace, wl.cptr64), at<int>(workspace, wl.ridx64), st));
    row_ptr = at<int>(workspace, wl.ptr64);
    col_idx = at<int>(workspace, wl.idx64);
    col_ptr = at<int>(workspace, wl.cptr64);
    row_idx = at<int>(workspace, wl.ridx64);
    if (coarse) {
      VSA2_CUDA(launch_expand_rows(n, n.Hq, false, saved->oc_hat, at<float>(workspace, wl.oc_hat64), st));
      oc_hat = at<float>(workspace, wl.oc_hat64);
    }
  }
  Geo fx = n;                                   // geometry of the fine kernels' block problem
  if (g.Lt > 0) {
    const TextMapLayout tl = text_map_layout(g, true);
    unsigned char* tbase = at<unsigned char>(workspace, bwd_base_bytes(g));
    fx = text_geo(n);
    VSA2_CUDA(launch_extend_map(n, text_blocks(g), row_ptr, col_idx, at<int>(tbase, tl.ptr), at<int>(tbase, tl.idx),
                                fx.nnz_cap, st));
    VSA2_CUDA(launch_extend_map(n, text_blocks(g), col_ptr, row_idx, at<int>(tbase, tl.cptr), at<int>(tbase, tl.ridx),
                                fx.nnz_cap, st));
    row_ptr = at<int>(tbase, tl.ptr);
    col_idx = at<int>(tbase, tl.idx);
    col_ptr = at<int>(tbase, tl.cptr);
    row_idx = at<int>(tbase, tl.ridx);
  }
  if (!coarse && dgate != nullptr)
    VSA2_CUDA(cudaMemsetAsync(dgate, 0, (size_t)g.batch * g.Hq * g.L * sizeof(float), st));
  const bf16* o_res = (saved != nullptr && !g.out_f32) ? reinterpret_cast<const bf16*>(saved->o_res) : nullptr;
  // (V is copied to fp16 for GQA groups only; O is of V's size or, a mean of up to a few thousand rows, well below it)
  const DsScale scale{at<float2>(workspace, lay.absmax), at<int>(workspace, lay.ds_exp), dkv_pass_gqa_f16(g) ? pow2i(-16) : 0.f};
  unsigned char* pooled_ws = at<unsigned char>(cube_ws, cl.pooled);
  const PooledInputs pooled = coarse && !wide ? pooled_bwd_inputs(g, saved->qc, saved->kc, saved->vc, nullptr, pooled_ws) : PooledInputs{};
  {
    ProfScope ps(VSA2_KERNEL_BWD_PRE, st);
    VSA2_CUDA(launch_bwd_preprocess(fx, dob, o, o_res, coarse ? gate : nullptr, oc_hat, delta, coarse ? dgate : nullptr,
                                    wide ? d_oc_hat : nullptr, coarse && !wide ? pooled.y[3] : nullptr, coarse && !wide ? pooled_bwd_delta(g, pooled_ws) : nullptr,
                                    dq_pass_f16(g) ? at<float2>(workspace, lay.absmax) : nullptr,
                                    reinterpret_cast<StatusBlock*>(workspace), st));
  }
  // dS kept from the dK/dV pass for the dQ pass, which then runs inside it; otherwise the dQ pass recomputes dS and runs first
  const DsLayout dl = ds_layout(g, scratch != nullptr ? scratch_bytes : 0, false);
  const int ds_groups = dl.groups;
  // (a few items per SM end together whatever their order)
  int sms = 0;
  VSA2_CUDA(sm_count(&sms));
  const Geo& dg = wide ? g : fx;                // geometry of the lists by which the tiles of dS are placed
  int* dkv_order = ds_groups > 0 && (long long)ds_groups * dg.N > 4 * sms ? at<int>(scratch, dl.order) : nullptr;
  // (64-token tiles; the dK/dV pass packs where it stores dS)
  const PackedCubes pk = ds_groups > 0 && !wide ? packed_cubes(fx, at<int>(workspace, lay.full)) : PackedCubes{};
  const StoredDs sd{at<unsigned char>(scratch, dl.tiles), at<int>(scratch, dl.pos), at<int>(scratch, dl.counters), dkv_order, ds_groups,
                    wide ? map->row_ptr : row_ptr, wide ? map->col_idx : col_idx, coarse ? dqc : nullptr, dq};
  // cubes of 128 tokens: both passes on 128 x 128 tiles
  const bool wide128 = wide && g.Lt == 0 && fine_bwd128_supported(n);
  {
    // what the passes below read beside the tensors (cubes of 128 tokens: the inputs of the coarse backward come from its own launches)
    ProfScope ps(VSA2_KERNEL_FINE_BWD_DQ, st);
    const PrepLists lists{sd.row_ptr, sd.col_idx, wide ? map->col_ptr : col_ptr, wide ? map->row_idx : row_idx, at<int>(scratch, dl.pos), sd.counters,
                          2 * g.batch * g.Hkv, pk.shift > 0 ? at<int>(workspace, lay.full) : nullptr, pk.first, dkv_order};
    const bool pooled_here = coarse && !wide;
    if (ds_groups > 0 || pooled_here)
      VSA2_CUDA(launch_bwd_prep(ds_groups > 0 ? &fx : nullptr, qb, at<unsigned char>(workspace, bwd_f16_offset(g)), kb,
                                at<unsigned char>(workspace, bwd_f16_offset(g) + bwd_q16_bytes(g)), scale,
                                &reinterpret_cast<StatusBlock*>(workspace)->pad[kRangeFlagSlot], ds_groups > 0 ? &dg : nullptr, lists,
                                pooled_here ? &pooled : nullptr, st));
  }
  if (coarse) {
    // pooled grid: dQ, dK/dV (+ two group spreads); cubes of 128 tokens: first the bf16 copies with the dense map and the pooled preprocess
    ProfScope ps(VSA2_KERNEL_COARSE_BWD, st);
    if (wide) VSA2_CUDA(launch_fold_sum(n, n.Hq, d_oc_hat, d_oc_hat_cube, st));
    VSA2_CUDA(launch_coarse_bwd_pooled(g, saved->qc, saved->kc, saved->vc, saved->oc_hat, saved->lse_c, wide ? d_oc_hat_cube : nullptr,
                                       dqc_cube, dkc_cube, dvc_cube, pooled_ws,
                                       reinterpret_cast<StatusBlock*>(workspace), st));
    if (wide) {
      VSA2_CUDA(launch_expand_rows(n, n.Hq, true, dqc_cube, dqc, st));
      VSA2_CUDA(launch_expand_rows(n, n.Hq, true, dkc_cube, dkc, st));
      VSA2_CUDA(launch_expand_rows(n, n.Hq, true, dvc_cube, dvc, st));
    }
  }
  if (ds_groups == 0) {
    const bool f16 = dq_pass_f16(g);     // the copy, the fp16 form, the (idle) fallback
    ProfScope ps(VSA2_KERNEL_FINE_BWD_DQ, st);
    if (wide128)
      VSA2_CUDA(launch_fine_bwd128_dq_tc(n, qb, kb, vb, dob, lse, delta, row_ptr, col_idx, coarse ? dqc : nullptr, dq,
                                         reinterpret_cast<StatusBlock*>(workspace), st,
                                         f16 ? at<unsigned char>(workspace, bwd_f16_offset(g)) : nullptr,
                                         f16 ? at<unsigned char>(workspace, bwd_f16_offset(g) + bwd_q16_bytes(g)) : nullptr, &scale));
    else
      VSA2_CUDA(launch_fine_bwd_dq_tc(fx, qb, kb, vb, dob, lse, delta, row_ptr, col_idx, coarse ? dqc : nullptr, dq,
                                      reinterpret_cast<StatusBlock*>(workspace), st,
                                      f16 ? at<unsigned char>(workspace, bwd_f16_offset(g)) : nullptr,
                                      f16 ? at<unsigned char>(workspace, bwd_f16_offset(g) + bwd_q16_bytes(g)) : nullptr, &scale));
  }
  {
    const bool dkv128 = wide128 && !fine_bwd_dkv_wants_pair(n);
    const bool two = !dkv128 && fine_bwd_dkv_splits_long_columns(fx, true);
    const bool gqa16 = !dkv128 && dkv_pass_gqa_f16(g);    // (the copy of V and dO, the all-fp16 form, the pair form as its fallback)
    const bool f16 = (two || gqa16 || ds_groups > 0) && dq_pass_f16(g);      // fp16 copies of Q and K have been made
    ProfScope ps(VSA2_KERNEL_FINE_BWD_DKV, st);
    unsigned char* v16 = gqa16 ? at<unsigned char>(workspace, bwd_f16_offset(g) + bwd_q16_bytes(g) + bwd_k16_bytes(g)) : nullptr;
    if (dkv128 && ds_groups > 0)
      VSA2_CUDA(launch_fine_bwd128_stored(n, qb, kb, vb, dob, lse, delta, row_ptr, col_idx, col_ptr, row_idx, coarse ? dqc : nullptr,
                                          coarse ? dkc : nullptr, coarse ? dvc : nullptr, dq, dk, dv,
                                          reinterpret_cast<StatusBlock*>(workspace), st, at<unsigned char>(workspace, bwd_f16_offset(g)),
                                          at<unsigned char>(workspace, bwd_f16_offset(g) + bwd_q16_bytes(g)), scale.exp, sd));
    else if (dkv128)
      VSA2_CUDA(launch_fine_bwd128_dkv_tc(n, qb, kb, vb, dob, lse, delta, col_ptr, row_idx, coarse ? dkc : nullptr,
                                          coarse ? dvc : nullptr, dk, dv, reinterpret_cast<StatusBlock*>(workspace), st,
                                          dq_pass_f16(g) ? at<unsigned char>(workspace, bwd_f16_offset(g)) : nullptr,
                                          dq_pass_f16(g) ? at<unsigned char>(workspace, bwd_f16_offset(g) + bwd_q16_bytes(g)) : nullptr,
                                          scale.exp));
    else
      VSA2_CUDA(launch_fine_bwd_dkv_tc(fx, qb, kb, vb, dob, lse, delta, col_ptr, row_idx, coarse ? dkc : nullptr,
                                       coarse ? dvc : nullptr, dk, dv, reinterpret_cast<StatusBlock*>(workspace), st, true,
                                       f16 ? at<unsigned char>(workspace, bwd_f16_offset(g)) : nullptr,
                                       f16 ? at<unsigned char>(workspace, bwd_f16_offset(g) + bwd_q16_bytes(g)) : nullptr, v16,
                                       gqa16 ? v16 + bwd_k16_bytes(g) : nullptr, ds_groups > 0 ? &sd : nullptr, scale.exp, pk));
  }
  return VSA2_OK;
}

int vsa2_permute_cube_major(const vsa2_params* p, int32_t heads, int32_t inverse, const void* src, void* dst,
                            void* cuda_stream) {
  Geo g;
  int rc = fill_geo(p, &g);
  if (rc != VSA2_OK) return rc;
  if (!src || !dst || heads <= 0 || heads > 65535) return VSA2_ERR_INVALID_ARG;
  if (!aligned16(src) || !aligned16(dst)) return VSA2_ERR_MISALIGNED;
  if ((rc = check_device()) != VSA2_OK) return rc;
  VSA2_CUDA(launch_permute(g, reinterpret_cast<const bf16*>(src), heads, inverse != 0, reinterpret_cast<bf16*>(dst),
                           reinterpret_cast<cudaStream_t>(cuda_stream)));
  return VSA2_OK;
}

int vsa2_gate_fwd(const vsa2_params* p, int32_t hidden, const void* x, const void* w_g, float* gate, void* cuda_stream) {
  Geo g;
  int rc = fill_geo(p, &g);
  if (rc != VSA2_OK) return rc;
  if (!x || !w_g || !gate) return VSA2_ERR_INVALID_ARG;
  if (!gate_supported(hidden, g.Hq)) return VSA2_ERR_UNSUPPORTED;
  if (!aligned16(x)) return VSA2_ERR_MISALIGNED;
  if ((rc = check_device()) != VSA2_OK) return rc;
  VSA2_CUDA(launch_gate_fwd(g.batch, g.L, hidden, g.Hq, reinterpret_cast<const bf16*>(x), reinterpret_cast<const bf16*>(w_g),
                            gate, reinterpret_cast<cudaStream_t>(cuda_stream)));
  return VSA2_OK;
}

size_t vsa2_gate_bwd_workspace_bytes(const vsa2_params* p, int32_t hidden) {
  Geo g;
  if (fill_geo(p, &g) != VSA2_OK || !gate_supported(hidden, g.Hq)) return 0;
  return gate_bwd_workspace_bytes(g.batch, g.L, hidden, g.Hq);
}

int vsa2_gate_bwd(const vsa2_params* p, int32_t hidden, const void* x, const void* w_g, const float* gate,
                  const float* dgate, float* d_w_g, void* dx, void* workspace, size_t workspace_bytes, void* cuda_stream) {
  Geo g;
  int rc = fill_geo(p, &g);
  if (rc != VSA2_OK) return rc;
  if (!x || !w_g || !gate || !dgate || !d_w_g || !dx || !workspace) return VSA2_ERR_INVALID_ARG;
  if (!gate_supported(hidden, g.Hq)) return VSA2_ERR_UNSUPPORTED;
  if (!aligned16(x) || !aligned16(dx) || !aligned256(workspace)) return VSA2_ERR_MISALIGNED;
  if (workspace_bytes < gate_bwd_workspace_bytes(g.batch, g.L, hidden, g.Hq)) return VSA2_ERR_WORKSPACE_TOO_SMALL;
  if ((rc = check_device()) != VSA2_OK) return rc;
  VSA2_CUDA(launch_gate_bwd(g.batch, g.L, hidden, g.Hq, g.out_f32, reinterpret_cast<const bf16*>(x),
                            reinterpret_cast<const bf16*>(w_g), gate, dgate, d_w_g, dx, workspace,
                            reinterpret_cast<cudaStream_t>(cuda_stream)));
  return VSA2_OK;
}

int vsa2_device_status(const void* workspace, void* cuda_stream, int32_t* status_out) {
  if (workspace == nullptr || status_out == nullptr) return VSA2_ERR_INVALID_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  VSA2_CUDA(cudaStreamSynchronize(st));
  int s = 0;
  VSA2_CUDA(cudaMemcpy(&s, workspace, sizeof(int), cudaMemcpyDeviceToHost));
  *status_out = s;
  return VSA2_OK;
}

const char* vsa2_strerror(int code) {
  switch (code) {
    case VSA2_OK: return "ok";
    case VSA2_ERR_INVALID_ARG: return "invalid argument";
    case VSA2_ERR_UNSUPPORTED: return "unsupported shape, dtype or device (needs sm_100)";
    case VSA2_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
    case VSA2_ERR_MISALIGNED: return "pointer not aligned (16 bytes for tensors, 256 bytes for workspaces)";
    case VSA2_ERR_CUDA: return "CUDA call or kernel launch failed";
    case VSA2_ERR_DEVICE_TIMEOUT: return "a bounded device-side wait ran out";
    case VSA2_ERR_MAP_OVERFLOW: return "more selected blocks than nnz_cap";
    case VSA2_ERR_STATIC_SCRATCH: return "problem needs more scratch than the library's built-in 8 MiB buffer (use vsa2_route)";
    default: return "unknown vsa2 error";
  }
}

}  // extern "C"
