// Shared device/host definitions of the VSA2 library: geometry of the latent grid, index
// maps between raster tokens and cubes (paper Sec. 2.2 "Permutation"), workspace layout.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "vsa2.h"

namespace vsa2 {

typedef __nv_bfloat16 bf16;

constexpr int kBlockTokens = 64;   // tokens per block handled by the kernels (a 128-token cube runs as two)

// Everything a kernel needs to know about the problem; passed by value.
struct Geo {
  int batch, Hq, Hkv, rep, D;
  int T, H, W, L;
  int Bt, Bh, Bw, Nt, Nh, Nw, N;
  int Rt, Rh, Rw, Gt, Gh, Gw, G;
  int K;            // TopK after clamping
  int mode;         // VSA2_PER_*
  int out_f32;      // 1: outputs are fp32, 0: bf16
  int flags;
  float scale;      // softmax scale
  long long nnz_cap;
  // Text tokens (the sentence after Eq. 12): every token tensor holds S = L + Lt rows per head, the L video tokens in raster
  // order followed by Lt text tokens.  The routing and coarse kernels see the video part only (N = Nvid cubes).  The fine
  // kernels and the backward preprocess run on the BLOCK problem: N = Nvid + ceil(Lt / 64) blocks, block j < Nvid is video
  // cube j, block j >= Nvid holds text tokens 64 (j - Nvid) .. ; their maps are the block maps extended by the text blocks.
  int Nvid, Lt, S;
  // ceil(2^32 / d) for d = Nw, Nh, Bw, Bh (geo_set_magics): the index arithmetic of the kernels divides by these with one
  // multiply instead of a reciprocal, which would run on the unit the softmax exponentials need
  unsigned mNw, mNh, mBw, mBh;
};
inline unsigned div_magic(int d) { return d <= 1 ? 0u : (unsigned)((0x100000000ull + (unsigned)d - 1ull) / (unsigned)d); }
// to be called wherever Nw, Nh, Bw or Bh of a Geo are set
inline void geo_set_magics(Geo& g) {
  g.mNw = div_magic(g.Nw);
  g.mNh = div_magic(g.Nh);
  g.mBw = div_magic(g.Bw);
  g.mBh = div_magic(g.Bh);
}

// Status block at the start of every workspace.
struct StatusBlock {
  int status;       // VSA2_OK / VSA2_ERR_DEVICE_TIMEOUT / VSA2_ERR_MAP_OVERFLOW
  int detail;
  int pad[62];
};

// Kernels of a call follow one another on one stream, up to 40 of them, and on small problems most take a few microseconds.  Each is
// launched so that its CTAs may be placed as soon as all CTAs of the kernel before it have started (and finds room), and waits
// in grid_enter for that kernel's completion and its writes: what is left between two kernels is that wait instead of a launch.
// Every kernel enters that way before it reads or writes global memory, also one that has nothing to do: its completion then stands
// for all before it.  A kernel with tensor memory lets its successor in only when it has allocated it (or exits): a successor
// that allocated first would keep it from ending.  The large ones also wait behind their set-up (barriers, tensor memory, tables).
// What a kernel reads may be written while it is already there, waiting: so none of it is read-only for the kernel's lifetime, and no kernel
// reads through __ldg or `const __restrict__` pointers (loads on the read-only path may be moved in front of the wait, and owe
// nothing to it).  `__restrict__` stands only on pointers that a kernel writes and never reads.
// 2048-token clip, 12 heads, training: 216 us without, 189 with the wait at the top of every kernel, 183 so; ragged clip 733, 709, 702.
void count_launch();      // (vsa2_launch_count)
template <typename T> struct NotDeduced { using type = T; };
template <typename... P>
inline cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 typename NotDeduced<P>::type... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  if (e == cudaSuccess) count_launch();
  return e;
}
__device__ __forceinline__ void grid_enter(bool early = true) {
  if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
// The attention kernels let their successor in when they end: beside them it finds no room or takes issue slots from them (all kernels early up to
// eight items per CTA / the router alone, us: 2048-token clip, training 176 / 168; toy grid, as a graph 72 / 62; 480p, 12 heads on 3 6093 / 6039;
// ragged clip 624 / 623; 13 x 27 x 47 tokens, 16 heads 1335 / 1331).  The router lets it in up to eight items per CTA (without: ragged clip 624 / 628).
__device__ __forceinline__ void grid_enter_items(int items) { grid_enter(items <= 8 * (int)gridDim.x); }

// Brackets the launches of one kernel group with the caller's timing events.
struct ProfScope {
  int id;
  cudaStream_t st;
  ProfScope(int kernel_id, cudaStream_t stream);
  ~ProfScope();
};

// Per kernel and device: the dynamic shared memory it has been allowed so far, and the CUDA context in which that was (the limit is a
// context's: another context of the device, or the primary one after a device reset, starts without it).  A launch asks the
// driver only when it needs more or the context is another (each such call costs the host as much as half a launch, and the
// kernels' needs are constants or grow with the problem).
constexpr int kMaxDevices = 64;
struct KernelAttr {
  std::mutex lock;
  std::atomic<unsigned long long> known[kMaxDevices] = {};      // context id << 20 | bytes
};
// `least_registers`: registers the launch has to allocate over all its threads (kernels that redistribute them wait for ever
// otherwise), checked with `threads` on the first call
cudaError_t prepare_kernel(const void* kernel, KernelAttr& attr, size_t smem, int threads = 0, int least_registers = 0);
// Whether the current context has room for a cluster of `ctas` CTAs of the kernel (a MIG slice or a green context may not have the SMs in one GPC):
// asked once per context, of the kernel's largest need `smem`, which is allowed it by this
struct ClusterRoom {
  KernelAttr attr;
  std::atomic<unsigned long long> known[kMaxDevices] = {};      // context id << 1 | answer
};
cudaError_t cluster_room(const void* kernel, ClusterRoom& room, int ctas, int threads, size_t smem, bool* fits);
// number of SMs of the current device (looked up once per device)
cudaError_t sm_count(int* sms);

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// q = n / d, r = n % d for 0 <= n < 2^22 and 0 < d < 2^10 with m = ceil(2^32 / d) (0 for d = 1): floor(n m / 2^32), exact
// while n d < 2^32 -- one multiply.  The tensor-core kernels decode cube and token indices several times per tile; the
// earlier form (a reciprocal and a fix-up) runs on the special-function unit, behind the exponentials of the softmax warps,
// which cost a service warp of the 128-token backward 4000 cycles per tile.  A translation unit that defines
// VSA2_RECIPROCAL_DIVMOD before including this header keeps the reciprocal form (where that measured faster).
// (host and device: vsa2_selftest_divmod checks the multiply form on the host, exhaustively for small divisors)
__host__ __device__ __forceinline__ int mulhi_div(int n, unsigned m) {
  return m == 0u ? n : (int)(((unsigned long long)(unsigned)n * m) >> 32);
}
__device__ __forceinline__ void fast_divmod(int n, int d, unsigned m, int& q, int& r) {
#ifdef VSA2_RECIPROCAL_DIVMOD
  (void)m;
  q = __float2int_rz(__fdividef((float)n, (float)d));
  r = n - q * d;
  if (r < 0) {
    --q;
    r += d;
  } else if (r >= d) {
    ++q;
    r -= d;
  }
#else
  q = mulhi_div(n, m);
  r = n - q * d;
#endif
}

// cube n -> (nt, nh, nw);  n = (nt*Nh + nh)*Nw + nw
__device__ __forceinline__ void cube_coords(const Geo& g, int n, int& nt, int& nh, int& nw) {
  int r;
  fast_divmod(n, g.Nw, g.mNw, r, nw);
  fast_divmod(r, g.Nh, g.mNh, nt, nh);
}

// position (bt, bh, bw) inside cube (nt, nh, nw) -> raster token index, or -1 if padding
__device__ __forceinline__ int cube_token_at(const Geo& g, int nt, int nh, int nw, int bt, int bh, int bw) {
  int t = nt * g.Bt + bt, h = nh * g.Bh + bh, w = nw * g.Bw + bw;
  if (t >= g.T || h >= g.H || w >= g.W) return -1;
  return (t * g.H + h) * g.W + w;
}

// position p in [0, B) inside a cube, ordered (bt, bh, bw) -> raster token index, or -1 if padding
__device__ __forceinline__ int cube_token(const Geo& g, int nt, int nh, int nw, int p) {
  int bw, bh, bt, r;
  fast_divmod(p, g.Bw, g.mBw, r, bw);
  fast_divmod(r, g.Bh, g.mBh, bt, bh);
  return cube_token_at(g, nt, nh, nw, bt, bh, bw);
}

// number of valid tokens of cube n (0 only for the empty trailing half-cubes of a 128-token-cube problem)
__device__ __forceinline__ int cube_count(const Geo& g, int n) {
  int nt, nh, nw;
  cube_coords(g, n, nt, nh, nw);
  int ct = min(g.Bt, g.T - nt * g.Bt), ch = min(g.Bh, g.H - nh * g.Bh), cw = max(0, min(g.Bw, g.W - nw * g.Bw));
  return ct * ch * cw;
}

// router sub-cube gsub of cube n: number of valid tokens (0 = the sub-cube is padding only)
__device__ __forceinline__ int subcube_count(const Geo& g, int n, int gsub) {
  int nt, nh, nw;
  cube_coords(g, n, nt, nh, nw);
  int gw = gsub % g.Gw;
  int r = gsub / g.Gw;
  int gh = r % g.Gh;
  int gt = r / g.Gh;
  int t0 = nt * g.Bt + gt * g.Rt, h0 = nh * g.Bh + gh * g.Rh, w0 = nw * g.Bw + gw * g.Rw;
  int ct = max(0, min(g.Rt, g.T - t0)), ch = max(0, min(g.Rh, g.H - h0)), cw = max(0, min(g.Rw, g.W - w0));
  return ct * ch * cw;
}

// ---- blocks of the fine kernels: video cubes followed by text blocks ---------------------------------------------------
__device__ __forceinline__ bool block_is_text(const Geo& g, int j) { return j >= g.Nvid; }
// TMA box coordinates (dimensions 1..3 of the 5-D maps) of block j: a video cube in the raster map, or 64 rows of the text map
__device__ __forceinline__ void block_box(const Geo& g, int j, int& c1, int& c2, int& c3) {
  if (j < g.Nvid) {
    int jt, jh, jw;
    cube_coords(g, j, jt, jh, jw);
    c1 = jw * g.Bw; c2 = jh * g.Bh; c3 = jt * g.Bt;
  } else {
    c1 = (j - g.Nvid) * kBlockTokens; c2 = 0; c3 = 0;
  }
}
// position p of block j -> row of the token tensors (0 .. S-1), or -1 if padding
__device__ __forceinline__ int block_token(const Geo& g, int j, int p) {
  if (j < g.Nvid) {
    int jt, jh, jw;
    cube_coords(g, j, jt, jh, jw);
    return cube_token(g, jt, jh, jw, p);
  }
  const int t = (j - g.Nvid) * kBlockTokens + p;
  return t < g.Lt ? g.L + t : -1;
}
// valid tokens of block j
__device__ __forceinline__ int block_count(const Geo& g, int j) {
  if (j < g.Nvid) return cube_count(g, j);
  return min(kBlockTokens, g.Lt - (j - g.Nvid) * kBlockTokens);
}
// work item -> (batch * heads index, block).  With text tokens the blocks of a head are handed out in descending order, so
// that the text blocks (whose lists are the longest by far) start first and the persistent CTAs do not end on them.
__device__ __forceinline__ void item_block(const Geo& g, int item, int& bh, int& i) {
  bh = item / g.N;
  const int r = item - bh * g.N;
  i = g.Lt > 0 ? g.N - 1 - r : r;
}
__device__ __forceinline__ int block_item(const Geo& g, int bh, int i) { return bh * g.N + (g.Lt > 0 ? g.N - 1 - i : i); }

__device__ __forceinline__ void store_out(void* base, size_t idx, float v, int out_f32) {
  if (out_f32) reinterpret_cast<float*>(base)[idx] = v;
  else reinterpret_cast<bf16*>(base)[idx] = __float2bfloat16_rn(v);
}

// ---------------------------------------------------------------------------------------------
// launchers implemented in the .cu files (all enqueue on `st`, return cudaGetLastError())
// ---------------------------------------------------------------------------------------------
// (`clear`: null, or a status block that the launch sets to zero for the kernels behind it)
cudaError_t launch_pool(const Geo& g, const bf16* x, int heads, bf16* xr, float* xc, StatusBlock* clear, cudaStream_t st);
cudaError_t launch_pool_router(const Geo& g, const bf16* q, const bf16* k, bf16* qr, bf16* kr, StatusBlock* clear, cudaStream_t st);
cudaError_t launch_pool_coarse(const Geo& g, const bf16* q, const bf16* k, const bf16* v, float* qc, float* kc, float* vc,
                               StatusBlock* clear, cudaStream_t st);

// raster <-> cube-major copy of a [batch, heads, L or N*B, D] bf16 tensor (pool.cu)
cudaError_t launch_permute(const Geo& g, const bf16* src, int heads, bool inverse, bf16* dst, cudaStream_t st);

cudaError_t launch_router_scores(const Geo& g, const bf16* qr, const bf16* kr, float* lse_r, float* pr,
                                 cudaStream_t st);

// tensor-core router (router_tc.cu), both passes in one launch; with `fold` (half-cubes of 8 sub-cubes, N even) the scores
// come out at the level of the 128-token cubes, bit for bit what launch_fold_scores makes of the others
bool router_tc_supported(const Geo& g);
// (`redo`: null, or the flag without which the launch does nothing)
cudaError_t launch_router_scores_tc(const Geo& g, bool fold, const bf16* qr, const bf16* kr, float* pr, int* redo, StatusBlock* status,
                                    cudaStream_t st);
// the one-pass form and the two-pass scores of listed pairs (router_tc.cu), where router_one_runs
bool router_one_runs(const Geo& g);
size_t router_one_park_bytes(const Geo& g, bool fold);
cudaError_t launch_router_one(const Geo& g, bool fold, const bf16* qr, const bf16* kr, float* pr, void* park, float* lse2, int* redo,
                              StatusBlock* status, cudaStream_t st);
cudaError_t launch_router_exact(const Geo& g, bool fold, const bf16* qr, const bf16* kr, const float* lse2, const int2* pairs,
                                const int* count, int cap, int heads, const int* redo, float* pr, StatusBlock* status, cudaStream_t st);

// up to this many cubes one block per head turns the selection into both maps (select.cu): 128 cubes 4.7 us against 12 us and
// five more launches; at 288 cubes the block takes 40 us and the six launches 18
constexpr int kSelOneBlockN = 128;
struct SelectScratch {
  unsigned* hist;        // [BH][3][2048]
  unsigned* state;       // [BH][8]
  float* row_tau;        // [BH][N]
  int* row_eq_take;      // [BH][N]
  int* row_cnt;          // [BH][N]
  int* row_gt;           // [BH][N]
  int* row_eq;           // [BH][N]
  unsigned* bitmap;      // [BH][N][words]   rows x column words
  unsigned* bitmap_t;    // [BH][N][words]   columns x row words
  int words;             // ceil(N/32)
};
// Selection on one-pass scores (select.cu): thresholds and the lists of what lies next to them (launch_select_band), the two-pass
// scores of those (launch_router_exact), the decision (launch_select_settle); then launch_select with `redo`, which finds
// everything in place or, should the flag be up, starts again from two-pass scores.
struct Settle {
  int* redo;           // raised when the two-pass form has to be run after all
  int* count;          // listed pairs
  int2* pairs;         // [cap] {(batch * Hq + head) * N + row, column}
  int cap;
  int* row_count;      // per-row modes: listed rows
  int* rows;           // [B * Hq * N]
};
cudaError_t launch_select_band(const Geo& g, const float* pr, const int* budgets, const SelectScratch& s, const Settle& se, cudaStream_t st);
cudaError_t launch_select_settle(const Geo& g, const float* pr, const int* budgets, const SelectScratch& s, const Settle& se,
                                 cudaStream_t st);
cudaError_t launch_select(const Geo& g, const float* pr, const int* budgets, const SelectScratch& s, const int* redo,
                          int* row_ptr, int* col_idx, int* col_ptr, int* row_idx, StatusBlock* status,
                          cudaStream_t st);

// coarse branch forward on the fp32 cube means, TF32 tensor-core products with register-resident accumulators
// (coarse_fwd_mma.cu)
cudaError_t launch_coarse_fwd_mma(const Geo& g, const float* qc, const float* kc, const float* vc, float* oc_hat,
                                  float* lse_c, cudaStream_t st);

cudaError_t launch_fine_fwd(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const float* gate,
                            const int* row_ptr, const int* col_idx, const float* oc_hat, void* o, bf16* o_res,
                            float* lse, cudaStream_t st);

// coarse branch through the fine-branch kernels on the pooled grid (coarse_pooled.cu); offsets into a scratch region
struct PooledLayout {
  size_t status, q16, k16, v16, ptr, idx, do16, delta, dk_kv, dv_kv, total;
};
Geo pooled_geo(const Geo& g);
PooledLayout pooled_layout(const Geo& g, bool backward);
cudaError_t launch_coarse_fwd_pooled(const Geo& g, const float* qc, const float* kc, const float* vc, float* oc_hat,
                                     float* lse_c, void* workspace, StatusBlock* caller_status, cudaStream_t st);
cudaError_t launch_coarse_bwd_pooled(const Geo& g, const float* qc, const float* kc, const float* vc, const float* oc_hat,
                                     const float* lse_c, const float* d_oc_hat, float* dqc, float* dkc, float* dvc,
                                     void* workspace, StatusBlock* caller_status, cudaStream_t st);

// cubes of 128 tokens as pairs of 64-token half-cubes (wide_cube.cu); `narrow` is narrow_geo() of the problem
bool wide_cube(const Geo& g);
Geo narrow_geo(const Geo& g);
cudaError_t launch_fold_scores(const Geo& narrow, const float* pr64, float* pr, cudaStream_t st);
// "group head" routing: replaces every block score by the sum over the query heads of its KV group (in place)
cudaError_t launch_group_sum_scores(const Geo& g, float* pr, const int* redo, cudaStream_t st);      // (`redo`: null, or the flag without which nothing happens)
cudaError_t launch_fold_mean(const Geo& narrow, int heads, const float* x64, float* x, cudaStream_t st);
cudaError_t launch_fold_sum(const Geo& narrow, int heads, const float* x64, float* x, cudaStream_t st);
cudaError_t launch_expand_rows(const Geo& narrow, int heads, bool by_count, const float* x, float* x64,
                               cudaStream_t st);
cudaError_t launch_expand_map(const Geo& narrow, const int* ptr, const int* idx, int* ptr64, int* idx64,
                              cudaStream_t st);
// block map of the video cubes (g: the video problem) -> block map with `text_blocks` text blocks appended to every row and
// all-ones text rows; capx = capacity per (batch, head) of idxx
cudaError_t launch_extend_map(const Geo& g, int text_blocks, const int* ptr, const int* idx, int* ptrx, int* idxx, long long capx,
                              cudaStream_t st);

// gate projection and its backward (gate.cu)
bool gate_supported(int hidden, int heads);
size_t gate_bwd_workspace_bytes(int batch, int L, int hidden, int heads);
cudaError_t launch_gate_fwd(int batch, int L, int C, int Hq, const bf16* x, const bf16* w, float* gate, cudaStream_t st);
cudaError_t launch_gate_bwd(int batch, int L, int C, int Hq, int out_f32, const bf16* x, const bf16* w, const float* gate,
                            const float* dgate, float* d_w, void* dx, void* workspace, cudaStream_t st);

// tensor-core forward (fine_fwd_tc.cu); `status` heads a workspace of fine_fwd_tc_workspace_bytes()
size_t fine_fwd_tc_workspace_bytes();
int fwd_rescue_capacity();
void set_fwd_rescue_capacity(int cap);
cudaError_t launch_fine_fwd_tc(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const float* gate,
                               const int* row_ptr, const int* col_idx, const float* oc_hat, void* o, bf16* o_res,
                               float* lse, StatusBlock* status, cudaStream_t st);

// tensor-core forward with the queries in the accumulator rows (fine_fwd_rows_tc.cu); same workspace as launch_fine_fwd_tc
bool fine_fwd_rows_supported(const Geo& g);
cudaError_t launch_fine_fwd_rows_tc(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const float* gate,
                                    const int* row_ptr, const int* col_idx, const float* oc_hat, void* o, bf16* o_res,
                                    float* lse, StatusBlock* status, cudaStream_t st);

// tensor-core forward with two query blocks (128 rows) per tile (fine_fwd_rows2_tc.cu): the halves of a 128-token cube, or one
// block of two heads that share their map.  `g`, the map and oc_hat are those of the half-cube problem (or, with pair_heads,
// of the ordinary 64-token problem); the workspace is the one of launch_fine_fwd_tc
bool fine_fwd_rows2_supported(const Geo& g, bool pair_heads);
cudaError_t launch_fine_fwd_rows2_tc(const Geo& g, bool pair_heads, const bf16* q, const bf16* k, const bf16* v, const float* gate,
                                     const int* row_ptr, const int* col_idx, const float* oc_hat, void* o, bf16* o_res,
                                     float* lse, StatusBlock* status, cudaStream_t st);

// Scale of dS in the passes that round it to fp16: 2^exp per KV group.  dS is a weight of about one over the kept keys times a
// sum over dO V, so an unscaled fp16 dS has lost its bits to the subnormals long before dO is small (dO of 1e-4, 4096 keys: a
// few per cent of dQ; of 1e-7: all of it).  The exponent lifts max|dO| max|O| of the group to 2^-3 (O is a mean of V rows, so it
// is of V's size wherever a weight is large) and is never negative: gradients of ordinary size keep exponent 0, and a dS that
// the scale takes beyond the fp16 range ends in the range fallback like any other.  It is folded into the row statistics
// (lse, or delta where dO itself is a scaled copy) and taken out again by the epilogues, both exact.
struct DsScale {
  const float2* absmax;   // [B, Hq, N of the block problem]: max |dO|, max |O| of each block (launch_bwd_preprocess)
  int* exp;               // [B, Hkv], written by launch_bwd_prep or launch_cast_qk
  // 0, or (where dP is formed from an fp16 copy of V) the max |O| below which a group's V counts as too small for that copy and
  // the range flag goes up: an element of it is then good to 2^-9 of V's size at worst
  float least_o;
};
__host__ __device__ __forceinline__ float pow2i(int e) {      // 2^e, |e| <= 126
  union { int i; float f; } u{(127 + e) << 23};
  return u.f;
}

// tensor-core backward passes for cubes of 128 tokens (fine_bwd128_tc.cu): `g` and the maps are those of the half-cube problem
bool fine_bwd128_supported(const Geo& g);
bool fine_bwd_dkv_wants_pair(const Geo& g);
cudaError_t launch_fine_bwd128_dq_tc(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const bf16* d_o,
                                     const float* lse, const float* delta, const int* row_ptr, const int* col_idx,
                                     const float* dqc, void* dq, StatusBlock* status, cudaStream_t st, void* q16, void* k16,
                                     const DsScale* scale);
cudaError_t launch_fine_bwd128_dkv_tc(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const bf16* d_o,
                                      const float* lse, const float* delta, const int* col_ptr, const int* row_idx,
                                      const float* dkc, const float* dvc, void* dk, void* dv, StatusBlock* status,
                                      cudaStream_t st, const void* q16, const void* k16, const int* ds_exp);

// tensor-core backward passes (fine_bwd_tc.cu)
cudaError_t launch_fine_bwd_dq_tc(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const bf16* d_o,
                                  const float* lse, const float* delta, const int* row_ptr, const int* col_idx,
                                  const float* dqc, void* dq, StatusBlock* status, cudaStream_t st, void* q16, void* k16,
                                  const DsScale* scale, StatusBlock* report = nullptr,       // (report: the status block written to, if not `status`)
                                  bool beside = false);      // the launch that comes next is a dK/dV pass with `beside`
bool fine_bwd_dq_uses_f16(const Geo& g);
// Slot of StatusBlock.pad that holds the range flag of the fp16 dQ passes (the slot behind it: the fallback launch's counter)
constexpr int kRangeFlagSlot = 8;
// fp16 copies of Q and K; a finite value beyond the fp16 range sets *range_flag.  Also forms scale->exp
cudaError_t launch_cast_qk(const Geo& g, const bf16* q, void* q16, const bf16* k, void* k16, const DsScale& scale, int* range_flag,
                           cudaStream_t st);
// fp16 copies of V and of dO times 2^ds_exp of its KV group, with the same flag
cudaError_t launch_cast_v_do(const Geo& g, const bf16* v, void* v16, const bf16* d_o, void* do16, const int* ds_exp, int* range_flag,
                             cudaStream_t st);
// Query cubes of a last layer of frames that the grid cuts, packed by the dK/dV pass: the tokens of such a cube are the first rows of
// its 64-row tile (positions run frame by frame), so 2^shift of them share one tile.  Grids of 4n + 1 latent frames, which causal
// video encoders make, leave one frame of four there: at 21 frames a sixth of all query blocks is a quarter of a tile.
struct PackedCubes {
  int shift;          // 1 or 2; 0: not packed
  int first;          // first cube of the layer; its cubes are the last of the video, and of every (ascending) list
  const int* full;    // [B, Hq, N]: entries of a column list in front of them
};
PackedCubes packed_cubes(const Geo& g, const int* full);
// dS kept between the two backward passes (fine_bwd_dq_ds_tc.cu, fine_bwd128_dq_ds_tc.cu): scratch for the pairs of `chunk_groups`
// KV groups at a time.  On 128 x 128 tiles every size and list below is that of the cube map.
struct StoredDs {
  void* scratch;        // chunk_groups * rep * nnz_cap tiles of 8 KB (64 queries x 64 keys, fp16), or of 32 KB (128 x 128)
  const int* pos;       // [B, Hq, nnz_cap], filled by launch_bwd_prep
  int* counters;        // two words per chunk, cleared by launch_bwd_prep
  int* order;           // null, or [B, Hkv, N]: items of the dK/dV pass, longest lists of a group first (launch_bwd_prep)
  int chunk_groups;
  const int* row_ptr;
  const int* col_idx;
  const float* dqc;
  void* dq;
};
// The backward's preparation in one launch (bwd_prep.cu), each part where its pointer is given: the fp16 copies of Q and K (`fine`: geometry of
// the fine passes) as launch_cast_qk makes them; the lists of the dS tiles; the inputs of the coarse backward.
struct PrepLists {
  const int *row_ptr, *col_idx, *col_ptr, *row_idx;
  int* pos;             // StoredDs::pos and counters
  int* counters;
  int n_counters;
  int* full;            // null, or PackedCubes::full, with the first cube of the layer
  int first;
  int* order;           // null, or StoredDs::order
};
struct PooledInputs;
cudaError_t launch_bwd_prep(const Geo* fine, const bf16* q, void* q16, const bf16* k, void* k16, const DsScale& scale, int* range_flag,
                            const Geo* lists_geo, const PrepLists& lists, const PooledInputs* pooled, cudaStream_t st);
cudaError_t launch_fine_bwd_dq_ds(const Geo& g, const void* k16, const void* ds, int head0, int heads, const int* row_ptr,
                                  const int* col_idx, const float* dqc, void* dq, StatusBlock* status, int* range_flag,
                                  int* item_counter, bool swizzled, const int* ds_exp, const PackedCubes& pk, cudaStream_t st);
cudaError_t launch_fine_bwd128_dq_ds(const Geo& g, long long cap, const void* k16, const void* ds, int head0, int heads,
                                     const int* row_ptr, const int* col_idx, const float* dqc, void* dq, StatusBlock* status,
                                     int* range_flag, int* item_counter, const int* ds_exp, cudaStream_t st);
cudaError_t launch_fine_bwd128_stored(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const bf16* d_o, const float* lse,
                                      const float* delta, const int* row_ptr, const int* col_idx, const int* col_ptr,
                                      const int* row_idx, const float* dqc, const float* dkc, const float* dvc, void* dq, void* dk,
                                      void* dv, StatusBlock* status, cudaStream_t st, const void* q16, const void* k16,
                                      const int* ds_exp, const StoredDs& sd);
cudaError_t launch_fine_bwd_dq_fallback(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const bf16* d_o, const float* lse,
                                        const float* delta, const int* row_ptr, const int* col_idx, const float* dqc, void* dq,
                                        StatusBlock* status, cudaStream_t st);
cudaError_t launch_fine_bwd_dkv_tc(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const bf16* d_o,
                                   const float* lse, const float* delta, const int* col_ptr, const int* row_idx,
                                   const float* dkc, const float* dvc, void* dk, void* dv, StatusBlock* status,
                                   cudaStream_t st, bool split_long_columns, const void* q16,
                                   const void* k16, void* v16, void* do16, const StoredDs* sd, const int* ds_exp,
                                   const PackedCubes& pk = PackedCubes{}, StatusBlock* report = nullptr,
                                   bool beside = false);     // it may run beside the dQ pass launched just before it with `beside` (same inputs)
bool fine_bwd_dkv_gqa_uses_f16(const Geo& g);
bool fine_bwd_dkv_splits_long_columns(const Geo& g, bool split_long_columns);

cudaError_t launch_bwd_preprocess(const Geo& g, const bf16* d_o, const void* o, const bf16* o_res, const float* gate,
                                  const float* oc_hat, float* delta, float* dgate, float* d_oc_hat, bf16* do_c, float* delta_c,
                                  float2* absmax, StatusBlock* clear, cudaStream_t st);
}  // namespace vsa2
