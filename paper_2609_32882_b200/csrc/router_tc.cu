// Router block scores (paper Eq. 6-7) on the Blackwell tensor cores, two passes as in the paper's kernel
// description (Sec. 2.2 "Kernel Implementation"): pass 1 accumulates the row log-sum-exp of
// Q_r K_r^T * scale, pass 2 recomputes the scores, applies the softmax and pools G x G sub-blocks on chip.
//
// A CTA owns 128 consecutive pooled queries (128/G query cubes) of one head and streams the head's pooled
// keys twice, in tiles of 128 through a TMA ring; S [128 q, 128 keys] lands in tensor memory (four buffers).
// Both passes over an item run in one launch: the row statistics stay in shared memory, and a problem of a few items pays the
// start of one kernel instead of two.
// Four compute threads own each query row, 32 key columns of every tile each (a single warp per scheduler keeps
// the exponential unit only half busy); pass 1 merges their running (max, sum) pairs once per item.  The G
// rows of a query cube sit in G adjacent lanes: their pooled sums are combined with warp shuffles.
// Both passes are bound by the exponential unit (one ex2 per score: 1024 cycles per tile of ~1250), not by the tensor pipe.
// A buffer of scores is given back as soon as they are in registers (720p, 40 heads: 3.27 -> 3.22 ms; fetching the next tile's
// scores before a tile is worked on made it 3.58).
#include "tc_attn.cuh"

namespace vsa2 {

constexpr int kRtParts = 4;        // compute threads per pooled query row (each owns 128 / kRtParts key columns of a tile)
constexpr int kRtThreads = 64 + 128 * kRtParts;    // TMA warp, MMA warp, 4 * kRtParts compute warps
constexpr int kRtSlots = 4;
constexpr int kRtTile = 128;
constexpr int kRtBufs = 4;         // score tiles in tensor memory (4 x 128 columns = all of it)

template <int D>
struct RouterTc {
  static constexpr int DH = D / 64;
  static constexpr uint32_t HALF = kRtTile * 128;          // 128 rows x 64 channels
  static constexpr uint32_t TILE = DH * HALF;
  static constexpr uint32_t OFF_Q = kRtSlots * TILE;
  static constexpr uint32_t OFF_MISC = OFF_Q + TILE;
  static constexpr uint32_t MISC_BYTES = 4096;
  static size_t smem_bytes(int valid_words) { return OFF_MISC + MISC_BYTES + (size_t)valid_words * 4 + 1024; }
};

struct RouterMisc {
  uint64_t q_full, q_empty;
  uint64_t k_full[kRtSlots], k_empty[kRtSlots];
  uint64_t s_full[kRtBufs], s_free[kRtBufs];
  uint64_t part_ready, lse_ready;   // between the passes: part_stats written, row_lse2 written
  uint32_t tmem_base;
  int abort_flag;
  float2 part_stats[kRtParts - 1][128];   // (running max, running sum) of the threads of parts 1 .. kRtParts-1
  float row_lse2[128];                    // log2 sum_{valid keys} 2^(s * scale * log2 e) of the item's rows
};

// tensor map over pooled operands [BH, N*G, D] bf16: box = 64 channels x 128 rows x 1
inline bool make_pooled_tmap(CUtensorMap* out, const void* base, int D, int rows_per_head, int heads_total) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)rows_per_head, (cuuint64_t)heads_total};
  cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)rows_per_head * D * 2};
  cuuint32_t box[3] = {64, kRtTile, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* m, uint64_t* bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(tc::smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(tc::smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

// Pass 1 on 32 scores of a row: running maximum (in the exponent's units) and sum.  The maximum is taken over the raw scores
// (the scale is positive) and the scale folded into the exponent's multiply-add.
__device__ __forceinline__ void rt_accumulate(uint32_t (&s)[32], uint32_t kbits, float c2, float& m_run, float& l_run) {
  float cmax = -INFINITY;
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    if (kbits != 0xffffffffu && !((kbits >> c) & 1u)) s[c] = 0xff800000u;      // -inf
    cmax = fmaxf(cmax, __uint_as_float(s[c]));
  }
  if (cmax > -INFINITY) {
    const float m_new = fmaxf(m_run, cmax * c2);
    float acc = 0.f;
#pragma unroll
    for (int c = 0; c < 32; ++c) acc += ex2_approx(fmaf(__uint_as_float(s[c]), c2, -m_new));
    l_run = l_run * ex2_approx(m_run - m_new) + acc;
    m_run = m_new;
  }
}

// Pass 2 on 32 scores of a row: softmax, column sums of the 32 / G key cubes, then the sum over the G rows of the query cube,
// which sit in G adjacent lanes: a butterfly that halves the values a lane carries at every step (4 shuffles instead of
// 3 per key cube) and leaves each total in one lane -- that of cube `mine` of the 32 / G.
template <int G>
__device__ __forceinline__ float rt_pool(const uint32_t (&s)[32], uint32_t kbits, float c2, float lse2, int lane, int& mine) {
  static_assert(G == 8 || G == 16, "router pooling layout");
  float p[32];
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    p[c] = ex2_approx(fmaf(__uint_as_float(s[c]), c2, -lse2));
    if (kbits != 0xffffffffu) p[c] = ((kbits >> c) & 1u) ? p[c] : 0.f;
  }
  float tv[32 / G];
#pragma unroll
  for (int cc = 0; cc < 32 / G; ++cc) {
    float tot = 0.f;
#pragma unroll
    for (int c = 0; c < G; ++c) tot += p[cc * G + c];
    tv[cc] = tot;
  }
  float t;
  if constexpr (G == 8) {
    const bool hi4 = lane & 4, hi2 = lane & 2;
    const float k0 = hi4 ? tv[2] : tv[0], k1 = hi4 ? tv[3] : tv[1];
    const float s0 = hi4 ? tv[0] : tv[2], s1 = hi4 ? tv[1] : tv[3];
    const float u0 = k0 + __shfl_xor_sync(0xffffffffu, s0, 4), u1 = k1 + __shfl_xor_sync(0xffffffffu, s1, 4);
    t = (hi2 ? u1 : u0) + __shfl_xor_sync(0xffffffffu, hi2 ? u0 : u1, 2);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    mine = (hi4 ? 2 : 0) + (hi2 ? 1 : 0);
  } else {
    const bool hi8 = lane & 8;
    t = (hi8 ? tv[1] : tv[0]) + __shfl_xor_sync(0xffffffffu, hi8 ? tv[0] : tv[1], 8);
    t += __shfl_xor_sync(0xffffffffu, t, 4);
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    mine = hi8 ? 1 : 0;
  }
  return t;
}

// Writes P_r of the blocks of `g` or, with FOLD (G = 8), of the 128-token cubes whose half-cubes those blocks are: the scores of the
// four pairs of halves, weighted with the valid query sub-cubes of each half (wide_cube.cu, fold_scores_kernel).
template <int D, int G, bool FOLD>
__global__ void __launch_bounds__(kRtThreads, 1)
router_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, Geo g,
                 float* __restrict__ pr, StatusBlock* status) {
  static_assert(!FOLD || G == 8, "half-cubes of 8 sub-cubes");
  using C = RouterTc<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* q_tile = smem + C::OFF_Q;
  RouterMisc* misc = reinterpret_cast<RouterMisc*>(smem + C::OFF_MISC);
  uint32_t* valid_bits = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC + C::MISC_BYTES);   // one bit per pooled token

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NG = g.N * g.G;
  const int row_tiles = (NG + kRtTile - 1) / kRtTile;
  const int total_items = g.batch * g.Hq * row_tiles;
  const int valid_words = (row_tiles * kRtTile) / 32;
  const float c2 = g.scale * 1.4426950408889634f;

  // validity of every pooled token of the sequence (a sub-cube that is padding only is invalid)
  for (int w = warp; w < valid_words; w += blockDim.x >> 5) {       // (a warp per word, a lane per token)
    const int r = w * 32 + lane;
    const uint32_t bits = __ballot_sync(0xffffffffu, r < NG && subcube_count(g, r / G, r % G) > 0);
    if (lane == 0) valid_bits[w] = bits;
  }
  if (tid == 0) {
    misc->abort_flag = 0;
    tc::mbar_init(&misc->q_full, 1);
    tc::mbar_init(&misc->q_empty, 1);
    for (int s = 0; s < kRtSlots; ++s) {
      tc::mbar_init(&misc->k_full[s], 1);
      tc::mbar_init(&misc->k_empty[s], 1);
    }
    for (int s = 0; s < kRtBufs; ++s) {
      tc::mbar_init(&misc->s_full[s], 1);
      tc::mbar_init(&misc->s_free[s], 4 * kRtParts);       // one arrival per compute warp
    }
    tc::mbar_init(&misc->part_ready, 128 * (kRtParts - 1));
    tc::mbar_init(&misc->lse_ready, 128);
    tc::fence_barrier_init();
    tc::prefetch_tmap(&tm_q);
    tc::prefetch_tmap(&tm_k);
  }
  if (warp == 1) {
    tc::tmem_alloc(&misc->tmem_base, 128 * kRtBufs);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = misc->tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      uint32_t seq = 0, n_items = 0;
      for (int item = blockIdx.x; item < total_items; item += gridDim.x, ++n_items) {
        const int rt = item % row_tiles, bhq = item / row_tiles;
        const int b = bhq / g.Hq, hq = bhq % g.Hq, bhk = b * g.Hkv + hq / g.rep;
        VSA2_WAIT(&misc->q_empty, (n_items & 1) ^ 1);
        tc::mbar_expect_tx(&misc->q_full, C::TILE);
        for (int h = 0; h < C::DH; ++h) tma_load_3d(q_tile + h * C::HALF, &tm_q, &misc->q_full, h * 64, rt * kRtTile, bhq);
        for (int step = 0; step < 2 * row_tiles; ++step, ++seq) {       // pass 1, then pass 2
          const int kt = step < row_tiles ? step : step - row_tiles;
          const uint32_t slot = seq % kRtSlots, par = (seq / kRtSlots) & 1;
          VSA2_WAIT(&misc->k_empty[slot], par ^ 1);
          tc::mbar_expect_tx(&misc->k_full[slot], C::TILE);
          for (int h = 0; h < C::DH; ++h)
            tma_load_3d(smem + slot * C::TILE + h * C::HALF, &tm_k, &misc->k_full[slot], h * 64, kt * kRtTile, bhk);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = tc::idesc_bf16(128, 128, false, false);
      const uint32_t q_addr = tc::smem_u32(q_tile), slot0 = tc::smem_u32(smem);
      uint32_t seq = 0, n_items = 0;
      for (int item = blockIdx.x; item < total_items; item += gridDim.x, ++n_items) {
        VSA2_WAIT(&misc->q_full, n_items & 1);
        for (int step = 0; step < 2 * row_tiles; ++step, ++seq) {
          const uint32_t slot = seq % kRtSlots, buf = seq % kRtBufs;
          VSA2_WAIT(&misc->k_full[slot], (seq / kRtSlots) & 1);
          VSA2_WAIT(&misc->s_free[buf], ((seq / kRtBufs) & 1) ^ 1);
          tc::tc_fence_after();
          const uint32_t k_addr = slot0 + slot * C::TILE;
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const uint32_t aa = q_addr + (ks / 4) * C::HALF + (ks % 4) * 32;
            const uint32_t bb = k_addr + (ks / 4) * C::HALF + (ks % 4) * 32;
            tc::mma_ss(tmem_base + buf * 128, tc::smem_desc_sw128(aa, 16, 1024), tc::smem_desc_sw128(bb, 16, 1024), idesc,
                       ks > 0);
          }
          tc::mma_commit(&misc->s_full[buf]);
          tc::mma_commit(&misc->k_empty[slot]);
          if (step == 2 * row_tiles - 1) tc::mma_commit(&misc->q_empty);
        }
      }
    }
  } else {
    const int quad = warp & 3;                   // tensor-memory lane quadrant of this warp
    const int part = (warp - 2) >> 2;            // which 32 key columns of every tile
    const int row = (quad << 5) | lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + part * 32;
    uint32_t seq = 0, n_items = 0;
    // this thread's 32 scores of tile `seq`
    uint32_t s[32];
    auto fetch = [&]() -> bool {
      const uint32_t buf = seq % kRtBufs;
      if (!tc::mbar_wait(&misc->s_full[buf], (seq / kRtBufs) & 1, &misc->abort_flag)) return false;
      tc::tc_fence_after();
      tc::tmem_ld32(lane_addr + buf * 128, s);
      tc::tmem_ld_wait();
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&misc->s_free[buf]);
      ++seq;
      return true;
    };
    for (int item = blockIdx.x; item < total_items; item += gridDim.x, ++n_items) {
      const int rt = item % row_tiles, bhq = item / row_tiles;
      const int r = rt * kRtTile + row;                          // pooled query index inside the head
      const bool q_valid = (valid_bits[r >> 5] >> (r & 31)) & 1u;
      float m_run = -INFINITY, l_run = 0.f;
      for (int kt = 0; kt < row_tiles; ++kt) {
        if (!fetch()) goto done;
        rt_accumulate(s, valid_bits[kt * 4 + part], c2, m_run, l_run);
      }
      // merge the four column quarters of the row
      if (part > 0) {
        misc->part_stats[part - 1][row] = make_float2(m_run, l_run);
        tc::mbar_arrive(&misc->part_ready);
      } else {
        VSA2_WAIT(&misc->part_ready, n_items & 1);
        float2 o[kRtParts - 1];
        float m_new = m_run;
#pragma unroll
        for (int pp = 0; pp < kRtParts - 1; ++pp) {
          o[pp] = misc->part_stats[pp][row];
          m_new = fmaxf(m_new, o[pp].x);
        }
        if (m_new > -INFINITY) {
          l_run *= ex2_approx(m_run - m_new);
#pragma unroll
          for (int pp = 0; pp < kRtParts - 1; ++pp) l_run += o[pp].y * ex2_approx(o[pp].x - m_new);
        }
        misc->row_lse2[row] = (l_run > 0.f) ? m_new + __log2f(l_run) : 0.f;
        tc::mbar_arrive(&misc->lse_ready);
      }
      VSA2_WAIT(&misc->lse_ready, n_items & 1);
      // (part_stats and row_lse2 need no barrier of their own for their next item: parts 1.. write the former after this wait, which
      //  part 0 has let pass after reading it; part 0 writes the latter after part_ready, on which every reader arrives later)
      const float my_lse2 = q_valid ? misc->row_lse2[row] : INFINITY;          // +inf => p = 0 for padding rows
      const uint32_t vb = __ballot_sync(0xffffffffu, q_valid);
      const int gi = __popc((vb >> (lane & ~(G - 1))) & ((1u << G) - 1u));     // valid rows of the query block
      const float inv_norm = gi > 0 ? 1.f / ((float)gi * (float)G) : 0.f;
      const int qi = r / G;                                      // query block of this row
      const int n_out = FOLD ? g.N / 2 : g.N;
      float* out = pr + ((size_t)bhq * n_out + (FOLD ? qi >> 1 : qi)) * n_out;
      float w0 = 0.f, w1 = 0.f;
      if (FOLD) {
        const int other = __shfl_xor_sync(0xffffffffu, gi, 8), vq0 = lane & 8 ? other : gi, vq1 = lane & 8 ? gi : other;
        w0 = (float)vq0 / (float)(2 * (vq0 + vq1));
        w1 = (float)vq1 / (float)(2 * (vq0 + vq1));
      }
      for (int kt = 0; kt < row_tiles; ++kt) {
        if (!fetch()) goto done;
        int mine;
        const float t = rt_pool<G>(s, valid_bits[kt * 4 + part], c2, my_lse2, lane, mine);
        const int kj = (kt * kRtTile + part * 32) / G + mine;
        if constexpr (FOLD) {
          // a lane holds one of the two key halves (lane bit 1) of one of the two query halves (lane bit 3) of a cube pair
          const float v = t * inv_norm;
          const float both = v + __shfl_xor_sync(0xffffffffu, v, 2);
          const float low = __shfl_xor_sync(0xffffffffu, both, 8);
          if (!(lane & 11) && qi < g.N && kj < g.N) out[kj >> 1] = w0 * both + w1 * low;
        } else {
          const bool owner = G == 8 ? !(lane & 1) : !(lane & 7);
          if (owner && qi < g.N && kj < g.N) out[kj] = t * inv_norm;
        }
      }
    }
  }

done:
  tc::tc_fence_before();
  __syncthreads();
  if (misc->abort_flag) {
    if (tid == 0) {
      atomicExch(&status->status, VSA2_ERR_DEVICE_TIMEOUT);
      const unsigned long long t0 = tc::global_timer_ns();
      while (tc::global_timer_ns() - t0 < 200000ull) {
      }
    }
    __syncthreads();
  }
  if (warp == 1) tc::tmem_dealloc(tmem_base, 128 * kRtBufs);
}

bool router_tc_supported(const Geo& g) { return g.G == 8 || g.G == 16; }

template <int D, int G, bool FOLD>
static cudaError_t launch_router(const CUtensorMap& tq, const CUtensorMap& tk, const Geo& g, float* pr, StatusBlock* status,
                                 cudaStream_t st) {
  const int row_tiles = (g.N * G + kRtTile - 1) / kRtTile;
  const size_t smb = RouterTc<D>::smem_bytes(row_tiles * kRtTile / 32);
  if (smb > 227 * 1024) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  static KernelAttr attr;
  if ((e = prepare_kernel((const void*)router_tc_kernel<D, G, FOLD>, attr, smb))) return e;
  const int total = g.batch * g.Hq * row_tiles;
  { ProfScope lse(VSA2_KERNEL_ROUTER_LSE, st, 0); }      // (both passes are timed as the second)
  ProfScope ps(VSA2_KERNEL_ROUTER_POOL, st, 1);
  router_tc_kernel<D, G, FOLD><<<total < sms ? total : sms, kRtThreads, smb, st>>>(tq, tk, g, pr, status);
  return cudaGetLastError();
}

cudaError_t launch_router_scores_tc(const Geo& g, bool fold, const bf16* qr, const bf16* kr, float* pr, StatusBlock* status,
                                    cudaStream_t st) {
  const int NG = g.N * g.G;
  CUtensorMap tq, tk;
  if (!make_pooled_tmap(&tq, qr, g.D, NG, g.batch * g.Hq) || !make_pooled_tmap(&tk, kr, g.D, NG, g.batch * g.Hkv))
    return cudaErrorInvalidValue;
  if (fold && g.G != 8) return cudaErrorInvalidValue;
  if (g.D == 128 && g.G == 8) return fold ? launch_router<128, 8, true>(tq, tk, g, pr, status, st) : launch_router<128, 8, false>(tq, tk, g, pr, status, st);
  if (g.D == 128 && g.G == 16) return launch_router<128, 16, false>(tq, tk, g, pr, status, st);
  if (g.D == 64 && g.G == 8) return fold ? launch_router<64, 8, true>(tq, tk, g, pr, status, st) : launch_router<64, 8, false>(tq, tk, g, pr, status, st);
  if (g.D == 64 && g.G == 16) return launch_router<64, 16, false>(tq, tk, g, pr, status, st);
  return cudaErrorInvalidValue;
}

}  // namespace vsa2
