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
// The two-pass form: both passes are bound by the exponential unit (one ex2 per score: 1024 cycles per tile of ~1250), not by the tensor pipe.
// ONE PASS (`ONE`): large problems form every exponential once.  A thread's sums over the 8 keys of a cube, taken against its running
// maximum, are parked in the caller's scratch (fp32, one factor per thread and row still missing); when the row's denominator is
// known they are fetched back, scaled and pooled -- tile by tile inside the next item's loop, the shuffles between the
// exponentials (behind one another they took 480 of 1820 cycles a tile).  435,600 tokens, 10 heads: 22.0 -> 13.4 ms (the card at its
// power cap; 1965 MHz before); 720p, 10 heads: 0.90 -> 0.58 ms.
// The denominators are those of the two-pass form bit for bit (same operations, same order).  A score differs from the two-pass
// score in its last bits (no further from 64 bits than that: 3.7e-7 against 3.8e-7 of the scores' norm at 1120 cubes), which can
// carry a pair across the threshold, so the selection settles the pairs next to it on their two-pass scores (router_exact_kernel
// below, select.cu) and the map is the two-pass map.  Where that cannot be done (too many pairs at the threshold, a score
// range beyond fp32 exponents) a flag runs the two-pass form behind.
// A buffer of scores is given back as soon as they are in registers (720p, 40 heads: 3.27 -> 3.22 ms; fetching the next tile's
// scores before a tile is worked on made it 3.58).
#include "tc_attn.cuh"

namespace vsa2 {

constexpr int kRtParts = 4;        // compute threads per pooled query row (each owns 128 / kRtParts key columns of a tile)
constexpr int kRtThreads = 64 + 128 * kRtParts;    // TMA warp, MMA warp, 4 * kRtParts compute warps
constexpr int kRtSlots = 4;
constexpr int kRtTile = 128;
// one-pass form: at most so many CTAs, those of a B200, on whatever it runs -- a caller asks for the scratch, a region per CTA, without a
// device at hand
constexpr int kRtOneCtas = 148;
constexpr int kRtAhead = 4;        // one-pass form: tiles of parked sums on their way
constexpr int kRtBufs = 4;         // score tiles in tensor memory (4 x 128 columns = all of it)

template <int D>
struct RouterTc {
  static constexpr int DH = D / 64;
  static constexpr uint32_t HALF = kRtTile * 128;          // 128 rows x 64 channels
  static constexpr uint32_t TILE = DH * HALF;
  static constexpr uint32_t OFF_Q = kRtSlots * TILE;
  static constexpr uint32_t OFF_MISC = OFF_Q + TILE;
  static constexpr uint32_t MISC_BYTES = 4096;
  static constexpr uint32_t OFF_VALID = OFF_MISC + MISC_BYTES;
  // the ring of fetched sums of the one-pass form lies behind the validity bits
  __host__ __device__ static constexpr uint32_t off_ring(int valid_words) { return OFF_VALID + (valid_words * 4 + 15) / 16 * 16; }
  static size_t smem_bytes(int valid_words, bool one) { return off_ring(valid_words) + (one ? kRtAhead * kRtParts * kRtTile * 16 : 0) + 1024; }
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

// what a thread parks per tile (a pair of half-cubes shares its sum)
template <bool FOLD> struct RtParked { using type = float4; };
template <> struct RtParked<true> { using type = float2; };
// that much global -> shared, asynchronously; groups of such copies of a thread complete in order
__device__ __forceinline__ void rt_copy_async(float4* dst, const float4* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(__cvta_generic_to_global(src)) : "memory");
}
__device__ __forceinline__ void rt_copy_async(float2* dst, const float2* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(tc::smem_u32(dst)), "l"(__cvta_generic_to_global(src)) : "memory");
}
__device__ __forceinline__ void rt_copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void rt_copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }

// What the one-pass form adds to a launch.
struct RouterOne {
  void* park;          // [CTA][key tile][part][row]: sums over the four key cubes of a thread's 32 columns (FOLD: the two 128-token cubes)
  float* lse2;         // [BH, N * G]: log2 of the row denominators
  int* redo;           // raised when the scores of this launch are not to be used; two-pass launch: runs only if it is up (or null)
};
// The reference of a thread's parked sums is the maximum of its first 32 valid keys.  The maximum may grow by a factor 2^48 along
// the row.  Where the reference lies more than 2^126 below the denominator all that a thread has of the row is lost: terms of less than
// 2^-78 each, little of any score of 2^-52 or more even when the terms are summed over the 16 heads of a group (select.cu)
constexpr float kRtMostGrowth = 48.f;
// 2^(a - b) with the rounding of the difference put back (exponents of 16 to 32 would lose 7e-7)
__device__ __forceinline__ float rt_exp2_diff(float a, float b) {
  const float d = a - b, t = d - a, lost = (a - (d - t)) - (b + t);
  const float p = ex2_approx(d);
  return fabsf(lost) < 1.f ? fmaf(p * lost, 0.6931471805599453f, p) : p;      // (infinities: no correction)
}

// the 2 x 2 fold of half-cube scores: spelled out, so that every kernel that folds rounds alike
__device__ __forceinline__ float rt_fold(float w0, float both0, float w1, float both1) { return __fmaf_rn(w0, both0, __fmul_rn(w1, both1)); }

// largest of three in one instruction (a NaN among them does not count, as with fmaxf)
__device__ __forceinline__ float rt_max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Pass 1 on 32 scores of a row: running maximum (in the exponent's units) and sum.  The maximum is taken over the raw scores
// (the scale is positive) and the scale folded into the exponent's multiply-add.
// (`s` is masked: rt_mask)
__device__ __forceinline__ void rt_mask(uint32_t (&s)[32], uint32_t kbits) {
  if (kbits != 0xffffffffu) {
#pragma unroll
    for (int c = 0; c < 32; ++c) s[c] = ((kbits >> c) & 1u) ? s[c] : 0xff800000u;      // -inf
  }
}
__device__ __forceinline__ float rt_max(const uint32_t (&s)[32]) {
  float a = __uint_as_float(s[0]), b = __uint_as_float(s[1]);
#pragma unroll
  for (int c = 2; c < 30; c += 4) {
    a = rt_max3(a, __uint_as_float(s[c]), __uint_as_float(s[c + 1]));
    b = rt_max3(b, __uint_as_float(s[c + 2]), __uint_as_float(s[c + 3]));
  }
  return rt_max3(fmaxf(a, b), __uint_as_float(s[30]), __uint_as_float(s[31]));
}
__device__ __forceinline__ void rt_accumulate(uint32_t (&s)[32], uint32_t kbits, float c2, float& m_run, float& l_run) {
  rt_mask(s, kbits);
  const float cmax = rt_max(s);
  if (cmax > -INFINITY) {
    const float m_new = fmaxf(m_run, cmax * c2);
    float acc = 0.f;
#pragma unroll
    for (int c = 0; c < 32; ++c) acc += ex2_approx(fmaf(__uint_as_float(s[c]), c2, -m_new));
    l_run = __fmaf_rn(l_run, ex2_approx(m_run - m_new), acc);
    m_run = m_new;
  }
}
// The same (bit for bit in m_run and l_run) without a branch, the sums of each 8 columns' exponentials in tv; step(0 .. 3) runs
// between the groups of 8: work that waits for shuffles goes there, while the exponential unit is busy.
template <bool PACKED, typename Step>
__device__ __forceinline__ void rt_accumulate_one(uint32_t (&s)[32], uint32_t kbits, float c2, float& m_run, float& l_run, float (&tv)[4],
                                                  Step&& step) {
  rt_mask(s, kbits);
  const float cmax = rt_max(s);
  const bool any = cmax > -INFINITY;
  const float m_new = fmaxf(m_run, cmax * c2), m_use = any ? m_new : 0.f;
  const float decay = ex2_approx(m_run - m_use);
  float acc = 0.f;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    float e[8];
#pragma unroll
    for (int c = 0; c < 8; c += 2) {
      float2 x = make_float2(__uint_as_float(s[8 * g + c]), __uint_as_float(s[8 * g + c + 1]));
      if constexpr (PACKED) x = __ffma2_rn(x, make_float2(c2, c2), make_float2(-m_use, -m_use));
      else x = make_float2(fmaf(x.x, c2, -m_use), fmaf(x.y, c2, -m_use));
      e[c] = ex2_approx(x.x);
      e[c + 1] = ex2_approx(x.y);
    }
    step(g);
#pragma unroll
    for (int c = 0; c < 8; ++c) acc += e[c];
    if constexpr (PACKED) {
      const float2 p = __fadd2_rn(__fadd2_rn(make_float2(e[0], e[1]), make_float2(e[2], e[3])), __fadd2_rn(make_float2(e[4], e[5]), make_float2(e[6], e[7])));
      tv[g] = p.x + p.y;
    } else {
      tv[g] = ((e[0] + e[1]) + (e[2] + e[3])) + ((e[4] + e[5]) + (e[6] + e[7]));
    }
  }
  l_run = any ? __fmaf_rn(l_run, decay, acc) : l_run;
  m_run = any ? m_new : m_run;
}

// Sums over the G rows of a query cube, which sit in G adjacent lanes, of the sums over 32 / G key cubes: a butterfly that halves the
// values a lane carries at every step (4 shuffles instead of 3 per key cube) and leaves each total in one lane -- that of cube
// `mine` of the 32 / G.  (The order of a total's additions does not depend on its place.)
template <int G>
__device__ __forceinline__ float rt_sum_rows(const float (&tv)[32 / G], int lane, int& mine) {
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

// Pass 2 on 32 scores of a row: softmax, column sums of the 32 / G key cubes, then the sum over the G rows of the query cube.
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
  return rt_sum_rows<G>(tv, lane, mine);
}

// Writes P_r of the blocks of `g` or, with FOLD (G = 8), of the 128-token cubes whose half-cubes those blocks are: the scores of the
// four pairs of halves, weighted with the valid query sub-cubes of each half (wide_cube.cu, fold_scores_kernel).
template <int D, int G, bool FOLD, bool ONE>
__global__ void __launch_bounds__(kRtThreads, 1)
router_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, Geo g,
                 float* pr, RouterOne one, StatusBlock* status) {
  static_assert(!FOLD || G == 8, "half-cubes of 8 sub-cubes");
  static_assert(!ONE || G == 8, "a thread parks the sums of four cubes");
  constexpr int PASSES = ONE ? 1 : 2;
  const bool redo = !ONE && one.redo != nullptr;
  if (redo) {
    grid_enter(false);
    if (*one.redo == 0) return;                  // (settled before this launch starts)
  }
  using C = RouterTc<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* q_tile = smem + C::OFF_Q;
  RouterMisc* misc = reinterpret_cast<RouterMisc*>(smem + C::OFF_MISC);
  uint32_t* valid_bits = reinterpret_cast<uint32_t*>(smem + C::OFF_VALID);   // one bit per pooled token

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
  if (!redo) grid_enter_items(total_items);

  if (warp == 0) {
    if (lane == 0) {
      uint32_t seq = 0, n_items = 0;
      for (int item = blockIdx.x; item < total_items; item += gridDim.x, ++n_items) {
        const int rt = item % row_tiles, bhq = item / row_tiles;
        const int b = bhq / g.Hq, hq = bhq % g.Hq, bhk = b * g.Hkv + hq / g.rep;
        VSA2_WAIT(&misc->q_empty, (n_items & 1) ^ 1);
        tc::mbar_expect_tx(&misc->q_full, C::TILE);
        for (int h = 0; h < C::DH; ++h) tma_load_3d(q_tile + h * C::HALF, &tm_q, &misc->q_full, h * 64, rt * kRtTile, bhq);
        for (int step = 0; step < PASSES * row_tiles; ++step, ++seq) {       // pass 1, then pass 2
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
        for (int step = 0; step < PASSES * row_tiles; ++step, ++seq) {
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
          if (step == PASSES * row_tiles - 1) tc::mma_commit(&misc->q_empty);
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
    // what the pooling of an item needs; ONE: of the item before, whose parked sums are fetched back tile by tile
    struct Pooling {
      float* out;          // the row of P_r of this thread's query cube
      float inv_norm, w0, w1, weight;
      int qi;
    } pool = {};
    using Parked = typename RtParked<FOLD>::type;
    Parked* const park = ONE ? static_cast<Parked*>(one.park) + ((size_t)blockIdx.x * row_tiles * kRtParts + part) * kRtTile + row : nullptr;
    auto write = [&](float t, int mine, int kt) {
      const int kj = (kt * kRtTile + part * 32) / G + mine;
      if constexpr (FOLD) {
        // a lane holds one of the two key halves (lane bit 1) of one of the two query halves (lane bit 3) of a cube pair
        const float v = t * pool.inv_norm;
        const float both = v + __shfl_xor_sync(0xffffffffu, v, 2);
        const float low = __shfl_xor_sync(0xffffffffu, both, 8);
        if (!(lane & 11) && pool.qi < g.N && kj < g.N) pool.out[kj >> 1] = rt_fold(pool.w0, both, pool.w1, low);
      } else {
        const bool owner = G == 8 ? !(lane & 1) : !(lane & 7);
        if (owner && pool.qi < g.N && kj < g.N) pool.out[kj] = t * pool.inv_norm;
      }
    };
    // ONE: tile `n` counts over the CTA's items.  The sums parked at tile n come back for tile n + row_tiles, by then in the ring:
    // each thread's own 16 bytes, asked for kRtAhead tiles before (a fetch from HBM takes longer than a tile)
    uint32_t n = 0;
    Parked* const ring = reinterpret_cast<Parked*>(smem + C::off_ring(valid_words)) + part * kRtTile + row;
    const uint32_t last = ONE ? (uint32_t)((total_items - 1 - (int)blockIdx.x) / (int)gridDim.x + 2) * row_tiles : 0;
    auto ask = [&](uint32_t at, int kt) {      // (at: from the second item on, below the end of the drain; kt = at % row_tiles)
      if (at >= (uint32_t)row_tiles && at < last)
        rt_copy_async(ring + (at % kRtAhead) * (kRtParts * kRtTile), park + (size_t)kt * (kRtParts * kRtTile));
      rt_copy_commit();
    };
    // the sums of tile `n` as they lie in the ring, and the request for those kRtAhead tiles on
    auto fetch_parked = [&](int kt) -> Parked {
      rt_copy_wait<kRtAhead - 1>();
      const Parked x = ring[(n % kRtAhead) * (kRtParts * kRtTile)];
      ask(n + kRtAhead, kt + kRtAhead < row_tiles ? kt + kRtAhead : kt + kRtAhead - row_tiles);
      return x;
    };
    // pools them in four steps: scaled and over lanes 4 apart, 2 apart, 1 apart (rt_sum_rows<8> in pieces), written.  FOLD: the two
    // sums stand for both key halves, and the lanes 8 apart have the query halves
    const bool hi4 = lane & 4, hi2 = lane & 2;
    auto pool_step = [&](int step, const Parked& x, int kt, float& u0, float& u1) {
      if (step == 0) {
        if constexpr (FOLD) {
          const float t0 = x.x * pool.weight, t1 = x.y * pool.weight;
          u0 = (hi4 ? t1 : t0) + __shfl_xor_sync(0xffffffffu, hi4 ? t0 : t1, 4);
        } else {
          const float t0 = x.x * pool.weight, t1 = x.y * pool.weight, t2 = x.z * pool.weight, t3 = x.w * pool.weight;
          u0 = (hi4 ? t2 : t0) + __shfl_xor_sync(0xffffffffu, hi4 ? t0 : t2, 4);
          u1 = (hi4 ? t3 : t1) + __shfl_xor_sync(0xffffffffu, hi4 ? t1 : t3, 4);
        }
      } else if (step == 1) {
        if constexpr (FOLD) u0 += __shfl_xor_sync(0xffffffffu, u0, 2);
        else u0 = (hi2 ? u1 : u0) + __shfl_xor_sync(0xffffffffu, hi2 ? u0 : u1, 2);
      } else if (step == 2) {
        u0 += __shfl_xor_sync(0xffffffffu, u0, 1);
        if constexpr (FOLD) {
          u0 *= pool.inv_norm;
          u1 = __shfl_xor_sync(0xffffffffu, u0, 8);
        }
      } else if (n >= (uint32_t)row_tiles) {
        if constexpr (FOLD) {
          const int kc = (kt * kRtTile + part * 32) / 16 + (hi4 ? 1 : 0);
          if (!(lane & 11) && pool.qi < g.N && kc < g.N / 2) pool.out[kc] = rt_fold(pool.w0, u0, pool.w1, u1);
        } else {
          write(u0, (hi4 ? 2 : 0) + (hi2 ? 1 : 0), kt);
        }
      }
    };
    if constexpr (ONE)
      for (int a = 0; a < kRtAhead; ++a) ask(a, a);
    for (int item = blockIdx.x; item < total_items; item += gridDim.x, ++n_items) {
      const int rt = item % row_tiles, bhq = item / row_tiles;
      const int r = rt * kRtTile + row;                          // pooled query index inside the head
      const bool q_valid = (valid_bits[r >> 5] >> (r & 31)) & 1u;
      float m_run = -INFINITY, l_run = 0.f;
      float ref = 0.f, factor = 0.f;                             // ONE: sums are parked as multiples of 2^ref
      for (int kt = 0; kt < row_tiles; ++kt) {
        float tv[4];
        if constexpr (ONE) {
          const uint32_t kbits = valid_bits[kt * 4 + part];
          if (kt == 0 || kt == row_tiles - kRtAhead) __threadfence();      // what was parked comes before what is asked for from here on
          const Parked parked = fetch_parked(kt);
          if (!fetch()) goto done;
          const float m_old = m_run;
          float u0 = 0.f, u1 = 0.f;
          rt_accumulate_one<FOLD>(s, kbits, c2, m_run, l_run, tv, [&](int step) { pool_step(step, parked, kt, u0, u1); });
          ++n;
          if (m_run != m_old) {
            if (m_old == -INFINITY) ref = m_run;
            factor = ex2_approx(m_run - ref);
          }
          if constexpr (FOLD) park[(size_t)kt * (kRtParts * kRtTile)] = make_float2((tv[0] + tv[1]) * factor, (tv[2] + tv[3]) * factor);
          else park[(size_t)kt * (kRtParts * kRtTile)] = make_float4(tv[0] * factor, tv[1] * factor, tv[2] * factor, tv[3] * factor);
        } else {
          if (!fetch()) goto done;
          rt_accumulate(s, valid_bits[kt * 4 + part], c2, m_run, l_run);
        }
      }
      // (a sum beyond the fp32 range, or close to it: the two-pass form does it)
      if (ONE && q_valid && !(m_run - ref <= kRtMostGrowth)) atomicExch(one.redo, 1);
      // merge the four column quarters of the row
      const float m_own = m_run;
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
        const float lse2 = (l_run > 0.f) ? m_new + __log2f(l_run) : 0.f;
        misc->row_lse2[row] = lse2;
        if (ONE && r < NG) {
          one.lse2[(size_t)bhq * NG + r] = lse2;
          // (a denominator that is not a number leaves lse2 = 0, and the two-pass form then has the bare exponentials)
          if (q_valid && !(l_run < INFINITY && fabsf(lse2) < INFINITY)) atomicExch(one.redo, 1);
        }
        tc::mbar_arrive(&misc->lse_ready);
      }
      VSA2_WAIT(&misc->lse_ready, n_items & 1);
      // (part_stats and row_lse2 need no barrier of their own for their next item: parts 1.. write the former after this wait, which
      //  part 0 has let pass after reading it; part 0 writes the latter after part_ready, on which every reader arrives later)
      const float my_lse2 = q_valid ? misc->row_lse2[row] : INFINITY;          // +inf => p = 0 for padding rows
      const uint32_t vb = __ballot_sync(0xffffffffu, q_valid);
      const int gi = __popc((vb >> (lane & ~(G - 1))) & ((1u << G) - 1u));     // valid rows of the query block
      pool.inv_norm = gi > 0 ? 1.f / ((float)gi * (float)G) : 0.f;
      pool.qi = r / G;                                           // query block of this row
      const int n_out = FOLD ? g.N / 2 : g.N;
      pool.out = pr + ((size_t)bhq * n_out + (FOLD ? pool.qi >> 1 : pool.qi)) * n_out;
      if (FOLD) {
        const int other = __shfl_xor_sync(0xffffffffu, gi, 8), vq0 = lane & 8 ? other : gi, vq1 = lane & 8 ? gi : other;
        pool.w0 = (float)vq0 / (float)(2 * (vq0 + vq1));
        pool.w1 = (float)vq1 / (float)(2 * (vq0 + vq1));
      }
      if constexpr (ONE) {
        pool.weight = m_own > -INFINITY ? rt_exp2_diff(ref, my_lse2) : 0.f;
      } else {
        for (int kt = 0; kt < row_tiles; ++kt) {
          if (!fetch()) goto done;
          int mine;
          const float t = rt_pool<G>(s, valid_bits[kt * 4 + part], c2, my_lse2, lane, mine);
          write(t, mine, kt);
        }
      }
    }
    if constexpr (ONE) {
      // the last item's, kRtAhead tiles side by side (one after the other: 390 cycles each)
      __threadfence();      // (as in the loop: its last kRtAhead tiles have been parked since the fence there)
      for (int k0 = 0; k0 < row_tiles; k0 += kRtAhead) {
        rt_copy_wait<0>();
        Parked x[kRtAhead];
        float u0[kRtAhead], u1[kRtAhead];
#pragma unroll
        for (int u = 0; u < kRtAhead; ++u) x[u] = ring[((n + u) % kRtAhead) * (kRtParts * kRtTile)];
#pragma unroll
        for (int u = 0; u < kRtAhead; ++u) ask(n + u + kRtAhead, min(k0 + u + kRtAhead, row_tiles - 1));      // (none beyond the last tile)
#pragma unroll
        for (int step = 0; step < 4; ++step)
#pragma unroll
          for (int u = 0; u < kRtAhead; ++u)
            if (step < 3 || k0 + u < row_tiles) pool_step(step, x[u], k0 + u, u0[u], u1[u]);
        n += kRtAhead;
      }
      rt_copy_wait<0>();
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

template <int D, int G, bool FOLD, bool ONE>
static cudaError_t launch_router(const CUtensorMap& tq, const CUtensorMap& tk, const Geo& g, float* pr, const RouterOne& one,
                                 StatusBlock* status, cudaStream_t st) {
  const int row_tiles = (g.N * G + kRtTile - 1) / kRtTile;
  const size_t smb = RouterTc<D>::smem_bytes(row_tiles * kRtTile / 32, ONE);
  if (smb > 227 * 1024) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  static KernelAttr attr;
  if ((e = prepare_kernel((const void*)router_tc_kernel<D, G, FOLD, ONE>, attr, smb))) return e;
  const int total = g.batch * g.Hq * row_tiles;
  if (ONE && sms > kRtOneCtas) sms = kRtOneCtas;
  launch_kernel(router_tc_kernel<D, G, FOLD, ONE>, total < sms ? total : sms, kRtThreads, smb, st, tq, tk, g, pr, one, status);
  return cudaGetLastError();
}

template <bool ONE>
static cudaError_t launch_router_any(const Geo& g, bool fold, const bf16* qr, const bf16* kr, float* pr, const RouterOne& one,
                                     StatusBlock* status, cudaStream_t st) {
  const int NG = g.N * g.G;
  CUtensorMap tq, tk;
  if (!make_pooled_tmap(&tq, qr, g.D, NG, g.batch * g.Hq) || !make_pooled_tmap(&tk, kr, g.D, NG, g.batch * g.Hkv))
    return cudaErrorInvalidValue;
  if (fold && g.G != 8) return cudaErrorInvalidValue;
  if (g.D == 128 && g.G == 8) return fold ? launch_router<128, 8, true, ONE>(tq, tk, g, pr, one, status, st) : launch_router<128, 8, false, ONE>(tq, tk, g, pr, one, status, st);
  if (g.D == 64 && g.G == 8) return fold ? launch_router<64, 8, true, ONE>(tq, tk, g, pr, one, status, st) : launch_router<64, 8, false, ONE>(tq, tk, g, pr, one, status, st);
  if constexpr (!ONE) {
    if (g.D == 128 && g.G == 16) return launch_router<128, 16, false, false>(tq, tk, g, pr, one, status, st);
    if (g.D == 64 && g.G == 16) return launch_router<64, 16, false, false>(tq, tk, g, pr, one, status, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_router_scores_tc(const Geo& g, bool fold, const bf16* qr, const bf16* kr, float* pr, int* redo, StatusBlock* status,
                                    cudaStream_t st) {
  return launch_router_any<false>(g, fold, qr, kr, pr, RouterOne{nullptr, nullptr, redo}, status, st);
}

// ---- the one-pass form ----------------------------------------------------------------------------------------------------
bool router_one_runs(const Geo& g) {
  const int row_tiles = (g.N * g.G + kRtTile - 1) / kRtTile;
  const size_t smb = g.D == 128 ? RouterTc<128>::smem_bytes(row_tiles * kRtTile / 32, true) : RouterTc<64>::smem_bytes(row_tiles * kRtTile / 32, true);
  return g.G == 8 && row_tiles >= 2 * kRtAhead && smb <= 227 * 1024;
}

size_t router_one_park_bytes(const Geo& g, bool fold) {
  const size_t row_tiles = ((size_t)g.N * g.G + kRtTile - 1) / kRtTile, items = (size_t)g.batch * g.Hq * row_tiles;
  return (items < (size_t)kRtOneCtas ? items : (size_t)kRtOneCtas) * row_tiles * kRtParts * kRtTile * (fold ? sizeof(float2) : sizeof(float4));
}

cudaError_t launch_router_one(const Geo& g, bool fold, const bf16* qr, const bf16* kr, float* pr, void* park, float* lse2, int* redo,
                              StatusBlock* status, cudaStream_t st) {
  return launch_router_any<true>(g, fold, qr, kr, pr, RouterOne{park, lse2, redo}, status, st);
}

// Two-pass scores of the listed pairs, written over the one-pass scores: the same products (the same instruction over the same
// operands), exponentials and sums in the same order as in router_tc_kernel, so the values are its values.  A tile of 128 x 128
// holds the sub-cubes of 16 pairs (FOLD: of 8 pairs of 128-token cubes, 16 rows each) of which the blocks on the diagonal are
// used; lists are short (a few pairs in a million lie at a threshold), so this is a launch of a few microseconds.
// `heads`: with a map shared by the query heads of a group a pair's score is the sum over them, in their order.
struct RouterExactArgs {
  const bf16* qr;
  const bf16* kr;
  const float* lse2;
  const int2* pairs;       // {(batch * Hq + head) * rows + row, column} of the score matrix
  const int* count;
  int cap, heads;
  const int* redo;         // up: the two-pass form does it all
  float* pr;
  StatusBlock* status;
};

template <int D, bool FOLD>
__global__ void __launch_bounds__(128) router_exact_kernel(Geo g, RouterExactArgs a) {
  grid_enter(false);
  using C = RouterTc<D>;
  constexpr int ROWS = FOLD ? 16 : 8, PAIRS = kRtTile / ROWS;      // sub-cubes of a pair's side, pairs of a tile
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  __shared__ uint64_t done_bar;
  __shared__ uint32_t tmem_addr;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int listed = *a.redo != 0 ? 0 : min(*a.count, a.cap);
  if ((int)blockIdx.x * PAIRS >= listed) return;
  const int NG = g.N * g.G, n_out = FOLD ? g.N / 2 : g.N;
  const float c2 = g.scale * 1.4426950408889634f;
  if (tid == 0) {
    abort_flag = 0;
    tc::mbar_init(&done_bar, 1);
    tc::fence_barrier_init();
  }
  if (warp == 0) {
    tc::tmem_alloc(&tmem_addr, 128);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = tmem_addr;
  uint32_t phase = 0;
  for (int first = blockIdx.x * PAIRS; first < listed; first += gridDim.x * PAIRS) {
    const int mine = first + tid / ROWS, sub = tid % ROWS;           // this thread's pair (its row of the tile), and row of it
    const bool live = mine < listed;
    const int2 pair = live ? a.pairs[mine] : make_int2(0, 0);
    const int bhq0 = pair.x / n_out, i = pair.x % n_out, j = pair.y;
    const int b = bhq0 / g.Hq, hk = bhq0 % g.Hq / g.rep, bhk = b * g.Hkv + hk;
    const int head0 = a.heads > 1 ? b * g.Hq + hk * g.rep : bhq0;    // first head of the sum
    const int q_row = i * ROWS + sub, k_row = j * ROWS + sub;        // (the two halves of a cube are neighbours)
    const bool q_valid = live && subcube_count(g, q_row / 8, q_row % 8) > 0;
    const uint32_t kbits = __ballot_sync(0xffffffffu, live && subcube_count(g, k_row / 8, k_row % 8) > 0);
    const uint32_t vb = __ballot_sync(0xffffffffu, q_valid);
    const int gi = __popc((vb >> (lane & ~7)) & 0xffu);
    const float inv_norm = gi > 0 ? 1.f / ((float)gi * 8.f) : 0.f;
    float total = 0.f;
    for (int hh = 0; hh < a.heads; ++hh) {
      // operand rows with the 128-byte swizzle of the TMA tiles
      const uint4* qs = reinterpret_cast<const uint4*>(a.qr + ((size_t)(head0 + hh) * NG + q_row) * D);
      const uint4* ks = reinterpret_cast<const uint4*>(a.kr + ((size_t)bhk * NG + k_row) * D);
#pragma unroll
      for (int c = 0; c < D / 8; ++c) {
        const uint32_t at = (c / 8) * C::HALF + tid * 128 + (((c % 8) ^ (tid & 7)) << 4);
        *reinterpret_cast<uint4*>(smem + at) = live ? qs[c] : make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(smem + C::TILE + at) = live ? ks[c] : make_uint4(0u, 0u, 0u, 0u);
      }
      tc::fence_proxy_async_smem();
      __syncthreads();
      if (tid == 0) {
        constexpr uint32_t idesc = tc::idesc_bf16(128, 128, false, false);
        const uint32_t q_addr = tc::smem_u32(smem), k_addr = q_addr + C::TILE;
        tc::tc_fence_after();
#pragma unroll
        for (int ks_ = 0; ks_ < D / 16; ++ks_) {
          const uint32_t off = (ks_ / 4) * C::HALF + (ks_ % 4) * 32;
          tc::mma_ss(tmem_base, tc::smem_desc_sw128(q_addr + off, 16, 1024), tc::smem_desc_sw128(k_addr + off, 16, 1024), idesc, ks_ > 0);
        }
        tc::mma_commit(&done_bar);
      }
      if (!tc::mbar_wait(&done_bar, phase & 1, &abort_flag)) goto done;
      ++phase;
      tc::tc_fence_after();
      uint32_t s[32];
      tc::tmem_ld32(tmem_base + ((uint32_t)(warp * 32) << 16) + warp * 32, s);
      tc::tmem_ld_wait();
      tc::tc_fence_before();
      {
        const float lse2 = q_valid ? a.lse2[(size_t)(head0 + hh) * NG + q_row] : INFINITY;
        float tv[4];
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          float tot = 0.f;
#pragma unroll
          for (int c = 8 * cc; c < 8 * cc + 8; ++c) {
            float p = ex2_approx(fmaf(__uint_as_float(s[c]), c2, -lse2));
            p = ((kbits >> c) & 1u) ? p : 0.f;
            tot += p;
          }
          tv[cc] = tot;
        }
        // sum over the eight rows of a (half-)cube, each with its own key columns
        float x = FOLD ? (lane & 16 ? tv[2] : tv[0]) : (lane & 16 ? (lane & 8 ? tv[3] : tv[2]) : (lane & 8 ? tv[1] : tv[0]));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        float score = x * inv_norm;
        if constexpr (FOLD) {
          float y = lane & 16 ? tv[3] : tv[1];
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
          const float both = score + y * inv_norm;
          const float low = __shfl_xor_sync(0xffffffffu, both, 8);
          const int other = __shfl_xor_sync(0xffffffffu, gi, 8);
          score = rt_fold((float)gi / (float)(2 * (gi + other)), both, (float)other / (float)(2 * (gi + other)), low);
        }
        total += score;
      }
      __syncthreads();               // the operands and the accumulator may be replaced
    }
    if (live && sub == 0) a.pr[(size_t)pair.x * n_out + j] = total;
  }
done:
  tc::tc_fence_before();
  __syncthreads();
  if (abort_flag && tid == 0) atomicExch(&a.status->status, VSA2_ERR_DEVICE_TIMEOUT);
  if (warp == 0) tc::tmem_dealloc(tmem_base, 128);
}

cudaError_t launch_router_exact(const Geo& g, bool fold, const bf16* qr, const bf16* kr, const float* lse2, const int2* pairs,
                                const int* count, int cap, int heads, const int* redo, float* pr, StatusBlock* status, cudaStream_t st) {
  if (g.G != 8) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  const RouterExactArgs a{qr, kr, lse2, pairs, count, cap, heads, redo, pr, status};
#define VSA2_LAUNCH_EXACT(DD, FF)                                                                        \
  do {                                                                                                   \
    const size_t smb = 2 * RouterTc<DD>::TILE + 1024;                                                    \
    static KernelAttr attr_;                                                                             \
    if ((e = prepare_kernel((const void*)router_exact_kernel<DD, FF>, attr_, smb))) return e;            \
    launch_kernel(router_exact_kernel<DD, FF>, sms, 128, smb, st, g, a);                                            \
  } while (0)
  if (g.D == 128 && fold) VSA2_LAUNCH_EXACT(128, true);
  else if (g.D == 128) VSA2_LAUNCH_EXACT(128, false);
  else if (fold) VSA2_LAUNCH_EXACT(64, true);
  else VSA2_LAUNCH_EXACT(64, false);
#undef VSA2_LAUNCH_EXACT
  return cudaGetLastError();
}

}  // namespace vsa2
