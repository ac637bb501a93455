// dQ of the fine branch from stored dS: dQ^T[D, 64 q] += K_pair^T[D, 128 kv] dS^T[128 kv, 64 q], one tcgen05 product per tile.
//
// The dK/dV pass (fine_bwd_dkv_tc.cu) forms dS of every kept pair anyway; it leaves the fp16 tile of 64 q x 64 kv in a scratch
// region at the pair's place in the row lists, and this pass streams a row's tiles with the K cubes.  A tile lies there as
// it is an operand here: rows of 64 keys with the 128-byte swizzle, as the dK/dV pass has it in shared memory, or (pair form of
// that pass, whose threads store it from registers) as [16-byte chunk of 8 keys][query]: a warp with a query row per lane then
// stores 512 contiguous bytes at a time -- rows of 128 bytes cost that pass 25 %, 32 lines per store -- and 8 queries of a
// chunk are one core matrix of an unswizzled operand.  Recomputing S and dP here
// instead (fine_bwd_tc.cu) costs two more products, the exponentials and the V and dO tiles: 224 KB of shared-memory
// traffic per tile against 96 KB, and under the power cap (all long cases) the work is the time.  The price is 8 KB per pair written to
// and read from HBM; the passes run head group by head group so that the scratch stays bounded (kStoredDsBytes).
// The tiles hold the values the recomputing pass would form (same operands, same order), so dQ is the same bit for bit -- but for the
// all-fp16 form of GQA groups, whose dP comes from fp16 copies of V and dO (an element below 2^-17 is 2^-25 off at most).
#include "fine_bwd_tc.cuh"

namespace vsa2 {

// 2 producer warps of K blocks, 1 of dS tiles, issuer; 2 x 4 epilogue warps; scheduler; with 128 channels 2 more K producers (a warp fetches some
// 24 bytes a cycle of such boxes and a tile needs 32 KB.  us, two / four: 480p, 12 heads 923 / 904; 720p, 5 heads with text 1035 / 1008; backward of 720p,
// 40 heads 24505 / 24190)
constexpr int ds_threads(int D) { return D == 128 ? 480 : 416; }
constexpr int kDsSets = 4;            // accumulators (64 columns each), used by item in turn

template <int D>
struct DqDs {
  static constexpr int DH = D / 64;
  static constexpr uint32_t KBYTES = 2 * DH * kSlab;      // a pair of K cubes, [half][A | B]
  static constexpr uint32_t DSBYTES = 2 * kSlab;          // a pair of dS tiles
  static constexpr uint32_t STAGE = KBYTES + DSBYTES;
  static constexpr int STAGES = D == 128 ? 4 : 6;
  static constexpr uint32_t OFF_MISC = STAGES * STAGE;
  static constexpr size_t smem_bytes = OFF_MISC + 2048 + 1024;
};

struct DqDsMisc {
  uint64_t full[6], empty[6];
  uint64_t o_full[kDsSets], o_empty[kDsSets];
  ListQueue queue;
  uint32_t tmem_base;
  int abort_flag;
  int tok[2][2][64];                  // raster tokens of an item's rows: per epilogue warpgroup, by parity of its items
};
static_assert(sizeof(DqDsMisc) <= 2048, "misc region too small");

__device__ __forceinline__ bool packed_query(const Geo& g, const PackedCubes& pk, int i) { return pk.shift > 0 && i >= pk.first && i < g.Nvid; }

template <int D>
__global__ void __launch_bounds__(ds_threads(D), 1)
fine_bwd_dq_ds_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_kt, Geo g,
                      DqDsArgs a) {
  using C = DqDs<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  DqDsMisc* misc = reinterpret_cast<DqDsMisc*>(smem + C::OFF_MISC);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    misc->abort_flag = 0;
    for (int s = 0; s < C::STAGES; ++s) {
      tc::mbar_init(&misc->full[s], D == 128 ? 5 : 3);       // the producers
      tc::mbar_init(&misc->empty[s], 1);
    }
    for (int s = 0; s < kDsSets; ++s) {
      tc::mbar_init(&misc->o_full[s], 1);
      tc::mbar_init(&misc->o_empty[s], 4);
    }
    list_queue_init(&misc->queue, 4 + 8 + (D == 128 ? 2 : 0));
    tc::fence_barrier_init();
    tc::prefetch_tmap(&tm_k);
  }
  if (warp == 3) {
    tc::tmem_alloc(&misc->tmem_base, 64 * kDsSets);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = misc->tmem_base;
  grid_enter(false);
  if (__syncthreads_or(tid == 0 && *a.range_flag != 0)) {       // the fallback computes dQ
    if (warp == 3) tc::tmem_dealloc(tmem_base, 64 * kDsSets);
    return;
  }

  if (warp < 3 || warp > 12) {
    const bool is_k = warp != 2;
    const int blk = warp > 12 ? warp - 13 : warp, my_h = D == 128 ? (warp > 12 ? 1 : 0) : lane;      // (D = 128: a warp per block and channel half)
    // ------------------------------------------------------------------ producers: first K block of a pair (warps 0 and 13), second (1, 14), dS pair (2)
    const uint64_t policy = tc::evict_first_policy();      // (the tiles pass through once, the K cubes stay)
    uint32_t tg = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      if (warp == 0 && lane == 0) tc::mbar_arrive(&misc->queue.taken);
      const int k = rec.z, nt = (k + 1) >> 1;
      if (k == 0) continue;
      const int b = rec.y / g.Hq, hq = rec.y % g.Hq, bhk = b * g.Hkv + hq / g.rep;
      const int* cols = a.col_idx + (size_t)rec.y * g.nnz_cap + rec.w;
      const unsigned char* tiles = a.ds + ((size_t)(rec.y - a.head0) * g.nnz_cap + rec.w) * kSlab;
      // (rows of a packed cube are the first of its tiles as the fp16 forms leave them; the other form has them in every chunk)
      const uint32_t tile_bytes = a.ds_swizzled && packed_query(g, a.pk, rec.x) ? kSlab >> a.pk.shift : kSlab;
      int j = is_k ? cols[(blk == 1 && k > 1) ? 1 : 0] : 0;
      for (int t = 0; t < nt; ++t, ++tg) {
        int c1 = 0, c2 = 0, c3 = 0;
        bool text = false;
        if (is_k) {
          block_box(g, j, c1, c2, c3);
          text = block_is_text(g, j);
          if (t + 1 < nt) j = cols[(blk == 1 && 2 * t + 3 < k) ? 2 * t + 3 : 2 * t + 2];   // next tile, fetched early
        }
        const uint32_t slot = tg % C::STAGES;
        const uint32_t ds_bytes = (t == nt - 1 && (k & 1)) ? tile_bytes : 2 * tile_bytes;
        int ok = 1;
        if (lane == 0) {
          ok = tc::mbar_wait_parked(&misc->empty[slot], ((tg / C::STAGES) & 1) ^ 1, &misc->abort_flag);
          if (ok) tc::mbar_expect_tx(&misc->full[slot], is_k ? (D == 128 ? C::KBYTES / 4 : C::KBYTES / 2) : ds_bytes);
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) goto done;
        unsigned char* stage = smem + slot * C::STAGE;
        if (is_k) {
          if (lane == 0)
            tc::tma_load_5d(stage + (2 * my_h + blk) * kSlab, text ? &tm_kt : &tm_k, &misc->full[slot], my_h * 64, c1, c2, c3, bhk);
        } else if (lane == 0) {
          tc::bulk_load(stage + C::KBYTES, tiles + (size_t)t * C::DSBYTES, tile_bytes == kSlab ? ds_bytes : tile_bytes, &misc->full[slot], policy);
          if (tile_bytes != kSlab && ds_bytes > tile_bytes)
            tc::bulk_load(stage + C::KBYTES + kSlab, tiles + (size_t)t * C::DSBYTES + kSlab, tile_bytes, &misc->full[slot], policy);
        }
      }
    }
  } else if (warp == 3) {
    // ------------------------------------------------------------------ issuer
    constexpr uint32_t idesc = tc::idesc_f16(128, 64, true, false);       // A = K_pair^T from key rows, B = dS, keys along K
    constexpr uint32_t lbo = (D == 128) ? 2 * kSlab : 0;                  // distance between the two 64-channel halves of K
    const uint32_t base = tc::smem_u32(smem);
    uint32_t tg = 0, n_items = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      const int k = rec.z, nt = (k + 1) >> 1;
      if (k == 0) continue;
      const uint32_t set = n_items % kDsSets, acc = tmem_base + set * 64;
      VSA2_WAIT_PARKED(&misc->o_empty[set], ((n_items / kDsSets) & 1) ^ 1);
      for (int t = 0; t < nt; ++t, ++tg) {
        const uint32_t slot = tg % C::STAGES;
        VSA2_WAIT_PARKED(&misc->full[slot], (tg / C::STAGES) & 1);
        tc::tc_fence_after();
        if (tc::elect_one()) {
          const uint64_t da = tc::smem_desc_sw128(base + slot * C::STAGE, lbo, 1024);
          const uint32_t b_addr = base + slot * C::STAGE + C::KBYTES;
          const uint64_t db = a.ds_swizzled ? tc::smem_desc_sw128(b_addr, 16, 1024) : tc::smem_desc_plain(b_addr, 1024, 128);
          const uint32_t b_step = a.ds_swizzled ? 32 : 2048;      // 16 keys on, inside a block of 64
          // (an odd list's last tile has one block)
          const int ksteps = (t == nt - 1 && (k & 1)) ? 4 : 8;
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {
            const uint64_t oa = (uint64_t)(((ks / 4) * kSlab + (ks % 4) * 2048) >> 4);
            const uint64_t ob = (uint64_t)(((ks / 4) * kSlab + (ks % 4) * b_step) >> 4);
            if (ks < ksteps) tc::mma_ss(acc, da + oa, db + ob, idesc, t > 0 || ks > 0);
          }
          tc::mma_commit(&misc->empty[slot]);
          if (t == nt - 1) tc::mma_commit(&misc->o_full[set]);
        }
        __syncwarp();
      }
      ++n_items;
    }
  } else if (warp < 12) {
    // ------------------------------------------------------------------ epilogue: two warpgroups take the items in turn, a thread
    // has one channel: dQ[l, d] = scale * dQ^T[d, q] + dQ_c[i, d] / count(i) (dS comes without the softmax scale and
    // with its own)
    const int wg = (warp - 4) >> 2;
    const int row = ((warp & 3) << 5) | lane;
    const uint32_t lane_addr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    uint32_t n_items = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      const int i = rec.x, k = rec.z;
      const uint32_t n = n_items;
      if (k > 0) ++n_items;
      if (k == 0 ? wg != 0 : (n & 1) != (uint32_t)wg) continue;
      const int tok0 = block_token(g, i, lane), tok1 = block_token(g, i, 32 + lane);
      const float coarse_d = (a.dqc != nullptr && row < D && !block_is_text(g, i))
                                 ? a.dqc[((size_t)rec.y * g.Nvid + i) * D + row] / (float)cube_count(g, i) : 0.f;
      const float out_scale = g.scale * pow2i(-a.ds_exp[rec.y / g.rep]);      // (rec.y / rep: batch * Hkv + KV head)
      const size_t head = (size_t)rec.y * g.S;
      if (k == 0) {                            // nothing kept: the coarse gradient only
#pragma unroll 1
        for (int c = 0; c < 64; ++c) {
          const int l = __shfl_sync(0xffffffffu, c < 32 ? tok0 : tok1, c & 31);
          if (l >= 0 && row < D) store_out(a.dq, (head + l) * D + row, coarse_d, g.out_f32);
        }
        continue;
      }
      const uint32_t set = n % kDsSets;
      VSA2_WAIT_PARKED(&misc->o_full[set], (n / kDsSets) & 1);
      tc::tc_fence_after();
      // The four warps write the same table: behind this wait all of them are through with the warpgroup's item two before,
      // whose table it was -- it used the same accumulator, which is given back after the last look at the table.
      int* tok = misc->tok[wg][(n >> 1) & 1];
      tok[lane] = tok0;
      tok[32 + lane] = tok1;
      __syncwarp();
      const int rows_in = packed_query(g, a.pk, i) ? 64 >> a.pk.shift : 64;       // (what lies behind a packed cube's rows is nobody's dS)
#pragma unroll 1
      for (int part = 0; part < 4; ++part) {
        uint32_t x[16];
        tc::tmem_ld16(lane_addr + set * 64 + part * 16, x);
        tc::tmem_ld_wait();
        // a dS that left the fp16 range is an infinity and has made every channel of its query column non-finite (one store per
        // warp: with all rows out of range one per thread took 2.7 ms for 8 heads of 720p)
        if (part * 16 >= rows_in) break;       // (a quarter or half of the rows)
        if (__any_sync(0xffffffffu, row < D && any_non_finite(x)) && lane == 0) *a.range_flag = 1;
        float v[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = fmaf(__uint_as_float(x[c]), out_scale, coarse_d);
        if (row < D) store_channels<D>(a.dq, g.out_f32, head, tok + part * 16, v, row);
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&misc->o_empty[set]);
    }
  } else {
    if (!schedule_lists(&misc->queue, g, a.first_item, a.items, 1, a.row_ptr, a.item_counter, nullptr, 0, 0x7fffffff, false, a.range_flag, lane,
                      &misc->abort_flag))
      goto done;
  }

done:
  tc::tc_fence_before();
  __syncthreads();
  if (misc->abort_flag) {
    if (tid == 0) {
      atomicExch(&a.status->status, VSA2_ERR_DEVICE_TIMEOUT);
      const unsigned long long t0 = tc::global_timer_ns();
      while (tc::global_timer_ns() - t0 < 200000ull) {
      }
    }
    __syncthreads();
  }
  if (warp == 3) tc::tmem_dealloc(tmem_base, 64 * kDsSets);
}

// dQ of the heads head0 .. head0 + heads - 1 (index batch * Hq) from their dS tiles
cudaError_t launch_fine_bwd_dq_ds(const Geo& g, const void* k16, const void* ds, int head0, int heads, const int* row_ptr,
                                  const int* col_idx, const float* dqc, void* dq, StatusBlock* status, int* range_flag,
                                  int* item_counter, bool swizzled, const int* ds_exp, const PackedCubes& pk, cudaStream_t st) {
  CUtensorMap tk, tkt;
  if (!make_cube_tmap(&tk, reinterpret_cast<const bf16*>(k16), g, g.Hkv) ||      // (same element size: the maps only move bytes)
      !make_text_tmap(&tkt, reinterpret_cast<const bf16*>(k16), g, g.Hkv))
    return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  DqDsArgs a{item_counter, row_ptr, col_idx, reinterpret_cast<const unsigned char*>(ds), swizzled ? 1 : 0, pk, dqc, dq, status, range_flag, ds_exp, head0, head0 * g.N, heads * g.N};
  const int grid = a.items < sms ? a.items : sms;
#define VSA2_LAUNCH_DQ_DS(DD)                                                                                                    \
  do {                                                                                                                           \
    static KernelAttr attr_;                                                                                                     \
    if ((e = prepare_kernel((const void*)fine_bwd_dq_ds_kernel<DD>, attr_, DqDs<DD>::smem_bytes))) return e;                     \
    launch_kernel(fine_bwd_dq_ds_kernel<DD>, grid, ds_threads(DD), DqDs<DD>::smem_bytes, st, tk, tkt, g, a);                               \
  } while (0)
  if (g.D == 128) VSA2_LAUNCH_DQ_DS(128);
  else VSA2_LAUNCH_DQ_DS(64);
#undef VSA2_LAUNCH_DQ_DS
  return cudaGetLastError();
}

}  // namespace vsa2
