// dQ of the fine branch from stored dS for cubes of 128 tokens: dQ [128 q, D] += dS [128 q, 128 kv] K [128 kv, D], one tcgen05
// product per 128 x 128 tile (fine_bwd_dq_ds_tc.cu is the same pass for 64-token cubes).
//
// The dK/dV pass (fine_bwd128_tc.cu) forms dS^T of every kept pair with a key per thread and stores it, fp16, as
// [chunk of 8 queries][128 keys][8 queries]: a warp then writes 512 contiguous bytes at a time, and 8 keys of a chunk are one core
// matrix of an unswizzled operand with the queries along M, so a tile is read with one 32 KB bulk copy and multiplied as it lies.
// Recomputing S and dP in a pass of its own (fine_bwd128_tc.cu, pass 0) takes two more products, the exponentials and the V and
// dO tiles; it remains for calls without scratch, for precision flags and as the range fallback.  The price here is 32 KB
// per pair written to and read from HBM, which bounds this pass: 10 heads of 219,600 tokens (top-64) are 40.3 GB in 7 ms, against 12.3
// for the recomputing pass; the dK/dV pass goes from 17.8 to 21 ms for writing them (the card is at its power cap throughout).
// The tiles hold the values the recomputing pass would form (same operands, same order), so dQ is the same bit for bit.
#include "fine_bwd_tc.cuh"

namespace vsa2 {

constexpr int kW2DsThreads = 288;      // 2 producer warps of K blocks, 1 of dS tiles, issuer; 4 epilogue warps; scheduler
constexpr int kW2DsSets = 2;           // accumulators, used by item in turn

template <int D>
struct DqDs128 {
  static constexpr int DH = D / 64;
  static constexpr uint32_t KBYTES = 2 * DH * kSlab;      // the two half-cubes of a key cube, [channel half][A | B]
  static constexpr uint32_t DSBYTES = 128 * 128 * 2;
  static constexpr uint32_t STAGE = KBYTES + DSBYTES;
  static constexpr int STAGES = D == 128 ? 3 : 4;
  static constexpr uint32_t OFF_MISC = STAGES * STAGE;
  static constexpr size_t smem_bytes = OFF_MISC + 1024 + 1024;
};

struct DqDs128Misc {
  uint64_t full[4], empty[4];
  uint64_t o_full[kW2DsSets], o_empty[kW2DsSets];
  ListQueue queue;
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(DqDs128Misc) <= 1024, "misc region too small");

// `g`: the half-cube geometry; the map, the items and the tiles are those of the cubes
template <int D>
__global__ void __launch_bounds__(kW2DsThreads, 1)
fine_bwd128_dq_ds_kernel(const __grid_constant__ CUtensorMap tm_k, Geo g, long long cap, DqDsArgs a) {
  using C = DqDs128<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  DqDs128Misc* misc = reinterpret_cast<DqDs128Misc*>(smem + C::OFF_MISC);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    misc->abort_flag = 0;
    for (int s = 0; s < C::STAGES; ++s) {
      tc::mbar_init(&misc->full[s], 3);       // the three producers
      tc::mbar_init(&misc->empty[s], 1);
    }
    for (int s = 0; s < kW2DsSets; ++s) {
      tc::mbar_init(&misc->o_full[s], 1);
      tc::mbar_init(&misc->o_empty[s], 4);
    }
    list_queue_init(&misc->queue, 8);
    tc::fence_barrier_init();
    tc::prefetch_tmap(&tm_k);
  }
  if (warp == 3) {
    tc::tmem_alloc(&misc->tmem_base, 128 * kW2DsSets);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = misc->tmem_base;
  grid_enter(false);
  if (__syncthreads_or(tid == 0 && *a.range_flag != 0)) {       // the fallback computes dQ
    if (warp == 3) tc::tmem_dealloc(tmem_base, 128 * kW2DsSets);
    return;
  }

  if (warp < 3) {
    // ------------------------------------------------------------------ producers: first half of a key cube, second, dS tile
    const uint64_t policy = tc::evict_first_policy();      // (the tiles pass through once, the K cubes stay)
    uint32_t tg = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      if (warp == 0 && lane == 0) tc::mbar_arrive(&misc->queue.taken);
      const int k = rec.z;
      if (k == 0) continue;
      const int b = rec.y / g.Hq, hq = rec.y % g.Hq, bhk = b * g.Hkv + hq / g.rep;
      const int* cols = a.col_idx + (size_t)rec.y * cap + rec.w;
      const unsigned char* tiles = a.ds + ((size_t)(rec.y - a.head0) * cap + rec.w) * C::DSBYTES;
      int j = warp < 2 ? cols[0] : 0;
      for (int t = 0; t < k; ++t, ++tg) {
        int c1 = 0, c2 = 0, c3 = 0;
        if (warp < 2) {
          block_box(g, 2 * j + warp, c1, c2, c3);
          if (t + 1 < k) j = cols[t + 1];          // the next entry is on its way while this warp waits
        }
        const uint32_t slot = tg % C::STAGES;
        int ok = 1;
        if (lane == 0) {
          ok = tc::mbar_wait_parked(&misc->empty[slot], ((tg / C::STAGES) & 1) ^ 1, &misc->abort_flag);
          if (ok) tc::mbar_expect_tx(&misc->full[slot], warp < 2 ? C::KBYTES / 2 : C::DSBYTES);
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) goto done;
        unsigned char* stage = smem + slot * C::STAGE;
        if (warp < 2) {
          if (lane < C::DH) tc::tma_load_5d(stage + (2 * lane + warp) * kSlab, &tm_k, &misc->full[slot], lane * 64, c1, c2, c3, bhk);
        } else if (lane == 0) {
          tc::bulk_load(stage + C::KBYTES, tiles + (size_t)t * C::DSBYTES, C::DSBYTES, &misc->full[slot], policy);
        }
      }
    }
  } else if (warp == 3) {
    // ------------------------------------------------------------------ issuer
    constexpr uint32_t idesc = tc::idesc_f16(128, D, true, true);         // A = dS with the queries along M, B = K with the channels along N
    constexpr uint32_t lbo = (D == 128) ? 2 * kSlab : 0;                  // distance between the two 64-channel halves of K
    const uint32_t base = tc::smem_u32(smem);
    uint32_t tg = 0, n_items = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      const int k = rec.z;
      if (k == 0) continue;
      const uint32_t set = n_items % kW2DsSets, acc = tmem_base + set * 128;
      VSA2_WAIT_PARKED(&misc->o_empty[set], ((n_items / kW2DsSets) & 1) ^ 1);
      for (int t = 0; t < k; ++t, ++tg) {
        const uint32_t slot = tg % C::STAGES;
        VSA2_WAIT_PARKED(&misc->full[slot], (tg / C::STAGES) & 1);
        tc::tc_fence_after();
        if (tc::elect_one()) {
          const uint64_t db = tc::smem_desc_sw128(base + slot * C::STAGE, lbo, 1024);
          // (queries along M: 8 keys of a chunk are one core matrix; chunks 2048 bytes apart, the next 8 keys 128)
          const uint64_t da = tc::smem_desc_plain(base + slot * C::STAGE + C::KBYTES, 128, 2048);
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {
            const uint64_t oa = (uint64_t)((ks * 256) >> 4);
            const uint64_t ob = (uint64_t)(((ks / 4) * kSlab + (ks % 4) * 2048) >> 4);
            tc::mma_ss(acc, da + oa, db + ob, idesc, t > 0 || ks > 0);
          }
          tc::mma_commit(&misc->empty[slot]);
          if (t == k - 1) tc::mma_commit(&misc->o_full[set]);
        }
        __syncwarp();
      }
      ++n_items;
    }
  } else if (warp < 8) {
    // ------------------------------------------------------------------ epilogue, a thread per query: dQ[l, d] = scale * dQ[q, d] +
    // dQ_c[block, d] / count(block) (dS comes without the softmax scale and with its own)
    const int row = ((warp & 3) << 5) | lane, member = row >> 6;
    const uint32_t lane_addr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    uint32_t n_items = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      const int k = rec.z, blk = 2 * rec.x + member;
      const int l_tok = block_token(g, blk, row & 63);
      const float inv_cnt = 1.f / (float)cube_count(g, blk);
      const float sc = g.scale * pow2i(-a.ds_exp[rec.y / g.rep]);      // (rec.y / rep: batch * Hkv + KV head)
      const uint32_t set = n_items % kW2DsSets;
      if (k > 0) {
        VSA2_WAIT_PARKED(&misc->o_full[set], (n_items / kW2DsSets) & 1);
        tc::tc_fence_after();
      }
#pragma unroll 1
      for (int col0 = 0; col0 < D; col0 += 32) {
        uint32_t acc[32];
        if (k > 0) {
          tc::tmem_ld32(lane_addr + set * 128 + col0, acc);
          tc::tmem_ld_wait();
          // a dS that left the fp16 range is an infinity and has made every channel of its query non-finite
          if (__any_sync(0xffffffffu, any_non_finite(acc)) && lane == 0) *a.range_flag = 1;
        } else {
#pragma unroll
          for (int e = 0; e < 32; ++e) acc[e] = 0u;
        }
        if (l_tok >= 0) {
          float val[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) val[e] = __uint_as_float(acc[e]) * sc;
          if (a.dqc != nullptr) {
            const float4* c4 = reinterpret_cast<const float4*>(a.dqc + ((size_t)rec.y * g.Nvid + blk) * D + col0);
#pragma unroll
            for (int e4 = 0; e4 < 8; ++e4) {
              const float4 cv = c4[e4];
              val[4 * e4 + 0] = fmaf(cv.x, inv_cnt, val[4 * e4 + 0]);
              val[4 * e4 + 1] = fmaf(cv.y, inv_cnt, val[4 * e4 + 1]);
              val[4 * e4 + 2] = fmaf(cv.z, inv_cnt, val[4 * e4 + 2]);
              val[4 * e4 + 3] = fmaf(cv.w, inv_cnt, val[4 * e4 + 3]);
            }
          }
          const size_t idx = ((size_t)rec.y * g.S + l_tok) * D + col0;
          if (g.out_f32) {
            float* dst = reinterpret_cast<float*>(a.dq) + idx;
#pragma unroll
            for (int e = 0; e < 32; e += 4) *reinterpret_cast<float4*>(dst + e) = make_float4(val[e], val[e + 1], val[e + 2], val[e + 3]);
          } else {
            bf16* dst = reinterpret_cast<bf16*>(a.dq) + idx;
#pragma unroll
            for (int e = 0; e < 32; e += 8)
              *reinterpret_cast<uint4*>(dst + e) = make_uint4(pack_bf16x2(val[e], val[e + 1]), pack_bf16x2(val[e + 2], val[e + 3]),
                                                              pack_bf16x2(val[e + 4], val[e + 5]), pack_bf16x2(val[e + 6], val[e + 7]));
          }
        }
        __syncwarp();
      }
      if (k > 0) {
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&misc->o_empty[set]);
        ++n_items;
      }
    }
  } else {
    Geo cubes = g;
    cubes.N = g.N / 2;
    if (!schedule_lists(&misc->queue, cubes, a.first_item, a.items, 1, a.row_ptr, a.item_counter, nullptr, 0, 0x7fffffff, false,
                      a.range_flag, lane, &misc->abort_flag))
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
  if (warp == 3) tc::tmem_dealloc(tmem_base, 128 * kW2DsSets);
}

// dQ of the heads head0 .. head0 + heads - 1 (index batch * Hq) from their dS tiles; `g`: the half-cube geometry, `cap`: entries of
// the cube map per head, row_ptr / col_idx: the cube map
cudaError_t launch_fine_bwd128_dq_ds(const Geo& g, long long cap, const void* k16, const void* ds, int head0, int heads,
                                     const int* row_ptr, const int* col_idx, const float* dqc, void* dq, StatusBlock* status,
                                     int* range_flag, int* item_counter, const int* ds_exp, cudaStream_t st) {
  CUtensorMap tk;
  if (!make_cube_tmap(&tk, reinterpret_cast<const bf16*>(k16), g, g.Hkv)) return cudaErrorInvalidValue;      // (same element size)
  int sms = 0;
  cudaError_t e;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  DqDsArgs a{item_counter, row_ptr, col_idx, reinterpret_cast<const unsigned char*>(ds), 0, PackedCubes{}, dqc, dq, status, range_flag, ds_exp,
             head0, head0 * (g.N / 2), heads * (g.N / 2)};
  const int grid = a.items < sms ? a.items : sms;
  if (g.D == 128) {
    static KernelAttr attr;
    if ((e = prepare_kernel((const void*)fine_bwd128_dq_ds_kernel<128>, attr, DqDs128<128>::smem_bytes))) return e;
    launch_kernel(fine_bwd128_dq_ds_kernel<128>, grid, kW2DsThreads, DqDs128<128>::smem_bytes, st, tk, g, cap, a);
  } else {
    static KernelAttr attr;
    if ((e = prepare_kernel((const void*)fine_bwd128_dq_ds_kernel<64>, attr, DqDs128<64>::smem_bytes))) return e;
    launch_kernel(fine_bwd128_dq_ds_kernel<64>, grid, kW2DsThreads, DqDs128<64>::smem_bytes, st, tk, g, cap, a);
  }
  return cudaGetLastError();
}

}  // namespace vsa2
