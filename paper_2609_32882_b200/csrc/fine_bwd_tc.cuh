// Shared pieces of the two backward passes of the fine branch (fine_bwd_tc.cu: dQ pass, fine_bwd_dkv_tc.cu: dK/dV pass):
// shared-memory plan, barriers, the ring producer.
#pragma once
#include "tc_attn.cuh"

namespace vsa2 {

constexpr int kDqThreads = 416;    // dQ pass: 4 service warps, 2 x 4 elementwise warps, 1 more issuer warp
constexpr int kDkvThreads = 768;   // dK/dV pass: 4 service warps, 2 x 4 elementwise warps, 4 row-statistics warps, 2 issuer warps,
                                   // a scheduler warp (and an idle one), 4 epilogue warps
constexpr int kRingA = 3;          // slots of the ring whose tiles are also an operand of the last product of a tile
constexpr int kRingB = 2;          // (the ring-B slot of a tile is also the index of its tensor-memory buffers)
static_assert(kRingB == 2, "ring B shares its slot index with the two accumulator buffers");

// Barriers of the dK/dV pass's rings where they have more slots than BwdMisc holds (behind it)
struct BwdRings {
  uint64_t a_full[6], a_empty[6], b_full[6], b_empty[6];
};

// Shared-memory plan of both passes (D = 128: 5 x 32 KB ring slots, 2 x 16 KB stationary tiles, 2 x 16 KB operand
// buffers, 2 KB of barriers and per-block vectors: exactly the 227 KB a block may use).  Ring A has 3 slots, ring B 2;
// each ring has one producing warp and fixed consuming roles.
// RA: slots of ring A; NP: 16 KB operand buffers (the dK/dV pass in its split mode trades one ring-A slot for the two
// buffers that hold the low-order parts of P and dS).
template <int D, int RA = kRingA, int NP = 2, int RB = kRingB>
struct BwdTc {
  static constexpr int DH = D / 64;
  static constexpr uint32_t SLOT = 2 * DH * kSlab;   // a pair of cube tiles, [half][A | B]
  static constexpr uint32_t TILE = DH * kSlab;       // one cube tile, [half]
  static constexpr uint32_t PBYTES = 128 * 128;      // 128 rows x 64 bf16
  static constexpr uint32_t OFF_RING_B = RA * SLOT;
  static constexpr uint32_t OFF_ST0 = (RA + RB) * SLOT;       // stationary tile 0 (Q or K)
  static constexpr uint32_t OFF_ST1 = OFF_ST0 + TILE;             // stationary tile 1 (dO or V)
  static constexpr uint32_t OFF_P = OFF_ST1 + TILE;               // the 16 KB operand buffers
  static constexpr uint32_t OFF_MISC = OFF_P + NP * PBYTES;
  static constexpr uint32_t MISC_BYTES = D == 64 ? 2048 + sizeof(BwdRings) : 2048;
  static constexpr size_t smem_bytes = OFF_MISC + MISC_BYTES + 1024;
};

// Stores 16 values per thread -- channel `row` of 16 tokens, the warp's lanes being 32 neighbouring channels -- to the token
// rows named by tok[0 .. 15] (shared memory, -1 = no token).  No exchange between lanes: shuffles and a transpose in shared
// memory both use the data pipe that bounds the passes, and a chain of them took the epilogue warps three times as long as
// storing 64 bytes per warp and token.  Sixteen tokens at a time in a rolled loop, because an epilogue's code passes through the
// instruction cache once per item (kernels of 52 and 29 KB instead of 70 and 40 with 32 tokens): backward, us, 13 x 27 x 47 tokens, 16 heads of
// 64 channels 728 -> 679; 8 heads on 2 with budgets 14135 -> 13693.
template <int D>
__device__ __forceinline__ void store_channels(void* out, int out_f32, size_t head, const int* tok, const float (&v)[16], int row) {
  if (out_f32) {
    float* base = reinterpret_cast<float*>(out) + head * D + row;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int l = tok[c];
      if (l >= 0) base[(size_t)l * D] = v[c];
    }
  } else {
    bf16* base = reinterpret_cast<bf16*>(out) + head * D + row;
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int l = tok[c];
      if (l >= 0) base[(size_t)l * D] = __float2bfloat16_rn(v[c]);
    }
  }
}

struct DqDsArgs {
  int* item_counter;    // global, zero before the launch
  const int* row_ptr;
  const int* col_idx;
  const unsigned char* ds;
  int ds_swizzled;      // layout of the tiles, see fine_bwd_dkv_tc.cu
  PackedCubes pk;       // as in the dK/dV pass: only the first rows of a tile of a packed query cube have been written
  const float* dqc;     // [B, Hq, N, D] or null
  void* dq;
  StatusBlock* status;
  int* range_flag;      // the launch runs if it is clear, and sets it if a dS had left the fp16 range
  const int* ds_exp;    // exponent of the scale of dS per KV group (DsScale)
  int head0;            // (batch * Hq) index of the first head of the dS scratch
  int first_item, items;
};

constexpr int kWholeBlock = -2;
struct BwdMisc {
  uint64_t st_full, st_empty, o_full[2], o_empty[2];       // (the dQ pass uses one accumulator)
  uint64_t a_full[kRingA], a_empty[kRingA], b_full[kRingB], b_empty[kRingB];
  uint64_t s_full[2], s_free[2], dp_full[2], dp_free[2];   // the two score / dP accumulators in tensor memory
  uint64_t p_ready, p_free;                                 // dK/dV pass: the P operand buffer; dQ pass: p_ready is the group barrier
                                                            // of its 256 elementwise threads
  uint64_t ds_ready[2], ds_free[2];                         // dS operand buffers (the dK/dV pass has one)
  uint64_t stat_full, stat_free;                            // dK/dV pass: the per-row statistics of a tile
  union {                                                   // work items of this CTA
    ItemQueue items;                                        // dQ pass (see tc_attn.cuh)
    ListQueue queue;                                         // dK/dV pass
  };
  uint32_t tmem_base;
  int abort_flag;
  // dQ pass: lse2[tb][c] = stats[tb * 64 + c], delta[tb][c] = stats[128 + tb * 64 + c]: per query column of the item with
  // parity tb, lse * log2(e) (+inf for padding) and delta.  dK/dV pass: (lse * log2(e), delta) of the 128 query rows of
  // the current tile, interleaved.
  alignas(16) float stats[256];
  union {
    unsigned char edge[kRingA][2];   // dQ pass: edge flags of the two key cubes in each ring-A slot (written by its producer)
    // dK/dV pass: places of the dS blocks of a tile's two halves in the scratch (-1: none), by tile index mod 3 (they are written at
    // most two tiles ahead of their last reader); a half that is one block has kWholeBlock in its second word
    int ds_slot[3][2][4];
  };
  int tok[128];                    // raster tokens of the rows of an item's block, by parity (dK/dV pass: of the items with entries)
};
static_assert(sizeof(BwdMisc) <= 2048, "misc region too small");

__device__ __forceinline__ void bwd_init_barriers(BwdMisc* misc) {
  misc->abort_flag = 0;
  tc::mbar_init(&misc->st_full, 1);
  tc::mbar_init(&misc->st_empty, 2);     // both first-stage issuers
  for (int s = 0; s < 2; ++s) {
    tc::mbar_init(&misc->o_full[s], 1);       // re-initialised by the dK/dV pass
    tc::mbar_init(&misc->o_empty[s], 256);
  }
  for (int s = 0; s < kRingA; ++s) {
    tc::mbar_init(&misc->a_full[s], 1);
    tc::mbar_init(&misc->a_empty[s], 1);
  }
  for (int s = 0; s < kRingB; ++s) {
    tc::mbar_init(&misc->b_full[s], 1);
    tc::mbar_init(&misc->b_empty[s], 1);
  }
  for (int s = 0; s < 2; ++s) {
    tc::mbar_init(&misc->s_full[s], 1);
    tc::mbar_init(&misc->s_free[s], 256);
    tc::mbar_init(&misc->dp_full[s], 1);
    tc::mbar_init(&misc->dp_free[s], 256);
    tc::mbar_init(&misc->ds_ready[s], 256);
    tc::mbar_init(&misc->ds_free[s], 1);
  }
  tc::mbar_init(&misc->p_ready, 256);
  tc::mbar_init(&misc->p_free, 1);
  tc::mbar_init(&misc->stat_full, 128);
  tc::mbar_init(&misc->stat_free, 256);
}

// One warp streams pairs of cube tiles into a ring of NS slots: lane 0 owns the barriers, lanes 0 .. 2*DH-1 issue one
// box each (half h = lane / 2 of block lane & 1).  C3, C2, C1: box coordinates of this lane's block in map TMAP, `bh`: its head.
// `LANE0_PRE`: statement lane 0 runs once the slot is free, before the loads are armed (may use slot_).
#define VSA2_RING_LOAD(FULL, EMPTY, NS, RING_BASE, TMAP, SEQ, CT, CH, CW, BH, LANE0_PRE, WAITFN)                  \
  do {                                                                                                            \
    const uint32_t slot_ = (SEQ) % (NS), par_ = ((SEQ) / (NS)) & 1;                                               \
    int ok_ = 1;                                                                                                  \
    if (lane == 0) {                                                                                              \
      ok_ = tc::WAITFN(&(EMPTY)[slot_], par_ ^ 1, &misc->abort_flag);                                             \
      if (ok_) {                                                                                                  \
        LANE0_PRE;                                                                                                \
        tc::mbar_expect_tx(&(FULL)[slot_], C::SLOT);                                                              \
      }                                                                                                           \
    }                                                                                                             \
    if (!__shfl_sync(0xffffffffu, ok_, 0)) goto done;                                                             \
    if (lane < 2 * C::DH)                                                                                         \
      tc::tma_load_5d((RING_BASE) + slot_ * C::SLOT + (2 * (lane >> 1) + (lane & 1)) * kSlab, (TMAP), &(FULL)[slot_], \
                      (lane >> 1) * 64, (CW), (CH), (CT), (BH));                                                  \
  } while (0)

// An exponent of max|dO| max|O| from which on a dS is taken to leave the fp16 range: a weight of 2^-8 in the row of the largest dO is
// enough.  The flag then goes up before the fp16 passes have run for nothing (720p, 8 heads, dO of 3e6: 14.6 -> 7 ms).
constexpr int kBeyondF16 = 22;
// DsScale::exp of the groups first, first + step, ... (the whole block calls it); true if the fp16 forms are not to run:
// O below least_o, or dS beyond the fp16 range
__device__ __forceinline__ bool form_ds_exp(const DsScale& s, int groups, int per_group, int first, int step) {
  __shared__ unsigned red[2][8];
  bool bad = false;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int grp = first; grp < groups; grp += step) {
    const uint2* m = reinterpret_cast<const uint2*>(s.absmax) + (size_t)grp * per_group;      // (bit patterns order like the numbers)
    unsigned d = 0u, o = 0u;
    for (int i = threadIdx.x; i < per_group; i += 256) {
      const uint2 v = m[i];
      d = max(d, v.x);
      o = max(o, v.y);
    }
    d = __reduce_max_sync(0xffffffffu, d);
    o = __reduce_max_sync(0xffffffffu, o);
    if (lane == 0) {
      red[0][warp] = d;
      red[1][warp] = o;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) {
        d = max(d, red[0][w]);
        o = max(o, red[1][w]);
      }
      const int e = (int)(d >> 23) - 127 + (int)(o >> 23) - 127;
      s.exp[grp] = d == 0u || o == 0u ? 0 : max(0, min(-3 - e, 100));
      bad |= o != 0u && (__uint_as_float(o) < s.least_o || (d != 0u && e >= kBeyondF16));
    }
    __syncthreads();
  }
  return bad;
}

struct CastJob {
  const uint4* xa;
  uint4* ya;
  size_t na;
  const uint4* xb;
  uint4* yb;
  size_t nb;
  const int* b_exp;
  unsigned b_group;
  int* range_flag;
};
constexpr int kCastBlocksPerSm = 16;
// (na, nb, b_group: elements, multiples of 8)
inline CastJob cast_job(const bf16* a, void* a16, size_t na, const bf16* b, void* b16, size_t nb, const int* b_exp, size_t b_group, int* range_flag) {
  return CastJob{reinterpret_cast<const uint4*>(a), reinterpret_cast<uint4*>(a16), na / 8, reinterpret_cast<const uint4*>(b), reinterpret_cast<uint4*>(b16),
                 nb / 8, b_exp, (unsigned)(b_group / 8), range_flag};
}
// Copies of two bf16 tensors in fp16 (8 elements per thread and step), b times 2^b_exp[its group of `b_group` steps] if there is one.
// A finite bf16 below 65520 in magnitude has an exact fp16 image if it is a multiple of 2^-24 (all of 2^-17 and more are: fp16
// keeps more mantissa bits), and one within 2^-25 otherwise; a finite value beyond that range sets `range_flag` and the caller's
// fp16 kernels stand back.
// SCALED: there is a b_exp.  (Without it the magnitudes are compared as the integers they are; a thread walks its groups by adding
// quotient and remainder of its stride: a division per step and products of 1 made the copies of 480p 30 us longer.)
template <bool SCALED>
__device__ __forceinline__ void cast_bf16_to_f16(const CastJob& job, unsigned block, unsigned blocks) {
  const size_t stride = (size_t)blocks * blockDim.x, n = job.na + job.nb, first = (size_t)block * blockDim.x + threadIdx.x;
  bool bad = false;
  constexpr int U = 4;      // 16-byte loads in flight per thread (a pure streaming kernel)
  unsigned grp = 0u, in_grp = 0u, step_q = 0u, step_r = 0u;      // SCALED: group of element group i of b, place in it; the same of a stride
  if (SCALED) {
    step_q = (unsigned)(stride / job.b_group);
    step_r = (unsigned)(stride % job.b_group);
  }
  bool in_b = false;
  for (size_t i0 = first; i0 < n; i0 += U * stride) {
    uint4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const size_t i = i0 + u * stride;
      v[u] = i < n ? (i < job.na ? job.xa[i] : job.xb[i - job.na]) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const size_t i = i0 + u * stride;
      if (i >= n) break;
      const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
      float f = 1.f;
      if (SCALED && i >= job.na) {
        if (!in_b) {
          in_b = true;
          grp = (unsigned)((i - job.na) / job.b_group);
          in_grp = (unsigned)((i - job.na) % job.b_group);
        } else {
          grp += step_q;
          in_grp += step_r;
          if (in_grp >= job.b_group) {
            in_grp -= job.b_group;
            ++grp;
          }
        }
        // (a scaled value stays finite: the exponent takes the largest of a group to 2^-2 / max |O| at most)
        f = pow2i(job.b_exp[grp]);
      }
      uint32_t r[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float x0 = __uint_as_float(w[e] << 16), x1 = __uint_as_float(w[e] & 0xffff0000u);
        if (SCALED) {
          x0 *= f;
          x1 *= f;
        }
        // magnitudes as bit patterns (65536 <= |x| < infinity)
        const uint32_t m0 = __float_as_uint(x0) & 0x7fffffffu, m1 = __float_as_uint(x1) & 0x7fffffffu;
        bad |= m0 - 0x47800000u < 0x38000000u || m1 - 0x47800000u < 0x38000000u;
        const __half2 h = __floats2half2_rn(x0, x1);
        r[e] = *reinterpret_cast<const uint32_t*>(&h);
      }
      const uint4 o = make_uint4(r[0], r[1], r[2], r[3]);
      if (i < job.na) job.ya[i] = o;
      else job.yb[i - job.na] = o;
    }
  }
  if (bad) atomicExch(job.range_flag, 1);
}

}  // namespace vsa2
