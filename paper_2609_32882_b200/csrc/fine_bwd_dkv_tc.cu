// dK/dV pass of the backward of the fine branch (gradient of paper Eq. 12) on the Blackwell tensor cores: the formulation,
// the shared-memory plan and the dQ pass are in fine_bwd_tc.cu / fine_bwd_tc.cuh.
//
// The pass runs at the edge of the SM's instruction cache (about 32 KB; a miss goes to a cache that the SMs of a GPC share
// and that saturates): with 87 KB of code its hit rate was 90 % and the time moved by several per cent with any change of
// the code's size or layout.  What is executed per tile and per item is therefore kept small: one query head per KV head
// is a template case of its own, the key-column mask comes from the token table, index divisions are multiplies.
#include "fine_bwd_tc.cuh"

namespace vsa2 {

// ================================================================================================
// dK/dV pass
// ================================================================================================
struct DkvArgs {
  int* item_counter;    // global, zero before the launch
  const float* lse;
  const float* delta;
  const int* col_ptr;
  const int* row_idx;
  const float* dkc;     // [B, Hq, N, D] per query head, or null
  const float* dvc;
  void* dk;
  void* dv;
  StatusBlock* status;
  int k_lo, k_hi;       // the launch handles the KV blocks whose column lists hold k_lo .. k_hi entries, and leaves the others alone
  int* range_flag;      // fp16 form and its fallback, as in DqArgs of the dQ pass (when = 0: the launch always runs)
  int when;
  int first_item, items;  // work items of the launch (block lists of a range of KV heads)
  unsigned char* ds;    // null, or the scratch for dS in fp16 (forms STORES_DS): [entry of the row lists of heads ds_head0 ..][8 chunks of 8 keys][64 q]
  const int* ds_pos;    // [B, Hq, nnz_cap]: place of every entry of the column lists in the row lists
  int ds_head0;
  const int* ds_exp;    // null, or the exponent of the scale of dS per KV group (DsScale; forms whose dS is rounded to fp16)
  const int* order;     // null, or the order in which the items are drawn
  PackedCubes pk;       // PACK
  int overlap;          // 1: the launch behind this one may start while this one runs; 2: this one may be running beside the one before it
};

constexpr int kMaxRep = 16;   // query heads per KV head the dK/dV pass supports

// entry e of the concatenated column lists of the group's query heads -> (query head, query block)
// (`cnt_prefix`, `col_beg`: per-head counts prefix and list starts of the item, read once per item so that this lookup
// costs a single global load)
// (`POS`: also its place in the row lists)
// PACK: entry e is a tile of 64 rows, `sub` the packed cube of it that is asked for (the last one again beyond the list's end);
// returns 0 for a block that fills the tile, 1 for a packed cube, 2 for one beyond the end.  `col_full`, `col_cnt`: entries of each
// head's list in front of the cut layer, and of all of it.
template <bool POS = false, bool PACK = false>
__device__ __forceinline__ int dkv_entry(const Geo& g, const DkvArgs& a, int rep, int b, int hk, const int* cnt_prefix,
                                         const int* col_beg, int e, int& bhq, int& i, int* pos = nullptr, int sub = 0,
                                         const int* col_full = nullptr, const int* col_cnt = nullptr) {
  int hh = 0;
  while (hh + 1 < rep && e >= cnt_prefix[hh + 1]) ++hh;
  bhq = b * g.Hq + hk * rep + hh;
  int v = e - cnt_prefix[hh], kind = 0;
  if (PACK && v >= col_full[hh]) {
    const int full = col_full[hh], end = col_cnt[hh] - (g.N - g.Nvid), groups = (end - full + (1 << a.pk.shift) - 1) >> a.pk.shift;
    if (v < full + groups) {
      v = full + ((v - full) << a.pk.shift) + sub;
      kind = v < end ? 1 : 2;
      v = min(v, end - 1);
    } else {
      v += end - full - groups;                  // (a text block)
    }
  }
  const size_t at = (size_t)bhq * g.nnz_cap + col_beg[hh] + v;
  i = a.row_idx[at];
  if (POS && a.ds != nullptr) *pos = a.ds_pos[at];
  return kind;
}

// Slots of the Q ring and of the dO ring.  With 64 channels a slot is 16 KB, half of what the plan is made for, and a short list's pass waits
// for its loads, so there are more of them.  Backward of 13 x 27 x 47 tokens, 16 heads of 64 channels, us: 3 + 2 slots 816, 4 + 3 767, 5 + 4 769,
// 6 + 4 777.
__host__ __device__ constexpr int dkv_ring_a(int D, bool split) { return D == 64 ? 4 : split ? 2 : kRingA; }
__host__ __device__ constexpr int dkv_ring_b(int D) { return D == 64 ? 3 : kRingB; }

// Roles: warp 0 = TMA producer of the Q pairs (ring A) and of the stationary K and V tiles, warp 1 = TMA producer of the
// dO pairs (ring B), warp 2 = issuer of S = Q_pair K^T, warp 3 = issuer of dP = dO_pair V^T, warp 16 = issuer of
// dV^T += dO_pair^T P (frees the dO slot), warp 17 = issuer of dK^T += Q_pair^T dS (frees the Q slot), warps 4..11 =
// elementwise stage (each half of the key columns): P is handed to the dV^T product before dS is formed;
// warps 12..15 = one thread per query row of the tile: they look up the row's (head, block, token) and fetch its lse and
// delta one tile ahead, so that the elementwise warps, which bound the pass, touch no global memory inside a tile; warp 18 =
// scheduler (ListQueue); warps 20..23 = epilogue.  The accumulators of dK^T and dV^T exist twice (without SPLIT), so the
// elementwise warps go from one KV block to the next while the epilogue warps read out and store the last one: with
// the epilogue on the elementwise warps, 9200 of 85000 cycles of a 720p item (top-64) went by between its last tile and the
// first of the next item (clock64 trace: 3900 epilogue, 3200 fetching the next item's record and lists, 2100 waits).
// SPLIT: P and dS are handed to the dV^T and dK^T products as [bf16(X) | bf16(X - bf16(X))] (N = 128 products into two
// accumulator halves that the epilogue adds), which removes their bf16 rounding from dV and dK: a KV block sums hundreds of
// query blocks (times the query heads of a GQA group), and with plain bf16 operands that noise alone passes 2e-2.  The two
// extra operand buffers take the place of the third ring-A slot.
// MHA: one query head per KV head (g.rep == 1): the per-head prefix of the column lists and the search in it fold away,
// which takes several KB out of every role's per-item code and out of the producers' and statistics warps' tile loops
// (the pass runs at the edge of the SM's instruction cache).
// F16 (without SPLIT): the maps of Q and K point at the fp16 copies the dQ pass has made and dS is rounded to fp16, so S and
// the dK^T product are fp16 x fp16 instructions; dP and the dV^T product keep bf16 operands (V and dO are not copied, P is
// rounded to bf16).  dK is where the rounding of the plain form shows (|dK| reaches 15 on the blocks most queries keep):
// with 11 bits in dS it stays below 1e-2 there, and the second launch for the long lists is not needed.  The launch stands
// back when the range flag is up: the dQ pass, which runs first, forms the same dS values and raises it if one of them (or
// a value of Q or K) leaves the fp16 range.
// With `a.ds` (the fp16 forms, and SPLIT for GQA groups) dS also goes to memory, rounded to fp16 without a clamp, for the dQ pass of
// fine_bwd_dq_ds_tc.cu: with SPLIT the elementwise threads
// store a pair's tile as [chunk of 8 keys][query]; the fp16 forms have it in shared memory as the dK product's operand, and warp
// 19 copies it as it stands, [query][64 keys] with the 128-byte swizzle (stored by the elementwise threads it cost the pass 14 %).  A dS beyond the fp16 range is an infinity there, which
// that pass finds and turns into the range flag; the fp16 forms then also use it unclamped (their result is redone).
// No key column is masked: the columns of positions without a token are accumulator columns that are never read out, and
// in dQ they meet zero rows of K (fine_bwd_tc.cu).
// dS is scaled by 2^ds_exp (DsScale).  The weights carry the scale, through the lse of a row, so P and dV^T are scaled as well (P is
// bf16 there, whose range has room); with F16 = 2 the copy of dO carries it and delta is multiplied.  The epilogue takes it out.
// F16 = 2: all four maps point at fp16 copies and P is rounded to fp16 as well (every product fp16 x fp16): the form for GQA
// groups, where a KV block sums the query blocks of several heads and bf16 P leaves dV at 1.4e-2 (480p sample, |dV| = 11).
// F16 = 3: the same without `a.ds`, dS clamped: the recomputing dQ pass forms dP from the bf16 originals, of which the copies of V and
// dO can be 2^-25 off, so of a dS next to the limit one pass may have 65504 and the other an infinity that no flag tells of.
// PACK: query cubes of a cut last layer (PackedCubes) share the 64-row halves of a tile: their boxes have fewer frames and lie one
// behind the other, row statistics and dS places go by cube.  Every grid of 4n + 1 frames runs fewer tiles for it (21 frames: an
// eighth); a form of its own, so that the others keep their code.  Backward, ms: 720p, 40 heads 26.3 -> 24.6, 8 heads on 2 with budgets
// 15.1 -> 14.2; 480p, 12 heads on 3 4.33 -> 4.23; 13 frames, 16 heads of 64 channels 0.913 -> 0.875.  The packed cubes' rows are whole
// steps of a contraction and stay in order, so the gradients are the same bit for bit.  (As KEYS such cubes are hardly ever
// kept -- their block score is a mean over sub-cubes they do not have -- so nothing is packed there.)
// The elementwise stage is the longest serial chain of a tile, so its arithmetic goes two values at a time (fma_bits2, ds_bits2).
// Backward, us, scalar -> packed: 480p, 12 heads on 3 4205 -> 4110; 720p, 5 heads with text 4308 -> 4197; 8 heads on 2 with budgets
// 14390 -> 14196; 13 x 27 x 47 tokens, 16 heads of 64 channels 866 -> 835.
template <int D, bool SPLIT, bool MHA, int F16, bool PACK = false>
__global__ void __launch_bounds__(kDkvThreads, 1)
fine_bwd_dkv_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                       const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
                       const __grid_constant__ CUtensorMap tm_qt, const __grid_constant__ CUtensorMap tm_kt,
                       const __grid_constant__ CUtensorMap tm_vt, const __grid_constant__ CUtensorMap tm_dot,
                       const __grid_constant__ CUtensorMap tm_qe, const __grid_constant__ CUtensorMap tm_doe, Geo g,
                       DkvArgs a) {
  constexpr int RA = dkv_ring_a(D, SPLIT), RB = dkv_ring_b(D);      // slots of the Q ring and of the dO ring
  // accumulators: without SPLIT two sets of dK^T, dV^T (64 columns each), used by item parity
  constexpr uint32_t TM_DK = 256, TM_DV = SPLIT ? 384 : 320, TM_SET = 128, SETS = SPLIT ? 1 : 2;
  using C = BwdTc<D, RA, SPLIT ? 4 : 2, RB>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* k_tile = smem + C::OFF_ST0;
  unsigned char* v_tile = smem + C::OFF_ST1;
  unsigned char* p_tile = smem + C::OFF_P;                                  // P  [128 q, 64 kv] (SPLIT: followed by its low part)
  unsigned char* ds_tile = smem + C::OFF_P + (SPLIT ? 2 : 1) * C::PBYTES;   // dS [128 q, 64 kv] (SPLIT: followed by its low part)
  BwdMisc* misc = reinterpret_cast<BwdMisc*>(smem + C::OFF_MISC);

  BwdRings* rings = reinterpret_cast<BwdRings*>(smem + C::OFF_MISC + 2048);      // (D = 64)
  uint64_t *ring_a_full = D == 64 ? rings->a_full : misc->a_full, *ring_a_empty = D == 64 ? rings->a_empty : misc->a_empty;
  uint64_t *ring_b_full = D == 64 ? rings->b_full : misc->b_full, *ring_b_empty = D == 64 ? rings->b_empty : misc->b_empty;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float c2 = g.scale * 1.4426950408889634f;
  const int rep = MHA ? 1 : g.rep;
  constexpr bool STORES_DS = F16 == 1 || F16 == 2 || (SPLIT && !MHA);
  static_assert(F16 == 0 || !SPLIT, "the fp16 forms carry no pairs");
  // The launch of the few long lists (overlap 1), or the dQ pass of the pooled problem, lets the launch of the others (2; disjoint outputs, nothing read from the first) take
  // the SMs as its CTAs leave them, once what both read is there; the second waits for the first at its end, so that what
  // follows waits for both.
  const bool second = !SPLIT && F16 == 0 && a.overlap == 2;
  const bool fallback = a.when == 2;             // hardly ever does anything, and then it needs no set-up
  if (fallback) {
    if (!second) grid_enter(false);
    if (*a.range_flag == 0) {                    // (final before this launch starts)
      if (second) grid_enter(false);
      return;
    }
  }

  if (tid == 0) {
    bwd_init_barriers(misc);
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(&misc->o_full[s], 2);                                     // two last-stage issuers
      tc::mbar_init(&misc->o_empty[s], 4);                                    // the epilogue warps
    }
    list_queue_init(&misc->queue, 2 + 4 + 8 + 4 + 4 + (STORES_DS && !SPLIT && a.ds != nullptr ? 1 : 0));
    if (STORES_DS && !SPLIT && a.ds != nullptr) tc::mbar_init(&misc->ds_free[0], 2);     // read by the dK product and by the copy
    if (D == 64) {
      for (int s = 0; s < RA; ++s) {
        tc::mbar_init(&ring_a_full[s], 1);
        tc::mbar_init(&ring_a_empty[s], 1);
      }
      for (int s = 0; s < RB; ++s) tc::mbar_init(&ring_b_full[s], 1);
    }
    for (int s = 0; s < RB; ++s) tc::mbar_init(&ring_b_empty[s], 2);     // a dO slot is read by dP and by dV^T
    tc::fence_barrier_init();
    tc::prefetch_tmap(&tm_q);
    tc::prefetch_tmap(&tm_k);
    tc::prefetch_tmap(&tm_v);
    tc::prefetch_tmap(&tm_do);
  }
  if (warp == 2) {
    tc::tmem_alloc(&misc->tmem_base, 512);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = misc->tmem_base;
  if (SPLIT && a.overlap == 1) {
    grid_enter(false);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  } else if (!second && !fallback) {
    grid_enter(false);
  }
  if (a.when == 1 && __syncthreads_or(tid == 0 && *a.range_flag != 0)) {
    if (warp == 2) tc::tmem_dealloc(tmem_base, 512);
    return;
  }
  // tensor-memory columns: S buffers 0, 64; dP buffers 128, 192; dK^T 256, dV^T 320 and 384, 448 (SPLIT: dK^T 256 + 320,
  // dV^T 384 + 448)

  // per item, for the roles that walk the list: prefix of the per-head column counts and the list starts
#define VSA2_DKV_ITEM_SETUP()                                                            \
  const int j = rec.x, bhk = rec.y, k = rec.z;                                           \
  const int b = bhk / g.Hkv, hk = bhk % g.Hkv;                                           \
  int cnt_prefix[(MHA ? 1 : kMaxRep) + 1], col_beg[MHA ? 1 : kMaxRep];                   \
  int col_full[MHA || !PACK ? 1 : kMaxRep], col_cnt[MHA || !PACK ? 1 : kMaxRep];         \
  cnt_prefix[0] = 0;                                                                     \
  col_beg[0] = rec.w;                                                                    \
  if (MHA) {                                                                             \
    cnt_prefix[1] = k;                                                                   \
    if (PACK) {                                                                          \
      col_full[0] = a.pk.full[(size_t)bhk * g.N + j];                                    \
      col_cnt[0] = a.col_ptr[(size_t)bhk * (g.N + 1) + j + 1] - rec.w;                   \
    }                                                                                    \
  } else if (PACK) {                                                                     \
    for (int hh = 0; hh < rep; ++hh) {                                                   \
      const size_t head_ = (size_t)(b * g.Hq + hk * rep + hh), base_ = head_ * (g.N + 1) + j; \
      col_beg[hh] = a.col_ptr[base_];                                                    \
      col_cnt[hh] = a.col_ptr[base_ + 1] - col_beg[hh];                                  \
      col_full[hh] = a.pk.full[head_ * g.N + j];                                         \
      const int text_ = g.N - g.Nvid;                                                    \
      cnt_prefix[hh + 1] = cnt_prefix[hh] + col_full[hh] + text_ +                       \
                           ((col_cnt[hh] - text_ - col_full[hh] + (1 << a.pk.shift) - 1) >> a.pk.shift); \
    }                                                                                    \
  } else {                                                                               \
    for (int hh = 0; hh < rep; ++hh) {                                                   \
      const size_t base_ = (size_t)(b * g.Hq + hk * rep + hh) * (g.N + 1) + j;           \
      col_beg[hh] = a.col_ptr[base_];                                                    \
      cnt_prefix[hh + 1] = cnt_prefix[hh] + (a.col_ptr[base_ + 1] - col_beg[hh]);        \
    }                                                                                    \
  }

  // (registers: the launch allocates 80 a thread; the elementwise and epilogue warps take what the service warps leave)
  if (warp < 4) {
    tc::reg_dec<48>();
    if (warp < 2) {
    // ------------------------------------------------------------------ TMA producers
    const int which = warp;                               // 0: Q pairs (ring A) + K, V tiles; 1: dO pairs (ring B)
    const CUtensorMap* tm = which == 0 ? &tm_q : &tm_do;
    const CUtensorMap* tm_text = which == 0 ? &tm_qt : &tm_dot;
    const int my_blk = lane & 1;
    const int my_h = (lane >> 1) % C::DH, my_sub = PACK ? ((lane >> 1) / C::DH) & ((1 << a.pk.shift) - 1) : 0;
    const CUtensorMap* tm_cut = which == 0 ? &tm_qe : &tm_doe;
    (void)my_h; (void)tm_cut;
    uint32_t tg = 0, n_items = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      if (warp == 0 && lane == 0) tc::mbar_arrive(&misc->queue.taken);
      if (rec.z == 0) continue;
      VSA2_DKV_ITEM_SETUP();
      if (which == 0) {
        int c1, c2, c3;
        block_box(g, j, c1, c2, c3);
        const bool ktext = block_is_text(g, j);
        int ok = 1;
        if (lane == 0) {
          ok = tc::mbar_wait_parked(&misc->st_empty, (n_items & 1) ^ 1, &misc->abort_flag);
          if (ok) tc::mbar_expect_tx(&misc->st_full, 2 * C::TILE);
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) goto done;
        if (lane < 2 * C::DH) {
          const int h = lane >> 1;
          if (lane & 1) tc::tma_load_5d(v_tile + h * kSlab, ktext ? &tm_vt : &tm_v, &misc->st_full, h * 64, c1, c2, c3, bhk);
          else tc::tma_load_5d(k_tile + h * kSlab, ktext ? &tm_kt : &tm_k, &misc->st_full, h * 64, c1, c2, c3, bhk);
        }
      }
      ++n_items;
      const int nt = (k + 1) >> 1;
      int bhq_l, i_l;           // this lane's entry of the tile, fetched one tile ahead of the slot wait
      int kind_l = dkv_entry<false, PACK>(g, a, rep, b, hk, cnt_prefix, col_beg, (my_blk == 1 && k > 1) ? 1 : 0, bhq_l, i_l, nullptr, my_sub, col_full, col_cnt);
      for (int t = 0; t < nt; ++t, ++tg) {
        int c1, c2, c3;
        block_box(g, i_l, c1, c2, c3);
        const CUtensorMap* tm_i = PACK && kind_l > 0 ? tm_cut : block_is_text(g, i_l) ? tm_text : tm;
        const int bhq_t = bhq_l, kind_t = kind_l;
        if (t + 1 < nt)
          kind_l = dkv_entry<false, PACK>(g, a, rep, b, hk, cnt_prefix, col_beg, (my_blk == 1 && 2 * t + 3 < k) ? 2 * t + 3 : 2 * t + 2, bhq_l, i_l, nullptr,
                                          my_sub, col_full, col_cnt);
        if constexpr (PACK) {
          const uint32_t nslots = which == 0 ? RA : RB, slot = tg % nslots, par = (tg / nslots) & 1;
          uint64_t* full = which == 0 ? &ring_a_full[slot] : &ring_b_full[slot];
          int ok = 1;
          if (lane == 0) {
            ok = tc::mbar_wait_parked(which == 0 ? &ring_a_empty[slot] : &ring_b_empty[slot], par ^ 1, &misc->abort_flag);
            if (ok) tc::mbar_expect_tx(full, C::SLOT);
          }
          if (!__shfl_sync(0xffffffffu, ok, 0)) goto done;
          if (lane < (kind_t > 0 ? 2 * C::DH << a.pk.shift : 2 * C::DH))
            tc::tma_load_5d(smem + (which == 0 ? 0 : C::OFF_RING_B) + slot * C::SLOT + (2 * my_h + my_blk) * kSlab +
                                (kind_t > 0 ? my_sub * (kSlab >> a.pk.shift) : 0),
                            tm_i, full, my_h * 64, c1, c2, c3, bhq_t);
        } else {
          if (which == 0) VSA2_RING_LOAD(ring_a_full, ring_a_empty, RA, smem, tm_i, tg, c3, c2, c1, bhq_t, {}, mbar_wait_parked);
          else VSA2_RING_LOAD(ring_b_full, ring_b_empty, RB, smem + C::OFF_RING_B, tm_i, tg, c3, c2, c1, bhq_t, {}, mbar_wait_parked);
        }
      }
    }
    } else {
    // ------------------------------------------------------------------ issuers of S = Q_pair K^T (warp 2) and
    // dP = dO_pair V^T (warp 3); whole warp in the loop, one elected lane issues (see the dQ pass)
    {
      const bool is_s = warp == 2;
      const uint32_t b_addr = tc::smem_u32(is_s ? k_tile : v_tile), base = tc::smem_u32(smem);
      uint32_t tg = 0, n_items = 0;
      for (uint32_t seq = 0;; ++seq) {
        VSA2_NEXT_REC(rec, seq);
        if (rec.z == 0) continue;
        const int nt = (rec.z + 1) >> 1;
        VSA2_WAIT_PARKED(&misc->st_full, n_items & 1);
        for (int t = 0; t < nt; ++t, ++tg) {
          const uint32_t sb = tg & 1, pb = (tg >> 1) & 1;
          if (is_s) {
            const uint32_t sa = tg % RA, pa = (tg / RA) & 1;
            VSA2_WAIT_PARKED(&ring_a_full[sa], pa);
            VSA2_WAIT_PARKED(&misc->s_free[sb], pb ^ 1);
            tc::tc_fence_after();
            if (tc::elect_one()) {
              mma_pair_kmajor<D, F16 != 0>(tmem_base + sb * 64, base + sa * C::SLOT, b_addr);
              tc::mma_commit(&misc->s_full[sb]);
              if (t == nt - 1) tc::mma_commit(&misc->st_empty);
            }
          } else {
            const uint32_t so = tg % RB;
            VSA2_WAIT_PARKED(&ring_b_full[so], (tg / RB) & 1);
            VSA2_WAIT_PARKED(&misc->dp_free[sb], pb ^ 1);
            tc::tc_fence_after();
            if (tc::elect_one()) {
              mma_pair_kmajor<D, F16 >= 2>(tmem_base + 128 + sb * 64, base + C::OFF_RING_B + so * C::SLOT, b_addr);
              tc::mma_commit(&misc->dp_full[sb]);
              tc::mma_commit(&ring_b_empty[so]);
              if (t == nt - 1) tc::mma_commit(&misc->st_empty);
            }
          }
          __syncwarp();
        }
        ++n_items;
      }
    }
    }
  } else if (warp >= 16 && warp < 20) {
    tc::reg_dec<48>();
    if (warp == 18 && !schedule_lists<PACK>(&misc->queue, g, a.first_item, a.items, rep, a.col_ptr, a.item_counter, a.order, a.k_lo,
                                    a.k_hi, SPLIT && MHA && a.k_lo > 1, nullptr, lane, &misc->abort_flag, a.pk))
      goto done;
    if (STORES_DS && !SPLIT && warp == 19 && a.ds != nullptr) {
      // ---------------------------------------------------------------- copies the dS tiles to the scratch as they stand
      const uint64_t policy = tc::evict_first_policy();
      uint32_t tg = 0;
      for (uint32_t seq = 0;; ++seq) {
        VSA2_NEXT_REC(rec, seq);
        const int nt = (rec.z + 1) >> 1;
        for (int t = 0; t < nt; ++t, ++tg) {
          VSA2_WAIT_PARKED(&misc->ds_ready[0], tg & 1);
          if (lane == 0) {
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
              const int* at = misc->ds_slot[tg % 3][h];
              if (!PACK || at[1] == kWholeBlock) {
                if (at[0] >= 0) tc::bulk_store(a.ds + (size_t)at[0] * kSlab, ds_tile + h * kSlab, kSlab, policy);
              } else {
                const uint32_t bytes = kSlab >> a.pk.shift;
#pragma unroll 1
                for (int c = 0; c < 1 << a.pk.shift; ++c)
                  if (at[c] >= 0) tc::bulk_store(a.ds + (size_t)at[c] * kSlab, ds_tile + h * kSlab + c * bytes, bytes, policy);
              }
            }
            tc::bulk_store_commit();
            tc::bulk_store_wait_read();
            tc::mbar_arrive(&misc->ds_free[0]);
          }
          __syncwarp();
        }
      }
      if (lane == 0) tc::bulk_store_wait();
    }
    if (warp < 18) {
    // ------------------------------------------------------------------ issuers of dV^T += dO_pair^T P (warp 16) and
    // dK^T += Q_pair^T dS (warp 17); whole warp in the loop, one elected lane issues
    {
      const bool is_v = warp == 16;
      const uint32_t b_addr = tc::smem_u32(is_v ? p_tile : ds_tile), base = tc::smem_u32(smem);
      uint32_t tg = 0, n_items = 0;
      for (uint32_t seq = 0;; ++seq) {
        VSA2_NEXT_REC(rec, seq);
        if (rec.z == 0) continue;
        const int nt = (rec.z + 1) >> 1;
        const uint32_t set = n_items % SETS, acc = tmem_base + (is_v ? TM_DV : TM_DK) + set * TM_SET;
        VSA2_WAIT_PARKED(&misc->o_empty[set], ((n_items / SETS) & 1) ^ 1);
        for (int t = 0; t < nt; ++t, ++tg) {
          if (is_v) {
            // P depends on S only, so it can be ready before the dO pair of the tile has landed: wait for that too
            const uint32_t sv = tg % RB;
            VSA2_WAIT_PARKED(&ring_b_full[sv], (tg / RB) & 1);
            VSA2_WAIT_PARKED(&misc->p_ready, tg & 1);
            tc::tc_fence_after();
            if (tc::elect_one()) {
              if constexpr (SPLIT) mma_pairT_mnmajor_n128<D>(acc, base + C::OFF_RING_B + sv * C::SLOT, b_addr, C::PBYTES, t > 0);
              else mma_pairT_mnmajor<D, F16 >= 2>(acc, base + C::OFF_RING_B + sv * C::SLOT, b_addr, t > 0);
              tc::mma_commit(&ring_b_empty[sv]);
              tc::mma_commit(&misc->p_free);
              if (t == nt - 1) tc::mma_commit(&misc->o_full[set]);
            }
          } else {
            const uint32_t sa = tg % RA;
            VSA2_WAIT_PARKED(&misc->ds_ready[0], tg & 1);
            tc::tc_fence_after();
            if (tc::elect_one()) {
              if constexpr (SPLIT) mma_pairT_mnmajor_n128<D>(acc, base + sa * C::SLOT, b_addr, C::PBYTES, t > 0);
              else mma_pairT_mnmajor<D, F16 != 0>(acc, base + sa * C::SLOT, b_addr, t > 0);
              tc::mma_commit(&ring_a_empty[sa]);
              tc::mma_commit(&misc->ds_free[0]);
              if (t == nt - 1) tc::mma_commit(&misc->o_full[set]);
            }
          }
          __syncwarp();
        }
        ++n_items;
      }
    }
    }
  } else if (warp >= 12 && warp < 16) {
    tc::reg_dec<48>();
    // ------------------------------------------------------------------ row statistics of the tiles (128 threads)
    const int r = tid - 384;                 // query row of the tile
    const int blk = r >> 6;
    const int sub = PACK ? (r & 63) >> (6 - a.pk.shift) : 0, cut_rows = PACK ? 64 >> a.pk.shift : 64;
    float2* rowstat = reinterpret_cast<float2*>(misc->stats);
    uint32_t tg = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      if (rec.z == 0) continue;
      VSA2_DKV_ITEM_SETUP();
      (void)j;
      const int ds_exp = a.ds_exp != nullptr ? a.ds_exp[bhk] : 0;
      const float lse_off = F16 >= 2 ? 0.f : (float)ds_exp, dlt_scale = F16 >= 2 ? pow2i(ds_exp) : 1.f;
      const int nt = (k + 1) >> 1;
      int bhq_n, i_n, pos_n = 0;
      int kind_n = dkv_entry<STORES_DS, PACK>(g, a, rep, b, hk, cnt_prefix, col_beg, (blk == 1 && k > 1) ? 1 : 0, bhq_n, i_n, &pos_n, sub, col_full, col_cnt);
      for (int t = 0; t < nt; ++t, ++tg) {
        const int slot = STORES_DS && a.ds != nullptr ? (bhq_n - a.ds_head0) * (int)g.nnz_cap + pos_n : -1;
        const bool dup = ((blk == 1) && (2 * t + 1 >= k)) || (PACK && kind_n == 2);
        const int kind = kind_n, row_in = PACK && kind > 0 ? r & (cut_rows - 1) : r & 63;
        const int l = dup ? -1 : block_token(g, i_n, row_in);
        const size_t idx = l >= 0 ? (size_t)bhq_n * g.S + l : 0;
        const float lse_raw = a.lse[idx], dlt_raw = a.delta[idx];
        if (t + 1 < nt)
          kind_n = dkv_entry<STORES_DS, PACK>(g, a, rep, b, hk, cnt_prefix, col_beg, (blk == 1 && 2 * t + 3 < k) ? 2 * t + 3 : 2 * t + 2, bhq_n, i_n, &pos_n,
                                              sub, col_full, col_cnt);
        VSA2_WAIT_PARKED(&misc->stat_free, (tg & 1) ^ 1);
        if (STORES_DS && row_in == 0) {
          misc->ds_slot[tg % 3][blk][PACK && kind > 0 ? sub : 0] = dup ? -1 : slot;
          if (PACK && kind == 0) misc->ds_slot[tg % 3][blk][1] = kWholeBlock;
        }
        rowstat[r] = make_float2(l >= 0 ? lse_raw * 1.4426950408889634f - lse_off : INFINITY, l >= 0 ? dlt_raw * dlt_scale : 0.f);
        tc::mbar_arrive(&misc->stat_full);
      }
    }
  } else if (warp < 12) {
    tc::reg_inc<120>();
    // ------------------------------------------------------------------ elementwise stage (256 threads):
    // warps 4..7 take key columns 0..31 of every tile, warps 8..11 columns 32..63
    const int quad = warp & 3;
    const int half = (warp - 4) >> 2;
    const int row = (quad << 5) | lane;      // query row of the tile
    const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
    uint32_t tg = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      const int k = rec.z;
      if (k > 0) {
        const int nt = (k + 1) >> 1;
        const float2* rowstat = reinterpret_cast<const float2*>(misc->stats);
        for (int t = 0; t < nt; ++t, ++tg) {
          const uint32_t s = tg & 1, par = (tg >> 1) & 1;
          VSA2_WAIT(&misc->stat_full, tg & 1);
          const float2 rs = rowstat[row];
          int ds_slot = -1, ds_row = row & 63;
          if (SPLIT && STORES_DS) {
            const int* at = misc->ds_slot[tg % 3][row >> 6];
            if (PACK && at[1] != kWholeBlock) {
              ds_slot = at[ds_row >> (6 - a.pk.shift)];
              ds_row &= (64 >> a.pk.shift) - 1;
            } else {
              ds_slot = at[0];
            }
          }
          tc::mbar_arrive(&misc->stat_free);
          const float lse2 = rs.x, dlt = rs.y;
          uint32_t sv[32];      // S, then P
          VSA2_WAIT(&misc->s_full[s], par);
          tc::tc_fence_after();
          tc::tmem_ld32(lane_addr + s * 64 + half * 32, sv);
          tc::tmem_ld_wait();
          tc::tc_fence_before();
          tc::mbar_arrive(&misc->s_free[s]);
          {
            uint32_t pp[16], pl[SPLIT ? 16 : 1];
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
              const float2 x = fma_bits2(sv[c], sv[c + 1], c2, -lse2, -lse2);
              const float p0 = ex2_approx(x.x), p1 = ex2_approx(x.y);
              sv[c] = __float_as_uint(p0);
              sv[c + 1] = __float_as_uint(p1);
              if constexpr (SPLIT) split_bf16x2(p0, p1, pp[c >> 1], pl[c >> 1]);
              else if constexpr (F16 >= 2) pp[c >> 1] = pack_f16x2_sat(p0, p1);
              else pp[c >> 1] = pack_bf16x2(p0, p1);
            }
            VSA2_WAIT(&misc->p_free, (tg & 1) ^ 1);
            unsigned char* prow = p_tile + row * 128;
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
              *reinterpret_cast<uint4*>(prow + (((half * 4 + ch) ^ (row & 7)) << 4)) =
                  make_uint4(pp[4 * ch], pp[4 * ch + 1], pp[4 * ch + 2], pp[4 * ch + 3]);
              if constexpr (SPLIT)
                *reinterpret_cast<uint4*>(prow + C::PBYTES + (((half * 4 + ch) ^ (row & 7)) << 4)) =
                    make_uint4(pl[4 * ch], pl[4 * ch + 1], pl[4 * ch + 2], pl[4 * ch + 3]);
            }
            tc::fence_proxy_async_smem();
            tc::mbar_arrive(&misc->p_ready);
          }
          {
            uint32_t dp[32], pd[16], pdl[SPLIT ? 16 : 1], ph[SPLIT && STORES_DS ? 16 : 1];
            VSA2_WAIT(&misc->dp_full[s], par);
            tc::tc_fence_after();
            tc::tmem_ld32(lane_addr + 128 + s * 64 + half * 32, dp);
            tc::tmem_ld_wait();
            tc::tc_fence_before();
            tc::mbar_arrive(&misc->dp_free[s]);
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
              const float2 d = ds_bits2(sv[c], sv[c + 1], dp[c], dp[c + 1], dlt, dlt);
              const float d0 = d.x, d1 = d.y;
              if constexpr (SPLIT) {
                split_bf16x2(d0, d1, pd[c >> 1], pdl[c >> 1]);
                if constexpr (STORES_DS) ph[c >> 1] = pack_f16x2(d0, d1);
              } else if constexpr (F16 == 3) {
                pd[c >> 1] = pack_f16x2_sat(d0, d1);
              } else if constexpr (F16 != 0) {
                // (a dS beyond the range: the recomputing dQ pass, which runs first, has met the same value and raised the flag,
                //  or the pass behind this one finds the infinity in the scratch)
                pd[c >> 1] = pack_f16x2(d0, d1);
              } else {
                pd[c >> 1] = pack_bf16x2(d0, d1);
              }
            }
            if (SPLIT && STORES_DS && ds_slot >= 0) {
              // [chunk of 8 keys][query row]: 512 contiguous bytes per warp and store
              uint4* dst = reinterpret_cast<uint4*>(a.ds + (size_t)ds_slot * kSlab) + half * 256 + ds_row;
#pragma unroll
              for (int ch = 0; ch < 4; ++ch) {
                if constexpr (SPLIT && STORES_DS) dst[ch * 64] = make_uint4(ph[4 * ch], ph[4 * ch + 1], ph[4 * ch + 2], ph[4 * ch + 3]);
              }
            }
            VSA2_WAIT(&misc->ds_free[0], (tg & 1) ^ 1);
            unsigned char* drow = ds_tile + row * 128;
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
              *reinterpret_cast<uint4*>(drow + (((half * 4 + ch) ^ (row & 7)) << 4)) =
                  make_uint4(pd[4 * ch], pd[4 * ch + 1], pd[4 * ch + 2], pd[4 * ch + 3]);
              if constexpr (SPLIT)
                *reinterpret_cast<uint4*>(drow + C::PBYTES + (((half * 4 + ch) ^ (row & 7)) << 4)) =
                    make_uint4(pdl[4 * ch], pdl[4 * ch + 1], pdl[4 * ch + 2], pdl[4 * ch + 3]);
            }
            tc::fence_proxy_async_smem();
            tc::mbar_arrive(&misc->ds_ready[0]);
          }
        }
      }
    }
  } else {
    tc::reg_inc<96>();
    // ------------------------------------------------------------------ epilogue (128 threads, one per channel):
    // dK[l, d] = scale * dK^T[d, kv] + sum_heads dK_c[j, d] / count(j) (dS goes to its product without the softmax scale),
    // dV the same without a scale
    const int row = tid - 640;
    const uint32_t lane_addr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    uint32_t n_items = 0;
    for (uint32_t seq = 0;; ++seq) {
      VSA2_NEXT_REC(rec, seq);
      const int j = rec.x, bhk = rec.y, k = rec.z;
      const int b = bhk / g.Hkv, hk = bhk % g.Hkv;
      const int tok0 = block_token(g, j, lane), tok1 = block_token(g, j, 32 + lane);
      float coarse[2] = {0.f, 0.f};            // dK, dV
      if (a.dkc != nullptr && row < D && !block_is_text(g, j)) {
        for (int hh = 0; hh < rep; ++hh) {
          const size_t cidx = ((size_t)(b * g.Hq + hk * rep + hh) * g.Nvid + j) * D + row;
          coarse[0] += a.dkc[cidx];
          coarse[1] += a.dvc[cidx];
        }
        const float inv_cnt = 1.f / (float)cube_count(g, j);
        coarse[0] *= inv_cnt;
        coarse[1] *= inv_cnt;
      }
      const float inv_scale = a.ds_exp != nullptr ? pow2i(-a.ds_exp[bhk]) : 1.f, k_scale = g.scale * inv_scale;
      const size_t head = (size_t)bhk * g.S;
      if (k == 0) {                            // nothing kept: the coarse gradients only
#pragma unroll 1
        for (int c = 0; c < 64; ++c) {
          const int l = __shfl_sync(0xffffffffu, c < 32 ? tok0 : tok1, c & 31);
          if (l < 0 || row >= D) continue;
          store_out(a.dk, (head + l) * D + row, coarse[0], g.out_f32);
          store_out(a.dv, (head + l) * D + row, coarse[1], g.out_f32);
        }
        continue;
      }
      const uint32_t set = n_items % SETS;
      VSA2_WAIT_PARKED(&misc->o_full[set], (n_items / SETS) & 1);
      tc::tc_fence_after();
      // The four warps write the same table.  Behind this wait every one of them is through with the item two before, whose
      // table this was: its accumulators were given back after the last look at it (SETS = 2), or those of the item in between
      // were (SETS = 1).
      int* tok = misc->tok + (n_items & 1) * 64;
      tok[lane] = tok0;
      tok[32 + lane] = tok1;
      __syncwarp();
#pragma unroll 1
      for (int part = 0; part < 8; ++part) {   // dK tokens 0..15, .., 48..63, dV the same
        const bool is_v = part >= 4;
        const uint32_t addr = lane_addr + set * TM_SET + (is_v ? TM_DV : TM_DK) + (part & 3) * 16;
        uint32_t x[16], lo[SPLIT ? 16 : 1];
        tc::tmem_ld16(addr, x);
        if constexpr (SPLIT) tc::tmem_ld16(addr + 64, lo);
        tc::tmem_ld_wait();
        if (SPLIT && part == 7) {              // everything has been read: the accumulators are free
          tc::tc_fence_before();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&misc->o_empty[0]);
        }
        const float add = is_v ? coarse[1] : coarse[0], factor = is_v ? inv_scale : k_scale;
        float v[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          v[c] = __uint_as_float(x[c]);
          if constexpr (SPLIT) v[c] += __uint_as_float(lo[c]);
          v[c] = fmaf(v[c], factor, add);
        }
        if (row < D) store_channels<D>(is_v ? a.dv : a.dk, g.out_f32, head, tok + (part & 3) * 16, v, row);
      }
      if constexpr (!SPLIT) {
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&misc->o_empty[set]);
      }
      ++n_items;
    }
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
  if (warp == 2) tc::tmem_dealloc(tmem_base, 512);
  if (!SPLIT && F16 == 0 && a.overlap == 2) asm volatile("griddepcontrol.wait;" ::: "memory");     // (what follows waits for both)
}

// ================================================================================================
// launcher
// ================================================================================================
// A column list longer than this many query blocks goes through the pair form (see below)
constexpr int kDkvLongColumn = 256;

// `split_long_columns`: when the pass would run with plain bf16 operands (one query head per KV head, no precision flag), the
// KV blocks that more than kDkvLongColumn query blocks keep are computed by a second launch that carries P and dS as bf16
// pairs.  The rounding of the plain form leaves a relative error of 1 - 2e-3 of the largest gradient of a block, whatever
// the list length (720p sample, fp32 outputs: 6.5e-3 at |dK| = 5.5 with 200 query blocks, 6.3e-3 at 3.0 with 260); the
// few blocks that nearly every query keeps reach |dK| = 15 and then 1.5e-2 .. 2.7e-2 depending on nothing but where the
// roundings fall (e.g. whether the softmax scale is applied before or after dS is rounded), i.e. across the stated 2e-2.
// As pairs they come out at 6e-3.  The pair launch comes first (a handful of 0.3 ms items on 148 CTAs: alone it would end with most
// SMs idle) and the plain launch fills the SMs as its CTAs leave them; each skips the other's items.
cudaError_t launch_fine_bwd_dkv_tc(const Geo& g, const bf16* q, const bf16* k, const bf16* v, const bf16* d_o,
                                   const float* lse, const float* delta, const int* col_ptr, const int* row_idx,
                                   const float* dkc, const float* dvc, void* dk, void* dv, StatusBlock* status,
                                   cudaStream_t st, bool split_long_columns, const void* q16,
                                   const void* k16, void* v16, void* do16, const StoredDs* sd, const int* ds_exp,
                                   const PackedCubes& pk, StatusBlock* report, bool beside) {
  if (g.rep > kMaxRep) return cudaErrorInvalidValue;
  CUtensorMap tq, tk, tv, tdo, tqt, tkt, tvt, tdot, tq16, tk16, tqt16, tkt16, tv16, tdo16, tvt16, tdot16;
  // GQA groups without a precision flag take the all-fp16 form when they are given scratch for fp16 copies of V and dO as
  // well (their fallback is the pair form over all lists)
  const bool gqa16 = fine_bwd_dkv_gqa_uses_f16(g) && split_long_columns && v16 != nullptr && do16 != nullptr;
  const bool f16 = q16 != nullptr && k16 != nullptr && (gqa16 || fine_bwd_dkv_splits_long_columns(g, split_long_columns));
  if (f16 && (!make_cube_tmap(&tq16, reinterpret_cast<const bf16*>(q16), g, g.Hq) ||       // (same element size and layout)
              !make_cube_tmap(&tk16, reinterpret_cast<const bf16*>(k16), g, g.Hkv) ||
              !make_text_tmap(&tqt16, reinterpret_cast<const bf16*>(q16), g, g.Hq) ||
              !make_text_tmap(&tkt16, reinterpret_cast<const bf16*>(k16), g, g.Hkv)))
    return cudaErrorInvalidValue;
  if (!make_cube_tmap(&tq, q, g, g.Hq) || !make_cube_tmap(&tk, k, g, g.Hkv) || !make_cube_tmap(&tv, v, g, g.Hkv) ||
      !make_cube_tmap(&tdo, d_o, g, g.Hq) || !make_text_tmap(&tqt, q, g, g.Hq) || !make_text_tmap(&tkt, k, g, g.Hkv) ||
      !make_text_tmap(&tvt, v, g, g.Hkv) || !make_text_tmap(&tdot, d_o, g, g.Hq))
    return cudaErrorInvalidValue;
  if (f16 && gqa16 && (!make_cube_tmap(&tv16, reinterpret_cast<const bf16*>(v16), g, g.Hkv) ||
                       !make_cube_tmap(&tdo16, reinterpret_cast<const bf16*>(do16), g, g.Hq) ||
                       !make_text_tmap(&tvt16, reinterpret_cast<const bf16*>(v16), g, g.Hkv) ||
                       !make_text_tmap(&tdot16, reinterpret_cast<const bf16*>(do16), g, g.Hq)))
    return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  const bool mha = g.rep == 1;
  // the main forms with stored dS have a packed version
  CUtensorMap tqe = {}, tdoe = {};
  const bool pack = pk.shift > 0 && sd != nullptr;
  if (pack) {
    const int frames = g.T - (g.Nt - 1) * g.Bt;
    if (!make_cube_tmap(&tqe, f16 ? reinterpret_cast<const bf16*>(q16) : q, g, g.Hq, frames) ||
        !make_cube_tmap(&tdoe, f16 && gqa16 ? reinterpret_cast<const bf16*>(do16) : d_o, g, g.Hq, frames))
      return cudaErrorInvalidValue;
  }
#define VSA2_LAUNCH_DKV(DD, SP, MH, F, PK, TQ, TK, TQT, TKT, TV, TDO, TVT, TDOT)                                                                         \
  do {                                                                                                                           \
    using L_ = BwdTc<DD, dkv_ring_a(DD, SP), SP ? 4 : 2, dkv_ring_b(DD)>;                                                         \
    static KernelAttr attr_;                                                                                                     \
    if ((e = prepare_kernel((const void*)fine_bwd_dkv_tc_kernel<DD, SP, MH, F, PK>, attr_, L_::smem_bytes, kDkvThreads,               \
                            128 * (48 + 2 * 120 + 2 * 48 + 96))))                                                                \
      return e;                                                                                                                  \
    if ((e = launch_kernel(fine_bwd_dkv_tc_kernel<DD, SP, MH, F, PK>, grid, kDkvThreads, L_::smem_bytes, st, TQ, TK, TV, TDO, TQT, TKT, TVT, TDOT, tqe, tdoe, g, a))) \
      return e;                                                                                                                  \
  } while (0)
  // `when`: see DkvArgs.
  // `group0`, `groups`: range of KV heads (batch * Hkv index); `ds`: the launch stores dS, counting on a counter of its own.
  // `overlap`: see DkvArgs.
  auto launch = [&](bool split, int* counter, int k_lo, int k_hi, int when, int group0, int groups,
                    bool ds, int overlap = 0) -> cudaError_t {
    const int items = groups * g.N, grid = items < sms ? items : sms;
    DkvArgs a{counter, lse, delta, col_ptr, row_idx, dkc, dvc, dk, dv, report != nullptr ? report : status, k_lo, k_hi, &status->pad[kRangeFlagSlot], when,
              group0 * g.N, items, ds ? reinterpret_cast<unsigned char*>(sd->scratch) : nullptr, ds ? sd->pos : nullptr,
              group0 * g.rep, when == 1 || ds ? ds_exp : nullptr, ds ? sd->order : nullptr, pk, overlap};
    if (ds && pack) {
#define VSA2_LAUNCH_PACKED(DD)                                                                                  \
      if (when == 1 && gqa16) VSA2_LAUNCH_DKV(DD, false, false, 2, true, tq16, tk16, tqt16, tkt16, tv16, tdo16, tvt16, tdot16); \
      else if (when == 1) VSA2_LAUNCH_DKV(DD, false, true, 1, true, tq16, tk16, tqt16, tkt16, tv, tdo, tvt, tdot);      \
      else VSA2_LAUNCH_DKV(DD, true, false, 0, true, tq, tk, tqt, tkt, tv, tdo, tvt, tdot)
      if (g.D == 128) { VSA2_LAUNCH_PACKED(128); }
      else { VSA2_LAUNCH_PACKED(64); }
#undef VSA2_LAUNCH_PACKED
    } else if (when == 1 && gqa16 && ds) { // every product in fp16
      if (g.D == 128) VSA2_LAUNCH_DKV(128, false, false, 2, false, tq16, tk16, tqt16, tkt16, tv16, tdo16, tvt16, tdot16);
      else VSA2_LAUNCH_DKV(64, false, false, 2, false, tq16, tk16, tqt16, tkt16, tv16, tdo16, tvt16, tdot16);
    } else if (when == 1 && gqa16) {
      if (g.D == 128) VSA2_LAUNCH_DKV(128, false, false, 3, false, tq16, tk16, tqt16, tkt16, tv16, tdo16, tvt16, tdot16);
      else VSA2_LAUNCH_DKV(64, false, false, 3, false, tq16, tk16, tqt16, tkt16, tv16, tdo16, tvt16, tdot16);
    } else if (when == 1) {         // S and the dK product in fp16 (one query head per KV head)
      if (g.D == 128) VSA2_LAUNCH_DKV(128, false, true, 1, false, tq16, tk16, tqt16, tkt16, tv, tdo, tvt, tdot);
      else VSA2_LAUNCH_DKV(64, false, true, 1, false, tq16, tk16, tqt16, tkt16, tv, tdo, tvt, tdot);
    } else if (g.D == 128) {
      if (split && mha) VSA2_LAUNCH_DKV(128, true, true, 0, false, tq, tk, tqt, tkt, tv, tdo, tvt, tdot);
      else if (split) VSA2_LAUNCH_DKV(128, true, false, 0, false, tq, tk, tqt, tkt, tv, tdo, tvt, tdot);
      else if (mha) VSA2_LAUNCH_DKV(128, false, true, 0, false, tq, tk, tqt, tkt, tv, tdo, tvt, tdot);
      else VSA2_LAUNCH_DKV(128, false, false, 0, false, tq, tk, tqt, tkt, tv, tdo, tvt, tdot);
    } else {
      if (split && mha) VSA2_LAUNCH_DKV(64, true, true, 0, false, tq, tk, tqt, tkt, tv, tdo, tvt, tdot);
      else if (split) VSA2_LAUNCH_DKV(64, true, false, 0, false, tq, tk, tqt, tkt, tv, tdo, tvt, tdot);
      else if (mha) VSA2_LAUNCH_DKV(64, false, true, 0, false, tq, tk, tqt, tkt, tv, tdo, tvt, tdot);
      else VSA2_LAUNCH_DKV(64, false, false, 0, false, tq, tk, tqt, tkt, tv, tdo, tvt, tdot);
    }
    return cudaGetLastError();
  };
#undef VSA2_LAUNCH_DKV
  constexpr int kAll = 0x7fffffff;
  const int all = g.batch * g.Hkv;
  int* range_flag = &status->pad[kRangeFlagSlot];
  // Launches over all items; or, with `sd`, over as many KV groups at a time as the scratch holds, the dQ pass of these groups
  // behind each
  auto main_pass = [&](bool split, int when) -> cudaError_t {
    if (sd == nullptr) return launch(split, &status->pad[3], 0, kAll, when, 0, all, false);
    cudaError_t r;
    for (int c = 0, g0 = 0; g0 < all; ++c, g0 += sd->chunk_groups) {
      const int n = all - g0 < sd->chunk_groups ? all - g0 : sd->chunk_groups;
      if ((r = launch(split, sd->counters + 2 * c, 0, kAll, when, g0, n, true)) != cudaSuccess) return r;
      if ((r = launch_fine_bwd_dq_ds(g, k16, sd->scratch, g0 * g.rep, n * g.rep, sd->row_ptr, sd->col_idx, sd->dqc, sd->dq, status,
                                     range_flag, sd->counters + 2 * c + 1, !split, ds_exp, pack ? pk : PackedCubes{}, st)) != cudaSuccess)
        return r;
    }
    // dQ again, from bf16 pairs, if a value left the fp16 range
    return launch_fine_bwd_dq_fallback(g, q, k, v, d_o, lse, delta, sd->row_ptr, sd->col_idx, sd->dqc, sd->dq, status, st);
  };
  if (f16 && gqa16) {
    if ((e = launch_cast_v_do(g, v, v16, d_o, do16, ds_exp, range_flag, st)) != cudaSuccess) return e;
    if ((e = main_pass(false, 1)) != cudaSuccess) return e;
    return launch(true, &status->pad[4], 0, kAll, 2, 0, all, false);
  }
  if (fine_bwd_dkv_wants_pair(g)) return main_pass(true, 0);
  if (!fine_bwd_dkv_splits_long_columns(g, split_long_columns))
    return launch(false, &status->pad[3], 0, kAll, 0, 0, all, false, beside ? 2 : 0);
  // With the fp16 copies of Q and K: one launch in the fp16 form; the two launches below then run only if the range flag
  // came up (in the dQ pass or in this launch), on counters of their own.
  int when = 0, slot_plain = 3;
  if (f16) {
    if ((e = main_pass(false, 1)) != cudaSuccess) return e;
    when = 2;
    slot_plain = 5;
  }
  // (no list is longer than the blocks of the problem)
  const bool long_lists = g.N > kDkvLongColumn;
  if (long_lists && (e = launch(true, &status->pad[4], kDkvLongColumn + 1, kAll, when, 0, all, false, 1)) != cudaSuccess) return e;
  return launch(false, &status->pad[slot_plain], 0, kDkvLongColumn, when, 0, all, false, long_lists ? 2 : 0);
}

// Packed where two or four cubes fill a tile.  Below 128 cubes the counts are a launch for nothing.
PackedCubes packed_cubes(const Geo& g, const int* full) {
  const int rows = (g.T - (g.Nt - 1) * g.Bt) * g.Bh * g.Bw;
  const int shift = rows == kBlockTokens / 4 ? 2 : rows == kBlockTokens / 2 ? 1 : 0;
  return PackedCubes{g.Nvid >= 128 && g.Nt > 1 ? shift : 0, (g.Nt - 1) * g.Nh * g.Nw, full};
}

// Whether the dK/dV pass of a GQA problem takes its all-fp16 form when it is given the scratch for the four copies.  Rows that
// keep only a few blocks have sharply peaked weights and gradients of 10 - 30 per element; a KV block then sums the heads of
// a group at magnitudes where the 11 bits of fp16 leave 2e-2 (a per-query top-1 case with 12:3 heads: dK 2.08e-2), so those
// problems (and per-row budgets, whose sizes the host does not know) keep the bf16 pairs.
constexpr int kGqaF16MinTopk = 8;
bool fine_bwd_dkv_gqa_uses_f16(const Geo& g) {
  return g.rep > 1 && !(g.flags & (VSA2_FLAG_FAST_BWD | VSA2_FLAG_PRECISE_BWD)) && g.K >= kGqaF16MinTopk;
}

// whether launch_fine_bwd_dkv_tc runs as two launches for this problem
bool fine_bwd_dkv_splits_long_columns(const Geo& g, bool split_long_columns) {
  return split_long_columns && !fine_bwd_dkv_wants_pair(g) && !(g.flags & VSA2_FLAG_FAST_BWD);
}

}  // namespace vsa2
