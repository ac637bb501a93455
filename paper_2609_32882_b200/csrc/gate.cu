// Gate projection of the gated merge (paper Eq. 13): gate = tanh(X W_g), one column of W_g per query head, and its
// backward.  X [batch, L, C] are the layer's hidden states (bf16, tokens in raster order), W_g [C, Hq] bf16, gate and
// dgate [batch, Hq, L] fp32 (the layout vsa2_attn_fwd / vsa2_attn_bwd use).
//
// All three kernels are bound by one pass over X or dX (2 L C bytes per batch entry against 2 L C Hq FLOP with Hq a few
// dozen), so they are written for wide, coalesced HBM access; the products run on mma.sync m16n8k16 (bf16 in, fp32
// accumulate) because the N or K extent (the heads) is far below a tcgen05 tile.
//   forward : gate^T[l, h] = tanh(sum_c X[l, c] W[c, h])                        M = tokens,  N = heads,    K = channels
//   dX      : dX[l, c]     = sum_h dz[l, h] W[c, h],  dz = dgate (1 - gate^2)   M = tokens,  N = channels, K = heads
//   dW_g    : dW[c, h]     = sum_{b, l} X[l, c] dz[l, h]                        M = channels, N = heads,   K = tokens
// dW_g is reduced over the tokens in two deterministic steps (per-split partial sums, then a sum over the splits in a
// fixed order): no floating-point atomics.
#include "common.cuh"

namespace vsa2 {

namespace {

constexpr int kGtTok = 64;        // tokens per CTA tile
constexpr int kGtCh = 128;        // channels per chunk
constexpr int kGtThreads = 128;   // four warps
constexpr int kGtSplits = 16;     // token ranges per batch entry in the dW_g pass
constexpr int kDxCh = 128;        // channels per chunk of the dX pass

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], const void* smem_row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(smem_row)));
}
__device__ __forceinline__ void ldmatrix_x2_trans(uint32_t& r0, uint32_t& r1, const void* smem_row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"((uint32_t)__cvta_generic_to_shared(smem_row)));
}
__device__ __forceinline__ uint32_t lds32(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

constexpr int kLdx = kGtCh + 8;   // 272-byte rows: 16-byte aligned, and eight consecutive rows cover all 32 banks

// Eight consecutive elements of W, the first of them element i of a chunk whose rows (channels) have Hq heads, into the rows
// row_of(channel) of a tile of LD elements a row.
template <int LD, typename RowOf>
__device__ __forceinline__ void scatter_w(bf16* ws, uint4 v, int i, int Hq, RowOf row_of) {
  const bf16* e = reinterpret_cast<const bf16*>(&v);
  int c = i / Hq, h = i - c * Hq;
  bf16* row = ws + row_of(c) * LD;
  if (Hq % 8 == 0) {
    *reinterpret_cast<uint4*>(row + h) = v;
    return;
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    row[h] = e[u];
    if (++h == Hq) {
      h = 0;
      row = ws + row_of(++c) * LD;
    }
  }
}

// dz = dgate (1 - gate^2) in bf16, once per backward, in the two layouts its products read:
//   dz_hm [batch][HP][Lp]  head-major  (HP = heads rounded up to 16, Lp = tokens rounded up to 64; zero padding)
//   dz_tm [batch][Lp][HP]  token-major
// grid (Lp / 64, batch)
__global__ void __launch_bounds__(kGtThreads) gate_dz_kernel(const float* gate, const float* dgate,
                                                             int L, int Lp, int Hq, int HP, bf16* __restrict__ dz_hm,
                                                             bf16* __restrict__ dz_tm) {
  grid_enter();
  extern __shared__ __align__(16) unsigned char gate_dz_smem[];
  bf16* tile = reinterpret_cast<bf16*>(gate_dz_smem);          // [HP][64 + 8]
  constexpr int LD = kGtTok + 8;
  const int l0 = blockIdx.x * kGtTok, b = blockIdx.y;
  const float* gb = gate + (size_t)b * Hq * L;
  const float* db = dgate + (size_t)b * Hq * L;
  for (int e = threadIdx.x; e < HP * kGtTok; e += kGtThreads) {
    const int h = e / kGtTok, tl = e % kGtTok;
    float v = 0.f;
    if (h < Hq && l0 + tl < L) {
      const float g = gb[(size_t)h * L + l0 + tl];
      v = db[(size_t)h * L + l0 + tl] * (1.f - g * g);
    }
    const bf16 vb = __float2bfloat16_rn(v);
    tile[h * LD + tl] = vb;
    dz_hm[((size_t)b * HP + h) * Lp + l0 + tl] = vb;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kGtTok * HP; e += kGtThreads) {
    const int tl = e / HP, h = e % HP;
    dz_tm[((size_t)b * Lp + l0 + tl) * HP + h] = tile[h * LD + tl];
  }
}

// ---------------------------------------------------------------------------------------------- forward
// MW warp rows of 16 tokens, each of HW warps that take NT / HW head tiles of 8; grid (ceil(L / (16 MW)), batch).
// X goes from global memory straight into the A fragments.  The k-steps run over the channels in order and one warp sums all of them,
// so a gate does not depend on how many tokens share the launch; inside a step the order is free.  Of a group of 32 channels a
// thread loads the 16 bytes of channels 8t .. 8t+7, trades 8 of them with thread t ^ 2 (the first two threads hold the first step's 16
// channels, the others the second's) and then has 4 channels of each step as its logical k = 2t, 2t+1, 2t+8, 2t+9; the rows
// of W lie in that order in shared memory, for ldmatrix.  (8-byte loads need no trade but twice the cache look-ups: 75,600 tokens of
// 5,120 channels, 40 heads 345 us against 296; 10 heads 168 both ways.)  The loads of the next chunk are in flight while a chunk is multiplied; warps beyond MW HW only
// stage W.  Least CTAs per SM where the compiler's own choice of registers is slower: 32 heads 213 us (240), 40 heads 293 (320).
template <int NT, int MW, int HW, int CH>
__global__ void __launch_bounds__(kGtThreads, MW != 4 ? 0 : NT == 4 ? 4 : NT == 5 ? 3 : 0) gate_fwd_kernel(const bf16* x, const bf16* w, int L,
                                                              int C, int Hq, float* __restrict__ gate) {
  grid_enter();
  static_assert(NT % HW == 0 && MW * HW * 32 <= kGtThreads, "warps of a CTA");
  constexpr int LDW = NT * 8 + 8;                           // 16-byte aligned rows, eight rows on different banks
  constexpr int NTW = NT / HW, GROUPS = CH / 32;
  __shared__ __align__(16) bf16 ws[CH * LDW];               // W chunk as stored: [channel][head]; read by ldmatrix.trans
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int mw = warp % MW, hw = warp / MW, h0 = hw * NTW * 8;
  const bool works = hw < HW;
  const int l0 = blockIdx.x * (16 * MW) + mw * 16, b = blockIdx.y;
  const bf16* xa = x + ((size_t)b * L + min(l0 + g, L - 1)) * C + t * 8;       // (rows behind the last token repeat it)
  const bf16* xc = x + ((size_t)b * L + min(l0 + g + 8, L - 1)) * C + t * 8;
  // (the rows of a chunk of W are contiguous: read as 16-byte vectors whatever the number of heads)
  const bool w_vec = (reinterpret_cast<uintptr_t>(w) & 15u) == 0;
  // channel of a chunk -> its row in ws (inside its step of 16: upper half, thread, parity)
  auto w_row = [](int c) { return (c & ~15) + ((c >> 1) & 1) * 8 + (((c >> 3) & 1) + ((c >> 2) & 1) * 2) * 2 + (c & 1); };
  float acc[NTW][4];
#pragma unroll
  for (int n = 0; n < NTW; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.f;
  constexpr int WV = CH * NT / kGtThreads;                  // vectors of a W chunk per thread
  uint4 ra[GROUPS], rc[GROUPS], rw[WV];
  for (int e = tid; e < CH * LDW / 8; e += kGtThreads) reinterpret_cast<uint4*>(ws)[e] = make_uint4(0, 0, 0, 0);   // (padding heads)
  auto load = [&](int c0) {
    if (w_vec) {
#pragma unroll
      for (int u = 0; u < WV; ++u) {
        const int e = tid + u * kGtThreads;
        rw[u] = e * 8 < CH * Hq && c0 * Hq + e * 8 < C * Hq ? reinterpret_cast<const uint4*>(w + (size_t)c0 * Hq)[e]
                                                            : make_uint4(0, 0, 0, 0);
      }
    }
    if (works) {
#pragma unroll
      for (int q = 0; q < GROUPS; ++q) {
        const bool in = c0 + q * 32 + t * 8 < C;
        ra[q] = in ? *reinterpret_cast<const uint4*>(xa + c0 + q * 32) : make_uint4(0, 0, 0, 0);
        rc[q] = in ? *reinterpret_cast<const uint4*>(xc + c0 + q * 32) : make_uint4(0, 0, 0, 0);
      }
    }
  };
  load(0);
  for (int c0 = 0; c0 < C; c0 += CH) {
    __syncthreads();
    if (w_vec) {
#pragma unroll
      for (int u = 0; u < WV; ++u) {
        const int e = tid + u * kGtThreads;
        if (e * 8 < CH * Hq) scatter_w<LDW>(ws, rw[u], e * 8, Hq, w_row);
      }
    } else {
      for (int e = tid; e < CH * NT * 8; e += kGtThreads) {
        const int c = e / (NT * 8), h = e % (NT * 8);
        ws[w_row(c) * LDW + h] = (h < Hq && c0 + c < C) ? w[(size_t)(c0 + c) * Hq + h] : __float2bfloat16_rn(0.f);
      }
    }
    __syncthreads();
    uint4 ca[GROUPS], cc[GROUPS];
#pragma unroll
    for (int q = 0; q < GROUPS; ++q) {
      ca[q] = ra[q];
      cc[q] = rc[q];
    }
    if (c0 + CH < C) load(c0 + CH);
    if (works) {
#pragma unroll
      for (int q = 0; q < GROUPS; ++q) {
        // (x, y) = this thread's half for the first step of the group, (z, w) for the second
        auto trade = [&](uint4 v) {
          const uint32_t r0 = __shfl_xor_sync(0xffffffffu, t < 2 ? v.z : v.x, 2), r1 = __shfl_xor_sync(0xffffffffu, t < 2 ? v.w : v.y, 2);
          return t < 2 ? make_uint4(v.x, v.y, r0, r1) : make_uint4(r0, r1, v.z, v.w);
        };
        const uint4 va = trade(ca[q]), vc = trade(cc[q]);
#pragma unroll
        for (int st = 0; st < 2; ++st) {
          const uint32_t a[4] = {st ? va.z : va.x, st ? vc.z : vc.x, st ? va.w : va.y, st ? vc.w : vc.y};
          const bf16* row = ws + (q * 32 + st * 16 + (lane & 15)) * LDW + h0;
#pragma unroll
          for (int n = 0; n + 1 < NTW; n += 2) {
            uint32_t bb[4];
            ldmatrix_x4_trans(bb, row + n * 8 + (lane >> 4) * 8);
            mma_bf16(acc[n], a, bb[0], bb[1]);
            mma_bf16(acc[n + 1], a, bb[2], bb[3]);
          }
          if constexpr (NTW % 2 == 1) {
            uint32_t b0, b1;
            ldmatrix_x2_trans(b0, b1, row + (NTW - 1) * 8);
            mma_bf16(acc[NTW - 1], a, b0, b1);
          }
        }
      }
    }
  }
  if (!works) return;
  float* gb = gate + (size_t)b * Hq * L;
  const int tok = l0 + g;
#pragma unroll
  for (int n = 0; n < NTW; ++n) {
    const int h = h0 + n * 8 + 2 * t;
    if (h < Hq) {
      if (tok < L) gb[(size_t)h * L + tok] = tanhf(acc[n][0]);
      if (tok + 8 < L) gb[(size_t)h * L + tok + 8] = tanhf(acc[n][2]);
    }
    if (h + 1 < Hq) {
      if (tok < L) gb[(size_t)(h + 1) * L + tok] = tanhf(acc[n][1]);
      if (tok + 8 < L) gb[(size_t)(h + 1) * L + tok + 8] = tanhf(acc[n][3]);
    }
  }
}

// ---------------------------------------------------------------------------------------------- dX
// grid (ceil(L / 64), batch, channel slices); KT = head tiles of 16 (the contraction).  Four column tiles of a group of 32
// channels are interleaved (column n of tile u is channel 8 (n / 2) + 2 u + n % 2), so that a thread's accumulators of the four
// are 8 neighbouring channels of a token and go to memory as one 16-byte store; no tile is staged for coalescing.
template <int KT>
__global__ void __launch_bounds__(kGtThreads) gate_bwd_dx_kernel(const bf16* w, const bf16* dz_tm,
                                                                 int L, int Lp, int C, int Hq, int per_slice, int out_f32,
                                                                 void* __restrict__ dx) {
  grid_enter();
  constexpr int LDZ = KT * 16 + 8;
  __shared__ __align__(16) bf16 az[kGtTok * LDZ];            // dz^T: [token][head]
  __shared__ __align__(16) bf16 ws[kDxCh * LDZ];             // W chunk: [channel][head]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int l0 = blockIdx.x * kGtTok, b = blockIdx.y;
  const int c_beg = blockIdx.z * per_slice, c_end = min(C, c_beg + per_slice);
  {
    // the tile's 64 rows of dz_tm are contiguous: 16-byte loads
    const uint4* src = reinterpret_cast<const uint4*>(dz_tm + ((size_t)b * Lp + l0) * (KT * 16));
    for (int e = threadIdx.x; e < kGtTok * KT * 2; e += kGtThreads) {
      const int tl = e / (KT * 2), ch = e % (KT * 2);
      *reinterpret_cast<uint4*>(az + tl * LDZ + ch * 8) = src[e];
    }
  }
  for (int e = threadIdx.x; e < kDxCh * LDZ / 8; e += kGtThreads) reinterpret_cast<uint4*>(ws)[e] = make_uint4(0, 0, 0, 0);   // (padding heads)
  __syncthreads();
  uint32_t a[KT][4];
  {
    const bf16* ar = az + (warp * 16 + g) * LDZ + 2 * t;
#pragma unroll
    for (int ks = 0; ks < KT; ++ks) {
      a[ks][0] = lds32(ar + ks * 16);
      a[ks][1] = lds32(ar + 8 * LDZ + ks * 16);
      a[ks][2] = lds32(ar + ks * 16 + 8);
      a[ks][3] = lds32(ar + 8 * LDZ + ks * 16 + 8);
    }
  }
  const int la = l0 + warp * 16 + g, lb = la + 8;
  // channel of a chunk -> its row in ws: the eight channels of a column tile lie together
  auto w_row = [](int c) { return (c & ~31) + ((c >> 1) & 3) * 8 + ((c >> 3) & 3) * 2 + (c & 1); };
  for (int c0 = c_beg; c0 < c_end; c0 += kDxCh) {
    __syncthreads();                                           // the previous chunk's products have read ws
    if ((reinterpret_cast<uintptr_t>(w) & 15u) == 0) {
      const uint4* src = reinterpret_cast<const uint4*>(w + (size_t)c0 * Hq);
      for (int e = threadIdx.x; e * 8 < kDxCh * Hq; e += kGtThreads)
        scatter_w<LDZ>(ws, c0 * Hq + e * 8 < C * Hq ? src[e] : make_uint4(0, 0, 0, 0), e * 8, Hq, w_row);
    } else {
      for (int e = threadIdx.x; e < kDxCh * KT * 16; e += kGtThreads) {
        const int c = e / (KT * 16), h = e % (KT * 16);
        ws[w_row(c) * LDZ + h] = (h < Hq && c0 + c < C) ? w[(size_t)(c0 + c) * Hq + h] : __float2bfloat16_rn(0.f);
      }
    }
    __syncthreads();
#pragma unroll 2
    for (int q = 0; q < kDxCh / 32; ++q) {
      float acc[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        acc[u][0] = acc[u][1] = acc[u][2] = acc[u][3] = 0.f;
        const bf16* wr = ws + (q * 32 + u * 8 + g) * LDZ + 2 * t;
#pragma unroll
        for (int ks = 0; ks < KT; ++ks) mma_bf16(acc[u], a[ks], lds32(wr + ks * 16), lds32(wr + ks * 16 + 8));
      }
      const int c = c0 + q * 32 + t * 8;                       // (C is a multiple of 8)
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int l = half ? lb : la;
        const size_t idx = ((size_t)b * L + l) * C + c;
        const float* v[4] = {acc[0] + 2 * half, acc[1] + 2 * half, acc[2] + 2 * half, acc[3] + 2 * half};
        if (c < c_end && l < L) {
          if (out_f32) {
            float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(dx) + idx);
            dst[0] = make_float4(v[0][0], v[0][1], v[1][0], v[1][1]);
            dst[1] = make_float4(v[2][0], v[2][1], v[3][0], v[3][1]);
          } else {
            __nv_bfloat162 p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) p[u] = __floats2bfloat162_rn(v[u][0], v[u][1]);
            *reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(dx) + idx) = *reinterpret_cast<const uint4*>(p);
          }
        }
      }
      __syncwarp();                                            // (together again for the next group's products)
    }
  }
}

// ---------------------------------------------------------------------------------------------- dW_g
// grid (ceil(C / 128), splits, batch): partial[(b * splits + s)][c][h] = sum over the split's tokens of X[l, c] dz[l, h]
template <int NT>
__global__ void __launch_bounds__(kGtThreads) gate_bwd_dw_kernel(const bf16* x, const bf16* dz_hm,
                                                                 int L, int Lp, int C, int Hq, int HP,
                                                                 float* __restrict__ partial) {
  grid_enter();
  constexpr int LDZ = kGtTok + 8;
  __shared__ __align__(16) bf16 xs[kGtTok * kLdx];           // [token][channel]; read transposed by ldmatrix
  __shared__ __align__(16) bf16 dz[NT * 8 * LDZ];            // [head][token]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int c0 = blockIdx.x * kGtCh, s = blockIdx.y, b = blockIdx.z, splits = gridDim.y;
  const int per = ((L + splits - 1) / splits + kGtTok - 1) / kGtTok * kGtTok;      // tokens per split, whole tiles
  const int l_beg = s * per, l_end = min(L, l_beg + per);
  const bf16* xb = x + (size_t)b * L * C;
  const bf16* zb = dz_hm + (size_t)b * HP * Lp;
  float acc[2][NT][4];                                        // this warp: channels 32 warp .. + 31 (two tiles of 16)
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
  // the next tile's loads are in flight while a tile is multiplied
  constexpr int XV = kGtTok * (kGtCh / 8) / kGtThreads, ZV = (NT * 8 * (kGtTok / 8) + kGtThreads - 1) / kGtThreads;
  uint4 rx[XV], rz[ZV];
  auto load = [&](int l0) {
#pragma unroll
    for (int u = 0; u < XV; ++u) {
      const int e = threadIdx.x + u * kGtThreads, r = e / (kGtCh / 8), ch = e % (kGtCh / 8);
      rx[u] = (l0 + r < L && c0 + ch * 8 < C) ? *reinterpret_cast<const uint4*>(xb + (size_t)(l0 + r) * C + c0 + ch * 8)
                                              : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int u = 0; u < ZV; ++u) {
      const int e = threadIdx.x + u * kGtThreads, h = e / (kGtTok / 8), ch = e % (kGtTok / 8);
      rz[u] = h < HP ? *reinterpret_cast<const uint4*>(zb + (size_t)h * Lp + l0 + ch * 8) : make_uint4(0, 0, 0, 0);
    }
  };
  if (l_beg < l_end) load(l_beg);
  for (int l0 = l_beg; l0 < l_end; l0 += kGtTok) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < XV; ++u) {
      const int e = threadIdx.x + u * kGtThreads;
      *reinterpret_cast<uint4*>(xs + (e / (kGtCh / 8)) * kLdx + (e % (kGtCh / 8)) * 8) = rx[u];
    }
#pragma unroll
    for (int u = 0; u < ZV; ++u) {
      const int e = threadIdx.x + u * kGtThreads, h = e / (kGtTok / 8), ch = e % (kGtTok / 8);
      if (h < NT * 8) *reinterpret_cast<uint4*>(dz + h * LDZ + ch * 8) = rz[u];
    }
    __syncthreads();
    if (l0 + kGtTok < l_end) load(l0 + kGtTok);
#pragma unroll
    for (int ks = 0; ks < kGtTok / 16; ++ks) {
      uint32_t a[2][4];
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        // four stored 8 x 8 blocks (tokens x channels) -> A fragment (rows = channels, k = tokens) of one 16 x 16 tile:
        // lanes 0-7: tokens 0-7 / channels 0-7, 8-15: tokens 0-7 / channels 8-15, 16-23 and 24-31: tokens 8-15
        const int tok = ks * 16 + (lane >> 4) * 8 + (lane & 7);
        const int ch = warp * 32 + m * 16 + ((lane >> 3) & 1) * 8;
        ldmatrix_x4_trans(a[m], xs + tok * kLdx + ch);
      }
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const bf16* zr = dz + (n * 8 + g) * LDZ + ks * 16 + 2 * t;
        const uint32_t b0 = lds32(zr), b1 = lds32(zr + 8);
        mma_bf16(acc[0][n], a[0], b0, b1);
        mma_bf16(acc[1][n], a[1], b0, b1);
      }
    }
  }
  float* out = partial + (size_t)(b * splits + s) * C * Hq;
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      const int c = c0 + warp * 32 + m * 16 + g, h = n * 8 + 2 * t;
      if (c < C) {
        if (h < Hq) out[(size_t)c * Hq + h] = acc[m][n][0];
        if (h + 1 < Hq) out[(size_t)c * Hq + h + 1] = acc[m][n][1];
      }
      if (c + 8 < C) {
        if (h < Hq) out[(size_t)(c + 8) * Hq + h] = acc[m][n][2];
        if (h + 1 < Hq) out[(size_t)(c + 8) * Hq + h + 1] = acc[m][n][3];
      }
    }
}

__global__ void gate_reduce_dw_kernel(const float* partial, int parts, size_t n, float* __restrict__ dw) {
  grid_enter();
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float acc = 0.f;
  for (int p = 0; p < parts; ++p) acc += partial[(size_t)p * n + i];
  dw[i] = acc;
}

}  // namespace

bool gate_supported(int hidden, int heads) { return hidden > 0 && hidden % 8 == 0 && heads > 0 && heads <= 64; }

namespace {
int padded_heads(int heads) { return (heads + 15) / 16 * 16; }
int padded_tokens(int L) { return (L + kGtTok - 1) / kGtTok * kGtTok; }
size_t dz_bytes(int batch, int L, int heads) { return align_up((size_t)batch * padded_tokens(L) * padded_heads(heads) * sizeof(bf16), 256); }
}  // namespace

// [partial sums of dW_g][dz head-major][dz token-major]
size_t gate_bwd_workspace_bytes(int batch, int L, int hidden, int heads) {
  return align_up((size_t)batch * kGtSplits * hidden * heads * sizeof(float), 256) + 2 * dz_bytes(batch, L, heads);
}

cudaError_t launch_gate_fwd(int batch, int L, int C, int Hq, const bf16* x, const bf16* w, float* gate, cudaStream_t st) {
  // 64 tokens a CTA; with fewer than two such CTAs per SM, 16 tokens and the head tiles split over the warps (2048 tokens of 1536
  // channels: 37 us with 64-token CTAs, which leave 116 of 148 SMs without one)
  int sms = 0;
  cudaError_t e;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  const bool few = (long long)batch * ((L + 63) / 64) < 2 * sms;
  dim3 grid((L + (few ? 15 : 63)) / (few ? 16 : 64), batch);
  const int nt = (Hq + 7) / 8;
#define VSA2_GATE_FWD(NT_, HW_)                                                                                  \
  do {                                                                                                           \
    if (few) launch_kernel(gate_fwd_kernel<NT_, 1, HW_, 256>, grid, kGtThreads, 0, st, x, w, L, C, Hq, gate);               \
    else launch_kernel(gate_fwd_kernel<NT_, 4, 1, 128>, grid, kGtThreads, 0, st, x, w, L, C, Hq, gate);                     \
  } while (0)
  if (nt <= 1) VSA2_GATE_FWD(1, 1);
  else if (nt <= 2) VSA2_GATE_FWD(2, 2);
  else if (nt <= 4) VSA2_GATE_FWD(4, 4);
  else if (nt <= 5) VSA2_GATE_FWD(5, 1);
  else if (nt <= 6) VSA2_GATE_FWD(6, 3);
  else VSA2_GATE_FWD(8, 4);
#undef VSA2_GATE_FWD
  return cudaGetLastError();
}

cudaError_t launch_gate_bwd(int batch, int L, int C, int Hq, int out_f32, const bf16* x, const bf16* w, const float* gate,
                            const float* dgate, float* d_w, void* dx, void* workspace, cudaStream_t st) {
  const int HP = padded_heads(Hq), Lp = padded_tokens(L);
  float* partial = reinterpret_cast<float*>(workspace);
  unsigned char* wsb = reinterpret_cast<unsigned char*>(workspace);
  bf16* dz_hm = reinterpret_cast<bf16*>(wsb + align_up((size_t)batch * kGtSplits * C * Hq * sizeof(float), 256));
  bf16* dz_tm = reinterpret_cast<bf16*>(reinterpret_cast<unsigned char*>(dz_hm) + dz_bytes(batch, L, Hq));
  launch_kernel(gate_dz_kernel, dim3(Lp / kGtTok, batch), kGtThreads, (size_t)HP * (kGtTok + 8) * sizeof(bf16), st, gate, dgate, L, Lp, Hq,
                                                                                                   HP, dz_hm, dz_tm);
  {
    // channel slices until there are eight CTAs per SM (a chunk is the least a CTA takes)
    const int tiles = (L + kGtTok - 1) / kGtTok * batch, chunks = (C + kDxCh - 1) / kDxCh;
    int sms = 0;
    cudaError_t e;
    if ((e = sm_count(&sms)) != cudaSuccess) return e;
    int slices = (8 * sms + tiles - 1) / tiles;
    if (slices > chunks) slices = chunks;
    const int per_slice = (chunks + slices - 1) / slices * kDxCh;
    dim3 grid((L + kGtTok - 1) / kGtTok, batch, (C + per_slice - 1) / per_slice);
    const int kt = (Hq + 15) / 16;
#define VSA2_GATE_DX(KT_) launch_kernel(gate_bwd_dx_kernel<KT_>, grid, kGtThreads, 0, st, w, dz_tm, L, Lp, C, Hq, per_slice, out_f32, dx)
    if (kt <= 1) VSA2_GATE_DX(1);
    else if (kt <= 2) VSA2_GATE_DX(2);
    else if (kt <= 3) VSA2_GATE_DX(3);
    else VSA2_GATE_DX(4);
#undef VSA2_GATE_DX
  }
  {
    dim3 grid((C + kGtCh - 1) / kGtCh, kGtSplits, batch);
    const int nt = (Hq + 7) / 8;
#define VSA2_GATE_DW(NT_) launch_kernel(gate_bwd_dw_kernel<NT_>, grid, kGtThreads, 0, st, x, dz_hm, L, Lp, C, Hq, HP, partial)
    if (nt <= 1) VSA2_GATE_DW(1);
    else if (nt <= 2) VSA2_GATE_DW(2);
    else if (nt <= 4) VSA2_GATE_DW(4);
    else if (nt <= 5) VSA2_GATE_DW(5);
    else if (nt <= 6) VSA2_GATE_DW(6);
    else VSA2_GATE_DW(8);
#undef VSA2_GATE_DW
  }
  const size_t n = (size_t)C * Hq;
  launch_kernel(gate_reduce_dw_kernel, (unsigned)((n + 255) / 256), 256, 0, st, partial, batch * kGtSplits, n, d_w);
  return cudaGetLastError();
}

}  // namespace vsa2
