// First step of the backward pass: the per-token quantities of the gated merge (paper Eq. 14) and of the fine softmax
// (Eq. 12) that the dQ and dK/dV passes (fine_bwd_tc.cu) and the coarse backward read:
//   delta = rowsum(dO * O_f), dGate = rowsum(dO * O_c), dO_c_hat[n] = sum_{l in n} gate_l dO_l (in fp32, or in bf16 with its row sum against O_c)
// and, for the scale of dS in the fp16 passes (DsScale in common.cuh), the largest |dO| and |O| of every block.
// HBM-bound: one pass over dO, O (and the bf16 rounding residual of O).
#include "common.cuh"

namespace vsa2 {

// One CTA of 256 threads per 64-token block: a thread has a 16-byte channel chunk of one token in 256 / (D / 8), two tokens at a time
// (six loads in flight; four CTAs per SM, five with 64 channels); the D / 8 threads of a token reduce its two row sums with shuffles.  The sum
// gate_l dO_l runs over the tokens in PARTS parts side by side, so the dO rows are left in shared memory.  (With
// one thread per chunk walking the block's tokens a small problem waited for sixteen rounds of loads, 21 us.)
// Issue slots (78 %) bound it before memory, so sums and products go two values at a time, and all warps take part in the sum over the tokens (one
// thread per channel walked 64 of them while half the CTA waited).  us, before -> after: 720p, 40 heads 685 -> 647; 480p, 12 heads 82 -> 78; 13 x 27 x 47
// tokens, 16 heads of 64 channels 34.5 -> 29.1 (four CTAs: 32); 2048-token clip 7.1 -> 6.5.  Five CTAs with 128 channels: 688, 84.
// F32: the type of O.  (As a branch in the loop it cost the loads of a token their place ahead of the first use: 720p, 40 heads, 646 us
// against 533 = 4.5 TB/s.)
__device__ __forceinline__ uint32_t word(const uint4& v, int e) { return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w; }
__device__ __forceinline__ float2 bf16_pair(uint32_t x) { return make_float2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }
template <int D, bool F32>
__global__ void __launch_bounds__(256, D == 64 ? 5 : 4) bwd_preprocess_kernel(const bf16* d_o, const void* o,
                                                             const bf16* o_res,
                                                             const float* gate,
                                                             const float* oc_hat, Geo g,
                                                             float* __restrict__ delta, float* __restrict__ dgate,
                                                             float* __restrict__ d_oc_hat, bf16* __restrict__ do_c, float* __restrict__ delta_c,
                                                             float2* __restrict__ absmax, StatusBlock* clear) {
  grid_enter();
  constexpr int CH = D / 8;                // threads per token = 16-byte chunks of a token row
  constexpr int PAR = 256 / CH;            // tokens at a time
  constexpr int TOK = 2;                   // tokens in flight per thread
  __shared__ __align__(16) bf16 rows[kBlockTokens * D];
  __shared__ __align__(16) float gates[kBlockTokens];
  constexpr int PARTS = 512 / D;           // parts of a block's tokens in the sum of gate * dO
  __shared__ __align__(8) float part_sum[PARTS][D];
  __shared__ unsigned warp_max[2][8];
  __shared__ float row_sum[D / 32];
  if (clear != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x < sizeof(StatusBlock) / 4)
    reinterpret_cast<int*>(clear)[threadIdx.x] = 0;      // (for the kernels behind this one)
  const int i = blockIdx.x, ch = threadIdx.x % CH, hq = blockIdx.y, b = blockIdx.z;
  const int lane = threadIdx.x & 31;
  const unsigned group_mask = (CH == 16 ? 0xffffu : 0xffu) << (lane & ~(CH - 1));
  const size_t bhq = (size_t)b * g.Hq + hq;
  // text blocks (i >= Nvid) take no part in the coarse branch or the gate: only delta is formed for them
  const bool coarse = !(g.flags & VSA2_FLAG_NO_COARSE) && gate != nullptr && !block_is_text(g, i);
  float ocv[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) ocv[e] = 0.f;
  if (coarse) {
    const float4* p4 = reinterpret_cast<const float4*>(oc_hat + (bhq * g.Nvid + i) * D + ch * 8);
    const float4 x = *p4, y = p4[1];
    ocv[0] = x.x; ocv[1] = x.y; ocv[2] = x.z; ocv[3] = x.w;
    ocv[4] = y.x; ocv[5] = y.y; ocv[6] = y.z; ocv[7] = y.w;
  }
  unsigned most = 0u;                      // largest |O| (cut to bf16, upper half) and |dO|: bit patterns order like the numbers
#pragma unroll 1
  for (int p0 = threadIdx.x / CH; p0 < kBlockTokens; p0 += TOK * PAR) {
    int l[TOK];
    float gt[TOK];
    uint4 dv[TOK], ov4[TOK][2];            // (O in fp32, or in bf16 and its residual: the same registers)
#pragma unroll
    for (int u = 0; u < TOK; ++u) {
      l[u] = block_token(g, i, p0 + u * PAR);
      gt[u] = 0.f;
      dv[u] = ov4[u][0] = ov4[u][1] = make_uint4(0, 0, 0, 0);
      if (l[u] >= 0) {
        const size_t base = (bhq * g.S + l[u]) * D + ch * 8;
        dv[u] = *reinterpret_cast<const uint4*>(d_o + base);
        if constexpr (F32) {
          ov4[u][0] = *reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(o) + base);
          ov4[u][1] = *reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(o) + base + 4);
        } else {
          ov4[u][0] = *reinterpret_cast<const uint4*>(reinterpret_cast<const bf16*>(o) + base);
          if (o_res != nullptr) ov4[u][1] = *reinterpret_cast<const uint4*>(o_res + base);
        }
        if (coarse) gt[u] = gate[bhq * g.L + l[u]];
      }
    }
#pragma unroll
    for (int u = 0; u < TOK; ++u) {
      const int p = p0 + u * PAR;
      if (coarse) {
        *reinterpret_cast<uint4*>(rows + p * D + ch * 8) = dv[u];
        if (ch == 0) gates[p] = gt[u];
      }
      const unsigned d2_max = __vmaxu2(__vmaxu2(dv[u].x & 0x7fff7fffu, dv[u].y & 0x7fff7fffu),
                                       __vmaxu2(dv[u].z & 0x7fff7fffu, dv[u].w & 0x7fff7fffu));
      unsigned o_max = 0u;
      float2 oo = make_float2(0.f, 0.f), oc = oo;      // even and odd channels apart
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 dd = bf16_pair(word(dv[u], e));
        float2 ov;
        if constexpr (F32) ov = make_float2(__uint_as_float(word(ov4[u][e >> 1], 2 * (e & 1))), __uint_as_float(word(ov4[u][e >> 1], 2 * (e & 1) + 1)));
        else ov = __fadd2_rn(bf16_pair(word(ov4[u][0], e)), bf16_pair(word(ov4[u][1], e)));     // (no residual: zero)
        oo = __ffma2_rn(dd, ov, oo);
        oc = __ffma2_rn(dd, make_float2(ocv[2 * e], ocv[2 * e + 1]), oc);
        o_max = max(max(o_max, __float_as_uint(ov.x) & 0x7fff0000u), __float_as_uint(ov.y) & 0x7fff0000u);
      }
      float s_oo = oo.x + oo.y, s_oc = oc.x + oc.y;
      most = __vmaxu2(most, o_max | max(d2_max >> 16, d2_max & 0xffffu));
#pragma unroll
      for (int off = CH / 2; off >= 1; off >>= 1) {
        s_oo += __shfl_xor_sync(group_mask, s_oo, off);
        s_oc += __shfl_xor_sync(group_mask, s_oc, off);
      }
      if (ch == 0 && l[u] >= 0) {
        delta[bhq * g.S + l[u]] = s_oo - gt[u] * s_oc;     // rowsum(dO * (O - gate*O_c)) = rowsum(dO * O_f)
        if (dgate != nullptr && coarse) dgate[bhq * g.L + l[u]] = s_oc;
      }
    }
  }
  const unsigned d_max = __reduce_max_sync(0xffffffffu, most << 16), o_max = __reduce_max_sync(0xffffffffu, most & 0xffff0000u);
  if (lane == 0) {
    warp_max[0][threadIdx.x >> 5] = d_max;
    warp_max[1][threadIdx.x >> 5] = o_max;
  }
  __syncthreads();
  if (absmax != nullptr && threadIdx.x < 8) {
    const unsigned dm = __reduce_max_sync(0xffu, warp_max[0][threadIdx.x]), om = __reduce_max_sync(0xffu, warp_max[1][threadIdx.x]);
    if (threadIdx.x == 0) absmax[bhq * g.N + i] = make_float2(__uint_as_float(dm), __uint_as_float(om));
  }
  if (!coarse) return;
  {
    constexpr int PT = kBlockTokens / PARTS;
    const int c = threadIdx.x % (D / 2), part = threadIdx.x / (D / 2);
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int p = 0; p < PT; p += 4) {
      const float4 g4 = *reinterpret_cast<const float4*>(gates + part * PT + p);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float w = u == 0 ? g4.x : u == 1 ? g4.y : u == 2 ? g4.z : g4.w;
        acc = __ffma2_rn(make_float2(w, w), bf16_pair(*reinterpret_cast<const uint32_t*>(rows + (part * PT + p + u) * D + 2 * c)), acc);
      }
    }
    *reinterpret_cast<float2*>(&part_sum[part][2 * c]) = acc;
  }
  __syncthreads();
  if (threadIdx.x < D) {
    float acc = part_sum[0][threadIdx.x];
#pragma unroll
    for (int q = 1; q < PARTS; ++q) acc += part_sum[q][threadIdx.x];
    const size_t at = (bhq * g.Nvid + i) * D + threadIdx.x;
    if (d_oc_hat != nullptr) d_oc_hat[at] = acc;
    if (do_c != nullptr) {
      // the coarse branch's backward reads dO_c_hat in bf16 and rowsum(dO_c_hat * O_c) of that
      const bf16 h = __float2bfloat16_rn(acc);
      do_c[at] = h;
      float s = __bfloat162float(h) * oc_hat[at];
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      if (lane == 0) row_sum[threadIdx.x >> 5] = s;
    }
  }
  if (do_c == nullptr) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < D / 32; ++w) s += row_sum[w];
    delta_c[bhq * g.Nvid + i] = s;
  }
}

cudaError_t launch_bwd_preprocess(const Geo& g, const bf16* d_o, const void* o, const bf16* o_res, const float* gate,
                                  const float* oc_hat, float* delta, float* dgate, float* d_oc_hat, bf16* do_c, float* delta_c,
                                  float2* absmax, StatusBlock* clear, cudaStream_t st) {
  dim3 grid(g.N, g.Hq, g.batch);
  if (g.D == 128 && g.out_f32) launch_kernel(bwd_preprocess_kernel<128, true>, grid, 256, 0, st, d_o, o, o_res, gate, oc_hat, g, delta, dgate, d_oc_hat, do_c, delta_c, absmax, clear);
  else if (g.D == 128) launch_kernel(bwd_preprocess_kernel<128, false>, grid, 256, 0, st, d_o, o, o_res, gate, oc_hat, g, delta, dgate, d_oc_hat, do_c, delta_c, absmax, clear);
  else if (g.out_f32) launch_kernel(bwd_preprocess_kernel<64, true>, grid, 256, 0, st, d_o, o, o_res, gate, oc_hat, g, delta, dgate, d_oc_hat, do_c, delta_c, absmax, clear);
  else launch_kernel(bwd_preprocess_kernel<64, false>, grid, 256, 0, st, d_o, o, o_res, gate, oc_hat, g, delta, dgate, d_oc_hat, do_c, delta_c, absmax, clear);
  return cudaGetLastError();
}

}  // namespace vsa2
