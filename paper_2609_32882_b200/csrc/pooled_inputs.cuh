// What the kernels on the pooled grid read (coarse_pooled.cu), made by blocks of a launch of its own or of the backward's preparation (bwd_prep.cu).
#pragma once
#include "common.cuh"

namespace vsa2 {

// dense map of np blocks for `heads` lists: ptr[h][i] = i * np, idx[h][i * np + j] = j (its transpose is the same map)
__device__ __forceinline__ void dense_map_entry(int* ptr, int* idx, int np, size_t e) {
  const size_t per = (size_t)np * np + np + 1, h = e / per;
  const int r = (int)(e - h * per);
  if (r <= np) ptr[h * (np + 1) + r] = r * np;
  else idx[h * np * np + r - np - 1] = (r - np - 1) % np;
}
// What the pooled kernels read: bf16 copies of up to four fp32 tensors, the dense map, a cleared status block
struct PooledInputs {
  const float* x[4];
  bf16* y[4];
  size_t n4[4];            // 16-byte groups of each tensor
  int* ptr;
  int* idx;
  int np;
  size_t map_words;        // heads * (np * np + np + 1)
  StatusBlock* status;
};
__device__ __forceinline__ void pooled_inputs(const PooledInputs& p, unsigned block, unsigned blocks) {
  if (block == 0 && threadIdx.x < sizeof(StatusBlock) / 4) reinterpret_cast<int*>(p.status)[threadIdx.x] = 0;
  const size_t stride = (size_t)blocks * blockDim.x, first = block * (size_t)blockDim.x + threadIdx.x;
#pragma unroll
  for (int t = 0; t < 4; ++t)
    for (size_t i = first; i < p.n4[t]; i += stride) {
      const float4 v = reinterpret_cast<const float4*>(p.x[t])[i];
      __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
      uint2 o;
      o.x = *reinterpret_cast<uint32_t*>(&a);
      o.y = *reinterpret_cast<uint32_t*>(&b);
      reinterpret_cast<uint2*>(p.y[t])[i] = o;
    }
  for (size_t i = first; i < p.map_words; i += stride) dense_map_entry(p.ptr, p.idx, p.np, i);
}
inline unsigned pooled_inputs_blocks(const PooledInputs& p, int sms) {
  size_t most = p.map_words;
  for (size_t n : p.n4) most = n > most ? n : most;
  const size_t blocks = (most + 255) / 256;
  return (unsigned)(blocks < (size_t)sms * 8 ? blocks : (size_t)sms * 8);
}
// Inputs of the backward on the pooled grid; without d_oc_hat its copy is not among them (launch_bwd_preprocess leaves it, and delta)
PooledInputs pooled_bwd_inputs(const Geo& g, const float* qc, const float* kc, const float* vc, const float* d_oc_hat, void* workspace);
float* pooled_bwd_delta(const Geo& g, void* workspace);

}  // namespace vsa2
