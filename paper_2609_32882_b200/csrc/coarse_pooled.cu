// Coarse branch (paper Eq. 2-3) and its backward on the Blackwell tensor cores, by running the fine-branch kernels on the
// POOLED grid: the N = Nt x Nh x Nw cube means form a small (Nt, Nh, Nw) token grid of their own, in raster order,
// and dense attention over them is block-sparse attention with every block selected.  The pooled fp32 means are
// rounded to bf16 (the precision of the model's other attention operands), the outputs stay fp32.
// This file holds the glue: the pooled problem's geometry, the dense block map, the casts and the launch sequence.
#include "pooled_inputs.cuh"

namespace vsa2 {

// geometry of the pooled problem: tokens = cubes of g, cubes of 4 x 4 x 4 pooled tokens, every block selected
Geo pooled_geo(const Geo& g) {
  Geo p = wide_cube(g) ? narrow_geo(g) : g;      // the kernels' blocks are 64 pooled tokens whatever the caller's cube
  p.T = g.Nt; p.H = g.Nh; p.W = g.Nw;
  p.L = g.N;
  p.Nt = (p.T + p.Bt - 1) / p.Bt; p.Nh = (p.H + p.Bh - 1) / p.Bh; p.Nw = (p.W + p.Bw - 1) / p.Bw;
  p.N = p.Nt * p.Nh * p.Nw;
  geo_set_magics(p);
  p.Nvid = p.N; p.Lt = 0; p.S = p.L;
  p.K = p.N;
  p.mode = VSA2_PER_QUERY;
  p.out_f32 = 1;
  p.flags = VSA2_FLAG_NO_COARSE;
  p.nnz_cap = (long long)p.N * p.N;
  return p;
}

PooledLayout pooled_layout(const Geo& g, bool backward) {
  const Geo p = pooled_geo(g);
  PooledLayout r;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
  const size_t BHq = (size_t)g.batch * g.Hq, BHk = (size_t)g.batch * g.Hkv;
  r.status = take(fine_fwd_tc_workspace_bytes());
  r.q16 = take(BHq * g.N * g.D * sizeof(bf16));
  r.k16 = take(BHk * g.N * g.D * sizeof(bf16));
  r.v16 = take(BHk * g.N * g.D * sizeof(bf16));
  r.ptr = take(BHq * (p.N + 1) * sizeof(int));
  r.idx = take(BHq * (size_t)p.N * p.N * sizeof(int));
  r.do16 = r.delta = r.dk_kv = r.dv_kv = 0;
  if (backward) {
    r.do16 = take(BHq * g.N * g.D * sizeof(bf16));
    r.delta = take(BHq * g.N * sizeof(float));
    r.dk_kv = take(BHk * g.N * g.D * sizeof(float));
    r.dv_kv = take(BHk * g.N * g.D * sizeof(float));
  }
  r.total = off;
  return r;
}

__global__ void __launch_bounds__(256) pooled_inputs_kernel(PooledInputs p) {
  grid_enter();
  pooled_inputs(p, blockIdx.x, gridDim.x);
}
static cudaError_t launch_pooled_inputs(const PooledInputs& p, cudaStream_t st) {
  int sms = 0;
  cudaError_t e;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  launch_kernel(pooled_inputs_kernel, pooled_inputs_blocks(p, sms), 256, 0, st, p);
  return cudaGetLastError();
}

// the recursive dK/dV pass returns one gradient per KV head; the epilogues of the main passes sum dK_c, dV_c over the
// query heads of a group, so the result goes to the group's first query head and zeros to the others
__global__ void spread_to_group_kernel(const float* x_kv, float* __restrict__ x_q, int rep, size_t per_head4,
                                       int heads_q) {
  grid_enter();
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const int hq = blockIdx.y;            // b * Hq + hq (Hq = Hkv * rep, so b * Hq + hq = (b * Hkv + hk) * rep + hh)
  if (i >= per_head4 || hq >= heads_q) return;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (hq % rep == 0) v = reinterpret_cast<const float4*>(x_kv)[(size_t)(hq / rep) * per_head4 + i];
  reinterpret_cast<float4*>(x_q)[(size_t)hq * per_head4 + i] = v;
}

// The pooled passes count their work items in a status block of their own (inside the scratch region).  The backward ones report to the
// caller's block; a non-zero status word that the forward leaves there (a bounded wait that ran out, a rescue list that overflowed) is copied
// into the caller's status word, which is the one vsa2_device_status reads.
__global__ void merge_status_kernel(const StatusBlock* from, StatusBlock* into) {
  grid_enter();
  const int s = from->status;
  if (s != 0) atomicCAS(&into->status, 0, s);
}

cudaError_t launch_coarse_fwd_pooled(const Geo& g, const float* qc, const float* kc, const float* vc, float* oc_hat,
                                     float* lse_c, void* workspace, StatusBlock* caller_status, cudaStream_t st) {
  const Geo p = pooled_geo(g);
  const PooledLayout lay = pooled_layout(g, false);
  unsigned char* ws = reinterpret_cast<unsigned char*>(workspace);
  const size_t BHq = (size_t)g.batch * g.Hq, BHk = (size_t)g.batch * g.Hkv;
  bf16* q16 = reinterpret_cast<bf16*>(ws + lay.q16);
  bf16* k16 = reinterpret_cast<bf16*>(ws + lay.k16);
  bf16* v16 = reinterpret_cast<bf16*>(ws + lay.v16);
  int* ptr = reinterpret_cast<int*>(ws + lay.ptr);
  int* idx = reinterpret_cast<int*>(ws + lay.idx);
  cudaError_t e;
  const PooledInputs in{{qc, kc, vc, nullptr}, {q16, k16, v16, nullptr}, {BHq * g.N * g.D / 4, BHk * g.N * g.D / 4, BHk * g.N * g.D / 4, 0},
                        ptr, idx, p.N, BHq * ((size_t)p.N * p.N + p.N + 1), reinterpret_cast<StatusBlock*>(ws + lay.status)};
  if ((e = launch_pooled_inputs(in, st)) != cudaSuccess) return e;
  if ((e = launch_fine_fwd_tc(p, q16, k16, v16, nullptr, ptr, idx, nullptr, oc_hat, nullptr, lse_c,
                              reinterpret_cast<StatusBlock*>(ws + lay.status), st)) != cudaSuccess)
    return e;
  launch_kernel(merge_status_kernel, 1, 1, 0, st, reinterpret_cast<const StatusBlock*>(ws + lay.status), caller_status);
  return cudaGetLastError();
}

PooledInputs pooled_bwd_inputs(const Geo& g, const float* qc, const float* kc, const float* vc, const float* d_oc_hat, void* workspace) {
  const PooledLayout lay = pooled_layout(g, true);
  unsigned char* ws = reinterpret_cast<unsigned char*>(workspace);
  const int np = pooled_geo(g).N;
  const size_t BHq = (size_t)g.batch * g.Hq, nq = BHq * g.N * g.D / 4, nk = (size_t)g.batch * g.Hkv * g.N * g.D / 4;      // (multiples of the head dimension)
  auto b16 = [&](size_t off) { return reinterpret_cast<bf16*>(ws + off); };
  return PooledInputs{{qc, kc, vc, d_oc_hat}, {b16(lay.q16), b16(lay.k16), b16(lay.v16), b16(lay.do16)}, {nq, nk, nk, d_oc_hat != nullptr ? nq : 0},
                      reinterpret_cast<int*>(ws + lay.ptr), reinterpret_cast<int*>(ws + lay.idx), np, BHq * ((size_t)np * np + np + 1),
                      reinterpret_cast<StatusBlock*>(ws + lay.status)};
}
float* pooled_bwd_delta(const Geo& g, void* workspace) { return reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(workspace) + pooled_layout(g, true).delta); }

cudaError_t launch_coarse_bwd_pooled(const Geo& g, const float* qc, const float* kc, const float* vc, const float* oc_hat,
                                     const float* lse_c, const float* d_oc_hat, float* dqc, float* dkc, float* dvc,
                                     void* workspace, StatusBlock* caller_status, cudaStream_t st) {
  const Geo p = pooled_geo(g);
  const PooledLayout lay = pooled_layout(g, true);
  const PooledInputs in = pooled_bwd_inputs(g, qc, kc, vc, d_oc_hat, workspace);
  unsigned char* ws = reinterpret_cast<unsigned char*>(workspace);
  const size_t BHq = (size_t)g.batch * g.Hq;
  const bf16 *q16 = in.y[0], *k16 = in.y[1], *v16 = in.y[2], *do16 = in.y[3];
  const int *ptr = in.ptr, *idx = in.idx;
  float* delta = pooled_bwd_delta(g, workspace);
  float* dk_kv = reinterpret_cast<float*>(ws + lay.dk_kv);
  float* dv_kv = reinterpret_cast<float*>(ws + lay.dv_kv);
  StatusBlock* status = in.status;
  cudaError_t e;
  if (d_oc_hat != nullptr) {
    if ((e = launch_pooled_inputs(in, st)) != cudaSuccess) return e;
    // delta_c = rowsum(dO_c * O_c) through the preprocess kernel of the pooled problem (no gate: only delta is written)
    if ((e = launch_bwd_preprocess(p, do16, oc_hat, nullptr, nullptr, nullptr, delta, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, st)) != cudaSuccess) return e;
  }
  // side by side where neither fills the GPU: whole passes as graphs, us, toy grid 59.5 -> 54.3, 2048-token clip with training 151.5 -> 145.5
  if ((e = launch_fine_bwd_dq_tc(p, q16, k16, v16, do16, lse_c, delta, ptr, idx, nullptr, dqc, status, st, nullptr, nullptr, nullptr,
                                 caller_status, true)) != cudaSuccess)
    return e;
  const bool grouped = g.rep > 1;
  if ((e = launch_fine_bwd_dkv_tc(p, q16, k16, v16, do16, lse_c, delta, ptr, idx, nullptr, nullptr, grouped ? dk_kv : dkc,
                                  grouped ? dv_kv : dvc, status, st, false, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, PackedCubes{},
                                  caller_status, true)) != cudaSuccess)
    return e;
  if (grouped) {
    const size_t per_head4 = (size_t)g.N * g.D / 4;
    dim3 grid((unsigned)((per_head4 + 255) / 256), (unsigned)BHq);
    launch_kernel(spread_to_group_kernel, grid, 256, 0, st, dk_kv, dkc, g.rep, per_head4, (int)BHq);
    launch_kernel(spread_to_group_kernel, grid, 256, 0, st, dv_kv, dvc, g.rep, per_head4, (int)BHq);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace vsa2
