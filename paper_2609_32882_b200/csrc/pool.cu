// Mean pooling over cubes (coarse branch, paper Eq. 1) and over router sub-cubes (Eq. 5).
// HBM-bound: every token row is read once with 16-byte loads.
// (one cube decode per thread: this file keeps the reciprocal form of the index divisions, which measured 7 % faster here)
#define VSA2_RECIPROCAL_DIVMOD 1
#include "common.cuh"

namespace vsa2 {

// Any router pool other than 2 x 2 x 2: one thread per (cube, 16-byte channel chunk) reads the cube's tokens sub-cube by
// sub-cube, so no tile is staged in shared memory and a warp's loads cover whole 256-byte token rows.
//   xr [b, h, N*G, D] bf16 : fp32 sum along w, then h, then t (each left to right; padding positions add +0), IEEE fp32
//                            division by the valid count, rounded to bf16 (nearest even).
//   xc [b, h, N, D]   fp32 : sum of the sub-cube sums / count.
// Up to three tensors per launch (grid.y runs over the heads of all of them).
struct PoolJob {
  const bf16* x;
  bf16* xr;
  float* xc;
  int heads;
};
struct PoolJobs {
  PoolJob job[3];
  int n;
  StatusBlock* clear;       // null, or a status block to set to zero for the kernels behind this one
};
__device__ __forceinline__ void clear_status(const PoolJobs& jobs) {
  if (jobs.clear != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x < sizeof(StatusBlock) / 4)
    reinterpret_cast<int*>(jobs.clear)[threadIdx.x] = 0;
}

__device__ __forceinline__ void add8(float (&acc)[8], const float (&v)[8], bool first) {
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = first ? v[i] : __fadd_rn(acc[i], v[i]);
}
__device__ __forceinline__ void load8(const bf16* base, int t, int h, int w, const Geo& g, int D, float (&f)[8]) {
  uint4 v = make_uint4(0, 0, 0, 0);
  if (t < g.T && h < g.H && w < g.W) v = *reinterpret_cast<const uint4*>(base + (size_t)((t * g.H + h) * g.W + w) * D);
  const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 x = __bfloat1622float2(h2[i]);
    f[2 * i] = x.x;
    f[2 * i + 1] = x.y;
  }
}

template <int D>
__global__ void __launch_bounds__(128) pool_kernel(PoolJobs jobs, Geo g) {
  grid_enter();
  constexpr int CH = D / 8;            // 16-byte chunks of a token row
  constexpr int CUBES = 128 / CH;      // cubes per CTA
  clear_status(jobs);
  int h = blockIdx.y;
  PoolJob jb = jobs.job[0];
  if (jobs.n > 1 && h >= jb.heads) {
    h -= jb.heads;
    jb = jobs.job[1];
    if (jobs.n > 2 && h >= jb.heads) {
      h -= jb.heads;
      jb = jobs.job[2];
    }
  }
  const int n = blockIdx.x * CUBES + threadIdx.x / CH, ch = threadIdx.x % CH, b = blockIdx.z;
  if (n >= g.N) return;
  const size_t bh = (size_t)b * jb.heads + h;
  const bf16* base = jb.x + bh * (size_t)g.S * D + ch * 8;
  int nt, nh, nw;
  cube_coords(g, n, nt, nh, nw);
  float tot[8];
  for (int gsub = 0; gsub < g.G; ++gsub) {
    const int gw = gsub % g.Gw, r = gsub / g.Gw, gh = r % g.Gh, gt = r / g.Gh;
    const int t0 = nt * g.Bt + gt * g.Rt, h0 = nh * g.Bh + gh * g.Rh, w0 = nw * g.Bw + gw * g.Rw;
    float ts[8];
    for (int it = 0; it < g.Rt; ++it) {
      float hs[8];
      for (int ih = 0; ih < g.Rh; ++ih) {
        float ws[8];
        for (int iw = 0; iw < g.Rw; ++iw) {
          float v[8];
          load8(base, t0 + it, h0 + ih, w0 + iw, g, D, v);
          add8(ws, v, iw == 0);
        }
        add8(hs, ws, ih == 0);
      }
      add8(ts, hs, it == 0);
    }
    add8(tot, ts, gsub == 0);
    if (jb.xr != nullptr) {
      const int cnt = subcube_count(g, n, gsub);
      uint4 o = make_uint4(0, 0, 0, 0);
      if (cnt > 0) {
        const float c = (float)cnt;
        __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
        for (int i = 0; i < 4; ++i) o2[i] = __floats2bfloat162_rn(__fdiv_rn(ts[2 * i], c), __fdiv_rn(ts[2 * i + 1], c));
      }
      *reinterpret_cast<uint4*>(jb.xr + ((bh * g.N + n) * g.G + gsub) * D + ch * 8) = o;
    }
  }
  if (jb.xc != nullptr) {
    const float cnt = (float)cube_count(g, n);
    float* dst = jb.xc + (bh * g.N + n) * D + ch * 8;
    float m[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) m[i] = cnt > 0.f ? tot[i] / cnt : 0.f;
    *reinterpret_cast<float4*>(dst) = make_float4(m[0], m[1], m[2], m[3]);
    *reinterpret_cast<float4*>(dst + 4) = make_float4(m[4], m[5], m[6], m[7]);
  }
}

// The same for the 2 x 2 x 2 router pool with one thread per (sub-cube, 16-byte chunk), for cubes of G = 8 sub-cubes: a CTA has
// kSubThreads / (D / 8) sub-cubes, whole cubes, whose sub-cube sums meet in shared memory and are added in order.
// Every load of a thread is in flight at once.  (One thread per cube walks eight sub-cubes one after another, 9 us on
// the smallest grids.)  The rest is kept short, since issue slots (84 to 88 %) bounded it, not memory: shifts for the sub-cube's place, one test per
// direction, two values per addition, a product for the quotient.  Means of Q, K / of Q, K, V, us, before -> after: 720p, 40 heads 279 -> 251 / 418 -> 362;
// 13 x 27 x 47 tokens, 16 heads of 64 channels 19.0 -> 15.2 / 63.7 -> 59.9 (the second starts beside its predecessor); 435,600 tokens, 10 heads
// 432 -> 388 / 3 x 204 -> 184.  The six CTAs leave the compiler the registers for eight loads at once: free to choose it took 48 and made 294 / 458 of
// the first.
constexpr int kSubThreads = 128;
template <int D>
__global__ void __launch_bounds__(kSubThreads, 6) pool_subcube_kernel(PoolJobs jobs, Geo g) {
  grid_enter();
  constexpr int CH = D / 8, SUB = kSubThreads / CH, CUBES = SUB / 8;
  __shared__ __align__(16) float sums[SUB * D];
  clear_status(jobs);
  int h = blockIdx.y;
  PoolJob jb = jobs.job[0];
  if (jobs.n > 1 && h >= jb.heads) {
    h -= jb.heads;
    jb = jobs.job[1];
    if (jobs.n > 2 && h >= jb.heads) {
      h -= jb.heads;
      jb = jobs.job[2];
    }
  }
  const int sub = threadIdx.x / CH, ch = threadIdx.x % CH, b = blockIdx.z;
  const int n = blockIdx.x * CUBES + (sub >> 3), gsub = sub & 7;
  const size_t bh = (size_t)b * jb.heads + h;
  if (n < g.N) {
    const bf16* base = jb.x + bh * (size_t)g.S * D + ch * 8;
    int nt, nh, nw;
    cube_coords(g, n, nt, nh, nw);
    // (Gw, Gh: their product with Gt is 8)
    const int lw = __ffs(g.Gw) - 1, lh = __ffs(g.Gh) - 1, gw = gsub & (g.Gw - 1), gh = (gsub >> lw) & (g.Gh - 1), gt = gsub >> (lw + lh);
    const int t0 = nt * g.Bt + gt * 2, h0 = nh * g.Bh + gh * 2, w0 = nw * g.Bw + gw * 2;
    const bool in0 = t0 < g.T && h0 < g.H && w0 < g.W, in_t = t0 + 1 < g.T, in_h = h0 + 1 < g.H, in_w = w0 + 1 < g.W;
    const bf16* at0 = base + (size_t)((t0 * g.H + h0) * g.W + w0) * D;
    const size_t row = (size_t)g.W * D, frame = g.H * row;
    uint4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const bool in = in0 && (!(k & 4) || in_t) && (!(k & 2) || in_h) && (!(k & 1) || in_w);
      v[k] = make_uint4(0, 0, 0, 0);
      if (in) v[k] = *reinterpret_cast<const uint4*>(at0 + (k & 4 ? frame : 0) + (k & 2 ? row : 0) + (k & 1 ? D : 0));
    }
    float2 ts[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      auto pair = [&](int k) {             // the two values of word i of token k
        const uint32_t x = i == 0 ? v[k].x : i == 1 ? v[k].y : i == 2 ? v[k].z : v[k].w;
        return make_float2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u));
      };
      ts[i] = __fadd2_rn(__fadd2_rn(__fadd2_rn(pair(0), pair(1)), __fadd2_rn(pair(2), pair(3))),
                         __fadd2_rn(__fadd2_rn(pair(4), pair(5)), __fadd2_rn(pair(6), pair(7))));
    }
    if (jb.xr != nullptr) {
      uint4 o = make_uint4(0, 0, 0, 0);
      if (in0) {
        // 1, 2, 4 or 8 tokens: the product with the reciprocal is the quotient
        const float inv = (in_t ? 0.5f : 1.f) * (in_h ? 0.5f : 1.f) * (in_w ? 0.5f : 1.f);
        __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
        for (int i = 0; i < 4; ++i) o2[i] = __floats2bfloat162_rn(__fmul_rn(ts[i].x, inv), __fmul_rn(ts[i].y, inv));
      }
      *reinterpret_cast<uint4*>(jb.xr + ((bh * g.N + n) * 8 + gsub) * D + ch * 8) = o;
    }
    if (jb.xc != nullptr) {
      float4* dst = reinterpret_cast<float4*>(sums + sub * D + ch * 8);
      dst[0] = make_float4(ts[0].x, ts[0].y, ts[1].x, ts[1].y);
      dst[1] = make_float4(ts[2].x, ts[2].y, ts[3].x, ts[3].y);
    }
  }
  if (jb.xc == nullptr) return;            // (the same for every thread of the CTA)
  __syncthreads();
  if (n < g.N) {
    // kSubThreads threads, CUBES * D means: one each
    const int cube = threadIdx.x / D, d = threadIdx.x % D, nn = blockIdx.x * CUBES + cube;
    if (nn < g.N) {
      float tot = sums[cube * 8 * D + d];
#pragma unroll
      for (int q = 1; q < 8; ++q) tot = __fadd_rn(tot, sums[(cube * 8 + q) * D + d]);
      const float cnt = (float)cube_count(g, nn);
      jb.xc[(bh * g.N + nn) * D + d] = cnt > 0.f ? tot / cnt : 0.f;
    }
  }
}

// Cube-major copy of a raster tensor (paper Sec. 2.2 "Permutation") and back.  One CTA per (cube, head, batch):
//   forward: y[b, h, n * B + p, :] = x[b, h, token(n, p), :], zero where position p of cube n lies outside the grid
//   inverse: x[b, h, token(n, p), :] = y[b, h, n * B + p, :] for the positions inside the grid
// The attention kernels never need this copy (they address cubes through tensor maps over the raster layout); it is for
// callers whose surrounding code works in the cube-major layout.
template <int D>
__global__ void __launch_bounds__(256) permute_kernel(const bf16* src, int heads, Geo g, int inverse,
                                                      bf16* __restrict__ dst) {
  grid_enter();
  const int n = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const size_t bh = (size_t)b * heads + h;
  const int B = g.Bt * g.Bh * g.Bw;
  int nt, nh, nw;
  cube_coords(g, n, nt, nh, nw);
  constexpr int CH = D / 8;
  for (int c = threadIdx.x; c < B * CH; c += blockDim.x) {
    const int p = c / CH, ch = c % CH;
    const int l = cube_token(g, nt, nh, nw, p);
    const size_t raster = (bh * g.S + (size_t)max(l, 0)) * D + ch * 8;
    const size_t cubed = ((bh * g.N + n) * B + p) * (size_t)D + ch * 8;
    if (!inverse) {
      uint4 v = make_uint4(0, 0, 0, 0);
      if (l >= 0) v = *reinterpret_cast<const uint4*>(src + raster);
      *reinterpret_cast<uint4*>(dst + cubed) = v;
    } else if (l >= 0) {
      *reinterpret_cast<uint4*>(dst + raster) = *reinterpret_cast<const uint4*>(src + cubed);
    }
  }
}

cudaError_t launch_permute(const Geo& g, const bf16* src, int heads, bool inverse, bf16* dst, cudaStream_t st) {
  dim3 grid(g.N, heads, g.batch);
  if (g.D == 128) launch_kernel(permute_kernel<128>, grid, 256, 0, st, src, heads, g, inverse ? 1 : 0, dst);
  else launch_kernel(permute_kernel<64>, grid, 256, 0, st, src, heads, g, inverse ? 1 : 0, dst);
  return cudaGetLastError();
}

static cudaError_t launch_pool_jobs(const Geo& g, const PoolJobs& jobs, cudaStream_t st) {
  int heads = 0;
  for (int i = 0; i < jobs.n; ++i) heads += jobs.job[i].heads;
  const int cubes = 128 / (g.D / 8);
  dim3 grid((g.N + cubes - 1) / cubes, heads, g.batch);
  const bool r222 = g.Rt == 2 && g.Rh == 2 && g.Rw == 2;
  if (r222 && g.G == 8) {          // (blocks of 64 tokens have eight such sub-cubes whatever the cube's shape)
    const int per_cta = kSubThreads / g.D;
    dim3 sub_grid((g.N + per_cta - 1) / per_cta, heads, g.batch);
    if (g.D == 128) launch_kernel(pool_subcube_kernel<128>, sub_grid, kSubThreads, 0, st, jobs, g);
    else launch_kernel(pool_subcube_kernel<64>, sub_grid, kSubThreads, 0, st, jobs, g);
    return cudaGetLastError();
  }
  if (g.D == 128) launch_kernel(pool_kernel<128>, grid, 128, 0, st, jobs, g);
  else launch_kernel(pool_kernel<64>, grid, 128, 0, st, jobs, g);
  return cudaGetLastError();
}

cudaError_t launch_pool(const Geo& g, const bf16* x, int heads, bf16* xr, float* xc, StatusBlock* clear, cudaStream_t st) {
  PoolJobs jobs{};
  jobs.clear = clear;
  jobs.job[0] = PoolJob{x, xr, xc, heads};
  jobs.n = 1;
  return launch_pool_jobs(g, jobs, st);
}

// router means of Q and K (Eq. 5) in one launch
cudaError_t launch_pool_router(const Geo& g, const bf16* q, const bf16* k, bf16* qr, bf16* kr, StatusBlock* clear, cudaStream_t st) {
  PoolJobs jobs{};
  jobs.clear = clear;
  jobs.job[0] = PoolJob{q, qr, nullptr, g.Hq};
  jobs.job[1] = PoolJob{k, kr, nullptr, g.Hkv};
  jobs.n = 2;
  return launch_pool_jobs(g, jobs, st);
}

// cube means of Q, K and V (Eq. 1) in one launch
cudaError_t launch_pool_coarse(const Geo& g, const bf16* q, const bf16* k, const bf16* v, float* qc, float* kc, float* vc,
                               StatusBlock* clear, cudaStream_t st) {
  PoolJobs jobs{};
  jobs.clear = clear;
  jobs.job[0] = PoolJob{q, nullptr, qc, g.Hq};
  jobs.job[1] = PoolJob{k, nullptr, kc, g.Hkv};
  jobs.job[2] = PoolJob{v, nullptr, vc, g.Hkv};
  jobs.n = 3;
  return launch_pool_jobs(g, jobs, st);
}

}  // namespace vsa2
