// What the backward's passes read beside their tensors, in one launch: the fp16 copies of Q and K with the exponents of dS, where every pair's
// dS tile lies, the counts of packed query cubes, the order of the dK/dV pass, and the inputs of the coarse branch's backward.
// These were five launches.  Each of the small ones waited for the one before it and kept a few SMs busy; here they run beside the copies, which
// are bound by HBM.  Training passes, us, five launches / one: 2048-token clip 171 / 163, 13 x 27 x 47 tokens, 16 heads 1350 / 1328, a toy grid 162 / 143 (as a
// graph 66 / 62); from 480p on no difference.
#include "fine_bwd_tc.cuh"
#include "pooled_inputs.cuh"

namespace vsa2 {

struct BwdPrepArgs {
  int exp_blocks, order_blocks, pooled_blocks, list_blocks;      // (the remaining blocks of the grid: copies)
  CastJob cast;
  DsScale scale;
  int groups, per_group;
  PooledInputs pooled;
  // block lists of dS (PrepLists): geometry by which the tiles are placed
  Geo g;
  PrepLists lists;
  int lists_per_head;                                            // blocks of 8 columns
};

// Places of the entries e0, e0 + 32, .. of column j of a head: U searches at once
template <int U>
__device__ __forceinline__ void find_places(const Geo& g, const int* rp, const int* ci, const int* list, int j, int e0, int end, int (&row)[U], int (&place)[U]) {
  int lo[U], hi[U], open = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) row[u] = e0 + 32 * u < end ? list[e0 + 32 * u] : -1;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    lo[u] = hi[u] = 0;
    if (row[u] >= 0) {                          // the entry j is in [lo, hi]
      lo[u] = rp[row[u]];
      hi[u] = rp[row[u] + 1] - 1;
    }
  }
  if (j >= g.Nvid) {                            // a text block: the last ones of every list
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int at = hi[u] + 1 - (g.N - j);
      if (row[u] >= 0 && at >= lo[u] && ci[at] == j) lo[u] = hi[u] = at;
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) open |= lo[u] < hi[u];
  while (open) {
    open = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (lo[u] < hi[u]) {
        const int mid = (lo[u] + hi[u]) >> 1;
        if (ci[mid] < j) lo[u] = mid + 1;
        else hi[u] = mid;
      }
      open |= lo[u] < hi[u];
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) place[u] = lo[u];
}

// One warp per column of the block map.  Place of every entry of the column's list in the row lists of its head: pos[bh][e] for entry
// e of row_idx (both kinds of lists ascend); and the entries in front of the cubes of a cut last layer -- or, of a list that does not have
// them at its end, all but the text blocks (nothing of it is packed then).
// A search is a chain of loads and a column can hold every query (the text blocks' do), so a lane has four under way at once where there are more
// than 32 entries, and text blocks are looked for where they lie.  The launch, us, one search at a time / this: 720p, 5 heads with text
// 182 / 71; 480p, 12 heads on 3 71 / 56; 8 heads on 2 with budgets 150 / 125.
__device__ __forceinline__ void prep_lists(const BwdPrepArgs& a, int block) {
  const Geo& g = a.g;
  const PrepLists& l = a.lists;
  if (block == 0)
    for (int c = threadIdx.x; c < l.n_counters; c += blockDim.x) l.counters[c] = 0;
  const int bh = block / a.lists_per_head, j = (block - bh * a.lists_per_head) * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= g.N) return;
  const long long cap = g.nnz_cap;
  const int* rp = l.row_ptr + (size_t)bh * (g.N + 1);
  const int* ci = l.col_idx + (size_t)bh * cap;
  const int* list = l.row_idx + (size_t)bh * cap;
  const int beg = l.col_ptr[(size_t)bh * (g.N + 1) + j], end = l.col_ptr[(size_t)bh * (g.N + 1) + j + 1], video_end = end - (g.N - g.Nvid);
  int n = 0, last = -1;                       // entries before the layer, and the last of them
  auto store = [&](int e, int i, int place) {
    if (e >= end) return;
    l.pos[(size_t)bh * cap + e] = min(place, (int)cap - 1);      // (column lists that are not the row lists' transpose stay inside the scratch)
    if (e < video_end && i < l.first) {
      ++n;
      last = e - beg;
    }
  };
  if (end - beg <= 32) {
    int row[1], place[1];
    find_places(g, rp, ci, list, j, beg + lane, end, row, place);
    store(beg + lane, row[0], place[0]);
  } else {
    for (int e0 = beg + lane; e0 < end; e0 += 128) {
      int row[4], place[4];
      find_places(g, rp, ci, list, j, e0, end, row, place);
#pragma unroll
      for (int u = 0; u < 4; ++u) store(e0 + 32 * u, row[u], place[u]);
    }
  }
  if (l.full == nullptr) return;
  n = __reduce_add_sync(0xffffffffu, n);
  last = __reduce_max_sync(0xffffffffu, last);
  if (lane == 0) l.full[(size_t)bh * g.N + j] = last + 1 == n ? n : video_end - beg;
}

// Items of the dK/dV pass in the order of their list lengths, longest first, group by group (groups stay in order: the CTAs work on
// one group's tensors at a time, which L2 holds).  A KV block's list can be ten times the mean, and a launch that draws such
// items last ends with most SMs idle (720p, budget of 16..256 cubes, four heads a group: 0.7 ms for the mean item of a
// 6 ms launch).  Counting sort by one block per group; the order of equal lengths depends on the run, the results do not.
__device__ __forceinline__ void prep_order(const BwdPrepArgs& a, int bhk) {
  __shared__ int hist[1024], warp_sums[8], longest;
  const Geo& g = a.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto length = [&](int r) {
    int bh, j, k = 0;
    item_block(g, bhk * g.N + r, bh, j);
    for (int hh = 0; hh < g.rep; ++hh) {
      const int* c = a.lists.col_ptr + ((size_t)bhk * g.rep + hh) * (g.N + 1) + j;
      k += c[1] - c[0];
    }
    return k;
  };
  for (int b = tid; b < 1024; b += 256) hist[b] = 0;
  if (tid == 0) longest = 0;
  __syncthreads();
  int m = 0;
  for (int r = tid; r < g.N; r += 256) m = max(m, length(r));
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) atomicMax(&longest, m);
  __syncthreads();
  const int shift = max(0, 22 - __clz(longest));          // bins of 2^shift entries: longest >> shift < 1024
  for (int r = tid; r < g.N; r += 256) atomicAdd(&hist[1023 - (length(r) >> shift)], 1);
  __syncthreads();
  int mine[4], sum = 0;                                   // four bins a thread
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    mine[b] = hist[4 * tid + b];
    sum += mine[b];
  }
  int incl = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  int before = incl - sum;
  for (int w = 0; w < warp; ++w) before += warp_sums[w];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    hist[4 * tid + b] = before;
    before += mine[b];
  }
  __syncthreads();
  for (int r = tid; r < g.N; r += 256) a.lists.order[bhk * g.N + atomicAdd(&hist[1023 - (length(r) >> shift)], 1)] = bhk * g.N + r;
}

__global__ void __launch_bounds__(256) bwd_prep_kernel(const __grid_constant__ BwdPrepArgs a) {
  grid_enter();
  int block = blockIdx.x;
  if (block < a.exp_blocks) {
    if (form_ds_exp(a.scale, a.groups, a.per_group, block, a.exp_blocks)) atomicExch(a.cast.range_flag, 1);
  } else if ((block -= a.exp_blocks) < a.order_blocks) {
    prep_order(a, block);
  } else if ((block -= a.order_blocks) < a.pooled_blocks) {
    pooled_inputs(a.pooled, block, a.pooled_blocks);
  } else if ((block -= a.pooled_blocks) < a.list_blocks) {
    prep_lists(a, block);
  } else {
    const unsigned before = a.exp_blocks + a.order_blocks + a.pooled_blocks + a.list_blocks;
    cast_bf16_to_f16<false>(a.cast, block - a.list_blocks, gridDim.x - before);
  }
}

cudaError_t launch_bwd_prep(const Geo* fine, const bf16* q, void* q16, const bf16* k, void* k16, const DsScale& scale, int* range_flag,
                            const Geo* lists_geo, const PrepLists& lists, const PooledInputs* pooled, cudaStream_t st) {
  int sms = 0;
  cudaError_t e;
  if ((e = sm_count(&sms)) != cudaSuccess) return e;
  BwdPrepArgs a{};
  int copies = 0;
  if (fine != nullptr) {
    const size_t head = (size_t)fine->S * fine->D;
    a.cast = cast_job(q, q16, (size_t)fine->batch * fine->Hq * head, k, k16, (size_t)fine->batch * fine->Hkv * head, nullptr, 8, range_flag);
    a.scale = scale;
    a.groups = fine->batch * fine->Hkv;
    a.per_group = fine->rep * fine->N;
    a.exp_blocks = a.groups < sms ? a.groups : sms;
    copies = sms * kCastBlocksPerSm;
  }
  if (lists_geo != nullptr) {
    a.g = *lists_geo;
    a.lists = lists;
    a.lists_per_head = (a.g.N + 7) / 8;
    a.list_blocks = a.lists_per_head * a.g.batch * a.g.Hq;
    a.order_blocks = lists.order != nullptr ? a.g.batch * a.g.Hkv : 0;
  }
  if (pooled != nullptr) {
    a.pooled = *pooled;
    a.pooled_blocks = (int)pooled_inputs_blocks(a.pooled, sms);
  }
  return launch_kernel(bwd_prep_kernel, a.exp_blocks + a.order_blocks + a.pooled_blocks + a.list_blocks + copies, 256, 0, st, a);
}

}  // namespace vsa2
