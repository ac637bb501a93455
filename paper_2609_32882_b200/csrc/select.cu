// TopK selection on the router block scores and construction of the block map
// (paper Eq. 8-9: the N*K largest of the flattened N*N scores; Sec. 2.1 for the per-row form).
// Scores are non-negative floats, so their bit patterns order like unsigned integers: the
// K-th largest value is found by a most-significant-digit radix select, ties at the threshold
// go to the lower flat index, and rows/columns are emitted in ascending order (deterministic,
// integer work only).
#include "common.cuh"

#include <cooperative_groups.h>

namespace vsa2 {

constexpr int kHistBins = 2048;
// digit positions of the three per-sequence passes: bits [31:21], [20:10], [9:0]
__device__ __forceinline__ int seq_shift(int pass) { return pass == 0 ? 21 : (pass == 1 ? 10 : 0); }
__device__ __forceinline__ unsigned seq_mask(int pass) { return pass == 2 ? 0x3FFu : 0x7FFu; }

// state[bh*8 + ..]: 0 prefix bits, 1 prefix mask, 2 remaining k, 3 tau bits, 4 eq_take
__global__ void sel_init_kernel(unsigned* state, unsigned* hist, int BH, unsigned keep, const int* redo) {
  grid_enter();
  if (redo != nullptr && *redo == 0) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < BH * 3 * kHistBins) hist[i] = 0u;
  if (i < BH) {
    state[i * 8 + 0] = 0u;
    state[i * 8 + 1] = 0u;
    state[i * 8 + 2] = keep;
    state[i * 8 + 3] = 0u;
    state[i * 8 + 4] = 0u;
  }
}

__global__ void __launch_bounds__(256) sel_hist_kernel(const float* pr, long long n_elems,
                                                       const unsigned* state, unsigned* hist, int pass,
                                                       const int* redo) {
  grid_enter();
  __shared__ unsigned sh[kHistBins];
  if (redo != nullptr && *redo == 0) return;
  const int bh = blockIdx.y;
  for (int i = threadIdx.x; i < kHistBins; i += blockDim.x) sh[i] = 0u;
  __syncthreads();
  const unsigned prefix = state[bh * 8 + 0], pmask = state[bh * 8 + 1];
  const int shift = seq_shift(pass);
  const unsigned dmask = seq_mask(pass);
  const unsigned* src = reinterpret_cast<const unsigned*>(pr) + (size_t)bh * n_elems;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x, nthr = (long long)gridDim.x * blockDim.x;
  long long done = 0;
  if ((n_elems & 3) == 0) {
    // 16-byte loads, two in flight per thread (the passes after the first count almost nothing: they are pure streaming reads)
    const uint4* src4 = reinterpret_cast<const uint4*>(src);
    const long long n4 = n_elems >> 2;
    for (long long i = tid; i < n4; i += 2 * nthr) {
      const uint4 a = src4[i];
      const bool two = i + nthr < n4;
      const uint4 b = two ? src4[i + nthr] : make_uint4(0, 0, 0, 0);
      const unsigned va[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if ((e < 4 || two) && (va[e] & pmask) == prefix) atomicAdd(&sh[(va[e] >> shift) & dmask], 1u);
    }
    done = n_elems;
  }
  for (long long i = done + tid; i < n_elems; i += nthr) {
    unsigned v = src[i];
    if ((v & pmask) == prefix) atomicAdd(&sh[(v >> shift) & dmask], 1u);
  }
  __syncthreads();
  unsigned* dst = hist + ((size_t)bh * 3 + pass) * kHistBins;
  for (int i = threadIdx.x; i < kHistBins; i += blockDim.x)
    if (sh[i]) atomicAdd(&dst[i], sh[i]);
}

// One warp per (batch, head): finds the digit whose bin holds the `remaining`-th largest entry.  Lane l owns the bins
// [l * nb/32, (l+1) * nb/32); a suffix sum over the lanes locates the lane, a short serial walk the bin.
__global__ void __launch_bounds__(32) sel_pick_kernel(unsigned* state, const unsigned* hist, int pass, const int* redo) {
  grid_enter();
  if (redo != nullptr && *redo == 0) return;
  const int bh = blockIdx.x, lane = threadIdx.x;
  const unsigned* hsrc = hist + ((size_t)bh * 3 + pass) * kHistBins;
  const unsigned remaining0 = state[bh * 8 + 2];
  const int nb = (int)seq_mask(pass) + 1, per = nb / 32;
  unsigned mine = 0u;
  for (int d = lane * per; d < (lane + 1) * per; ++d) mine += hsrc[d];
  // above = entries in the bins of all higher lanes
  unsigned incl = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned up = __shfl_down_sync(0xffffffffu, incl, o);
    if (lane + o < 32) incl += up;
  }
  const unsigned above = incl - mine;
  // the threshold bin lies in the highest lane whose suffix count reaches `remaining0`
  const bool here = above < remaining0 && incl >= remaining0;
  const unsigned vote = __ballot_sync(0xffffffffu, here);
  if (vote == 0u) {                    // fewer entries than requested (cannot happen for keep <= N*N): keep everything
    if (lane == 0) {
      const int shift = seq_shift(pass);
      state[bh * 8 + 1] |= seq_mask(pass) << shift;
      state[bh * 8 + 2] = remaining0 - incl;      // lane 0's inclusive suffix = all entries
      if (pass == 2) { state[bh * 8 + 3] = state[bh * 8 + 0]; state[bh * 8 + 4] = state[bh * 8 + 2]; }
    }
    return;
  }
  if (lane == 31 - __clz(vote)) {
    unsigned remaining = remaining0 - above;
    int bin = lane * per;
    for (int d = (lane + 1) * per - 1; d >= lane * per; --d) {
      const unsigned c = hsrc[d];
      if (c >= remaining) { bin = d; break; }
      remaining -= c;
    }
    const int shift = seq_shift(pass);
    const unsigned prefix = state[bh * 8 + 0] | ((unsigned)bin << shift);
    state[bh * 8 + 0] = prefix;
    state[bh * 8 + 1] |= seq_mask(pass) << shift;
    state[bh * 8 + 2] = remaining;
    if (pass == 2) {
      state[bh * 8 + 3] = prefix;      // tau: the smallest kept value
      state[bh * 8 + 4] = remaining;   // how many entries equal to tau are kept
    }
  }
}

// ---- scores of the one-pass router -----------------------------------------------------------------------------------------
// A one-pass score x stands for a two-pass score within a factor 1 +- e.  With t the K-th largest x, entries above t (1 + 2e) are
// among the K largest two-pass scores and entries below t (1 - 2e) are not, so only those between -- the band -- need their
// two-pass scores, and only where the band holds more entries than are still wanted.
// e: of a term that counts in a score of at least kBandLeast = 2^-52, either form rounds an exponent below 128 once (half an ulp,
// 2^-18); the one-pass form also rounds the growth of the row's maximum, at most 48 (2^-19), while its reference against the
// denominator keeps what rounding takes from it (router_tc.cu).  (2 2^-18 + 2^-19) ln 2 = 6.6e-6, with five approximations of
// ex2 (2^-22 each) and at most 40 additions of 2^-24 on either side 1.26e-5.  A query cube's other rows, and other heads of a group, may
// have lost terms of 2^-78 (router_tc.cu): 2^-74 of a sum over 16 heads, 2^-22 of kBandLeast.  Together less than 1.4e-5.  kBandUlps = 512 units of the last place of t
// are at least 3.05e-5 of t, more than 2e.
// Below kBandLeast the bound does not hold (a thread's sums may be lost altogether), so entries may lie anywhere: a head or row with
// such a threshold goes back to the two-pass form whatever its band holds, unless everything is kept.  About one entry in 10^5 lies in a
// band.
constexpr unsigned kBandUlps = 512, kBandLeast = 0x25800000u, kBandMost = 0x7f000000u;
__device__ __forceinline__ unsigned band_lo(unsigned tau) { return tau > kBandUlps ? tau - kBandUlps : 0u; }
__device__ __forceinline__ unsigned band_hi(unsigned tau) { return tau < 0xffffffffu - kBandUlps ? tau + kBandUlps : 0xffffffffu; }
__device__ __forceinline__ bool band_usable(unsigned tau) { return tau >= kBandLeast && tau <= kBandMost; }
constexpr int kBandHead = 2048;      // entries of a head's band that sel_settle_kernel ranks
__device__ __forceinline__ void settle_list(const Settle& se, int row, int column) {
  if (*reinterpret_cast<volatile int*>(se.redo) != 0) return;      // (a million ties would wait for one counter: the list is full, or not used)
  const int at = atomicAdd(se.count, 1);
  if (at < se.cap) se.pairs[at] = make_int2(row, column);
  else atomicExch(se.redo, 1);
}

// The same for the lanes of a warp with `in`, with one addition to the counter (one a pair: where every key is equal, 480p, 12 heads, a route
// call of 741 us instead of 602, of which the two forms of the router are 400; per query, where few rows list anything, it costs
// 5 us of 273).
__device__ __forceinline__ void settle_list_warp(const Settle& se, bool in, int row, int column) {
  const unsigned votes = __ballot_sync(0xffffffffu, in);
  if (votes == 0u) return;
  const int lane = threadIdx.x & 31;
  int first = -1;
  if (lane == 0 && *reinterpret_cast<volatile int*>(se.redo) == 0) {
    first = atomicAdd(se.count, __popc(votes));
    if (first + __popc(votes) > se.cap) atomicExch(se.redo, 1);
  }
  first = __shfl_sync(0xffffffffu, first, 0);
  const int at = first + __popc(votes & ((1u << lane) - 1u));
  if (in && first >= 0 && at < se.cap) se.pairs[at] = make_int2(row, column);
}

// per-sequence, one read of P_r for both the counts and the emission: one warp per row writes the row's bitmap words of the
// entries above tau (`bits_gt`) and equal to tau (`bits_eq`) and the two counts.  grid (ceil(N/8), BH), 256 threads
// BAND: entries above and in the band instead, the latter also listed for router_exact_kernel.
template <bool BAND>
__global__ void __launch_bounds__(256) sel_row_bits_kernel(const float* pr, int N, int words,
                                                           const unsigned* state, unsigned* bits_gt,
                                                           unsigned* bits_eq, int* row_gt, int* row_eq, Settle se) {
  grid_enter();
  if (!BAND && se.redo != nullptr && *se.redo == 0) return;
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int bh = blockIdx.y;
  if (i >= N) return;
  const unsigned tau = state[bh * 8 + 3];
  const unsigned hi = BAND ? band_hi(tau) : tau, lo = BAND ? band_lo(tau) : tau;
  const unsigned* src = reinterpret_cast<const unsigned*>(pr) + ((size_t)bh * N + i) * N;
  int gt = 0, eq = 0;
  constexpr int U = 8;                 // words in flight per warp (the kernel is a pure streaming read)
  for (int w0 = 0; w0 < words; w0 += U) {
    unsigned v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = (w0 + u) * 32 + lane;
      v[u] = j < N ? src[j] : 0u;      // (scores are non-negative: 0 is never above tau, and equal only if tau = 0
    }                                          //  -- excluded by the j < N test below)
    unsigned mine_g = 0u, mine_e = 0u;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = (w0 + u) * 32 + lane;
      const bool in = j < N && v[u] >= lo && v[u] <= hi;
      const unsigned gb = __ballot_sync(0xffffffffu, j < N && v[u] > hi);
      const unsigned eb = __ballot_sync(0xffffffffu, in);
      if (lane == u) { mine_g = gb; mine_e = eb; }
      gt += __popc(gb);
      eq += __popc(eb);
      if constexpr (BAND) settle_list_warp(se, in, bh * N + i, j);
    }
    if (lane < U && w0 + lane < words) {       // lanes 0..U-1 write one word each: consecutive addresses
      bits_gt[((size_t)bh * N + i) * words + w0 + lane] = mine_g;
      bits_eq[((size_t)bh * N + i) * words + w0 + lane] = mine_e;
    }
  }
  if (lane == 0) {
    row_gt[(size_t)bh * N + i] = gt;
    row_eq[(size_t)bh * N + i] = eq;
  }
}

// inclusive prefix sum over the lanes of a warp
__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// per-sequence: ordered emission of the kept columns from the two bitmaps (`bitmap` holds the entries above tau on entry and
// the kept entries on return).  One warp per row, one LANE per bitmap word: the lanes count their bits, a warp scan gives every
// word its position in the row's list, and each lane writes its own few entries (a warp per word spent 30 instructions on
// every word, 45 words a row).  Ties at tau go to the lower column: a lane keeps the equal entries whose rank in the row is
// below the row's quota.  grid (ceil(N/8), BH), 256 threads
__global__ void __launch_bounds__(256) sel_emit_rows_bits_kernel(int N, int words, const unsigned* bits_eq,
                                                                 const int* row_eq_take,
                                                                 const int* row_ptr, int* col_idx,
                                                                 unsigned* bitmap, long long nnz_cap) {
  grid_enter();
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int bh = blockIdx.y;
  if (i >= N) return;
  const int take = row_eq_take[(size_t)bh * N + i];
  int pos = row_ptr[(size_t)bh * (N + 1) + i];
  int eq_seen = 0;
  int* out = col_idx + (size_t)bh * nnz_cap;
  const size_t base = ((size_t)bh * N + i) * words;
  for (int w0 = 0; w0 < words; w0 += 32) {
    const int w = w0 + lane;
    const unsigned gb = w < words ? bitmap[base + w] : 0u;
    unsigned eb = w < words ? bits_eq[base + w] : 0u;
    const int ce = __popc(eb);
    const int ce_incl = warp_incl_scan(ce, lane);
    int rank = eq_seen + ce_incl - ce;             // equal entries of the row before this word
    unsigned keep = 0u;
    while (eb != 0u && rank < take) {
      keep |= eb & (0u - eb);
      eb &= eb - 1u;
      ++rank;
    }
    unsigned sel = gb | keep;
    const int c = __popc(sel);
    const int c_incl = warp_incl_scan(c, lane);
    int p = pos + c_incl - c;
    unsigned kept = 0u;                              // (entries past the capacity of the map are dropped from the bitmap too,
    while (sel != 0u) {                              //  so that the transposed map lists exactly the pairs emitted here)
      if (p < nnz_cap) {
        out[p] = w * 32 + (__ffs(sel) - 1);
        kept |= sel & (0u - sel);
      }
      sel &= sel - 1u;
      ++p;
    }
    if (w < words && kept != gb) bitmap[base + w] = kept;
    pos += __shfl_sync(0xffffffffu, c_incl, 31);
    eq_seen += __shfl_sync(0xffffffffu, ce_incl, 31);
  }
}

// Threshold of a row that keeps nothing: above every score as a bit pattern, also one that is not a number.  (Infinity is not: a row of NaNs that
// keeps nothing then wrote its columns over the lists of the rows behind it.)
constexpr unsigned kNoEntry = 0xffffffffu;
// The k-th largest (1 <= k <= entries) of a row that a warp holds in registers, U a lane (0 where there is none), by bisection over the bits
template <int U>
__device__ __forceinline__ unsigned row_threshold(const unsigned (&v)[U], int k) {
  unsigned tau = 0u;            // the largest value with at least k entries >= it
  for (int bit = 31; bit >= 0; --bit) {
    const unsigned cand = tau | (1u << bit);
    int c = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) c += v[u] >= cand;
    c = __reduce_add_sync(0xffffffffu, c);
    if (c >= k) tau = cand;
    if (c == k) {               // exactly the kept entries: the threshold is the smallest of them
      unsigned m = 0xffffffffu;
#pragma unroll
      for (int u = 0; u < U; ++u) m = v[u] >= cand ? min(m, v[u]) : m;
      tau = __reduce_min_sync(0xffffffffu, m);
      break;
    }
  }
  return tau;
}

// per-row modes: the k_i-th largest of row i by bisection over the bits of the threshold, a warp per row with the row in registers
// (U a lane): rounds of U compares and a warp sum until the kept entries are apart from the others (about 20; 32 with ties), no
// shared memory, no atomics, no block barrier.  grid (ceil(N / 8), BH)
// (a block per row with 8-bit histograms: 104 us for 7,488 rows of 624, most of it one thread walking the bins)
// U is the smallest of 8, 20, 32, 48, 64 that holds the row: a round costs U compares whatever the row's length, so the forms are
// close enough together (1.3 - 1.6 times, below 640 entries 2.5) for the padding not to outweigh the launch.
// MODE kBand: a row whose band holds more entries than it still wants is listed (se.rows), and its band's entries (se.pairs).
// MODE kListed: the listed rows alone, now with their two-pass scores (any grid).
constexpr int kAllRows = 0, kBand = 1, kListed = 2;
template <int U, int MODE>
__global__ void __launch_bounds__(256) sel_row_topk_warp_kernel(const float* pr, int N, int K,
                                                                const int* budgets, float* row_tau,
                                                                int* row_eq_take, int* row_cnt, Settle se) {
  grid_enter();
  if (MODE == kAllRows && se.redo != nullptr && *se.redo == 0) return;
  const int lane = threadIdx.x & 31, i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= (MODE == kListed ? *se.row_count : N)) return;
  const size_t o = MODE == kListed ? (size_t)se.rows[i] : (size_t)blockIdx.y * N + i;
  const unsigned* src = reinterpret_cast<const unsigned*>(pr) + o * N;
  unsigned v[U];
#pragma unroll
  for (int u = 0; u < U; ++u) v[u] = u * 32 + lane < N ? src[u * 32 + lane] : 0u;      // (0 is never above a candidate)
  const int asked = budgets ? budgets[o] : K, k = max(0, min(asked, N));
  if (k == 0) {
    if (lane == 0) { row_tau[o] = __uint_as_float(kNoEntry); row_eq_take[o] = 0; row_cnt[o] = 0; }
    return;
  }
  const unsigned tau = row_threshold<U>(v, k);
  int gt = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) gt += v[u] > tau;
  gt = __reduce_add_sync(0xffffffffu, gt);
  if (lane == 0) {
    row_tau[o] = __uint_as_float(tau);
    row_eq_take[o] = k - gt;
    row_cnt[o] = k;
  }
  if constexpr (MODE == kBand) {
    const unsigned lo = band_lo(tau), hi = band_hi(tau);
    int from = 0;                     // entries above the lower end of the band: more than k, and the band matters
#pragma unroll
    for (int u = 0; u < U; ++u) from += u * 32 + lane < N && v[u] >= lo;
    from = __reduce_add_sync(0xffffffffu, from);
    if (!band_usable(tau)) {
      // (not `k < N` or `k == N`: nvcc 12.9.86 compiles the latter to true here, whatever the clamped k is)
      if (lane == 0 && asked < N) atomicExch(se.redo, 1);
    } else if (from > k) {
      if (lane == 0) se.rows[atomicAdd(se.row_count, 1)] = (int)o;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (u * 32 + lane < N && v[u] >= lo && v[u] <= hi) settle_list(se, (int)o, u * 32 + lane);
    }
  }
}

// per-row modes, rows of more than 2048 entries: radix select of the k_i-th largest of row i.  grid (N, BH), 256 threads
// MODE as above
template <int MODE>
__global__ void __launch_bounds__(256) sel_row_topk_kernel(const float* pr, int N, int K,
                                                           const int* budgets, float* row_tau,
                                                           int* row_eq_take, int* row_cnt, Settle se) {
  grid_enter();
  __shared__ unsigned sh[256];
  __shared__ unsigned s_prefix, s_mask, s_remaining;
  if (MODE == kAllRows && se.redo != nullptr && *se.redo == 0) return;
  const size_t listed = MODE == kListed ? (size_t)*se.row_count : 1;
  for (size_t n = MODE == kListed ? blockIdx.x : 0; n < listed; n += gridDim.x) {
  const size_t o = MODE == kListed ? (size_t)se.rows[n] : (size_t)blockIdx.y * N + blockIdx.x;
  const unsigned* src = reinterpret_cast<const unsigned*>(pr) + o * N;
  const int asked = budgets ? budgets[o] : K, k = max(0, min(asked, N));
  if (k == 0) {
    if (threadIdx.x == 0) { row_tau[o] = __uint_as_float(kNoEntry); row_eq_take[o] = 0; row_cnt[o] = 0; }
    continue;
  }
  if (threadIdx.x == 0) { s_prefix = 0u; s_mask = 0u; s_remaining = (unsigned)k; }
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    sh[threadIdx.x] = 0u;
    __syncthreads();
    const unsigned prefix = s_prefix, pmask = s_mask;
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
      unsigned v = src[j];
      if ((v & pmask) == prefix) atomicAdd(&sh[(v >> shift) & 0xFFu], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned remaining = s_remaining;
      int bin = 0;
      for (int d = 255; d >= 0; --d) {
        unsigned c = sh[d];
        if (c >= remaining) { bin = d; break; }
        remaining -= c;
      }
      s_prefix = prefix | ((unsigned)bin << shift);
      s_mask = pmask | (0xFFu << shift);
      s_remaining = remaining;
    }
    __syncthreads();
  }
  const unsigned tau = s_prefix;
  if (threadIdx.x == 0) {
    row_tau[o] = __uint_as_float(tau);
    row_eq_take[o] = (int)s_remaining;
    row_cnt[o] = k;
  }
  if constexpr (MODE == kBand) {
    const unsigned lo = band_lo(tau), hi = band_hi(tau);
    int from = 0;
    for (int j = threadIdx.x; j < N; j += blockDim.x) from += src[j] >= lo;
    if (threadIdx.x == 0) sh[0] = 0u;
    __syncthreads();
    if (from > 0) atomicAdd(&sh[0], (unsigned)from);
    __syncthreads();
    if (!band_usable(tau)) {
      if (threadIdx.x == 0 && asked < N) atomicExch(se.redo, 1);
    } else if (sh[0] > (unsigned)k) {
      if (threadIdx.x == 0) se.rows[atomicAdd(se.row_count, 1)] = (int)o;
      for (int j = threadIdx.x; j < N; j += blockDim.x) {
        const unsigned v = src[j];
        if (v >= lo && v <= hi) settle_list(se, (int)o, j);
      }
    }
  }
  __syncthreads();
  }
}

// exclusive scan of v over the block (up to 1024 threads, whole warps); returns the prefix, total in `total`
template <int THREADS = 1024>
__device__ __forceinline__ int block_excl_scan(int v, int* warp_sums, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int w = lane < THREADS / 32 ? warp_sums[lane] : 0;
    int wi = w;
    for (int o = 1; o < 32; o <<= 1) {
      int t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    warp_sums[lane] = wi - w;        // exclusive prefix of the warp sums
    if (lane == 31) warp_sums[32] = wi;
  }
  __syncthreads();
  int res = warp_sums[warp] + incl - v;
  total = warp_sums[32];
  __syncthreads();
  return res;
}

// one block per (batch, head): per-sequence tie quota per row, then row_ptr = exclusive scan of counts
__global__ void __launch_bounds__(1024) sel_scan_rows_kernel(int N, int per_sequence, const unsigned* state,
                                                             const int* row_gt, const int* row_eq,
                                                             float* row_tau, int* row_eq_take, int* row_cnt, int* row_ptr,
                                                             long long nnz_cap, StatusBlock* status) {
  grid_enter();
  __shared__ int ws[33];
  const int bh = blockIdx.x;
  const size_t base = (size_t)bh * N;
  if (per_sequence) {
    const unsigned tau = state[bh * 8 + 3];
    const int quota = (int)state[bh * 8 + 4];
    int carry = 0;
    for (int i0 = 0; i0 < N; i0 += blockDim.x) {
      int i = i0 + threadIdx.x;
      int eq = i < N ? row_eq[base + i] : 0;
      int tot;
      int before = carry + block_excl_scan(eq, ws, tot);
      if (i < N) {
        int take = max(0, min(eq, quota - before));
        row_eq_take[base + i] = take;
        row_cnt[base + i] = row_gt[base + i] + take;
        row_tau[base + i] = __uint_as_float(tau);
      }
      carry += tot;
    }
    __syncthreads();
  }
  int carry = 0;
  for (int i0 = 0; i0 < N; i0 += blockDim.x) {
    int i = i0 + threadIdx.x;
    int c = i < N ? row_cnt[base + i] : 0;
    int tot;
    int pre = carry + block_excl_scan(c, ws, tot);
    // (an overflowing selection is reported below; its row pointers stop at the capacity, so that every later reader of
    // the map stays inside col_idx: rows past the capacity are empty, the row that crosses it is cut)
    if (i < N) row_ptr[(size_t)bh * (N + 1) + i] = (int)min((long long)pre, nnz_cap);
    carry += tot;
  }
  if (threadIdx.x == 0) {
    row_ptr[(size_t)bh * (N + 1) + N] = (int)min((long long)carry, nnz_cap);
    if ((long long)carry > nnz_cap) atomicExch(&status->status, VSA2_ERR_MAP_OVERFLOW);
  }
}

// one warp per row: ordered emission of the kept columns and of the row's bitmap words
__global__ void __launch_bounds__(256) sel_emit_rows_kernel(const float* pr, int N, int words,
                                                            const float* row_tau,
                                                            const int* row_eq_take,
                                                            const int* row_ptr, int* col_idx,
                                                            unsigned* bitmap, long long nnz_cap) {
  grid_enter();
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int bh = blockIdx.y;
  if (i >= N) return;
  const unsigned* src = reinterpret_cast<const unsigned*>(pr) + ((size_t)bh * N + i) * N;
  const unsigned tau = __float_as_uint(row_tau[(size_t)bh * N + i]);
  const int take = row_eq_take[(size_t)bh * N + i];
  int pos = row_ptr[(size_t)bh * (N + 1) + i];
  int eq_seen = 0;
  int* out = col_idx + (size_t)bh * nnz_cap;
  const unsigned lt = (1u << lane) - 1u;
  for (int w = 0; w < words; ++w) {
    int j = w * 32 + lane;
    unsigned v = j < N ? src[j] : 0u;
    bool gt = j < N && v > tau;
    bool eq = j < N && v == tau;
    unsigned eqb = __ballot_sync(0xffffffffu, eq);
    bool sel = gt || (eq && (eq_seen + __popc(eqb & lt)) < take);
    unsigned selb = __ballot_sync(0xffffffffu, sel);
    const int p = pos + __popc(selb & lt);
    const bool emit = sel && p < nnz_cap;            // (entries past the capacity of the map are dropped from the bitmap too,
    if (emit) out[p] = j;                            //  so that the transposed map lists exactly the pairs emitted here)
    const unsigned keptb = __ballot_sync(0xffffffffu, emit);
    pos += __popc(selb);
    eq_seen += __popc(eqb);
    if (lane == 0) bitmap[((size_t)bh * N + i) * words + w] = keptb;
  }
}

// bitmap [BH][N rows][words] -> bitmap_t [BH][N columns][words] (bit i of row-word set <-> bit of column-word set):
// one warp per 32 x 32 bit tile, transposed with 32 ballots.  grid (words, ceil(words/8), BH), 256 threads
__global__ void __launch_bounds__(256) sel_transpose_bitmap_kernel(const unsigned* bitmap, int N, int words,
                                                                   unsigned* __restrict__ bitmap_t) {
  grid_enter();
  const int lane = threadIdx.x & 31;
  const int wj = blockIdx.x;                                   // word column of the source: columns 32 wj .. 32 wj + 31
  const int wi = blockIdx.y * 8 + (threadIdx.x >> 5);          // word row of the source: rows 32 wi .. 32 wi + 31
  const int bh = blockIdx.z;
  if (wi >= words) return;
  const int i = wi * 32 + lane;
  const unsigned v = i < N ? bitmap[((size_t)bh * N + i) * words + wj] : 0u;
  unsigned mine = 0u;
#pragma unroll
  for (int bit = 0; bit < 32; ++bit) {
    const unsigned col_word = __ballot_sync(0xffffffffu, (v >> bit) & 1u);   // rows 32 wi .. of column 32 wj + bit
    if (lane == bit) mine = col_word;
  }
  const int j = wj * 32 + lane;
  if (j < N) bitmap_t[((size_t)bh * N + j) * words + wi] = mine;
}

// one warp per column: number of kept rows.  grid (ceil(N/8), BH), 256 threads
__global__ void __launch_bounds__(256) sel_col_count_kernel(const unsigned* bitmap_t, int N, int words,
                                                            int* col_cnt) {
  grid_enter();
  const int lane = threadIdx.x & 31;
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5), bh = blockIdx.y;
  if (j >= N) return;
  const unsigned* bm = bitmap_t + ((size_t)bh * N + j) * words;
  int c = 0;
  for (int w = lane; w < words; w += 32) c += __popc(bm[w]);
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) col_cnt[(size_t)bh * N + j] = c;
}

__global__ void __launch_bounds__(1024) sel_scan_cols_kernel(int N, const int* col_cnt, int* col_ptr,
                                                             long long nnz_cap) {
  grid_enter();
  __shared__ int ws[33];
  const int bh = blockIdx.x;
  int carry = 0;
  for (int j0 = 0; j0 < N; j0 += blockDim.x) {
    int j = j0 + threadIdx.x;
    int c = j < N ? col_cnt[(size_t)bh * N + j] : 0;
    int tot;
    int pre = carry + block_excl_scan(c, ws, tot);
    if (j < N) col_ptr[(size_t)bh * (N + 1) + j] = (int)min((long long)pre, nnz_cap);      // (as for the rows)
    carry += tot;
  }
  if (threadIdx.x == 0) col_ptr[(size_t)bh * (N + 1) + N] = (int)min((long long)carry, nnz_cap);
}

// one warp per column, one lane per bitmap word: ordered emission of the rows that keep it.  grid (ceil(N/8), BH), 256 threads
__global__ void __launch_bounds__(256) sel_emit_cols_kernel(const unsigned* bitmap_t, int N, int words,
                                                            const int* col_ptr, int* row_idx,
                                                            long long nnz_cap) {
  grid_enter();
  const int lane = threadIdx.x & 31;
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5), bh = blockIdx.y;
  if (j >= N) return;
  const unsigned* bm = bitmap_t + ((size_t)bh * N + j) * words;
  int pos = col_ptr[(size_t)bh * (N + 1) + j];
  int* out = row_idx + (size_t)bh * nnz_cap;
  for (int w0 = 0; w0 < words; w0 += 32) {
    // one lane per word, as in sel_emit_rows_bits_kernel
    unsigned word = w0 + lane < words ? bm[w0 + lane] : 0u;
    const int c = __popc(word);
    const int c_incl = warp_incl_scan(c, lane);
    int p = pos + c_incl - c;
    while (word != 0u) {
      if (p < nnz_cap) out[p] = (w0 + lane) * 32 + (__ffs(word) - 1);
      word &= word - 1u;
      ++p;
    }
    pos += __shfl_sync(0xffffffffu, c_incl, 31);
  }
}

// per-sequence, one-pass scores: of every head whose band holds more entries than are still wanted, ranks the band by its two-pass
// scores (ties to the lower index) and takes what is not kept out of the bitmap and the counts.  One block per head.
__global__ void __launch_bounds__(1024) sel_settle_kernel(const float* pr, int N, int words, unsigned keep, unsigned* state,
                                                          const int* row_gt, int* row_eq, unsigned* bits_eq, Settle se) {
  grid_enter();
  __shared__ int ws[33];
  __shared__ int n_rows;
  __shared__ int2 at[kBandHead];            // {row, column}: their flat index need not fit an int (46,341 cubes and more)
  __shared__ unsigned val[kBandHead];
  __shared__ int2 rows[kBandHead];          // (no more than entries)
  const int bh = blockIdx.x, tid = threadIdx.x;
  const size_t base = (size_t)bh * N;
  int above = 0, band = 0, tot;
  for (int i = tid; i < N; i += blockDim.x) {
    above += row_gt[base + i];
    band += row_eq[base + i];
  }
  block_excl_scan(above, ws, tot);
  const int need = (int)keep - tot;
  block_excl_scan(band, ws, band);
  if (tid == 0) state[bh * 8 + 4] = (unsigned)need;
  const bool usable = band_usable(state[bh * 8 + 3]);
  if (band == need && (usable || keep == (unsigned)((size_t)N * N))) return;
  if (band > kBandHead || !usable) {
    if (tid == 0) atomicExch(se.redo, 1);
    return;
  }
  // the rows that have such entries and the place of their first; then a warp per row, a lane per word of its bitmap
  if (tid == 0) n_rows = 0;
  int carry = 0;
  for (int i0 = 0; i0 < N; i0 += blockDim.x) {
    const int i = i0 + tid, eq = i < N ? row_eq[base + i] : 0;
    const int pos = carry + block_excl_scan(eq, ws, tot);
    carry += tot;
    if (eq > 0) rows[atomicAdd(&n_rows, 1)] = make_int2(i, pos);
  }
  __syncthreads();
  const int lane = tid & 31;
  for (int r = tid >> 5; r < n_rows; r += blockDim.x >> 5) {
    const int i = rows[r].x;
    int pos = rows[r].y;
    for (int w0 = 0; w0 < words; w0 += 32) {
      const unsigned bits = w0 + lane < words ? bits_eq[(base + i) * words + w0 + lane] : 0u;
      const int c = __popc(bits), incl = warp_incl_scan(c, lane);
      int p = pos + incl - c;
      for (unsigned b = bits; b != 0u; b &= b - 1u, ++p) {
        const int j = (w0 + lane) * 32 + (__ffs(b) - 1);
        at[p] = make_int2(i, j);
        val[p] = __float_as_uint(pr[(base + i) * N + j]);
      }
      pos += __shfl_sync(0xffffffffu, incl, 31);
    }
  }
  __syncthreads();
  for (int e = tid; e < band; e += blockDim.x) {
    const unsigned v = val[e];
    int rank = 0;
    for (int f = 0; f < band; ++f) rank += val[f] > v || (val[f] == v && f < e);
    if (rank >= need) {
      const int i = at[e].x, j = at[e].y;
      atomicAnd(&bits_eq[(base + i) * words + (j >> 5)], ~(1u << (j & 31)));
      atomicSub(&row_eq[base + i], 1);
    }
  }
}

// Up to kSelOneBlockN cubes, per-row modes: the selection in one launch (row_tau: null, or the thresholds are there), or everything behind the counts of the kept entries, a block per head with both bitmaps in
// shared memory (the six launches below take 2 us and a gap each and keep a few SMs busy).  Same rules: rows in order, ties at the
// threshold to the lower column, both maps cut at the capacity.
__global__ void __launch_bounds__(1024) sel_maps_kernel(const float* pr, int N, int words, int per_sequence,
                                                        const unsigned* state, const int* row_gt,
                                                        const int* row_eq, const float* row_tau,
                                                        const int* row_eq_take, const int* row_cnt,
                                                        const unsigned* bits_gt, const unsigned* bits_eq, int K, const int* budgets,
                                                        int* row_ptr, int* col_idx, int* col_ptr, int* row_idx, long long nnz_cap,
                                                        StatusBlock* status) {
  grid_enter();
  constexpr int W = kSelOneBlockN / 32;
  __shared__ unsigned tau_s[kSelOneBlockN];
  __shared__ unsigned bm[kSelOneBlockN * W], bt[kSelOneBlockN * W];
  __shared__ int take_s[kSelOneBlockN], ptr_s[kSelOneBlockN], ws[33];
  const int bh = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t base = (size_t)bh * N;
  int cnt = 0, take = 0, tot;
  if (per_sequence) {
    const int eq = tid < N ? row_eq[base + tid] : 0;
    const int before = block_excl_scan(eq, ws, tot);
    if (tid < N) {
      take = max(0, min(eq, (int)state[bh * 8 + 4] - before));
      cnt = row_gt[base + tid] + take;
    }
  } else if (row_tau != nullptr) {
    if (tid < N) {
      take = row_eq_take[base + tid];
      cnt = row_cnt[base + tid];
      tau_s[tid] = __float_as_uint(row_tau[base + tid]);
    }
  } else {
    // the thresholds as well (as sel_row_topk_warp_kernel): a launch less, and its wait
    for (int i = warp; i < N; i += 32) {
      const unsigned* src = reinterpret_cast<const unsigned*>(pr) + (base + i) * N;
      unsigned v[W];
#pragma unroll
      for (int w = 0; w < W; ++w) v[w] = w * 32 + lane < N ? src[w * 32 + lane] : 0u;
      const int k = max(0, min(budgets ? budgets[base + i] : K, N));
      const unsigned tau = k > 0 ? row_threshold<W>(v, k) : kNoEntry;
      int gt = 0;
#pragma unroll
      for (int w = 0; w < W; ++w) gt += v[w] > tau;
      gt = __reduce_add_sync(0xffffffffu, gt);
      if (lane == 0) {
        tau_s[i] = tau;
        take_s[i] = k > 0 ? k - gt : 0;
        ptr_s[i] = k;
      }
    }
    __syncthreads();
    if (tid < N) {
      take = take_s[tid];
      cnt = ptr_s[tid];
    }
  }
  int pre = block_excl_scan(cnt, ws, tot);
  if (tid < N) {
    take_s[tid] = take;
    ptr_s[tid] = pre;
    row_ptr[(size_t)bh * (N + 1) + tid] = (int)min((long long)pre, nnz_cap);
  }
  if (tid == 0) {
    row_ptr[(size_t)bh * (N + 1) + N] = (int)min((long long)tot, nnz_cap);
    if ((long long)tot > nnz_cap) atomicExch(&status->status, VSA2_ERR_MAP_OVERFLOW);
  }
  __syncthreads();
  int* out = col_idx + (size_t)bh * nnz_cap;
  const unsigned lt = (1u << lane) - 1u;
  for (int i = warp; i < N; i += 32) {
    const unsigned* src = reinterpret_cast<const unsigned*>(pr) + (base + i) * N;
    const unsigned tau = per_sequence ? 0u : tau_s[i];
    int pos = (int)min((long long)ptr_s[i], nnz_cap), left = take_s[i];
    // (the whole row is read first: a row's words one after another waited for memory every time)
    unsigned v[W], gw = 0u, ew = 0u;
    if (per_sequence) {
      if (lane < words) {
        gw = bits_gt[(base + i) * words + lane];
        ew = bits_eq[(base + i) * words + lane];
      }
    } else {
#pragma unroll
      for (int w = 0; w < W; ++w) v[w] = w * 32 + lane < N ? src[w * 32 + lane] : 0u;
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
      if (w >= words) break;
      const int j = w * 32 + lane;
      bool gt, eq;
      if (per_sequence) {
        gt = (__shfl_sync(0xffffffffu, gw, w) >> lane) & 1u;
        eq = (__shfl_sync(0xffffffffu, ew, w) >> lane) & 1u;
      } else {
        gt = j < N && v[w] > tau;
        eq = j < N && v[w] == tau;
      }
      const unsigned eqb = __ballot_sync(0xffffffffu, eq);
      const bool sel = gt || (eq && __popc(eqb & lt) < left);
      const unsigned selb = __ballot_sync(0xffffffffu, sel);
      const int p = pos + __popc(selb & lt);
      const bool emit = sel && p < nnz_cap;
      if (emit) out[p] = j;
      const unsigned keptb = __ballot_sync(0xffffffffu, emit);
      pos += __popc(selb);
      left -= __popc(eqb);
      if (lane == 0) bm[i * W + w] = keptb;
    }
  }
  __syncthreads();
  for (int t = warp; t < words * words; t += 32) {
    const int wi = t / words, wj = t - wi * words;
    const unsigned v = wi * 32 + lane < N ? bm[(wi * 32 + lane) * W + wj] : 0u;
    unsigned mine = 0u;
#pragma unroll
    for (int bit = 0; bit < 32; ++bit) {
      const unsigned col_word = __ballot_sync(0xffffffffu, (v >> bit) & 1u);
      if (lane == bit) mine = col_word;
    }
    if (wj * 32 + lane < N) bt[(wj * 32 + lane) * W + wi] = mine;
  }
  __syncthreads();
  cnt = 0;
  if (tid < N)
    for (int w = 0; w < words; ++w) cnt += __popc(bt[tid * W + w]);
  pre = block_excl_scan(cnt, ws, tot);
  if (tid < N) {
    ptr_s[tid] = (int)min((long long)pre, nnz_cap);
    col_ptr[(size_t)bh * (N + 1) + tid] = ptr_s[tid];
  }
  if (tid == 0) col_ptr[(size_t)bh * (N + 1) + N] = (int)min((long long)tot, nnz_cap);
  __syncthreads();
  int* rows = row_idx + (size_t)bh * nnz_cap;
  for (int j = warp; j < N; j += 32) {
    int pos = ptr_s[j];
    for (int w = 0; w < words; ++w) {
      const unsigned word = bt[j * W + w];
      const int p = pos + __popc(word & lt);
      if (((word >> lane) & 1u) && p < nnz_cap) rows[p] = w * 32 + lane;
      pos += __popc(word);
    }
  }
}

// ---- a head in one launch ----------------------------------------------------------------------------------------------------
// Per sequence, mid sizes: a cluster of eight CTAs per head, each with an eighth of the rows.  Behind the router the steps above are 14
// launches of a few microseconds of work each, every one of them a wait for the one before, and the scores are read four times; here a
// head's scores are read once into the cluster's shared memory, the histograms and the counts of the parts meet through distributed
// shared memory, and both maps are written at the end.  What bounds it is latency: nine cluster barriers with reads of the other parts' memory
// behind them (about 10 of 22 us at 288 cubes).  Everything is counted in integers and placed by prefix sums in row and column
// order, so the maps are those of the other form, ties and truncation included.
// Route calls, us, the launches above / this: 180 cubes, 12 heads 84 / 59; 288 cubes, 2 heads 79 / 64, 24 heads 183 / 158; 336 cubes, 16
// heads 180 / 163, 32 heads behind the one-pass router 270 / 229; 384 cubes, 16 heads 204 / 184; 480 cubes, 2 heads 99.6 / 96.3, 32
// heads 409 / 407; 528 cubes, 2 heads 109 / 111, 32 heads 475 / 481: eight CTAs a head are too few from there on, hence kSelHeadN.
// Where a context has no room for a cluster (cluster_room) the launches over all heads run at every size.
// (Below 129 cubes the launches above are nine.  For the maps of the per-row modes, and from bitmaps, a cluster was slower: 480p, 12 heads 264 / 279.)
// MAPS: the maps are written.  Without: bitmaps, counts and threshold as sel_row_bits_kernel leaves them, for one-pass scores (BAND: as there).
constexpr int kSelParts = 8, kSelHeadThreads = 512, kSelHeadN = 480;
struct SelHead {
  const float* pr;
  int N, words;
  unsigned keep;
  unsigned* state;
  unsigned *bits_gt, *bits_eq;
  int *row_gt, *row_eq;
  int *row_ptr, *col_idx, *col_ptr, *row_idx;
  long long nnz_cap;
  StatusBlock* status;
};
// shared memory in words: the part's scores (kScores); then two histograms, in whose place afterwards the part's kept bits by row and by
// column, its counts by column and the places of its entries in the columns' lists lie; then per row the kept entries' position and the entries
// taken at the threshold
struct SelHeadSmem {
  int rows, groups, hist, bm, eq, bt, cnt, col, pos, take, total;
  __host__ __device__ SelHeadSmem(int N, int words) {
    rows = (N + kSelParts - 1) / kSelParts;
    groups = (rows + 31) / 32;
    hist = (rows * N + 3) & ~3;
    bm = hist;
    eq = bm + rows * words;
    bt = eq + rows * words;
    cnt = bt + groups * N;
    col = cnt + N;
    pos = col + N;
    if (pos < hist + 2 * kHistBins) pos = hist + 2 * kHistBins;
    take = pos + rows;
    total = take + rows;
  }
};

template <bool BAND, bool MAPS>
__global__ void __cluster_dims__(kSelParts, 1, 1) __launch_bounds__(kSelHeadThreads) sel_head_kernel(SelHead a, Settle se) {
  grid_enter();
  if (!BAND && !MAPS && *se.redo == 0) return;      // (the whole grid)
  extern __shared__ unsigned sm[];
  constexpr int T = kSelHeadThreads, WARPS = T / 32;
  __shared__ int ws[33], part_tot[2], base[4];
  __shared__ unsigned pick[2];
  __shared__ alignas(16) unsigned slice[kHistBins / kSelParts];
  const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int part = (int)cluster.block_rank(), bh = blockIdx.x / kSelParts;
  const int N = a.N, words = a.words, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SelHeadSmem L(N, words);
  const int r0 = part * L.rows, rows = max(0, min(L.rows, N - r0));
  const size_t row0 = (size_t)bh * N + r0;
  const unsigned* src = reinterpret_cast<const unsigned*>(a.pr) + row0 * N;
  unsigned tau = 0u;
  int quota = 0;

  {
    // threshold: three digits, most significant first; the first histogram is taken while the scores come in
    const int n = rows * N;
    unsigned remaining = a.keep, mask = 0u;
    for (int c = tid; c < 2 * kHistBins; c += T) sm[L.hist + c] = 0u;
    __syncthreads();
    for (int e = tid; e < n; e += 8 * T) {
      unsigned v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = e + u * T < n ? src[e + u * T] : 0u;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (e + u * T < n) {
          sm[e + u * T] = v[u];
          atomicAdd(&sm[L.hist + (v[u] >> seq_shift(0))], 1u);
        }
    }
    for (int pass = 0;; ++pass) {
      // Every part adds up an eighth of the bins over all of them, then every part reads the sums, the highest digits in the first threads.
      // (Each part reading all eight histograms: 11,500 cycles a pass.)
      const int nb = (int)seq_mask(pass) + 1, per_part = nb / kSelParts;
      unsigned* hist = sm + L.hist + (pass & 1) * kHistBins;
      cluster.sync();
      if (tid < per_part) {
        unsigned c = 0u;
#pragma unroll
        for (int p = 0; p < kSelParts; ++p) c += cluster.map_shared_rank(hist, p)[part * per_part + tid];
        slice[tid] = c;
      }
      cluster.sync();
      const int per = nb / T, lo = nb - per * (tid + 1);          // this thread's bins: four, in the last pass two
      const unsigned* sums = cluster.map_shared_rank(slice, lo / per_part) + lo % per_part;
      uint4 c;
      if (per == 4) {
        c = *reinterpret_cast<const uint4*>(sums);
      } else {
        const uint2 two = *reinterpret_cast<const uint2*>(sums);
        c = make_uint4(two.x, two.y, 0u, 0u);
      }
      const unsigned mine = c.x + c.y + c.z + c.w;
      int tot;
      const unsigned above = (unsigned)block_excl_scan<T>((int)mine, ws, tot);
      if (above < remaining && remaining <= above + mine) {
        const unsigned left = remaining - above;        // the left-th largest of this thread's entries
        const unsigned a3 = c.w, a2 = a3 + c.z, a1 = a2 + c.y;
        const int b = left <= a3 ? 3 : left <= a2 ? 2 : left <= a1 ? 1 : 0;
        pick[0] = (unsigned)(lo + b);
        pick[1] = left - (b == 3 ? 0u : b == 2 ? a3 : b == 1 ? a2 : a1);
      }
      __syncthreads();
      tau |= pick[0] << seq_shift(pass);
      mask |= seq_mask(pass) << seq_shift(pass);
      remaining = pick[1];
      if (pass == 2) break;
      // (the first histogram is cleared for its second use behind the barriers that its readers have passed)
      hist = sm + L.hist + ((pass + 1) & 1) * kHistBins;
      if (pass == 1) {
        for (int c_ = tid; c_ < kHistBins; c_ += T) hist[c_] = 0u;
        __syncthreads();
      }
      const int shift = seq_shift(pass + 1);
      const unsigned dmask = seq_mask(pass + 1);
#pragma unroll 4
      for (int e = tid; e < n; e += T) {
        const unsigned v = sm[e];
        if ((v & mask) == tau) atomicAdd(&hist[(v >> shift) & dmask], 1u);
      }
    }
    quota = (int)remaining;
    if (!MAPS && part == 0 && tid == 0) {
      a.state[bh * 8 + 3] = tau;
      a.state[bh * 8 + 4] = remaining;
    }
    cluster.sync();            // (the histograms have been read: their place is used again)
  }

  // entries above the threshold (or its band) and at it, by row
  const unsigned hi = BAND ? band_hi(tau) : tau, lo = BAND ? band_lo(tau) : tau;
  unsigned* gt_bits = MAPS ? sm + L.bm : a.bits_gt + row0 * words;
  unsigned* eq_bits = MAPS ? sm + L.eq : a.bits_eq + row0 * words;
  for (int r = warp; r < rows; r += WARPS) {
    int gt = 0, eq = 0;
    constexpr int U = 4;
    for (int w0 = 0; w0 < words; w0 += U) {
      unsigned mine_g = 0u, mine_e = 0u;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = (w0 + u) * 32 + lane;
        const unsigned v = j < N ? sm[r * N + j] : 0u;
        const bool in = j < N && v >= lo && v <= hi;
        const unsigned gb = __ballot_sync(0xffffffffu, j < N && v > hi), eb = __ballot_sync(0xffffffffu, in);
        if (lane == u) { mine_g = gb; mine_e = eb; }
        gt += __popc(gb);
        eq += __popc(eb);
        if constexpr (BAND) settle_list_warp(se, in, (int)row0 + r, j);
      }
      if (lane < U && w0 + lane < words) {
        gt_bits[r * words + w0 + lane] = mine_g;
        eq_bits[r * words + w0 + lane] = mine_e;
      }
    }
    if (lane == 0) {
      if constexpr (MAPS) {
        sm[L.pos + r] = (unsigned)gt;
        sm[L.take + r] = (unsigned)eq;
      } else {
        a.row_gt[row0 + r] = gt;
        a.row_eq[row0 + r] = eq;
      }
    }
  }
  if constexpr (MAPS) {
    // positions of the rows: sums over the rows before, in this part and in the parts before.  Ties go to the lower row: of the
    // entries at the threshold the first `quota` are kept, so the kept entries before a row are those above it and min(quota, those at it)
    __syncthreads();
    int gt = 0, eq = 0, gt_tot, eq_tot;
    if (tid < rows) {
      gt = (int)sm[L.pos + tid];
      eq = (int)sm[L.take + tid];
    }
    int gt_before = block_excl_scan<T>(gt, ws, gt_tot), eq_before = block_excl_scan<T>(eq, ws, eq_tot);
    if (tid == 0) {
      part_tot[0] = gt_tot;
      part_tot[1] = eq_tot;
    }
    cluster.sync();
    if (warp == 0) {
      const int* t = cluster.map_shared_rank(part_tot, lane % kSelParts);
      const int tg = lane < kSelParts ? t[0] : 0, te = lane < kSelParts ? t[1] : 0;
      const int bg = __reduce_add_sync(0xffffffffu, lane < part ? tg : 0), be = __reduce_add_sync(0xffffffffu, lane < part ? te : 0);
      const int ag = __reduce_add_sync(0xffffffffu, tg), ae = __reduce_add_sync(0xffffffffu, te);
      if (lane == 0) {
        base[0] = bg;
        base[1] = be;
        base[2] = ag;
        base[3] = ae;
      }
    }
    __syncthreads();
    gt_before += base[0];
    eq_before += base[1];
    const long long kept = (long long)base[2] + min(base[3], quota);
    if (tid < rows) {
      const int pre = gt_before + min(eq_before, quota);
      sm[L.pos + tid] = (unsigned)min((long long)pre, a.nnz_cap);
      sm[L.take + tid] = (unsigned)max(0, min(eq, quota - eq_before));
    }
    __syncthreads();
    // the rows' kept bits (without entries beyond the capacity), a lane per word
    for (int r = warp; r < rows; r += WARPS) {
      int pos = (int)sm[L.pos + r], left = (int)sm[L.take + r];
      for (int w0 = 0; w0 < words; w0 += 32) {
        const int w = w0 + lane;
        unsigned sel = w < words ? sm[L.bm + r * words + w] : 0u;
        unsigned eb = w < words ? sm[L.eq + r * words + w] : 0u;
        const int ce = __popc(eb), ce_incl = warp_incl_scan(ce, lane);
        for (int rank = ce_incl - ce; eb != 0u && rank < left; ++rank) {
          sel |= eb & (0u - eb);
          eb &= eb - 1u;
        }
        const int c = __popc(sel), c_incl = warp_incl_scan(c, lane);
        for (long long p = (long long)pos + c_incl; p > a.nnz_cap && sel != 0u; --p) sel &= ~(0x80000000u >> __clz(sel));
        if (w < words) sm[L.bm + r * words + w] = sel;
        pos += __shfl_sync(0xffffffffu, c_incl, 31);
        left -= __shfl_sync(0xffffffffu, ce_incl, 31);
      }
    }
    __syncthreads();
    // the part's bits by column, 32 x 32 at a time, and their counts
    for (int t = warp; t < L.groups * words; t += WARPS) {
      const int rg = t / words, w = t - rg * words, r = rg * 32 + lane;
      const unsigned v = r < rows ? sm[L.bm + r * words + w] : 0u;
      unsigned mine = 0u;
#pragma unroll
      for (int bit = 0; bit < 32; ++bit) {
        const unsigned col_word = __ballot_sync(0xffffffffu, (v >> bit) & 1u);
        if (lane == bit) mine = col_word;
      }
      if (w * 32 + lane < N) sm[L.bt + rg * N + w * 32 + lane] = mine;
    }
    __syncthreads();
    for (int j = tid; j < N; j += T) {
      int c = 0;
      for (int rg = 0; rg < L.groups; ++rg) c += __popc(sm[L.bt + rg * N + j]);
      sm[L.cnt + j] = (unsigned)c;
    }
    cluster.sync();
    // where this part's entries of a column begin: behind the columns before, the rows of the parts before first
    int carry = 0;
    for (int j0 = 0; j0 < N; j0 += T) {
      const int j = j0 + tid;
      int c = 0, before = 0, tot;
      if (j < N) {
#pragma unroll
        for (int p = 0; p < kSelParts; ++p) {
          const int cp = (int)cluster.map_shared_rank(sm + L.cnt, p)[j];
          if (p < part) before += cp;
          c += cp;
        }
      }
      const int pre = carry + block_excl_scan<T>(c, ws, tot);
      carry += tot;
      if (j < N) {
        sm[L.col + j] = (unsigned)(pre + before);
      }
    }
    // (no part ends while another reads its counts.  Nothing is written to global memory before this last barrier, whose release would
    // wait for it.)
    cluster.sync();
    // maps: the rows' lists with a lane per word, the columns' with a lane per row
    const unsigned lt = (1u << lane) - 1u;
    int* out = a.col_idx + (size_t)bh * a.nnz_cap;
    for (int r = warp; r < rows; r += WARPS) {
      int pos = (int)sm[L.pos + r];
      if (lane == 0) a.row_ptr[(size_t)bh * (N + 1) + r0 + r] = pos;
      for (int w0 = 0; w0 < words; w0 += 32) {
        unsigned sel = w0 + lane < words ? sm[L.bm + r * words + w0 + lane] : 0u;
        const int c = __popc(sel), c_incl = warp_incl_scan(c, lane);
        for (int p = pos + c_incl - c; sel != 0u; sel &= sel - 1u, ++p) out[p] = (w0 + lane) * 32 + (__ffs(sel) - 1);
        pos += __shfl_sync(0xffffffffu, c_incl, 31);
      }
    }
    int* lists = a.row_idx + (size_t)bh * a.nnz_cap;
#pragma unroll 4
    for (int j = warp; j < N; j += WARPS) {
      int p = (int)sm[L.col + j];
      if (part == 0 && lane == 0) a.col_ptr[(size_t)bh * (N + 1) + j] = (int)min((long long)p, a.nnz_cap);
      for (int rg = 0; rg < L.groups; ++rg) {
        const unsigned b = sm[L.bt + rg * N + j];
        const int at = p + __popc(b & lt);
        if (((b >> lane) & 1u) && at < a.nnz_cap) lists[at] = r0 + rg * 32 + lane;
        p += __popc(b);
      }
    }
    if (part == 0 && tid == 0) {
      a.col_ptr[(size_t)bh * (N + 1) + N] = (int)min((long long)carry, a.nnz_cap);
      a.row_ptr[(size_t)bh * (N + 1) + N] = (int)min(kept, a.nnz_cap);
      if (kept > a.nnz_cap) atomicExch(&a.status->status, VSA2_ERR_MAP_OVERFLOW);
    }
  }
}

template <int MODE>
static void launch_row_topk(const Geo& g, const float* pr, const int* budgets, const SelectScratch& s, const Settle& se, cudaStream_t st) {
  const int BH = g.batch * g.Hq, N = g.N;
  const int* bud = g.mode == VSA2_PER_QUERY_BUDGET ? budgets : nullptr;
  const dim3 grid = MODE == kListed ? dim3((unsigned)(((long long)BH * N + 7) / 8)) : dim3((N + 7) / 8, BH);
#define VSA2_ROW_TOPK(U) launch_kernel(sel_row_topk_warp_kernel<U, MODE>, grid, 256, 0, st, pr, N, g.K, bud, s.row_tau, s.row_eq_take, s.row_cnt, se)
  if (N <= 256) VSA2_ROW_TOPK(8);
  else if (N <= 640) VSA2_ROW_TOPK(20);
  else if (N <= 1024) VSA2_ROW_TOPK(32);
  else if (N <= 1536) VSA2_ROW_TOPK(48);
  else if (N <= 2048) VSA2_ROW_TOPK(64);
  else
    launch_kernel(sel_row_topk_kernel<MODE>, MODE == kListed ? dim3(592) : dim3(N, BH), 256, 0, st, pr, N, g.K, bud, s.row_tau, s.row_eq_take, s.row_cnt, se);
#undef VSA2_ROW_TOPK
}

// Per sequence, up to kSelHeadN cubes: the selection of the heads in clusters, if the context has room for one of the largest; *done: it was launched
template <bool BAND, bool MAPS>
static cudaError_t launch_sel_head(const Geo& g, const float* pr, const SelectScratch& s, int* row_ptr, int* col_idx, int* col_ptr, int* row_idx,
                                   StatusBlock* status, const Settle& se, cudaStream_t st, bool* done) {
  *done = false;
  if (g.mode != VSA2_PER_SEQUENCE || g.N > kSelHeadN || (g.flags & VSA2_FLAG_SELECT_NO_CLUSTERS)) return cudaSuccess;
  static ClusterRoom room;
  cudaError_t e;
  if ((e = cluster_room((const void*)sel_head_kernel<BAND, MAPS>, room, kSelParts, kSelHeadThreads,
                        (size_t)SelHeadSmem(kSelHeadN, (kSelHeadN + 31) / 32).total * 4, done)) != cudaSuccess || !*done)
    return e;
  const SelHead a{pr, g.N, s.words, (unsigned)((long long)g.N * g.K), s.state, s.bitmap, s.bitmap_t, s.row_gt, s.row_eq,
                  row_ptr, col_idx, col_ptr, row_idx, g.nnz_cap, status};
  return launch_kernel(sel_head_kernel<BAND, MAPS>, kSelParts * g.batch * g.Hq, kSelHeadThreads, (size_t)SelHeadSmem(g.N, s.words).total * 4, st, a, se);
}

// thresholds, counts and (per sequence) bitmaps of all heads; `se.redo`: null, or the flag without which nothing happens
template <bool BAND>
static cudaError_t launch_thresholds(const Geo& g, const float* pr, const int* budgets, const SelectScratch& s, const Settle& se, cudaStream_t st) {
  const int BH = g.batch * g.Hq, N = g.N;
  if (g.mode == VSA2_PER_SEQUENCE) {
    const long long n_elems = (long long)N * N;
    const unsigned keep = (unsigned)((long long)N * g.K);
    const int* redo = BAND ? nullptr : se.redo;
    if (BAND || redo != nullptr) {
      bool done;
      const cudaError_t e = launch_sel_head<BAND, false>(g, pr, s, nullptr, nullptr, nullptr, nullptr, nullptr, se, st, &done);
      if (e != cudaSuccess || done) return e;
    }
    int init_n = BH * 3 * kHistBins;
    launch_kernel(sel_init_kernel, (init_n + 255) / 256, 256, 0, st, s.state, s.hist, BH, keep, redo);
    int chunks = (int)((n_elems + 256 * 16 - 1) / (256 * 16));
    if (chunks > 256) chunks = 256;
    for (int pass = 0; pass < 3; ++pass) {
      launch_kernel(sel_hist_kernel, dim3(chunks, BH), 256, 0, st, pr, n_elems, s.state, s.hist, pass, redo);
      launch_kernel(sel_pick_kernel, BH, 32, 0, st, s.state, s.hist, pass, redo);
    }
    // counts and bitmaps in one read of P_r (the bitmap of the entries equal to tau borrows the transposed bitmap's space)
    launch_kernel(sel_row_bits_kernel<BAND>, dim3((N + 7) / 8, BH), 256, 0, st, pr, N, s.words, s.state, s.bitmap, s.bitmap_t, s.row_gt, s.row_eq, se);
  } else {
    launch_row_topk<BAND ? kBand : kAllRows>(g, pr, budgets, s, se, st);
  }
  return cudaGetLastError();
}

cudaError_t launch_select_band(const Geo& g, const float* pr, const int* budgets, const SelectScratch& s, const Settle& se, cudaStream_t st) {
  return launch_thresholds<true>(g, pr, budgets, s, se, st);
}

cudaError_t launch_select_settle(const Geo& g, const float* pr, const int* budgets, const SelectScratch& s, const Settle& se,
                                 cudaStream_t st) {
  const int BH = g.batch * g.Hq, N = g.N;
  if (g.mode == VSA2_PER_SEQUENCE)
    launch_kernel(sel_settle_kernel, BH, 1024, 0, st, pr, N, s.words, (unsigned)((long long)N * g.K), s.state, s.row_gt, s.row_eq, s.bitmap_t, se);
  else
    launch_row_topk<kListed>(g, pr, budgets, s, se, st);
  return cudaGetLastError();
}

cudaError_t launch_select(const Geo& g, const float* pr, const int* budgets, const SelectScratch& s, const int* redo, int* row_ptr,
                          int* col_idx, int* col_ptr, int* row_idx, StatusBlock* status, cudaStream_t st) {
  const int BH = g.batch * g.Hq, N = g.N;
  Settle se{};
  se.redo = const_cast<int*>(redo);
  cudaError_t e;
  if (redo == nullptr) {
    bool done;
    if ((e = launch_sel_head<false, true>(g, pr, s, row_ptr, col_idx, col_ptr, row_idx, status, se, st, &done)) != cudaSuccess || done) return e;
  }
  const bool per_sequence = g.mode == VSA2_PER_SEQUENCE, small = N <= kSelOneBlockN;
  const bool with_thresholds = small && !per_sequence && redo == nullptr;      // (the block per head finds them itself)
  if (!with_thresholds && (e = launch_thresholds<false>(g, pr, budgets, s, se, st)) != cudaSuccess) return e;
  if (small) {
    launch_kernel(sel_maps_kernel, BH, 1024, 0, st, pr, N, s.words, per_sequence, s.state, s.row_gt, s.row_eq, with_thresholds ? nullptr : s.row_tau,
                  s.row_eq_take, s.row_cnt, s.bitmap, s.bitmap_t, g.K, g.mode == VSA2_PER_QUERY_BUDGET ? budgets : nullptr, row_ptr, col_idx,
                  col_ptr, row_idx, g.nnz_cap, status);
    return cudaGetLastError();
  }
  launch_kernel(sel_scan_rows_kernel, BH, 1024, 0, st, N, g.mode == VSA2_PER_SEQUENCE, s.state, s.row_gt, s.row_eq, s.row_tau,
                                            s.row_eq_take, s.row_cnt, row_ptr, g.nnz_cap, status);
  if (g.mode == VSA2_PER_SEQUENCE)
    launch_kernel(sel_emit_rows_bits_kernel, dim3((N + 7) / 8, BH), 256, 0, st, N, s.words, s.bitmap_t, s.row_eq_take, row_ptr, col_idx,
                                                                     s.bitmap, g.nnz_cap);
  else
    launch_kernel(sel_emit_rows_kernel, dim3((N + 7) / 8, BH), 256, 0, st, pr, N, s.words, s.row_tau, s.row_eq_take, row_ptr,
                                                                col_idx, s.bitmap, g.nnz_cap);
  // columns: transposed bitmap, then counts (row_gt reused as scratch), scan, ordered emission
  launch_kernel(sel_transpose_bitmap_kernel, dim3(s.words, (s.words + 7) / 8, BH), 256, 0, st, s.bitmap, N, s.words, s.bitmap_t);
  launch_kernel(sel_col_count_kernel, dim3((N + 7) / 8, BH), 256, 0, st, s.bitmap_t, N, s.words, s.row_gt);
  launch_kernel(sel_scan_cols_kernel, BH, 1024, 0, st, N, s.row_gt, col_ptr, g.nnz_cap);
  launch_kernel(sel_emit_cols_kernel, dim3((N + 7) / 8, BH), 256, 0, st, s.bitmap_t, N, s.words, col_ptr, row_idx, g.nnz_cap);
  return cudaGetLastError();
}

}  // namespace vsa2
