// Per-head top-n (Eq. 3; Algorithm 1's "topk(B^l)") under the total order (score descending, position
// ascending), and the digits that it shares with the global top-K of Eq. 4.  One thread block per (sample, KV head).
//
// Scores are non-negative floats, so their bit patterns order like unsigned integers.  A score's DIGIT is its exponent
// and six mantissa bits, clamped to 2048 values around the range scores live in (a score is a sum of at most 256
// probabilities): neighbouring digits are 1.6 % apart, so the digit that holds the n-th largest score holds few others.
//   1  histogram of the digits (shared memory) -> the digit d that holds the n-th largest score;
//   2  the scores with digit >= d (n and a few percent more) are collected into a list; where that does not fit the
//      list, digit d is divided further, down to single values and the lowest positions among equal ones;
//   3  the list is put in order by a counting sort: 4096 bins of equal width over the list's own range of bit patterns
//      (a bin then holds a run of equal pooled scores or little more), and every entry ranks itself within its bin.
//      A list with a bin of more than kMaxBin entries (many equal scores) goes through a bitonic network instead.
// The result is the order Algorithm 1's topk() returns and stores positions in; a later truncation to a smaller
// budget is a prefix of it.
//
// Latency-bound: chains of block-wide steps over L2-resident scores.  Two blocks of 512 threads share an SM, so that
// one's barriers overlap the other's work.
#pragma once
#include <cooperative_groups.h>
#include "common.cuh"
#include "compact.cuh"

namespace dkv {

constexpr int kSelThreads = 512;
constexpr int kBins = 2048;                  // digits
constexpr int kDigitBase = (127 - 24) << 6;  // digit 0: everything below 2^-24; digit 2047: from 2^8 (63/64) up
constexpr int kSortBins = 4096;
constexpr int kMaxBin = 128;
constexpr int kMaxCountingList = 8192;       // longest list that is sorted by counting (twice 8 bytes an entry)

__device__ __forceinline__ int digit_of(uint32_t bits) { return min(max((int)(bits >> 17) - kDigitBase, 0), kBins - 1); }
// The bit patterns of digit d are [digit_low(d), digit_last(d)].
__device__ __forceinline__ uint32_t digit_low(int d) { return d == 0 ? 0u : (uint32_t)(kDigitBase + d) << 17; }
__device__ __forceinline__ uint32_t digit_last(int d) { return d == kBins - 1 ? 0xFFFFFFFFu : ((uint32_t)(kDigitBase + d + 1) << 17) - 1u; }
// A range of patterns longer than 2048 is divided by its leading 11 bits: how far to shift an offset into it.
__device__ __forceinline__ int range_shift(uint32_t low, uint32_t last) { const int bits = 32 - __clz(last - low); return bits > 11 ? bits - 11 : 0; }
__device__ __forceinline__ void range_part(uint32_t& low, uint32_t& last, int part, int shift) {
  low += (uint32_t)part << shift;
  last = min(last, low + (1u << shift) - 1u);
}

// Exclusive prefix sum of one int per thread over the block; *total gets the block sum.
// sm must hold 33 ints.  Ends with a barrier.
__device__ __forceinline__ int block_excl_scan(int v, int* sm, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xFFFFFFFFu, inc, o); if (lane >= o) inc += t; }
  __syncthreads();
  if (lane == 31) sm[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < nw ? sm[lane] : 0;
    int s = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xFFFFFFFFu, s, o); if (lane >= o) s += t; }
    sm[lane] = s - w;
    if (lane == 31) sm[32] = s;
  }
  __syncthreads();
  const int r = sm[warp] + inc - v;
  *total = sm[32];
  __syncthreads();
  return r;
}

// Given hist[nbins] in shared memory (counts per digit, `total` entries in all), find the digit d
// holding the need-th largest entry: (#entries with digit > d) < need <= that + hist[d].
// Results go to out[0] = d, out[1] = need - (#entries with digit > d).  Every thread owns
// nbins / blockDim.x consecutive digits; every warp adds up the warps' totals for itself, so that two barriers suffice.
// sm: 32 ints.  Ends with a barrier; hist is unchanged.
__device__ __forceinline__ void find_digit(const unsigned int* hist, int nbins, int total, int need, int* sm, volatile int* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = nbins / (int)blockDim.x, b0 = threadIdx.x * per;
  int mine = 0;
  for (int j = 0; j < per; ++j) mine += (int)hist[b0 + j];
  int inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xFFFFFFFFu, inc, o); if (lane >= o) inc += t; }
  if (lane == 31) sm[warp] = inc;
  __syncthreads();
  const int before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? sm[lane] : 0);
  int above = total - before - (inc - mine);               // entries with this thread's first digit or a larger one
  for (int j = 0; j < per; ++j) {
    const int c = (int)hist[b0 + j];
    above -= c;
    if (c > 0 && above < need && need <= above + c) { out[0] = b0 + j; out[1] = need - above; }
  }
  __syncthreads();
}

// Counter bump without a return value for digits that come in runs (pooled scores: neighbouring positions share
// their digit): a run of equal digits in adjacent lanes makes one atomicAdd of its length.  Equal digits that are
// not adjacent are added separately.  Must be called by all 32 lanes.
__device__ __forceinline__ void run_bump(unsigned int* counters, unsigned int digit, bool active) {
  const unsigned int lane = threadIdx.x & 31;
  const unsigned int key = active ? digit : 0xFFFFFFFFu;
  const unsigned int prev = __shfl_up_sync(0xFFFFFFFFu, key, 1);
  const bool head = lane == 0 || prev != key;
  const unsigned int heads = __ballot_sync(0xFFFFFFFFu, head);
  if (head && active) {
    const unsigned int later = heads & ~((2u << lane) - 1u);       // run heads after this lane (lane 31: none)
    const int next = later ? __ffs(later) - 1 : 32;
    atomicAdd(&counters[digit], (unsigned int)(next - (int)lane));
  }
}

// One compare-exchange step of a bitonic network on the 64 keys a warp holds in registers: lane j has
// a = key[base + j] and b = key[base + 32 + j].  `s` is the stride (32, 16, ..., 1), `size` the length of the
// bitonic sequences being merged; a block of `size` keys is sorted ascending if its first index has bit `size` clear.
__device__ __forceinline__ void bitonic_step64(unsigned long long& a, unsigned long long& b, int base, int lane, int s, int size) {
  if (s == 32) {
    const bool up = ((base + lane) & size) == 0;
    if ((a > b) == up) { const unsigned long long t = a; a = b; b = t; }
  } else {
    const unsigned long long pa = __shfl_xor_sync(0xFFFFFFFFu, a, s), pb = __shfl_xor_sync(0xFFFFFFFFu, b, s);
    const bool lower = (lane & s) == 0;                       // this lane holds the lower index of its pair
    const bool up_a = ((base + lane) & size) == 0, up_b = ((base + 32 + lane) & size) == 0;
    a = (lower == up_a) ? (a < pa ? a : pa) : (a > pa ? a : pa);
    b = (lower == up_b) ? (b < pb ? b : pb) : (b > pb ? b : pb);
  }
}

// Bitonic sort of keys[0 .. sort_n) ascending; sort_n a power of two >= 2.  Strides of 64 and more are
// done by the whole block in shared memory with a barrier per stage; the strides below that stay inside
// 64-key blocks, each owned by one warp, which holds its block in registers (two keys per lane) and
// exchanges by shuffles; the first six merge lengths (2 .. 64) run entirely in registers.  Arrays of
// fewer than 64 keys use shared memory throughout.  Ends with a block barrier.
__device__ __forceinline__ void bitonic_sort(unsigned long long* keys, int sort_n) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  if (sort_n < 64) {
    for (int size = 2; size <= sort_n; size <<= 1) {
      for (int s = size >> 1; s > 0; s >>= 1) {
        for (int t = threadIdx.x; t < (sort_n >> 1); t += blockDim.x) {
          const int lo = ((t & ~(s - 1)) << 1) | (t & (s - 1)), hi = lo + s;
          const bool up = ((lo & size) == 0);
          const unsigned long long a = keys[lo], b = keys[hi];
          if ((a > b) == up) { keys[lo] = b; keys[hi] = a; }
        }
        __syncthreads();
      }
    }
    return;
  }
  __syncthreads();
  for (int base = warp * 64; base < sort_n; base += nwarps * 64) {      // merge lengths 2 .. 64 in registers
    unsigned long long a = keys[base + lane], b = keys[base + 32 + lane];
    for (int size = 2; size <= 64; size <<= 1)
      for (int s = size >> 1; s > 0; s >>= 1) bitonic_step64(a, b, base, lane, s, size);
    keys[base + lane] = a; keys[base + 32 + lane] = b;
  }
  __syncthreads();
  for (int size = 128; size <= sort_n; size <<= 1) {
    for (int stride = size >> 1; stride >= 64; stride >>= 1) {
      for (int t = threadIdx.x; t < (sort_n >> 1); t += blockDim.x) {
        const int lo = ((t & ~(stride - 1)) << 1) | (t & (stride - 1));
        const int hi = lo + stride;
        const bool up = ((lo & size) == 0);
        const unsigned long long a = keys[lo], b = keys[hi];
        if ((a > b) == up) { keys[lo] = b; keys[hi] = a; }
      }
      __syncthreads();
    }
    for (int base = warp * 64; base < sort_n; base += nwarps * 64) {
      unsigned long long a = keys[base + lane], b = keys[base + 32 + lane];
#pragma unroll
      for (int s = 32; s > 0; s >>= 1) bitonic_step64(a, b, base, lane, s, size);
      keys[base + lane] = a; keys[base + 32 + lane] = b;
    }
    __syncthreads();
  }
}

// The `n` best positions of one head (1 <= n <= P), in order, in sel[0 .. n) (shared memory, returned).
// v: the head's scores.  gh: if not null, the head's digit counts are added to these 2048 counters (global).
// kShared: a cluster of `parts` blocks works on the head, each on an equal share of the positions; block 0 gets the list and
// the result, the others nullptr.
// `cap`: entries of the list, a power of two; at least n.  Dynamic shared memory `dyn`: select_smem(cap) bytes.
// Ends with a barrier.
__host__ __device__ inline size_t select_smem(int cap) {
  return (size_t)cap * 8 * (cap <= kMaxCountingList ? 2 : 1) + sizeof(unsigned int) * kSortBins;
}
// A block's share of a head's positions.
template <bool kShared>
__device__ __forceinline__ void select_share(int P, int part, int parts, int& lo, int& hi) {
  const int share = kShared ? ((P + parts - 1) / parts + 31) & ~31 : P;
  lo = min(P, part * share); hi = min(P, lo + share);
}
constexpr int kSelUnroll = 8;                              // scores a thread has in flight
__device__ __forceinline__ unsigned int* select_bins(unsigned char* dyn, int cap) {
  return reinterpret_cast<unsigned int*>(dyn + (size_t)cap * 8 * (cap <= kMaxCountingList ? 2 : 1));
}
// The first step, which does not depend on n: the share's digits are counted in `bins` [kBins].  Ends with a barrier.
template <bool kShared>
__device__ __forceinline__ void count_digits(const uint32_t* v, int P, unsigned int* bins, int part, int parts) {
  const int tid = threadIdx.x;
  int lo, hi;
  select_share<kShared>(P, part, parts, lo, hi);
  const int hi32 = lo + ((hi - lo + 31) & ~31);
  for (int i = tid; i < kBins; i += kSelThreads) bins[i] = 0;
  __syncthreads();
  for (int p0 = lo + tid; p0 < hi32; p0 += kSelThreads * kSelUnroll) {
    uint32_t u[kSelUnroll];
#pragma unroll
    for (int j = 0; j < kSelUnroll; ++j) { const int p = p0 + j * kSelThreads; u[j] = p < hi ? v[p] : 0u; }
#pragma unroll
    for (int j = 0; j < kSelUnroll; ++j) {
      const int p = p0 + j * kSelThreads;
      if (p < hi32) run_bump(bins, digit_of(u[j]), p < hi);   // warp-uniform: neighbours share digits after pooling
    }
  }
  __syncthreads();
}
// The other steps; count_digits has been called.
template <bool kShared>
__device__ __forceinline__ int* select_head(const uint32_t* v, int P, int n, int cap, unsigned char* dyn, unsigned int* gh, int part,
                                            int parts) {
  namespace cg = cooperative_groups;
  __shared__ int sm_scan[33];
  __shared__ int found[2];
  __shared__ unsigned int s_n, s_max, s_full;
  const int tid = threadIdx.x, lane = tid & 31;
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(dyn);
  unsigned long long* sorted = keys + (cap <= kMaxCountingList ? cap : 0);
  unsigned int* bins = select_bins(dyn, cap);
  unsigned int* sums = kShared ? bins + kBins : bins;      // the whole head's counts
  int lo, hi;
  select_share<kShared>(P, part, parts, lo, hi);
  const int hi32 = lo + ((hi - lo + 31) & ~31);
  auto add_up = [&]() {                                    // bins of all blocks -> sums
    if constexpr (kShared) {
      cg::this_cluster().sync();
      for (int i = tid; i < kBins; i += kSelThreads) {
        unsigned int s = 0;
        for (int r = 0; r < parts; ++r) s += cg::this_cluster().map_shared_rank(bins, r)[i];
        sums[i] = s;
      }
      cg::this_cluster().sync();                           // nobody's bins change before all have read them
    } else {
      __syncthreads();
    }
  };

  // 1: the digit of the n-th largest score
  if (tid == 0) { s_n = 0; s_max = 0; s_full = 0; }        // barriers follow before these are counted up
  if (gh) for (int i = tid; i < kBins; i += kSelThreads) { const unsigned int c = bins[i]; if (c) atomicAdd(&gh[i], c); }
  add_up();
  find_digit(sums, kBins, P, n, sm_scan, found);
  uint32_t low = digit_low(found[0]), last = digit_last(found[0]);
  int need = found[1], inside = (int)sums[found[0]];       // `need` of the `inside` scores in the range are kept
  while (n - need + inside > cap && last > low) {          // too many for the list: divide the range
    const int shift = range_shift(low, last);
    __syncthreads();
    for (int i = tid; i < kBins; i += kSelThreads) bins[i] = 0;
    __syncthreads();
    for (int p = lo + tid; p < hi; p += kSelThreads) {
      const uint32_t u = v[p];
      if (u >= low && u <= last) atomicAdd(&bins[(u - low) >> shift], 1u);
    }
    add_up();
    find_digit(sums, kBins, inside, need, sm_scan, found);
    inside = (int)sums[found[0]]; need = found[1];
    range_part(low, last, found[0], shift);
  }
  __syncthreads();

  // 2: everything in or above the range; if equal scores alone overflow the list (one pattern), the first `need` of them
  const bool some_equal = n - need + inside > cap;
  const uint32_t from = low + (some_equal ? 1u : 0u);
  unsigned long long* to = keys;
  unsigned int *to_n = &s_n, *to_max = &s_max;
  if constexpr (kShared) {
    to = cg::this_cluster().map_shared_rank(keys, 0);
    to_n = cg::this_cluster().map_shared_rank(&s_n, 0);
    to_max = cg::this_cluster().map_shared_rank(&s_max, 0);
  }
  for (int p0 = lo + tid; p0 < hi32; p0 += kSelThreads * kSelUnroll) {
    uint32_t u[kSelUnroll];
#pragma unroll
    for (int j = 0; j < kSelUnroll; ++j) { const int p = p0 + j * kSelThreads; u[j] = p < hi ? v[p] : 0u; }
#pragma unroll
    for (int j = 0; j < kSelUnroll; ++j) {
      const int p = p0 + j * kSelThreads;
      const bool take = p < hi && u[j] >= from;
      const unsigned int m = __ballot_sync(0xFFFFFFFFu, take);
      if (m) {                                             // warp-uniform: most rows of 32 positions keep nothing
        unsigned int base = 0;
        if (lane == 0) base = atomicAdd(to_n, (unsigned int)__popc(m));
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if (take) to[base + __popc(m & ((1u << lane) - 1u))] = ((unsigned long long)(~u[j]) << 32) | (unsigned int)p;
        const unsigned int mx = __reduce_max_sync(0xFFFFFFFFu, take ? u[j] : 0u);
        if (lane == 0) atomicMax(to_max, mx);
      }
    }
  }
  if constexpr (kShared) {
    cg::this_cluster().sync();
    if (part != 0) return nullptr;
  } else {
    __syncthreads();
  }
  int list = (int)s_n;
  if (some_equal) {
    int have = 0;                                          // equal scores taken so far, in position order
    for (int p0 = 0; p0 < P && have < need; p0 += kSelThreads) {
      const bool eq = p0 + tid < P && v[p0 + tid] == low;
      int tot;
      const int at = have + block_excl_scan(eq ? 1 : 0, sm_scan, &tot);
      if (eq && at < need) keys[list + at] = ((unsigned long long)(~low) << 32) | (unsigned int)(p0 + tid);
      have += tot;
    }
    list += need;
    if (list == need && tid == 0) s_max = low;
    __syncthreads();
  }

  // 3: order
  bool counting = cap <= kMaxCountingList;
  if (counting) {
    const uint32_t top = s_max, range = top - low;
    const int shift = range < kSortBins ? 0 : 32 - __clz(range) - 12;
    for (int i = tid; i < kSortBins; i += kSelThreads) bins[i] = 0;
    __syncthreads();
    for (int i = tid; i < list; i += kSelThreads) atomicAdd(&bins[(top - ~(uint32_t)(keys[i] >> 32)) >> shift], 1u);
    __syncthreads();
    constexpr int kPer = kSortBins / kSelThreads;
    unsigned int c[kPer], mine = 0, most = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) { c[j] = bins[tid * kPer + j]; mine += c[j]; most = max(most, c[j]); }
    if (most > kMaxBin) s_full = 1;                           // any writer will do
    int tot;
    unsigned int off = (unsigned int)block_excl_scan((int)mine, sm_scan, &tot);
#pragma unroll
    for (int j = 0; j < kPer; ++j) { bins[tid * kPer + j] = off; off += c[j]; }
    __syncthreads();
    counting = s_full == 0;
    if (counting) {
      for (int i = tid; i < list; i += kSelThreads) {
        const unsigned long long k = keys[i];
        sorted[atomicAdd(&bins[(top - ~(uint32_t)(k >> 32)) >> shift], 1u)] = k;      // bins: from starts to ends
      }
      __syncthreads();
      int* sel = reinterpret_cast<int*>(keys);             // the unsorted list is done with
      for (int i = tid; i < list; i += kSelThreads) {
        const unsigned long long k = sorted[i];
        const unsigned int b = (top - ~(uint32_t)(k >> 32)) >> shift, b0 = b ? bins[b - 1] : 0, b1 = bins[b];
        if ((int)b0 >= n) continue;
        int r = (int)b0;
        for (unsigned int j = b0; j < b1; ++j) r += sorted[j] < k;
        if (r < n) sel[r] = (int)(uint32_t)k;
      }
      __syncthreads();
      return sel;
    }
  }
  int sort_n = 2;
  while (sort_n < list) sort_n <<= 1;
  for (int i = list + tid; i < sort_n; i += kSelThreads) keys[i] = ~0ull;
  __syncthreads();
  bitonic_sort(keys, sort_n);
  int* sel = reinterpret_cast<int*>(keys);
  for (int i0 = 0; i0 < n; i0 += kSelThreads) {            // in place: entry i moves to the front half, read before it is overwritten
    const int i = i0 + tid;
    const int p = i < n ? (int)(uint32_t)keys[i] : 0;
    __syncthreads();
    if (i < n) sel[i] = p;
    __syncthreads();
  }
  return sel;
}

// dkv_select_topk: the `keep` best of every head of one layer.  idx: [Bt*Hkv][keep], in order.  Adds the heads' digit
// counts to layer_hist [Bt][2048] and records count[b][layer] = keep.  One block a head, or a cluster of `parts` blocks (the
// launch says when).  grid Bt*Hkv*parts.
template <bool kShared>
__global__ void __launch_bounds__(kSelThreads, 2)
select_topk_kernel(const float* scores, int* idx, unsigned int* layer_hist, int P,
                   int keep, int cap, int* count, int Hkv, int L, int layer, int parts) {
  extern __shared__ __align__(16) unsigned char dyn[];
  const int head = blockIdx.x / parts, b = head / Hkv;
  pdl_launch();
  pdl_wait();
  if (threadIdx.x == 0 && blockIdx.x % (Hkv * parts) == 0) count[b * L + layer] = keep;
  const uint32_t* v = reinterpret_cast<const uint32_t*>(scores) + (size_t)head * P;
  count_digits<kShared>(v, P, select_bins(dyn, cap), blockIdx.x % parts, parts);
  const int* sel = select_head<kShared>(v, P, keep, cap, dyn, layer_hist + (size_t)b * kBins, blockIdx.x % parts, parts);
  if (sel) for (int i = threadIdx.x; i < keep; i += kSelThreads) idx[(size_t)head * keep + i] = sel[i];
}

// The end of a pass, for every layer and head at once: with the final counts known (count[b][layer], at most B^l), a
// block selects its head's best `count` positions, writes them to idx [layer][Bt*Hkv][stride] and copies those rows and
// the ws window rows of K and V into the layer's buffers.  Selecting and copying the final rows once replaces a
// selection and copy of B^l rows per layer and a truncation per update: 32K prompt with B^l = 4 N: 71 MB of rows read
// instead of 272, and no block of the scoring kernel gives way to it while keys are streamed.
// The scores' digits are counted while the last update still runs (rb_finish_kernel; see rb_collect_kernel for why the scores
// are complete by then): only launched right behind it.
// grid (Bt*Hkv, layers).
__global__ void __launch_bounds__(kSelThreads, 2)
select_gather_kernel(const __grid_constant__ PassPtrs ptrs, const float* scores, int* idx,
                     const int* count, int* held, int P, int ws, int stride, int cap, int S, int vec, int Hkv, int L) {
  extern __shared__ __align__(16) unsigned char dyn[];
  const int bh = blockIdx.x, b = bh / Hkv, layer = blockIdx.y, tid = threadIdx.x;
  const size_t head = (size_t)layer * gridDim.x + bh;
  const uint32_t* v = reinterpret_cast<const uint32_t*>(scores) + head * P;
  count_digits<false>(v, P, select_bins(dyn, cap), 0, 1);
  pdl_wait();
  pdl_launch();
  const int n = count[b * L + layer];
  if (tid == 0 && bh % Hkv == 0) held[b * L + layer] = n;
  const int* sel = nullptr;
  if (n > 0) {
    sel = select_head<false>(v, P, n, cap, dyn, nullptr, 0, 1);
    for (int i = tid; i < n; i += kSelThreads) idx[head * stride + i] = sel[i];
  }
  gather_rows(static_cast<const uint4*>(ptrs.k[layer]), static_cast<const uint4*>(ptrs.v[layer]), static_cast<uint4*>(ptrs.kb[layer]),
              static_cast<uint4*>(ptrs.vb[layer]), sel, n, bh, S, P, ws, stride + ws, vec, tid, kSelThreads, 0, 1);
}

// The same with a cluster a head, whose blocks share the selection and the copying.  grid (Bt*Hkv*cluster size, layers).
__global__ void __launch_bounds__(kSelThreads, 2)
select_gather_cluster_kernel(const __grid_constant__ PassPtrs ptrs, const float* scores, int* idx,
                             const int* count, int* held, int P, int ws, int stride, int cap, int S, int vec, int Hkv,
                             int L) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char dyn[];
  const int parts = cg::this_cluster().num_blocks(), part = blockIdx.x % parts, bh = blockIdx.x / parts;
  const int b = bh / Hkv, layer = blockIdx.y, tid = threadIdx.x;
  const size_t head = (size_t)layer * (gridDim.x / parts) + bh;
  const uint32_t* v = reinterpret_cast<const uint32_t*>(scores) + head * P;
  count_digits<true>(v, P, select_bins(dyn, cap), part, parts);
  pdl_wait();
  pdl_launch();
  const int n = count[b * L + layer];
  if (tid == 0 && part == 0 && bh % Hkv == 0) held[b * L + layer] = n;
  const int* sel = nullptr;
  if (n > 0) {
    select_head<true>(v, P, n, cap, dyn, nullptr, part, parts);
    cg::this_cluster().sync();                             // the first block's list (at the start of `dyn`) is complete
    sel = cg::this_cluster().map_shared_rank(reinterpret_cast<int*>(dyn), 0);
    for (int i = part * kSelThreads + tid; i < n; i += parts * kSelThreads) idx[head * stride + i] = sel[i];
  }
  gather_rows(static_cast<const uint4*>(ptrs.k[layer]), static_cast<const uint4*>(ptrs.v[layer]), static_cast<uint4*>(ptrs.kb[layer]),
              static_cast<uint4*>(ptrs.vb[layer]), sel, n, bh, S, P, ws, stride + ws, vec, tid, kSelThreads, part, parts);
  cg::this_cluster().sync();                               // the list is read until here
}

// The positions idx[b,h,0..n) of one layer ascending (sorted_out) and the place each had in idx (rank_out), either
// may be null.  n = held[b][layer], or `keep` where held is null.  Output rows are idx_stride apart, like idx's.
// One thread block per head; dynamic shared memory: 8 bytes for each of the power of two >= n entries.
__global__ void __launch_bounds__(kSelThreads)
sort_positions_kernel(const int* __restrict__ idx, const int* __restrict__ held, int keep, int* __restrict__ sorted_out,
                      int* __restrict__ rank_out, int idx_stride, int Hkv, int L, int layer) {
  extern __shared__ __align__(16) unsigned long long pos_keys[];
  const int tid = threadIdx.x, n = held ? held[(blockIdx.x / Hkv) * L + layer] : keep;
  int sort_n = 2;
  while (sort_n < n) sort_n <<= 1;
  const size_t row = (size_t)blockIdx.x * idx_stride;
  for (int i = tid; i < sort_n; i += kSelThreads)
    pos_keys[i] = i < n ? ((unsigned long long)(uint32_t)idx[row + i] << 32) | (unsigned int)i : ~0ull;
  __syncthreads();
  bitonic_sort(pos_keys, sort_n);
  for (int i = tid; i < n; i += kSelThreads) {
    if (sorted_out) sorted_out[row + i] = (int)(pos_keys[i] >> 32);
    if (rank_out) rank_out[row + i] = (int)(uint32_t)pos_keys[i];
  }
}

}  // namespace dkv
