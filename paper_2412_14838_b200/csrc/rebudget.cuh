// Update_Buffer_Length (Eq. 4-6) on the device: the K-th largest of all scores of the layers processed
// so far, the number of top-K hits per layer, then the integer budget arithmetic.
//
// Only per-layer counts leave the selection.  Every layer's scores were histogrammed by their digit (select.cuh) when
// they were computed or selected, so:
//   rb_locate   adds up the histograms of layers [0, l), finds the digit that holds the K-th largest score and
//               counts each layer's scores above it (no score is read);
//   rb_collect  streams the history once and lists the scores with that digit (1 or 2 % of it) with their layers;
//   rb_finish   fixes the exact threshold T from the list, gives the entries equal to T to the lowest layers first
//               (flat-index tie rule), and evaluates Eq. 5-6 in exact integers.
// Counts only ever shrink (count_i = min over the updates that include layer i), so a pass runs all its updates
// together when every layer has been scored: one launch of each kernel for up to kRbUpdates updates, one read of the
// history instead of one per update.
#pragma once
#include <cooperative_groups.h>
#include "common.cuh"
#include "select.cuh"

namespace dkv {

constexpr int kRbUpdates = 8;      // updates worked on together
constexpr int kRbThreads = 256;
constexpr int kRbChunk = 4096;     // scores of a block's slice read at a time
constexpr int kRbCluster = 8;      // blocks that share a long candidate list
constexpr unsigned int kRbSolo = 32768;   // candidates one block works through by itself (32 per thread)

struct RbBatch {                   // updates u = 0 .. n-1, l ascending
  int n;
  int l[kRbUpdates];               // layers [0, l) take part
  long long k[kRbUpdates];         // the K of the global top-K
};

struct RbState {                   // per update and sample
  int digit;                       // digit of T
  int need;                        // entries still to take inside it
  int inside;                      // entries with that digit over all layers and heads
  int pad;
};

// grid (updates, Bt).  layer_hist: [L][Bt][2048].  state: [updates][Bt].  above: [updates][Bt][L] scores above the digit
// per layer.  Clears cand_n [Bt]; fill > 0: count[b][.] starts at `fill` (a pass selects after the updates).
__global__ void __launch_bounds__(1024)
rb_locate_kernel(const __grid_constant__ RbBatch batch, const unsigned int* layer_hist, RbState* state,
                 unsigned int* above, unsigned int* cand_n, int* count, int fill, int Bt,
                 int Hkv, int L, int P) {
  __shared__ unsigned int hist[kBins];
  __shared__ int sm_scan[33];
  __shared__ int found[2];
  const int u = blockIdx.x, b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, l = batch.l[u];
  pdl_wait();
  pdl_launch();                                              // after the wait: see rb_collect_kernel
  {
    // two digits per thread, summed over the layers (consecutive threads read consecutive words)
    uint2 a = make_uint2(0, 0);
#pragma unroll 8
    for (int i = 0; i < l; ++i) {
      const uint2 x = reinterpret_cast<const uint2*>(layer_hist + ((size_t)i * Bt + b) * kBins)[tid];
      a.x += x.x; a.y += x.y;
    }
    hist[2 * tid] = a.x; hist[2 * tid + 1] = a.y;
  }
  if (u == 0) {
    if (tid == 0) cand_n[b] = 0;
    if (fill > 0) for (int e = tid; e < L; e += 1024) count[b * L + e] = fill;
  }
  __syncthreads();
  find_digit(hist, kBins, (int)((long long)l * Hkv * P), (int)batch.k[u], sm_scan, found);
  const int d = found[0];
  if (tid == 0) { RbState st; st.digit = d; st.need = found[1]; st.inside = (int)hist[d]; st.pad = 0; state[u * Bt + b] = st; }
  // one warp per layer: the layer's scores in the digits above
  for (int i = warp; i < l; i += 32) {
    const unsigned int* lh = layer_hist + ((size_t)i * Bt + b) * kBins;
    unsigned int a = 0;
#pragma unroll 8
    for (int bin = d + 1 + lane; bin < kBins; bin += 32) a += lh[bin];
    a = __reduce_add_sync(0xFFFFFFFFu, a);
    if (lane == 0) above[((size_t)u * Bt + b) * L + i] = a;
  }
}

// grid (slices, layers, Bt): one pass over the scores of the batch's layers.  A score whose digit is that of an update
// that includes its layer goes to the sample's candidate list as (pattern, layer).  The list has room for every score
// (cand_stride pairs per sample); its order is arbitrary, only counts are taken from it.  Matches are parked in shared
// memory, then the block reserves a range of the list with one atomic and copies them out.
// The update's three kernels, and in a pass the selection after them, are chains of block-wide steps that occupy few SMs, so each
// does what does not depend on the one before it while that runs.  To that end every one of them lets its successor start only
// after its own wait: a successor then knows, before it waits itself, that whatever came before its predecessor is complete and
// visible.  Here the scores, the first chunk of which is loaded before the wait.  (Passes of 4 layers of 1K 41.9 -> 38.3 us, of
// 14 layers of 3 x 5003 136.5 -> 130.0, of 32 of 8K 276.6 -> 268.1, together with select_gather_kernel
// counting digits early.)
__global__ void __launch_bounds__(kRbThreads)
rb_collect_kernel(const __grid_constant__ RbBatch batch, const float* scores, const RbState* state,
                  uint2* cand, unsigned int* cand_n, int Bt, size_t per_layer /* Hkv*P */, size_t cand_stride) {
  __shared__ uint32_t parked[kRbChunk];
  __shared__ unsigned int wanted[kBins / 32];
  __shared__ unsigned int s_cnt, s_base;
  const int b = blockIdx.z, i = blockIdx.y;
  const uint32_t* v = reinterpret_cast<const uint32_t*>(scores) + ((size_t)i * Bt + b) * per_layer;
  const size_t per_block = (per_layer + gridDim.x - 1) / gridDim.x;
  const size_t e0 = (size_t)blockIdx.x * per_block, e1 = e0 + per_block < per_layer ? e0 + per_block : per_layer;
  uint2* list = cand + (size_t)b * cand_stride;
  if (threadIdx.x < kBins / 32) wanted[threadIdx.x] = 0;
  uint32_t u[kRbChunk / kRbThreads];
  auto load = [&](size_t c0) {                                 // all loads of the chunk in flight together
#pragma unroll
    for (int j = 0; j < kRbChunk / kRbThreads; ++j) {
      const size_t e = c0 + threadIdx.x + (size_t)j * kRbThreads;
      u[j] = e < e1 ? v[e] : 0u;
    }
  };
  load(e0);
  pdl_wait();
  pdl_launch();
  __syncthreads();
  if (threadIdx.x < batch.n && batch.l[threadIdx.x] > i) {
    const int d = state[threadIdx.x * Bt + b].digit;
    atomicOr(&wanted[d >> 5], 1u << (d & 31));
  }
  for (size_t c0 = e0; c0 < e1; c0 += kRbChunk) {
    if (threadIdx.x == 0) s_cnt = 0;
    if (c0 > e0) load(c0);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kRbChunk / kRbThreads; ++j) {
      const size_t e = c0 + threadIdx.x + (size_t)j * kRbThreads;
      const int d = digit_of(u[j]);
      if (e < e1 && (wanted[d >> 5] >> (d & 31) & 1u)) parked[atomicAdd(&s_cnt, 1u)] = u[j];
    }
    __syncthreads();
    const unsigned int n = s_cnt;
    if (n) {
      if (threadIdx.x == 0) s_base = atomicAdd(&cand_n[b], n);
      __syncthreads();
      for (unsigned int x = threadIdx.x; x < n; x += kRbThreads) list[s_base + x] = make_uint2(parked[x], (unsigned int)i);
    }
    __syncthreads();
  }
}

// One cluster of kRbCluster blocks of 1024 threads per update and sample: exact T, per-layer hits, Eq. 5-6.  A list of
// up to kRbSolo candidates is left to the cluster's first block, a longer one (flat scores, many ties) is shared.
// cnt_i = hits of layer i among the K largest (ties at T to the lowest layers first);
// Z_i = floor(Bl*cnt_i/max cnt); Z'_i = floor(Z_i*N*L/sum Z); count_i = min(count_i, Z'_i).
// grid (kRbCluster, updates, Bt).  dbg_*: [Bt][L], of update `shown` (-1: none).  counts_out (single updates only): a copy.
__global__ void __launch_bounds__(1024)
rb_finish_kernel(const __grid_constant__ RbBatch batch, const RbState* state, const unsigned int* above,
                 const uint2* cand, const unsigned int* cand_n, size_t cand_stride, int* count,
                 int* dbg_cnt, int* dbg_z, int* dbg_zp, int shown, int* counts_out,
                 int Bt, int L, int Bl, int N, int prorata, int minmax) {
  namespace cg = cooperative_groups;
  __shared__ unsigned int hist[kBins], total_hist[kBins];
  __shared__ int sm_scan[33];
  __shared__ int found[2];
  __shared__ long long s_gt[128], s_eq[128];
  const int u = blockIdx.y, b = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, l = batch.l[u];
  const int rank = blockIdx.x;
  pdl_wait();
  pdl_launch();
  const RbState st = state[u * Bt + b];
  const unsigned int n = cand_n[b];
  const bool shared = n > kRbSolo;                           // the same for the whole cluster
  if (!shared && rank > 0) return;
  const unsigned int first = (shared ? rank * 1024 : 0) + tid, step = shared ? kRbCluster * 1024 : 1024;
  const uint2* list = cand + (size_t)b * cand_stride;
  // a counter array of every block in the cluster, added up in each block
  auto add_up = [&](const unsigned int* mine, unsigned int* sum, int len) {
    if (shared) cg::this_cluster().sync(); else __syncthreads();
    for (int j = tid; j < len; j += 1024) {
      unsigned int s = 0;
      if (shared) { for (int r = 0; r < kRbCluster; ++r) s += cg::this_cluster().map_shared_rank(const_cast<unsigned int*>(mine), r)[j]; }
      else s = mine[j];
      sum[j] = s;
    }
    if (shared) cg::this_cluster().sync(); else __syncthreads();
  };
  const uint32_t low0 = digit_low(st.digit), last0 = digit_last(st.digit);
  uint32_t low = low0, last = last0;
  int need = st.need, inside = st.inside;
  while (last > low) {
    const int shift = range_shift(low, last);
    hist[tid] = 0; hist[tid + 1024] = 0;
    __syncthreads();
#pragma unroll 4
    for (unsigned int e = first; e < n; e += step) {
      const uint2 c = list[e];
      if (c.x >= low && c.x <= last && (int)c.y < l) atomicAdd(&hist[(c.x - low) >> shift], 1u);
    }
    add_up(hist, total_hist, kBins);
    find_digit(total_hist, kBins, inside, need, sm_scan, found);
    inside = (int)total_hist[found[0]]; need = found[1];
    range_part(low, last, found[0], shift);
    __syncthreads();
  }
  const uint32_t T = low;
  long long ties = need;                                     // entries equal to T that are taken, lowest layers first
  for (int j = tid; j < 256; j += 1024) hist[j] = 0;         // [0, 128): above T inside the digit, [128, 256): equal to T
  __syncthreads();
#pragma unroll 4
  for (unsigned int e = first; e < n; e += step) {
    const uint2 c = list[e];
    if (c.x >= T && c.x <= last0 && (int)c.y < l) atomicAdd(&hist[c.y + (c.x == T ? 128 : 0)], 1u);
  }
  add_up(hist, total_hist, 256);
  if (rank > 0 || warp != 0) return;
  for (int i = lane; i < l; i += 32) {
    s_gt[i] = (long long)above[((size_t)u * Bt + b) * L + i] + total_hist[i];
    s_eq[i] = total_hist[128 + i];
  }
  __syncwarp();
  // Eq. 5-6 with one lane per layer (layers lane, lane + 32, ...): the ties go to the lowest layers first, i.e. layer i
  // takes min(eq_i, ties - sum of eq below i).
  const bool show = u == shown;
  long long carry = 0, cmax = 0, cmin = 0x7FFFFFFFFFFFFFFFll;
  for (int i0 = 0; i0 < l; i0 += 32) {
    const int i = i0 + lane;
    const long long eq = i < l ? s_eq[i] : 0;
    long long incl = eq;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o); if (lane >= o) incl += y; }
    const long long before = carry + incl - eq;
    long long take = ties - before;
    take = take < 0 ? 0 : (take < eq ? take : eq);
    if (i < l) {
      s_gt[i] += take;                      // = cnt_i
      if (show) dbg_cnt[b * L + i] = (int)s_gt[i];
      cmax = s_gt[i] > cmax ? s_gt[i] : cmax;
      cmin = s_gt[i] < cmin ? s_gt[i] : cmin;
    }
    carry += __shfl_sync(0xFFFFFFFFu, incl, 31);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { const long long y = __shfl_xor_sync(0xFFFFFFFFu, cmax, o); cmax = y > cmax ? y : cmax; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { const long long y = __shfl_xor_sync(0xFFFFFFFFu, cmin, o); cmin = y < cmin ? y : cmin; }
  if (cmax <= 0) cmax = 1;
  long long sumz = 0;
  for (int i = lane; i < l; i += 32) {
    // Z_i: counts scaled by their maximum, or (variant) min-max scaled; all layers equal under min-max -> Bl each
    if (minmax) s_eq[i] = cmax == cmin ? (long long)Bl : ((long long)Bl * (s_gt[i] - cmin)) / (cmax - cmin);
    else s_eq[i] = ((long long)Bl * s_gt[i]) / cmax;
    if (show) dbg_z[b * L + i] = (int)s_eq[i];
    sumz += s_eq[i];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sumz += __shfl_xor_sync(0xFFFFFFFFu, sumz, o);
  if (sumz <= 0) sumz = 1;
  const long long B = (long long)N * (prorata ? l : L);      // Eq. 6's budget (variant: of the layers seen so far)
  for (int i = lane; i < l; i += 32) {
    const long long zp = (s_eq[i] * B) / sumz;              // Z'_i
    const int zpi = zp > 0x7FFFFFFF ? 0x7FFFFFFF : (int)zp;
    if (show) dbg_zp[b * L + i] = zpi;
    atomicMin(&count[b * L + i], zpi);                       // other updates of the batch do the same
  }
  if (show) for (int i = l + lane; i < L; i += 32) { dbg_cnt[b * L + i] = 0; dbg_z[b * L + i] = 0; dbg_zp[b * L + i] = 0; }
  if (counts_out) {
    __threadfence();
    for (int i = lane; i < L; i += 32) counts_out[b * L + i] = *(volatile int*)&count[b * L + i];   // lanes read what they wrote
  }
}

}  // namespace dkv
