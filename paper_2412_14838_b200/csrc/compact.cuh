// Algorithm 1's buffer build (gather kept rows + window rows) and its progressive truncation
// (keep the best count_i of the held rows, window last).  Rows are kept in the order Algorithm 1's
// topk() yields them: score descending, ties by position.
#pragma once
#include "common.cuh"

namespace dkv {

constexpr int kGatherRows = 4;      // rows per thread, all loads issued before the stores

// One head's buffer rows: row r < n is source row sel[r] (shared or global memory), the ws window rows P .. S-1 follow.
// 16 bytes of K and of V per thread and row, `threads` threads (a multiple of vec = 16-byte pieces per row); `part` of
// `parts` sets of threads share the head.
__device__ __forceinline__ void gather_rows(const uint4* k_src, const uint4* v_src, uint4* kb,
                                            uint4* vb, const int* sel, int n, int bh, int S, int P, int ws,
                                            int row_stride /* rows per head in kb/vb */, int vec, int tid, int threads, int part, int parts) {
  const int per_pass = threads / vec, c = tid % vec, rows = n + ws;
  const size_t src0 = (size_t)bh * S * vec + c, dst0 = (size_t)bh * row_stride * vec + c;
  for (int row0 = part * per_pass * kGatherRows + tid / vec; row0 < rows; row0 += parts * per_pass * kGatherRows) {
    uint4 kv[kGatherRows], vv[kGatherRows];
#pragma unroll
    for (int j = 0; j < kGatherRows; ++j) {
      const int row = row0 + j * per_pass;
      if (row < rows) {
        const size_t from = src0 + (size_t)(row < n ? sel[row] : P + (row - n)) * vec;
        kv[j] = __ldcs(&k_src[from]);                             // read once: first in line for eviction from L2
        vv[j] = __ldcs(&v_src[from]);
      }
    }
#pragma unroll
    for (int j = 0; j < kGatherRows; ++j) {
      const int row = row0 + j * per_pass;
      if (row < rows) { kb[dst0 + (size_t)row * vec] = kv[j]; vb[dst0 + (size_t)row * vec] = vv[j]; }
    }
  }
}

// Gather of one layer with its current count: n = min(count[b][layer], sel_n) rows per head of idx, idx_stride apart;
// records held[b][layer] = n.  grid (row blocks, Bt*Hkv).
constexpr int kGatherThreads = 256;
__global__ void __launch_bounds__(kGatherThreads)
gather_rows_kernel(const uint4* k_src, const uint4* v_src, uint4* kb,
                   uint4* vb, const int* idx, const int* count, int sel_n, int idx_stride,
                   int S, int P, int ws, int row_stride, int vec, int* held, int Hkv, int L, int layer) {
  const int bh = blockIdx.y, b = bh / Hkv;
  pdl_launch();
  pdl_wait();
  const int n = min(count[b * L + layer], sel_n);
  if (threadIdx.x == 0 && blockIdx.x == 0 && bh % Hkv == 0) held[b * L + layer] = n;
  gather_rows(k_src, v_src, kb, vb, idx + (size_t)bh * idx_stride, n, bh, S, P, ws, row_stride, vec, threadIdx.x, kGatherThreads,
              blockIdx.x, gridDim.x);
}

// Per-layer device pointers of a pass.
struct PassPtrs {
  const void* k[128];
  const void* v[128];
  void* kb[128];
  void* vb[128];
};

// The valid rows (held[b][layer] + ws of the fixed stride) of every layer's and head's buffers from ptrs.k, ptrs.v to ptrs.kb, ptrs.vb, as the
// host-buffer pass delivers them into page-locked host memory: one launch, and the host need not know the counts.  (64 strided
// copies for 32 layers, which have to wait for the counts, took 0.2 ms of 6.7 longer.)  Bound by the bus.
// grid (row blocks of kGatherThreads / vec * kGatherRows, Bt*Hkv, layers).
__global__ void __launch_bounds__(kGatherThreads)
copy_valid_kernel(const __grid_constant__ PassPtrs ptrs, const int* held, int ws, int rows, int vec, int Hkv, int L) {
  const int bh = blockIdx.y, layer = blockIdx.z, per_pass = kGatherThreads / vec, c = threadIdx.x % vec;
  pdl_launch();
  pdl_wait();
  const int n = held[bh / Hkv * L + layer] + ws, row0 = blockIdx.x * per_pass * kGatherRows + threadIdx.x / vec;
  const size_t at = (size_t)bh * rows * vec + c;
  const uint4 *k = static_cast<const uint4*>(ptrs.k[layer]) + at, *v = static_cast<const uint4*>(ptrs.v[layer]) + at;
  uint4 *kb = static_cast<uint4*>(ptrs.kb[layer]) + at, *vb = static_cast<uint4*>(ptrs.vb[layer]) + at;
  uint4 kv[kGatherRows], vv[kGatherRows];
#pragma unroll
  for (int j = 0; j < kGatherRows; ++j) {
    const int row = row0 + j * per_pass;
    if (row < n) { kv[j] = k[(size_t)row * vec]; vv[j] = v[(size_t)row * vec]; }
  }
#pragma unroll
  for (int j = 0; j < kGatherRows; ++j) {
    const int row = row0 + j * per_pass;
    if (row < n) { kb[(size_t)row * vec] = kv[j]; vb[(size_t)row * vec] = vv[j]; }
  }
}

constexpr int kShrinkThreads = 256;

// In-place truncation of one (layer, sample, head, tensor): grid (Bt*Hkv, layers, 2).
// The buffers are in Algorithm 1's own order (score descending), so cutting a layer from `have` to
// `want` kept rows keeps the first `want` rows where they are; only the ws window rows move, from
// [have, have+ws) to [want, want+ws).  The two ranges may overlap (dst < src): rows are moved in
// blocks, each block read completely before it is written.  The last block of a (layer, sample) to arrive (a ticket
// each, zero between launches) records held[b][layer] = want: everyone has read the old value by then.
__global__ void __launch_bounds__(kShrinkThreads)
shrink_kernel(LayerPtrs ptrs, int layer0, const int* count, int* held, unsigned int* tickets,
              int Hkv, int L, int ws, int row_stride, int vec_per_row) {
  const int layer = layer0 + blockIdx.y;
  const int bh = blockIdx.x, b = bh / Hkv;
  pdl_launch();
  pdl_wait();
  const int have = held[b * L + layer];
  const int want = min(count[b * L + layer], have);
  if (want == have) return;                                  // the same for every block of the (layer, sample)
  uint4* buf = reinterpret_cast<uint4*>(blockIdx.z == 0 ? ptrs.kb[layer] : ptrs.vb[layer]) + (size_t)bh * row_stride * vec_per_row;
  const uint4* src = buf + (size_t)have * vec_per_row;
  uint4* dst = buf + (size_t)want * vec_per_row;
  const int n = ws * vec_per_row;
  for (int base = 0; base < n; base += kShrinkThreads) {
    const int e = base + threadIdx.x;
    uint4 val = make_uint4(0, 0, 0, 0);
    if (e < n) val = src[e];
    __syncthreads();
    if (e < n) dst[e] = val;
    __syncthreads();
  }
  if (threadIdx.x == 0) {                                    // the barriers above: the whole block has read `held`
    __threadfence();
    if (atomicAdd(&tickets[b * L + layer], 1u) == (unsigned int)(2 * Hkv - 1)) {
      tickets[b * L + layer] = 0;
      held[b * L + layer] = want;
    }
  }
}

// len_out[b][h] = held[b][layer] + ws
__global__ void write_len_kernel(int* __restrict__ len_out, const int* __restrict__ held, int Bt, int Hkv, int L, int layer, int ws) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= Bt * Hkv) return;
  len_out[e] = held[(e / Hkv) * L + layer] + ws;
}

}  // namespace dkv
