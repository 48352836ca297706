// Decoding over the compressed cache (Section 4.3: the decoding phase is the model's own attention, Eq. 1,
// run over what the prefill phase kept).  After Algorithm 1 every layer holds, per head, count_i kept rows
// followed by the ws window rows in a fixed-stride buffer, and count_i differs from layer to layer: the
// lengths are read from the device-side counts, nothing comes back to the host.
//
// The bytes that must move are the valid K and V rows, once; a step over one layer (2 MB) is bound by latency, one
// over all layers (50-70 MB) by HBM.  What kept the first version (dot products finished by warp shuffles, five per
// row and query; 200 us for four queries over 67 MB, 47 us for one over 47 MB, 13 us a call over one layer) from
// either was its instruction count, so both contractions run on the tensor pipe, in the warp-wide
// form (mma.sync m16n8k16): with 4 to 16 queries against blocks of 16 rows there is no 128-row tile to give to
// tcgen05, and operands go from global memory to registers without shared memory or a barrier.
//   S = Q K^T   A = queries (bf16 as given), B = K.  The order of the contracted dims is free, so a lane takes whole
//               16-byte chunks of a K row (4 lanes cover 64 contiguous bytes) and the queries are permuted alike.
//   O = P V     P is fp32.  It is split by truncation into three bf16 parts that add up to it exactly, so nothing is
//               lost against fp32 weights: up to 8 queries put the first two parts in the two halves of the 16-row
//               operand (one MMA) and the third in a second MMA; up to 16 queries take three MMAs.
// A warp works on 16 rows at a time with all its loads (K and V, 8 KB) in flight, keeps a running (max, sum) per
// query and the 16 x D result in registers; warps, blocks and clusters are then merged in a fixed order.
#pragma once
#include <cooperative_groups.h>
#include "common.cuh"

namespace dkv {

constexpr int kDecMaxLayers = 64;  // layers per launch (the pointers travel as a kernel argument)
constexpr int kDecRowBlock = 16;   // rows a warp takes at a time
constexpr int kDecMaxPairs = 1024; // (layer, sample) pairs whose lengths the split kernel can hold

struct DecodePtrs {                // per-layer device pointers, indexed by layer - layer0
  const void* q[kDecMaxLayers];
  const void* kb[kDecMaxLayers];
  const void* vb[kDecMaxLayers];
  float* out[kDecMaxLayers];
};

struct DecodeArgs {
  int layer0, nl, Bt, Hkv, GQ, L, ws, row_stride;
  float scale2;                    // log2(e) / sqrt(D)
  const int* held;                 // [Bt][L] kept rows of every layer; valid rows = held + ws
  float* scratch;                  // split kernel: [warps][2] partial results (DecodeWarp::save)
  unsigned int* tickets;           // split kernel: [nl][Bt*Hkv], zero before and after every launch
};

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// The upper halves (bf16 by truncation) of two floats, `a` in the low half; and what truncation leaves of a float.
__device__ __forceinline__ uint32_t pack_hi(float a, float b) { return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632); }
__device__ __forceinline__ float rest_of(float a) { return a - __uint_as_float(__float_as_uint(a) & 0xFFFF0000u); }
__device__ __forceinline__ uint4 ld_row16(const uint16_t* p) { return *reinterpret_cast<const uint4*>(p); }

// Asks for a 128-byte line to be brought to L2.  Nothing is read: a write that comes later finds its line there, so this may
// stand before pdl_wait.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// State of one warp: QB (8 or 16) queries against the rows it has seen.  Lane (g, t) = (lane / 4, lane % 4) holds
// queries g (and g + 8), output dims 64*(j/8) + 16 t + {j%8, 8 + j%8}, j < D/8.
template <int D, int QB>
struct DecodeWarp {
  static constexpr int kChunks = D / 32;       // 16-byte chunks of a row per lane in S = Q K^T
  static constexpr int kTiles = D / 8;         // 8-column tiles of the result
  static constexpr int kHalves = QB / 8;       // queries per lane
  uint4 q[kHalves][kChunks];
  float acc[kTiles][4];
  float m[kHalves], l[kHalves];

  // Queries [c0, c0 + QB) of the head group, those past GQ as zeros.
  __device__ __forceinline__ void start(const uint16_t* qbase, int c0, int GQ, int g, int t) {
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      const int row = c0 + g + 8 * h;
#pragma unroll
      for (int c = 0; c < kChunks; ++c)
        q[h][c] = row < GQ ? *reinterpret_cast<const uint4*>(qbase + (size_t)row * D + (c * 4 + t) * 8) : make_uint4(0, 0, 0, 0);
    }
    clear();
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int h = 0; h < kHalves; ++h) { m[h] = -INFINITY; l[h] = 0.f; }
#pragma unroll
    for (int j = 0; j < kTiles; ++j) { acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f; }
  }

  // The K and V chunks this lane takes of rows [r, r + 16); rows past `last` are read as `last`.
  struct Rows {
    uint4 kf[2][kChunks], vf[4][D / 64];
    __device__ __forceinline__ void load(const uint16_t* kbase, const uint16_t* vbase, int r, int last, int g, int t) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint16_t* kr = kbase + (size_t)min(r + 8 * i + g, last) * D + t * 8;
#pragma unroll
        for (int c = 0; c < kChunks; ++c) kf[i][c] = ld_row16(kr + c * 32);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {            // rows 2t, 2t + 1, 2t + 8, 2t + 9: the pairs an operand register holds
        const uint16_t* vr = vbase + (size_t)min(r + 2 * t + (i & 1) + (i >> 1) * 8, last) * D + g * 8;
#pragma unroll
        for (int c = 0; c < D / 64; ++c) vf[i][c] = ld_row16(vr + c * 64);
      }
    }
    // Values of rows from r1 on become zero (what the buffers hold there is unspecified and could be a NaN).
    __device__ __forceinline__ void clear_past(int r, int r1, int t) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (r + 2 * t + (i & 1) + (i >> 1) * 8 >= r1) {
#pragma unroll
          for (int c = 0; c < D / 64; ++c) vf[i][c] = make_uint4(0, 0, 0, 0);
        }
    }
  };

  // Rows [r, min(r + 16, r1)), r < r1, from x.
  __device__ __forceinline__ void add(const Rows& x, int r, int r1, float scale2, int t) {
    float s[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      s[i][0] = s[i][1] = s[i][2] = s[i][3] = 0.f;
#pragma unroll
      for (int c = 0; c < kChunks; ++c) {
        const uint4 q0 = q[0][c], q1 = QB == 16 ? q[kHalves - 1][c] : make_uint4(0, 0, 0, 0);
        mma_bf16_16816(s[i], q0.x, q1.x, q0.y, q1.y, x.kf[i][c].x, x.kf[i][c].y);
        mma_bf16_16816(s[i], q0.z, q1.z, q0.w, q1.w, x.kf[i][c].z, x.kf[i][c].w);
      }
    }
    uint32_t ph[kHalves][2], pm[kHalves][2], pl[kHalves][2];    // three parts of the weights: [query half][rows 2t / 2t + 8]
    float corr[kHalves];
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      float p[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = r + 2 * t + (i & 1) + (i >> 1) * 8;
        p[i] = row < r1 ? s[i >> 1][2 * h + (i & 1)] * scale2 : -INFINITY;
      }
      float mn = fmaxf(fmaxf(p[0], p[1]), fmaxf(p[2], p[3]));
      mn = fmaxf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, 1));
      mn = fmaxf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, 2));
      mn = fmaxf(mn, m[h]);
      corr[h] = fast_exp2(m[h] - mn);          // 0 on the first rows (m = -inf)
      m[h] = mn;
#pragma unroll
      for (int i = 0; i < 4; ++i) p[i] = fast_exp2(p[i] - mn);
      l[h] = l[h] * corr[h] + ((p[0] + p[1]) + (p[2] + p[3]));
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float a = p[2 * i], b = p[2 * i + 1], ra = rest_of(a), rb = rest_of(b);
        ph[h][i] = pack_hi(a, b); pm[h][i] = pack_hi(ra, rb); pl[h][i] = pack_hi(rest_of(ra), rest_of(rb));
      }
    }
#pragma unroll
    for (int j = 0; j < kTiles; ++j) {
      const int c = j >> 3, w = (j & 7) >> 1;
      const uint32_t sel = j & 1 ? 0x7632 : 0x5410;
      auto word = [&](int i) { return w == 0 ? x.vf[i][c].x : w == 1 ? x.vf[i][c].y : w == 2 ? x.vf[i][c].z : x.vf[i][c].w; };
      const uint32_t b0 = __byte_perm(word(0), word(1), sel), b1 = __byte_perm(word(2), word(3), sel);
      acc[j][0] *= corr[0]; acc[j][1] *= corr[0]; acc[j][2] *= corr[kHalves - 1]; acc[j][3] *= corr[kHalves - 1];
      if constexpr (QB == 8) {
        mma_bf16_16816(acc[j], ph[0][0], pm[0][0], ph[0][1], pm[0][1], b0, b1);
        mma_bf16_16816(acc[j], pl[0][0], 0u, pl[0][1], 0u, b0, b1);
      } else {
        mma_bf16_16816(acc[j], ph[0][0], ph[1][0], ph[0][1], ph[1][1], b0, b1);
        mma_bf16_16816(acc[j], pm[0][0], pm[1][0], pm[0][1], pm[1][1], b0, b1);
        mma_bf16_16816(acc[j], pl[0][0], pl[1][0], pl[0][1], pl[1][1], b0, b1);
      }
    }
  }

  // Every lane's sums become those of all rows the warp has seen.
  __device__ __forceinline__ void finish() {
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      l[h] += __shfl_xor_sync(0xFFFFFFFFu, l[h], 1);
      l[h] += __shfl_xor_sync(0xFFFFFFFFu, l[h], 2);
    }
    if constexpr (QB == 8) {
#pragma unroll
      for (int j = 0; j < kTiles; ++j) { acc[j][0] += acc[j][2]; acc[j][1] += acc[j][3]; }
    }
  }
  // Piece k (four consecutive dims of query g + 8 h) of the finished result, k = 0 .. kTiles/2 - 1, and its first dim.
  __device__ __forceinline__ float4 piece(int h, int k) const {
    const int j = (k >> 1) * 4, i = 2 * h + (k & 1);
    return make_float4(acc[j][i], acc[j + 1][i], acc[j + 2][i], acc[j + 3][i]);
  }
  __device__ __forceinline__ static int piece_dim(int k, int t) { const int j = (k >> 1) * 4; return 64 * (j >> 3) + 16 * t + (j & 7) + 8 * (k & 1); }
  // Results as rows in part[QB][D + 4], and (max, sum) per query.
  __device__ __forceinline__ void park(float* part, float2* ml, int g, int t) {
    finish();
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      if (t == 0) ml[g + 8 * h] = make_float2(m[h], l[h]);
#pragma unroll
      for (int k = 0; k < kTiles / 2; ++k) *reinterpret_cast<float4*>(part + (g + 8 * h) * (D + 4) + piece_dim(k, t)) = piece(h, k);
    }
  }
  // Finished results of queries [c0, c0 + QB) to out [GQ][D].
  __device__ __forceinline__ void store(float* out, int c0, int GQ, int g, int t) const {
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      const int row = c0 + g + 8 * h;
      if (row < GQ) {
        const float inv = 1.f / l[h];
#pragma unroll
        for (int k = 0; k < kTiles / 2; ++k) {
          const float4 v = piece(h, k);
          *reinterpret_cast<float4*>(out + (size_t)row * D + piece_dim(k, t)) = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
        }
      }
    }
  }
  // A finished result as it lies in the registers: [kHalves][kTiles/2][32] pieces, then [kHalves][8] (max, sum).
  static constexpr int kPartFloats = QB * D + QB * 2;
  __device__ __forceinline__ void save(float* part, int c0, int GQ, int lane, int g, int t) const {
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      if (c0 + g + 8 * h >= GQ) continue;
      if (t == 0) *reinterpret_cast<float2*>(part + QB * D + (h * 8 + g) * 2) = make_float2(m[h], l[h]);
#pragma unroll
      for (int k = 0; k < kTiles / 2; ++k) __stcg(reinterpret_cast<float4*>(part) + (h * (kTiles / 2) + k) * 32 + lane, piece(h, k));
    }
  }
  // Merges a saved result; all its loads are in flight together (one warp merges a head's parts, so the latencies add
  // up: 17 parts of 16 queries took 15 us with half of a part in flight).
  __device__ __forceinline__ void add_saved(const float* part, int c0, int GQ, int lane, int g) {
    float4 v[kHalves][kTiles / 2];
    float2 ml[kHalves];
#pragma unroll
    for (int h = 0; h < kHalves; ++h)
      if (c0 + g + 8 * h < GQ) {
        ml[h] = __ldcg(reinterpret_cast<const float2*>(part + QB * D + (h * 8 + g) * 2));
#pragma unroll
        for (int k = 0; k < kTiles / 2; ++k) v[h][k] = __ldcg(reinterpret_cast<const float4*>(part) + (h * (kTiles / 2) + k) * 32 + lane);
      }
#pragma unroll
    for (int h = 0; h < kHalves; ++h)
      if (c0 + g + 8 * h < GQ) {
        const float mn = fmaxf(m[h], ml[h].x), s0 = fast_exp2(m[h] - mn), s1 = fast_exp2(ml[h].x - mn);   // every part has rows: finite
        m[h] = mn;
        l[h] = l[h] * s0 + ml[h].y * s1;
#pragma unroll
        for (int k = 0; k < kTiles / 2; ++k) {
          const int j = (k >> 1) * 4, x = 2 * h + (k & 1);
          const float4 y = v[h][k];
          acc[j][x] = acc[j][x] * s0 + y.x * s1; acc[j + 1][x] = acc[j + 1][x] * s0 + y.y * s1;
          acc[j + 2][x] = acc[j + 2][x] * s0 + y.z * s1; acc[j + 3][x] = acc[j + 3][x] * s0 + y.w * s1;
        }
      }
  }
};

// One 4-value piece x (query qi = x / (D/4)) of the warps' parked results, merged in warp order: value sums, and the
// query's (max, sum); max = -inf: no rows.
template <int D, int QB, int NW>
__device__ __forceinline__ float2 merge_warps(const float* part, const float2* ml, int x, float4& v) {
  const int qi = x / (D / 4), d = x % (D / 4) * 4;
  float mm = -INFINITY, l = 0.f;
  float2 p[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) { p[w] = ml[w * QB + qi]; mm = fmaxf(mm, p[w].x); }
  v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (mm > -INFINITY) {
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float s = fast_exp2(p[w].x - mm);
      const float4 y = *reinterpret_cast<const float4*>(part + (w * QB + qi) * (D + 4) + d);
      v.x = fmaf(y.x, s, v.x); v.y = fmaf(y.y, s, v.y); v.z = fmaf(y.z, s, v.z); v.w = fmaf(y.w, s, v.w);
      l = fmaf(p[w].y, s, l);
    }
  }
  return make_float2(mm, l);
}

// Running merge of partial results (value sums relative to their max, max, sum).
struct DecodeMerge {
  float m = -INFINITY, l = 0.f;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  __device__ __forceinline__ void add(float2 ml, float4 y) {
    const float mn = fmaxf(m, ml.x);
    if (mn == -INFINITY) return;
    const float s0 = fast_exp2(m - mn), s1 = fast_exp2(ml.x - mn);
    v.x = v.x * s0 + y.x * s1; v.y = v.y * s0 + y.y * s1; v.z = v.z * s0 + y.z * s1; v.w = v.w * s0 + y.w * s1;
    l = l * s0 + ml.y * s1;
    m = mn;
  }
  __device__ __forceinline__ void store(float* out) const {
    *reinterpret_cast<float4*>(out) = make_float4(v.x / l, v.y / l, v.z / l, v.w / l);
  }
};

// Few heads (a step over one layer or a few): one cluster of gridDim.x blocks per head, its row blocks dealt out to
// all warps of the cluster.  Every block pushes the pieces of its result into the shared memory of the block that
// owns the piece, so one cluster barrier is all the merge waits for.  With 8 heads of 500 rows every warp has at most
// one or two row blocks: a call is one round of loads plus the merge.  It is the device that bounds a step made of such
// calls: 5.1 us a call with the queue full (8 heads of about 500 rows, colder than L2), where the host needs 3.1.  A block that
// starts while the kernel before it still runs asks for its rows to be brought to L2 meanwhile (5.4 -> 5.1).
// grid (cluster size <= 8, Bt*Hkv, layers).
template <int D, int QB, int NW>
__global__ void __launch_bounds__(NW * 32)
decode_cluster_kernel(const __grid_constant__ DecodePtrs ptrs, const __grid_constant__ DecodeArgs a) {
  namespace cg = cooperative_groups;
  constexpr int kPieces = QB * D / 4;
  __shared__ __align__(16) float part_s[NW * QB * (D + 4)];
  __shared__ float2 ml_s[NW * QB];
  __shared__ __align__(16) float4 recv_v[kPieces + 8];       // [block][piece of this block's share]
  __shared__ float2 recv_ml[kPieces + 8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int cs = gridDim.x, rank = blockIdx.x, bh = blockIdx.y, lz = blockIdx.z, b = bh / a.Hkv;
  pdl_launch();
  if (cs > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // the others have started: see below
  const uint16_t* kbase = static_cast<const uint16_t*>(ptrs.kb[lz]) + (size_t)bh * a.row_stride * D;
  const uint16_t* vbase = static_cast<const uint16_t*>(ptrs.vb[lz]) + (size_t)bh * a.row_stride * D;
  const uint16_t* qbase = static_cast<const uint16_t*>(ptrs.q[lz]) + (size_t)bh * a.GQ * D;
  {
    // the warp's first rows, on their way to L2 while the kernel before this one ends: whoever writes them writes there
    const int r0 = (rank * NW + warp) * kDecRowBlock, lines = (min(r0 + kDecRowBlock, a.row_stride) - r0) * D / 64;   // < 0: no rows
    for (int i = lane; i < lines; i += 32) {
      prefetch_l2(kbase + (size_t)r0 * D + i * 64);
      prefetch_l2(vbase + (size_t)r0 * D + i * 64);
    }
    if (rank == 0 && threadIdx.x * 64 < a.GQ * D) prefetch_l2(qbase + threadIdx.x * 64);
  }
  pdl_wait();
  float* out = ptrs.out[lz] + (size_t)bh * a.GQ * D;
  const int step = cs * NW * kDecRowBlock;
  for (int c0 = 0; c0 < a.GQ; c0 += QB) {
    DecodeWarp<D, QB> w;
    typename DecodeWarp<D, QB>::Rows x;
    int r = (rank * NW + warp) * kDecRowBlock;
    // the first rows are requested together with the head's length, without waiting for it
    x.load(kbase, vbase, r, a.row_stride - 1, g, t);
    const int len = a.held[b * a.L + a.layer0 + lz] + a.ws;
    w.start(qbase, c0, a.GQ, g, t);
    if (r < len && r + kDecRowBlock > len) x.clear_past(r, len, t);
    for (; r < len; r += step) {
      typename DecodeWarp<D, QB>::Rows next;
      if (r + step < len) next.load(kbase, vbase, r + step, len - 1, g, t);
      w.add(x, r, len, a.scale2, t);
      x = next;
    }
    w.park(part_s + warp * QB * (D + 4), ml_s + warp * QB, g, t);
    __syncthreads();
    // no block writes into another before that one has started (first chunk) or read what it last got (later ones)
    if (cs > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    const int pieces = min(QB, a.GQ - c0) * (D / 4), share = (pieces + cs - 1) / cs;
    for (int x = threadIdx.x; x < pieces; x += NW * 32) {
      float4 v;
      const float2 ml = merge_warps<D, QB, NW>(part_s, ml_s, x, v);
      const int to = x / share, at = rank * share + x % share;
      float4* dv = cs > 1 ? cg::this_cluster().map_shared_rank(recv_v, to) : recv_v;
      float2* dm = cs > 1 ? cg::this_cluster().map_shared_rank(recv_ml, to) : recv_ml;
      dv[at] = v; dm[at] = ml;
    }
    if (cs > 1) cg::this_cluster().sync(); else __syncthreads();
    for (int x = rank * share + threadIdx.x; x < min(pieces, (rank + 1) * share); x += NW * 32) {
      DecodeMerge r;
#pragma unroll
      for (int p = 0; p < 8; ++p) if (p < cs) r.add(recv_ml[p * share + x - rank * share], recv_v[p * share + x - rank * share]);
      r.store(out + (size_t)c0 * D + x * 4);
    }
    if (c0 + QB < a.GQ) {
      if (cs > 1) asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
      __syncthreads();
    }
  }
}

// Many heads (a step over all layers): the 16-row blocks of all heads form one sequence, (layer, sample) pairs in
// order, cut into one equal slice per WARP, so that the layers' different lengths leave nothing idle and nothing waits
// at a block barrier (with a slice per thread block, two thirds of the instructions of a step over short heads went
// into merging warps).  A head counts kDecHeadCost blocks more than it has: its set-up and its results.  A head that
// lies in one slice is finished there; of the others every warp leaves its part in scratch, as it lies in its
// registers, and the warp that arrives last for a head (a ticket per head) merges the parts in slice order.
// Two blocks of four warps an SM: at the 255 registers that leaves (254 used at most) nothing spills; three at 168 were
// 8 % slower, and requesting the next row block before the current one is worked on gains nothing here.  Measured (32
// layers, caches colder than L2): 32 us for four queries over 67 MB, 21 us for one over 47 MB of 1024 short heads, where
// the launch, the lengths' prefix sums and two or three heads' load latencies per warp are most of the time.
// Dynamic shared memory: nl*Bt + 1 integers.
constexpr int kDecHeadCost = 2;   // 1 to 4 measured: within 1 %, 3 and 4 slower for short heads
template <int D, int QB, int NW>
__global__ void __launch_bounds__(NW * 32, 2)
decode_split_kernel(const __grid_constant__ DecodePtrs ptrs, const __grid_constant__ DecodeArgs a) {
  using Warp = DecodeWarp<D, QB>;
  extern __shared__ int prefix_s[];                        // units (blocks and head costs) before pair i
  __shared__ int scan_s[NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int pairs = a.nl * a.Bt, BH = a.Bt * a.Hkv;
  pdl_launch();
  pdl_wait();
  auto units_of = [&](int i) {
    const int len = a.held[(i % a.Bt) * a.L + a.layer0 + i / a.Bt] + a.ws;
    return ((len + kDecRowBlock - 1) / kDecRowBlock + kDecHeadCost) * a.Hkv;
  };
  {
    const int per = (pairs + NW * 32 - 1) / (NW * 32), i0 = min(pairs, tid * per), i1 = min(pairs, i0 + per);
    int mine = 0;
    for (int i = i0; i < i1; ++i) mine += units_of(i);
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int y = __shfl_up_sync(0xFFFFFFFFu, inc, o); if (lane >= o) inc += y; }
    if (lane == 31) scan_s[warp] = inc;
    __syncthreads();
    int at = inc - mine;
    for (int w = 0; w < warp; ++w) at += scan_s[w];
    for (int i = i0; i < i1; ++i) { prefix_s[i] = at; at += units_of(i); }
    if (i0 < i1 && i1 == pairs) prefix_s[pairs] = at;
    __syncthreads();
  }
  // no more slices than units: an empty slice would leave no part, and whoever merges a head counts on one from each
  const int total = prefix_s[pairs], slices = min((int)gridDim.x * NW, total), own = blockIdx.x * NW + warp;
  if (own >= slices) return;
  auto slice = [&](int c) { return (int)((long long)total * c / slices); };
  auto owner = [&](int u) { return (int)(((long long)(u + 1) * slices + total - 1) / total) - 1; };   // slice that holds u
  const int u1 = slice(own + 1), chunks = (a.GQ + QB - 1) / QB;
  for (int u = slice(own); u < u1;) {
    int lo = 0, hi = pairs - 1;
    while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (prefix_s[mid] <= u) lo = mid; else hi = mid - 1; }
    const int units = (prefix_s[lo + 1] - prefix_s[lo]) / a.Hkv, h = (u - prefix_s[lo]) / units;
    const int row0 = prefix_s[lo] + h * units + kDecHeadCost;             // unit of the head's first row block
    const int e = min(u1, row0 - kDecHeadCost + units), lz = lo / a.Bt, b = lo % a.Bt, bh = b * a.Hkv + h;
    const int first = max(0, u - row0), after = e - row0;                 // row blocks [first, after) of the head
    u = e;
    if (after <= 0) continue;                                             // this slice has the head's cost only
    const bool whole = first == 0 && after == units - kDecHeadCost;
    const int len = a.held[b * a.L + a.layer0 + lz] + a.ws, r_end = min(len, after * kDecRowBlock);
    const uint16_t* kbase = static_cast<const uint16_t*>(ptrs.kb[lz]) + (size_t)bh * a.row_stride * D;
    const uint16_t* vbase = static_cast<const uint16_t*>(ptrs.vb[lz]) + (size_t)bh * a.row_stride * D;
    const uint16_t* qbase = static_cast<const uint16_t*>(ptrs.q[lz]) + (size_t)bh * a.GQ * D;
    float* out = ptrs.out[lz] + (size_t)bh * a.GQ * D;
    // parts: slot 0 of a slice continues a head, slot 1 begins one that others continue
    auto part = [&](int c, int slot, int chunk) { return a.scratch + ((size_t)(2 * c + slot) * chunks + chunk) * Warp::kPartFloats; };
    for (int c0 = 0, ch = 0; c0 < a.GQ; c0 += QB, ++ch) {
      Warp w;
      w.start(qbase, c0, a.GQ, g, t);
      for (int r = first * kDecRowBlock; r < r_end; r += kDecRowBlock) {
        typename Warp::Rows x;
        x.load(kbase, vbase, r, r_end - 1, g, t);
        w.add(x, r, r_end, a.scale2, t);
      }
      w.finish();
      if (whole) w.store(out, c0, a.GQ, g, t);
      else w.save(part(own, first == 0, ch), c0, a.GQ, lane, g, t);
    }
    if (whole) continue;
    const int c_lo = owner(row0), c_hi = owner(row0 - kDecHeadCost + units - 1);
    unsigned int* ticket = a.tickets + (size_t)lz * BH + bh;
    __threadfence();
    __syncwarp();
    unsigned int arrived = 0;
    if (lane == 0) arrived = atomicAdd(ticket, 1u);
    if (__shfl_sync(0xFFFFFFFFu, arrived, 0) != (unsigned int)(c_hi - c_lo)) continue;
    __threadfence();
    for (int c0 = 0, ch = 0; c0 < a.GQ; c0 += QB, ++ch) {
      Warp w;
      w.clear();
      for (int c = c_lo; c <= c_hi; ++c) w.add_saved(part(c, c == c_lo, ch), c0, a.GQ, lane, g);
      w.store(out, c0, a.GQ, g, t);
    }
    if (lane == 0) *ticket = 0;
  }
}

// ------------------------------------------------------------------------------------------------------
// Fixed-pattern budgets (the methods the paper compares with, Section 5.1 "Baselines", as policies only).

// count[b][i] = min(count[b][i], schedule_i); schedule: policy 0 = N in every layer, policy 1 = the pyramid
// N + floor(N (L-1-2i) / (2 (L-1))) (floor towards minus infinity; N when L = 1).
__global__ void policy_counts_kernel(int* __restrict__ count, int* __restrict__ counts_out, int Bt, int L, int N, int policy) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= Bt * L) return;
  const int i = e % L;
  long long want = N;
  if (policy == 1 && L > 1) {
    const long long num = (long long)N * (L - 1 - 2 * i), den = 2ll * (L - 1);
    want = N + (num >= 0 ? num / den : -((-num + den - 1) / den));
  }
  const int c = count[e];
  const int v = want < c ? (int)want : c;
  count[e] = v;
  if (counts_out) counts_out[e] = v;
}

// Kept positions without scores: the first n_sink and the last n_recent prefix positions of every head,
// ascending (sinks plus a window of the most recent tokens).  idx [Bt*Hkv][idx_stride]; count[b][layer] = n.
__global__ void positions_kernel(int* __restrict__ idx, int* __restrict__ count, int P, int idx_stride, int n_sink,
                                 int first_recent, int n, int Hkv, int L, int layer) {
  const int bh = blockIdx.y;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e == 0 && bh % Hkv == 0) count[(bh / Hkv) * L + layer] = n;
  if (e >= n) return;
  idx[(size_t)bh * idx_stride + e] = e < n_sink ? e : first_recent + (e - n_sink);
}

}  // namespace dkv
