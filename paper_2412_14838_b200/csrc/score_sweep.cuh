// Window scoring (Eq. 1-2) of many heads: row sums, then key sums, each one launch over the keys of up to 32 layers.
//
// A token's score is sum over window rows r of 2^(t_rj) / l_r with l_r = sum over keys of 2^(t_rj): the normalisers are only
// known when a head's last key has been seen, so the keys are swept twice (once where the caller has the log-denominators).
//
//   tile      128 keys of one head: logits^T = K . Q_win^T on the tensor cores, one TMEM lane a key, one column a window row
//             (at most 128 rows, rounded up to 16; up to 256 rows are two PLANES whose sums are added by pool_kernel).  Rounded up
//             to 32, 72 and 224 rows cost more: 14 layers of 3 x 5003 131.4 us against 124.0, 28 of 16K 454 against 390.
//   pipes     a block has two, each with its own contiguous range of the tiles, in SEGMENTS of one head, its own slots, copies,
//             MMAs, accumulator stages and eight warps for exponentials.
//   warps     0-7 and 8-15 exponentials of either pipe, 16 and 17 its copies, 18 and 19 its MMAs, 20 and 21 log-denominators of
//             its next segment, 22 and 23 publish its row sums.
//
// Tensor memory is read in the 16x256b shape: a thread has 2 keys x 2 rows of a block of 16 lanes x 8 columns.  Row sums of a
// warp (32 keys of a tile x half of the rows) are relative to references that are in registers, and are added in registers for
// a whole segment; key sums need 2 shuffles a tile.
//
// Row sums are e = 2^(t - m) with m the logit of the first key that the warp has seen in the segment: as that key counts with
// e = 1, no maximum is searched, and a sum only fails where another logit is 127 bits above it (or is infinite, or a NaN).  It is
// infinite or a NaN then, and the pipe sweeps that segment twice more when it has come to its end, for the largest logits and for
// sums relative to them (a pass of 32 layers of 32K, 8 heads of 128, 128 rows: 0.83 ms, with one such head 1.12, with all of them
// 3.15; by the ordinary cores, row by row on the block that had the segment, 18.8 and 70).
//
// What bounds it: a tile takes an SM 0.7 (row sums) and 0.8 us (key sums), 5.9-6.8 TB/s, near the 6.5 of a copy, in the launches
// of eight layers of 32K; a whole pass over 32K runs at the power limit, 0.95 us a tile.  The softmax loops bound what is in L2:
// 32 layers of 16K that share one K, 8 heads of 128, 128 rows, take 0.69 us a tile for the row sums, of which the special-function
// unit alone needs 0.55 (1024 clocks of 1.8-1.9 GHz); from HBM 0.76.  A launch takes 5 us to its first logits and
// about 10 in all beside its tiles, most of it instructions that are fetched for the first time: with the loops unrolled over
// a whole tile it took 15, and with two streams of long loops (row sums in one pipe, key sums in the other) a tile took twice as long.
//
// Against score_tc.cuh (us a pass): 14 layers of 3 x 5003, 6 heads of 64, 72 rows 166 -> 131; 16 layers of 16K, 4 heads of 64,
// 32 / 96 / 128 / 192 rows 118 / 149 / 155 / 220 -> 107 / 123 / 139 / 186; 28 of 2 x 2K, 4 heads of 128, 96 / 192 / 256 rows
// 114 / 153 / 162 -> 102 / 138 / 151; 32 layers of 32K, 8 heads of 128, with log-denominators 572 -> 530-554.  28 layers of 16K, 4 heads
// of 128, 224 rows: 415-423 -> 388-422, mostly at the power limit, where they are equal.
#pragma once
#include <limits.h>
#include <type_traits>
#include "score_tc.cuh"

namespace dkv {
namespace sweep {

using namespace tc;

constexpr int kTile = kTileKeys;
constexpr int kLaneWarps = 8;                    // warps on a tile, 16 lanes each
constexpr int kSoftWarps = 16, kCopyWarp = 16, kMmaWarp = 18, kRowWarp = 20, kPublishWarp = 22;
constexpr int kWarps = 24, kOneThreads = kWarps * 32;
// Registers a thread: 80 at launch; the four warpgroups with the exponentials take what the other two give (4 x 96 + 2 x 48 = 6 x 80).
constexpr int kSoftRegs = 96, kOtherRegs = 48;
// kGivenSums: key sums with the caller's log-denominators; kLongRowSums: row sums of heads with more than kRowTiles tiles
enum Sweep { kRowSums, kKeySums, kGivenSums, kLongRowSums };

// Tiles whose row sums a thread adds one after the other, four additions each; longer segments are cut there and their parts added by
// the warps that publish them.  296 heads of 262144 keys, logits of standard deviation 3: error of the scores (2-norm) 6.9e-6 uncut,
// 8.7e-7 cut (score_tc.cuh 1.2e-6); of 32768 keys 9.2e-7.  A build of its own, as the cut in that of shorter heads made a pass of
// four layers of 1K 0.7 us longer (39.5 -> 40.2).
constexpr int kRowTiles = 256;

constexpr int kSlots = 3, kSlotBytes = 2 * kHalfBytes;      // of a pipe: queries, two tiles of keys

// NB: 8-column blocks of window rows (even, at most 16)
template <int NB>
struct Shape1 {
  static constexpr int kCols = 8 * NB;                                      // accumulator columns of a tile
  static constexpr int kPer = NB <= 8 ? 4 : 2;                              // accumulator stages of a pipe,
  static constexpr int kStage = (kCols + 31) / 32 * 32;                     // this many columns apart
  static constexpr int kQBytes = kCols * 128;                               // window rows x 64 dims
  static constexpr int kPipeBars = 2 * kSlots + 2 * kPer + 6, kBars = 2 * kPipeBars;
  static constexpr int kSmem = 1024 + 2 * kSlots * kSlotBytes + 2 * 4 * kCols * 8 + 3 * 2 * kCols * 4 + kBars * 8;
  static_assert(kSmem + 1024 <= 227 * 1024 && 2 * kPer * kStage <= 512, "shared and tensor memory of an SM");
};

struct Args {
  int S, P, ws, M, D;
  int planes, plane_rows;       // 1 or 2; window rows of a plane: of two the first plane_rows and the last
  int tph;                      // tiles of a head
  int hpl, vheads;              // heads of a layer; (head, plane) pairs of the launch
  float scale2;                 // log2(e) / sqrt(D)
  float post;                   // factor on the sums before they are written
  uint32_t idesc;
  float* raw;                   // [vheads][tph * 128] unpooled scores
  float2* stats;                // [vheads][slots][plane_rows] (m, sum) of a head's segments
  int slots;
  unsigned int* hist;           // null, or counters to clear
  size_t hist_n;
  int* status;
  long long wait_cycles, segment_cycles;      // limits of a wait, for a tile and for a segment
  int withhold_tile;            // test hook: block 0 never loads its tile of this number (-1: off)
};

struct Layers {                                // by layer of the launch
  CUtensorMap q[kMaxGroup], k[kMaxGroup];
  const float* lse[kMaxGroup];
};

// ------------------------------------------------------------------------------------------ PTX
// N = 1 to 8 blocks of 8 columns x 16 lanes (N that are no power of two by several loads).  Register 4 b + 2 i + j: block b, lane (key) laneid / 4 + 8 i, column 2 (laneid % 4) + j.
template <int N>
__device__ __forceinline__ void ld_block(uint32_t a, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  if constexpr (N > 4 && N < 8) {
    ld_block<4>(a, v);
    ld_block<N - 4>(a + 32, v + 16);
  } else if constexpr (N == 3) {
    ld_block<2>(a, v);
    ld_block<1>(a + 16, v + 8);
  } else if constexpr (N == 1)
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
  else if constexpr (N == 2)
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(a));
  else if constexpr (N == 4)
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(a));
  else
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]) : "r"(a));
}

// ------------------------------------------------------------------------------------------ order of work
// The segments of a range of the tiles: the range cut at the heads, and after kMost tiles of one.
template <int kMost>
struct Segs {
  int g, end, tph;                              // what is left of the range
  int vh, t0, n;                                // the segment: (head, plane), first tile, tiles
  __device__ Segs(int g_, int end_, int tph_) : g(g_), end(end_), tph(tph_), n(0) {
    vh = g / tph;
    t0 = g - vh * tph;
    --vh;                                       // next() begins with it
  }
  // those of one pipe
  __device__ Segs(const Args& a, int pipe, int pipes)
      : Segs((int)((long long)a.vheads * a.tph * pipe / pipes), (int)((long long)a.vheads * a.tph * (pipe + 1) / pipes), a.tph) {}
  __device__ bool next() {
    if (g >= end) return false;
    if (kMost < INT_MAX && n && t0 + n < tph) {
      t0 += n;
    } else {
      if (n) t0 = 0;
      ++vh;
    }
    n = min(min(tph - t0, kMost), end - g);
    g += n;
    return true;
  }
};
// Places [0, n) in turn, and the parity of the phase to wait for.
struct Ring {
  int s, ph, n;
  __device__ Ring(int n_, int ph_) : s(0), ph(ph_), n(n_) {}
  __device__ void next() { if (++s == n) { s = 0; ph ^= 1; } }
};

// A sum of 2^64 or more hands its exponent to its reference.  Parts are added relative to the largest reference, whose own sum is at
// least 1: with sums below 2^64 no number of them reaches infinity, and what is lost where a factor is below the smallest normal
// float (2^-126) is below 2^-62 of the result.
__device__ __forceinline__ void lower_sum(float& ref, float& sum) {
  if (sum >= 0x1p64f && sum < INFINITY) {
    const int e = (__float_as_int(sum) >> 23) - 127;
    sum = __int_as_float(__float_as_int(sum) - (e << 23));
    ref += (float)e;
  }
}

// ------------------------------------------------------------------------------------------ kernel
template <int NB, int kSweep>
__global__ void __launch_bounds__(kOneThreads, 1)
score_sweep_kernel(const __grid_constant__ Layers maps, const __grid_constant__ Args a) {
  using C = Shape1<NB>;
  constexpr bool kLong = kSweep == kLongRowSums, kRows = kSweep == kRowSums || kLong;
  constexpr int kCols = C::kCols, kPer = C::kPer, kStage = C::kStage;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);     // [2 pipes][kSlots][half][128][128 B]
  float* sum_s = reinterpret_cast<float*>(ring + 2 * kSlots * kSlotBytes);  // [2 pipes][4 quads][kCols] a segment's row sums
  float* ref_s = sum_s + 2 * 4 * kCols;                                     // [2 pipes][4 quads][kCols] what they are relative to
  float* c_s = ref_s + 2 * 4 * kCols;                              // [2 pipes][2][kCols] minus a segment's log-denominators
  int* last_s = reinterpret_cast<int*>(c_s + 4 * kCols);                    // [2][kCols] last key that a plane's row sees
  uint64_t* bars = reinterpret_cast<uint64_t*>(last_s + 2 * kCols);
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  __shared__ int again_s[2][2];                 // a pipe's tiles from the first to the last segment with a sum that is not finite
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grid = gridDim.x;
  const int pipe = warp < kSoftWarps ? warp / kLaneWarps : warp & 1;
  const uint32_t bar0 = smem_u32(bars), pbar = bar0 + 8u * (pipe * C::kPipeBars);
  auto FULL = [&](int s) { return pbar + 8u * s; };                         // the slot's copy has landed
  auto EMPTY = [&](int s) { return pbar + 8u * (kSlots + s); };             // what was in it has been multiplied
  auto TFULL = [&](int s) { return pbar + 8u * (2 * kSlots + s); };         // logits are complete
  auto TEMPTY = [&](int s) { return pbar + 8u * (2 * kSlots + kPer + s); }; // the stage is free
  // by the parity of a segment's number
  auto CFULL = [&](int i) { return pbar + 8u * (2 * kSlots + 2 * kPer + i); };        // references or log-denominators are there
  auto CEMPTY = [&](int i) { return pbar + 8u * (2 * kSlots + 2 * kPer + 2 + i); };   // the segment is done (row sums are in sum_s)
  const uint32_t SUMFREE = pbar + 8u * (2 * kSlots + 2 * kPer + 4);         // row sums have been read
  const uint32_t DRAIN = pbar + 8u * (2 * kSlots + 2 * kPer + 5);           // all MMAs have ended
  volatile int* abort_flag = &abort_s;

  if (threadIdx.x == 0) {
    abort_s = 0;
    for (int p = 0; p < 2; ++p) {
      const uint32_t b = bar0 + 8u * (p * C::kPipeBars);
      for (int s = 0; s < 2 * kSlots + kPer; ++s) mbar_init(b + 8u * s, 1);             // FULL, EMPTY, TFULL
      for (int s = 0; s < kPer; ++s) mbar_init(b + 8u * (2 * kSlots + kPer + s), kLaneWarps);
      for (int i = 0; i < 2; ++i) { mbar_init(b + 8u * (2 * kSlots + 2 * kPer + i), 1); mbar_init(b + 8u * (2 * kSlots + 2 * kPer + 2 + i), kLaneWarps); }
      for (int i = 4; i < 6; ++i) mbar_init(b + 8u * (2 * kSlots + 2 * kPer + i), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
  }
  if (kRows && threadIdx.x < 4) again_s[threadIdx.x >> 1][threadIdx.x & 1] = 0;
  if (kRows && threadIdx.x < 2 * kCols) last_s[threadIdx.x] = a.P + (threadIdx.x / kCols * (a.M - a.plane_rows) + threadIdx.x % kCols) % a.ws;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // Key sums follow row sums over the same queries and keys, and row sums let them start only after their own wait for the inputs:
  // copies and MMAs begin at once, and the other warps wait for the end of the row sums.  So do copies and MMAs before the first of
  // their own waits that needs those warps: the limit is not for the time that another launch takes.
  if (kSweep == kKeySums) {
    pdl_launch();
    if (warp < kCopyWarp || warp >= kRowWarp) pdl_wait();
  } else {
    pdl_wait();
    pdl_launch();
  }
  const uint32_t tmem_base = tmem_base_s;
  // where the row sums go of the segment that a pipe of this block has of a (head, plane): its place among those of the head
  auto sums_of = [&](int vh, int p) {
    const int place = 2 * blockIdx.x + p - tile_owner((long long)vh * a.tph, (long long)a.vheads * a.tph, 2 * grid);
    return a.stats + ((size_t)vh * a.slots + place) * a.plane_rows;
  };
  // A plane's first row.  Of two planes neither has a column without a row: what both have (fewer than 32 rows) counts in the first.  An
  // empty column's logits are 0 times a key, which is no number where the key is infinite.
  auto row0_of = [&](int vh) { return (vh & (a.planes - 1)) * (a.M - a.plane_rows); };
  // What whole warps wait for they go on without once a wait has run out, as no wait blocks any more then: whether it had come is for
  // each lane to see, and lanes that left a loop alone would be missing from its next shuffle.  Single lanes stop.
  auto wait = [&](uint32_t bar, uint32_t parity, int code) { return mbar_wait(bar, parity, abort_flag, a.status, code, a.wait_cycles); };
  // for a segment of the warps with the exponentials
  auto wait_segment = [&](uint32_t bar, uint32_t parity) { mbar_wait(bar, parity, abort_flag, a.status, 107, a.segment_cycles); };
  const long long tiles = (long long)a.vheads * a.tph;
  using Segments = Segs<kLong ? kRowTiles : INT_MAX>;
  // Row sums: all warps of the block meet after the pipes' segments, and those of a pipe with a sum that is not finite go round a second
  // time, over its segments from the first to the last such one.
  auto second_round = [&](Segments& sg) {
    __syncwarp();
    asm volatile("bar.sync 3, %0;" ::"n"(kOneThreads) : "memory");
    if (!again_s[pipe][1]) return false;
    sg = Segments(again_s[pipe][0], again_s[pipe][1], a.tph);
    return true;
  };
  // f(segments, round) for each round, in two copies: what only the second round does, in the way of the first, made a pass of four
  // layers of 1K 0.4 to 1 us longer (of 38).
  auto rounds = [&](auto f) {
    Segments sg(a, 2 * blockIdx.x + pipe, 2 * grid);
    f(sg, std::integral_constant<int, 0>());
    if constexpr (kRows) if (second_round(sg)) f(sg, std::integral_constant<int, 1>());
  };
  // Minus the log-denominators of rows [r, r + 16) of a (head, plane), two lanes a row -> to[]: from the parts that the head's
  // segments have left, four in flight a lane, or the caller's.
  auto fill = [&](float* to, int vh, int r) {
    const int head = vh >> (a.planes - 1), layer = head / a.hpl, row0 = row0_of(vh), row = r + (lane >> 1);
    const bool in = row < a.plane_rows && (row0 == 0 || row0 + row >= a.plane_rows);
    float c = -INFINITY;
    if constexpr (kSweep == kKeySums) {
      const int n = tile_owner((long long)(vh + 1) * a.tph - 1, tiles, 2 * grid) - tile_owner((long long)vh * a.tph, tiles, 2 * grid) + 1;
      const float2* st = a.stats + (size_t)vh * a.slots * a.plane_rows + row;
      float m = -INFINITY, l = 0.f;
      for (int j = lane & 1; j < n; j += 8) {
        float2 x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = in && j + 2 * i < n ? st[(size_t)(j + 2 * i) * a.plane_rows] : make_float2(-INFINITY, 0.f);
        const float top = fmaxf(fmaxf(m, fmaxf(x[0].x, x[1].x)), fmaxf(x[2].x, x[3].x));
        l = l == 0.f ? 0.f : l * fast_exp2(m - top);
#pragma unroll
        for (int i = 0; i < 4; ++i) l += x[i].y == 0.f ? 0.f : x[i].y * fast_exp2(x[i].x - top);
        m = top;
      }
      const float m2 = __shfl_xor_sync(0xFFFFFFFFu, m, 1), l2 = __shfl_xor_sync(0xFFFFFFFFu, l, 1), top = fmaxf(m, m2);
      l = (l == 0.f ? 0.f : l * fast_exp2(m - top)) + (l2 == 0.f ? 0.f : l2 * fast_exp2(m2 - top));
      if (in) c = -(top + log2f(l));
    } else {
      if (in) c = -maps.lse[layer][(size_t)(head - layer * a.hpl) * a.M + row0 + row] * kLog2e;
    }
    if (!(lane & 1)) to[row] = c;
  };

  // The warps of a warpgroup have to change their registers by the same instruction: here, before the roles part.
  if (warp >= kSoftWarps) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
  if (warp < kSoftWarps) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftRegs));
    // ------------------------------------------------------------------ exponentials and sums
    const int part = warp & (kLaneWarps - 1), quad = warp & 3, half = warp >> 2 & 1;
    const uint64_t scale22 = pack2(a.scale2, a.scale2);
    // The bodies of the loops over a tile are kept short, and c and sums of a thread few: the instructions of all warps share the caches,
    // and a launch starts with none of them there.
    // Row sums: a warp has 32 lanes (keys) x half of the columns, 16 lanes at a time.  Key sums: 16 lanes x all columns, four blocks at a time.
    constexpr int kHalf = NB / 2, kSet = 4;
    const int c0 = kRows ? half * kHalf * 8 : 0, first = quad * 32 + (kRows ? 0 : half * 16);
    const uint32_t addr = tmem_base + ((uint32_t)first << 16) + (uint32_t)(pipe * kPer * kStage + c0);
    const int col2 = c0 + 2 * (lane & 3), key = first + (lane >> 2);        // the thread's keys: key, key + 8 (, key + 16, key + 24)
    if (kSweep != kKeySums) for (size_t n = blockIdx.x * (kSoftWarps * 32) + threadIdx.x; n < a.hist_n; n += grid * (kSoftWarps * 32)) a.hist[n] = 0;
    Ring st(kPer, 0);
    int i = 0;                                          // segments so far
    rounds([&](Segments& sg, auto round_) {
      constexpr int round = decltype(round_)::value;
      for (; sg.next(); ++i) {
        const int slot = i & 1;
        if (kRows) {
        } else if (i == 0) {                              // the first segment's are needed soon: 16 rows a warp
          if (16 * part < kCols) fill(c_s + 2 * pipe * kCols, sg.vh, 16 * part);
          asm volatile("bar.sync %0, 256;" ::"r"(1 + pipe) : "memory");
        } else {
          wait(CFULL(slot), i >> 1 & 1, 106);
        }
        if constexpr (kRows) {
          uint64_t c[kHalf], sum[kHalf];                  // minus the references; sums over the thread's keys so far, by columns
#pragma unroll
          for (int b = 0; b < kHalf; ++b) c[b] = sum[b] = 0ull;
          auto mask = [&](float (&x)[4 * kHalf], int t, int h) {              // row r sees keys 0 .. P + r % ws
            if ((sg.t0 + t + 1) * kTile - 1 <= a.P) return;
            const int *last = last_s + (sg.vh & (a.planes - 1)) * kCols + col2, k0 = (sg.t0 + t) * kTile + key + 16 * h;
#pragma unroll
            for (int b = 0; b < kHalf; ++b) {
              const int2 to = *reinterpret_cast<const int2*>(&last[8 * b]);
              x[4 * b] = k0 > to.x ? -INFINITY : x[4 * b]; x[4 * b + 1] = k0 > to.y ? -INFINITY : x[4 * b + 1];
              x[4 * b + 2] = k0 + 8 > to.x ? -INFINITY : x[4 * b + 2]; x[4 * b + 3] = k0 + 8 > to.y ? -INFINITY : x[4 * b + 3];
            }
          };
          auto read = [&](float (&x)[4 * kHalf], int h) {                     // the tile's lanes 16 h on
            ld_block<kHalf>(addr + (uint32_t)(st.s * kStage + (h << 20)), x);
            tc_wait_ld();
            if (h) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(TEMPTY(st.s));
            }
          };
          if constexpr (round > 0) {                      // the largest logits
            float m[2 * kHalf];
#pragma unroll
            for (int b = 0; b < 2 * kHalf; ++b) m[b] = -INFINITY;
            for (int t = 0; t < sg.n; ++t) {
              wait(TFULL(st.s), st.ph, 106);
              tc_fence_after();
#pragma unroll 1
              for (int h = 0; h < 2; ++h) {
                float x[4 * kHalf];
                read(x, h);
                mask(x, t, h);
#pragma unroll
                for (int b = 0; b < 2 * kHalf; ++b) m[b] = fmax3(m[b], x[2 * b - b % 2], x[2 * b - b % 2 + 2]);
              }
              st.next();
            }
#pragma unroll
            for (int b = 0; b < 2 * kHalf; ++b) {
#pragma unroll
              for (int o = 4; o <= 16; o <<= 1) m[b] = fmaxf(m[b], __shfl_xor_sync(0xFFFFFFFFu, m[b], o));
              m[b] = m[b] == -INFINITY ? 0.f : m[b] * -a.scale2;              // (no key of this warp counts for the row)
            }
#pragma unroll
            for (int b = 0; b < kHalf; ++b) c[b] = pack2(m[2 * b], m[2 * b + 1]);
          }
          for (int t = 0; t < sg.n; ++t) {
            wait(TFULL(st.s), st.ph, 106);
            tc_fence_after();
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
              float x[4 * kHalf];
              read(x, h);
              if (t + h + round == 0) {
#pragma unroll
                for (int b = 0; b < kHalf; ++b) {
                  const float r0 = __shfl_sync(0xFFFFFFFFu, x[4 * b], lane & 3), r1 = __shfl_sync(0xFFFFFFFFu, x[4 * b + 1], lane & 3);
                  c[b] = pack2(r0 * -a.scale2, r1 * -a.scale2);
                }
              }
              mask(x, t, h);
#pragma unroll
              for (int b = 0; b < kHalf; ++b)
#pragma unroll
                for (int j = 0; j < 2; ++j) sum[b] = exp2_acc2(false, sum[b], x[4 * b + 2 * j], x[4 * b + 2 * j + 1], scale22, c[b]);
            }
            st.next();
          }
          // Over the 8 lanes that have a column's keys: halves are exchanged, so that a lane ends with one pair of columns of four blocks.
          auto swap = [&](int o, uint64_t lo_v, uint64_t hi_v) { return add2(lane & o ? hi_v : lo_v, __shfl_xor_sync(0xFFFFFFFFu, lane & o ? lo_v : hi_v, o)); };
          wait(SUMFREE, (i & 1) ^ 1, 106);
          float* my_sum = sum_s + (pipe * 4 + quad) * kCols + col2;
          if (lane < 4)
#pragma unroll
            for (int b = 0; b < kHalf; ++b) *reinterpret_cast<uint64_t*>(&ref_s[(pipe * 4 + quad) * kCols + col2 + 8 * b]) = c[b] ^ 0x8000000080000000ull;
#pragma unroll
          for (int b = 0; b + 4 <= kHalf; b += 4) {
            uint64_t u = swap(8, swap(16, sum[b], sum[b + 2]), swap(16, sum[b + 1], sum[b + 3]));
            u = add2(u, __shfl_xor_sync(0xFFFFFFFFu, u, 4));
            if (!(lane & 4)) *reinterpret_cast<uint64_t*>(&my_sum[8 * (b + (lane >> 3))]) = u;
          }
          if constexpr (kHalf & 2) {
            constexpr int b = kHalf & ~3;
            uint64_t u = swap(16, sum[b], sum[b + 1]);
            u = add2(u, __shfl_xor_sync(0xFFFFFFFFu, u, 8));
            u = add2(u, __shfl_xor_sync(0xFFFFFFFFu, u, 4));
            if (!(lane & 12)) *reinterpret_cast<uint64_t*>(&my_sum[8 * (b + (lane >> 4))]) = u;
          }
          if constexpr (kHalf & 1) {
            uint64_t u = sum[kHalf - 1];
#pragma unroll
            for (int o = 16; o >= 4; o >>= 1) u = add2(u, __shfl_xor_sync(0xFFFFFFFFu, u, o));
            if (lane < 4) *reinterpret_cast<uint64_t*>(&my_sum[8 * (kHalf - 1)]) = u;
          }
        } else {
          const float* my_c = c_s + (2 * pipe + slot) * kCols + col2;
          float* raw = a.raw + ((size_t)sg.vh * a.tph + sg.t0) * kTile + key + (lane & 1) * 8;
          for (int t = 0; t < sg.n; ++t, raw += kTile) {
            wait(TFULL(st.s), st.ph, 106);
            tc_fence_after();
            uint64_t sum[4] = {0ull, 0ull, 0ull, 0ull};   // over the columns so far, by key and parity of the block
            const uint32_t at = addr + (uint32_t)(st.s * kStage);
            auto blocks = [&](auto count, int b0) {
              constexpr int kN = decltype(count)::value;
              float x[4 * kN];
              ld_block<kN>(at + (uint32_t)(8 * b0), x);
              uint64_t c[kN];
#pragma unroll
              for (int b = 0; b < kN; ++b) c[b] = *reinterpret_cast<const uint64_t*>(&my_c[8 * (b0 + b)]);
              tc_wait_ld();
              if (b0 + kN == NB) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(TEMPTY(st.s));
              }
#pragma unroll
              for (int b = 0; b < kN; ++b)
#pragma unroll
                for (int j = 0; j < 2; ++j) sum[2 * j + (b & 1)] = exp2_acc2(false, sum[2 * j + (b & 1)], x[4 * b + 2 * j], x[4 * b + 2 * j + 1], scale22, c[b]);
            };
#pragma unroll 1
            for (int b0 = 0; b0 + kSet <= NB; b0 += kSet) blocks(std::integral_constant<int, kSet>(), b0);
            if constexpr (NB % kSet) blocks(std::integral_constant<int, NB % kSet>(), NB - NB % kSet);
            st.next();
            // over all columns; a lane pair ends with one key
            float s0, s1, u, v;
            unpack2(add2(sum[0], sum[1]), u, v);
            s0 = u + v;
            unpack2(add2(sum[2], sum[3]), u, v);
            s1 = u + v;
            const bool h = lane & 1;
            float r = (h ? s1 : s0) + __shfl_xor_sync(0xFFFFFFFFu, h ? s0 : s1, 1);
            r += __shfl_xor_sync(0xFFFFFFFFu, r, 2);
            if (!(lane & 2)) *raw = r * a.post;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(CEMPTY(slot));
      }
    });
  } else if (warp < kMmaWarp) {
    // ------------------------------------------------------------------ copies
    const int halves = a.D / 64;
    const uint64_t first = l2_policy_evict_first();
    const bool once = a.planes == 1;                                      // the sweep reads the keys once
    const uint32_t slot0 = smem_u32(ring + pipe * kSlots * kSlotBytes);
    Ring kr(2, 1);
    unsigned int used = 0, parity = 0;                                    // slots with a copy of this block's, its phase
    int n = 0, qph = 1;
    bool ok = true;
    auto arm = [&](int s, int ph, int bytes) {
      mbar_expect_tx(FULL(s), (uint32_t)bytes);
      used |= 1u << s;
      parity = (parity & ~(1u << s)) | (unsigned int)(ph ^ 1) << s;
    };
    rounds([&](Segments& sg, auto round_) {
      constexpr int round = decltype(round_)::value;
      if (lane) return;
      while (ok && sg.next()) {
        const int head = sg.vh >> (a.planes - 1), layer = head / a.hpl, hh = head - layer * a.hpl;
        const CUtensorMap* k_map = &maps.k[layer];
        ok = wait(EMPTY(0), qph, 101);
        if (!ok) break;
        arm(0, qph, halves * C::kQBytes);
        for (int h = 0; h < halves; ++h) tma_load_3d(slot0 + h * kHalfBytes, &maps.q[layer], FULL(0), 64 * h, row0_of(sg.vh), hh);
        qph ^= 1;
        for (int u = round ? -sg.n : 0; u < sg.n; ++u) {
          const int row = (sg.t0 + (u < 0 ? u + sg.n : u)) * kTile;
          const int s = 1 + kr.s;
          ok = wait(EMPTY(s), kr.ph, 102);
          if (!ok) break;
          if (n == a.withhold_tile && blockIdx.x == 0 && pipe == 0) {       // test hook: this tile never arrives
            used &= ~(1u << s);
          } else {
            arm(s, kr.ph, halves * kHalfBytes);
            const uint32_t dst = slot0 + s * kSlotBytes;
            if (once) for (int h = 0; h < halves; ++h) tma_load_3d_hint(dst + h * kHalfBytes, k_map, FULL(s), 64 * h, row, hh, first);
            else for (int h = 0; h < halves; ++h) tma_load_3d(dst + h * kHalfBytes, k_map, FULL(s), 64 * h, row, hh);
          }
          kr.next();
          if (++n == kPer + 1 && kSweep == kKeySums) pdl_wait();            // (the queries' slot may be waited for next)
        }
      }
      // Copies land before this block's shared memory is given up, and MMAs (below) end before its tensor memory is, whenever another
      // warp's wait has run out.
      for (int s = 0; s < kSlots; ++s) if (used >> s & 1u) mbar_drain(FULL(s), parity >> s & 1u);
    });
  } else if (warp < kRowWarp) {
    // ------------------------------------------------------------------ MMAs
    const uint64_t desc = smem_desc(smem_u32(ring + pipe * kSlots * kSlotBytes));
    const uint32_t hi = (uint32_t)(desc >> 32), q_lo = (uint32_t)desc;
    Ring kr(2, 0), st(kPer, 1);
    int qph = 0;
    bool ok = true;
    rounds([&](Segments& sg, auto round_) {
      constexpr int round = decltype(round_)::value;
      if (lane) return;
      while (ok && sg.next()) {
        ok = wait(FULL(0), qph, 103);
        qph ^= 1;
        for (int u = round ? -sg.n : 0; ok && u < sg.n; ++u) {
          const int s = 1 + kr.s;
          ok = wait(FULL(s), kr.ph, 104) && wait(TEMPTY(st.s), st.ph, 105);
          if (!ok) break;
          tc_fence_after();
          const uint32_t d = tmem_base + (uint32_t)((pipe * kPer + st.s) * kStage), k_lo = q_lo + ((uint32_t)(s * kSlotBytes) >> 4);
          if (a.D == 128) {
            tc_mma_x8<(kHalfBytes >> 4), (kHalfBytes >> 4)>(d, k_lo, q_lo, hi, a.idesc);
          } else {
            for (int i = 0; i < 4; ++i)
              tc_mma(d, ((uint64_t)hi << 32) | (k_lo + 2 * i), ((uint64_t)hi << 32) | (q_lo + 2 * i), a.idesc, i > 0);
          }
          tc_commit(EMPTY(s));
          tc_commit(TFULL(st.s));
          kr.next();
          st.next();
          if (kSweep == kKeySums && st.s == 0) pdl_wait();                  // all stages have been used
        }
        if (ok) tc_commit(EMPTY(0));
      }
      tc_commit(DRAIN);
      mbar_drain(DRAIN, round);
    });
  } else if (warp < kPublishWarp) {
    // ------------------------------------------------------------------ log-denominators of the segments but the first
    int i = 0;
    rounds([&](Segments& sg, auto) {
      for (; !kRows && sg.next(); ++i) {
        const int slot = i & 1;
        wait_segment(CEMPTY(slot), (i >> 1 & 1) ^ 1);                            // the segment before last is done with its own
        if (i > 0)
#pragma unroll 1
          for (int r = 0; r < kCols; r += 16) fill(c_s + (2 * pipe + slot) * kCols, sg.vh, r);
        __syncwarp();
        if (lane == 0) mbar_arrive(CFULL(slot));
      }
    });
  } else {
    // ------------------------------------------------------------------ a segment's row sums -> the rows' counters
    if constexpr (kRows) {
      int i = 0;
      Segments sg(a, 2 * blockIdx.x + pipe, 2 * grid);
      int round = 0, part = 0;                            // first tile of what the pipe has of the head
      do {
        for (int vh = -1; sg.next(); ++i) {
          const bool more = kLong && sg.vh == vh;
          vh = sg.vh;
          if (!more) part = sg.g - sg.n;
          float2* to = sums_of(sg.vh, pipe);
          bool finite = true;
          wait_segment(CEMPTY(i & 1), i >> 1 & 1);
#pragma unroll 1
          for (int row = lane; row < a.plane_rows; row += 32) {
            float m[4], l[4], top = -INFINITY, sum = 0.f;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
              m[w] = ref_s[(pipe * 4 + w) * kCols + row];
              l[w] = sum_s[(pipe * 4 + w) * kCols + row];
              lower_sum(m[w], l[w]);
              if (l[w] != 0.f) top = fmaxf(top, m[w]);    // (0: no key of this quad counts for the row)
            }
#pragma unroll
            for (int w = 0; w < 4; ++w) sum += l[w] == 0.f ? 0.f : l[w] * fast_exp2(m[w] - top);
            if (more) {
              const float2 before = to[row];
              const float most = fmaxf(top, before.x);
              sum = (sum == 0.f ? 0.f : sum * fast_exp2(top - most)) + (before.y == 0.f ? 0.f : before.y * fast_exp2(before.x - most));
              top = most;
            }
            finite = finite && sum < INFINITY;
            to[row] = make_float2(top, sum);
          }
          finite = __all_sync(0xFFFFFFFFu, finite);
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(SUMFREE);
            if (!round && !finite) {
              if (!again_s[pipe][1]) again_s[pipe][0] = part;
              again_s[pipe][1] = sg.g;
            }
          }
        }
      } while (!round++ && second_round(sg));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512));
  }
}

// ------------------------------------------------------------------------------------------ pooling
// Eq. 2's pooling of the unpooled scores (the sum over a head's planes), and the digits of the result for the updates.
// raw: [heads * planes][raw_stride].  scores: [heads][P].  layer_hist: [layers][samples][kBins] counters that a sweep before has cleared.  grid heads * segs, segs = ceil(P / seg), seg
// (a multiple of the threads, kPoolSeg at most): as many as give every SM two blocks.  Bound by instructions (neighbours,
// digits, counters), not by memory: 16 layers of 32K, 17 MB in from L2 and as much out, took 22 us where a copy of it takes 5.
// Neighbours outside a head are NaNs in shared memory, which no maximum takes, so that none is checked for (a pass of 32 layers of
// 32K with log-denominators 515.4 -> 512.6 us, 14 layers of 3 x 5003 123.9 -> 123.1, 4 of 1K 38.7 -> 38.3).
constexpr int kPoolThreads = 256, kPoolSeg = 2048;
__global__ void __launch_bounds__(kPoolThreads)
pool_kernel(const float* raw, float* scores, unsigned int* layer_hist, int P, int raw_stride, int planes, int half, int avg, int hkv, int seg, int segs) {
  __shared__ float v[kPoolSeg + 256];
  __shared__ unsigned int hist[kBins];
  const int head = blockIdx.x / segs, o0 = (blockIdx.x - head * segs) * seg, o1 = min(P, o0 + seg), lo = o0 - half, hi = o1 + half;
  for (int i = threadIdx.x; i < kBins; i += kPoolThreads) hist[i] = 0;
  pdl_launch();
  pdl_wait();
  const float* r = raw + (size_t)head * planes * raw_stride;
  for (int i = lo + (int)threadIdx.x; i < hi; i += kPoolThreads) {
    float x = NAN;                                         // outside the head: no maximum takes it
    if (i >= 0 && i < P) {
      x = r[i];
      for (int p = 1; p < planes; ++p) x += r[(size_t)p * raw_stride + i];
    }
    v[i - lo] = x;
  }
  __syncthreads();
  for (int b = o0; b < o1; b += kPoolThreads) {
    const int o = b + threadIdx.x, x = o - lo;
    const bool ok = o < o1;
    float s = 0.f;
    if (ok) {
      s = v[x];
      if (avg) {
        int n = 1;
        for (int d = 1; d <= half; ++d) {
          if (o - d >= 0) { s += v[x - d]; ++n; }
          if (o + d < P) { s += v[x + d]; ++n; }
        }
        s = s / (float)n;
      } else {
#pragma unroll 4
        for (int d = 1; d <= half; ++d) s = fmaxf(s, fmaxf(v[x - d], v[x + d]));
      }
      scores[(size_t)head * P + o] = s;
    }
    run_bump(hist, digit_of(__float_as_uint(s)), ok);
  }
  __syncthreads();
  unsigned int* to = layer_hist + (size_t)(head / hkv) * kBins;
  for (int i = threadIdx.x; i < kBins; i += kPoolThreads) { const unsigned int n = hist[i]; if (n) atomicAdd(&to[i], n); }
}

}  // namespace sweep
}  // namespace dkv
