// libdkv: context, argument checking and the C ABI declared in include/dkv.h.
// The method's steps (Algorithm 1 of arXiv 2412.14838) live in the kernel headers included here.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>
#include <algorithm>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/dkv.h"
#include "common.cuh"
#include "compact.cuh"
#include "decode.cuh"
#include "rebudget.cuh"
#include "score_sweep.cuh"
#include "score_tc.cuh"
#include "select.cuh"

using namespace dkv;
using sweep::pool_kernel;
using sweep::score_sweep_kernel;

struct ProfRec { cudaEvent_t a, b; int step; int launches; };

struct dkv_ctx {
  dkv_config cfg;
  Shape s;
  int device;
  // device state
  float* d_scores;      // [L][Bt][Hkv][P]  pooled scores, the history A^b
  int* d_idx;           // [L][Bt][Hkv][Blc] kept positions, in buffer order
  int* d_count;         // [Bt][L] budget of each layer
  int* d_held;          // [Bt][L] rows the layer's buffers hold
  int* d_dbg;           // 3 x [Bt][L] : cnt, Z, Z' of the last update
  unsigned int* d_layer_hist; // [L][Bt][2048] digit histogram of every layer's scores (all heads of a sample)
  uint2* d_cand;              // [Bt][L*Hkv*P] (score bits, layer) of the scores with the digit of a global top-K's threshold;
                              // while a pass scores, its unpooled scores: float [layers of a launch][heads][planes][tiles * 128]
  unsigned int* d_cand_n;     // [Bt]
  RbState* d_rb_state;        // [kRbUpdates][Bt]
  unsigned int* d_rb_above;   // [kRbUpdates][Bt][L]
  unsigned int* d_shrink_tickets;   // [Bt][L], zero between launches
  int* d_status;        // [8]
  int sel_cap;          // entries of the select kernels' list
  // tensor-core scoring
  int n_sms;
  size_t stats_rows;    // (head, slot) pairs of a job, at most
  int pass_group;       // layers per scoring launch of dkv_run_prefill_pass (1..tc::kMaxGroup)
  bool emit_backward;   // sweep 2 walks every CTA's slice from the end to the start
  bool host_v_staged;   // dkv_run_prefill_pass_host copies V in full even where the gather could read its rows in place
  long long host_h2d, host_d2h;   // bytes the last dkv_run_prefill_pass_host moved in either direction
  int retain_mb;        // MB of a sweep-1 job's keys (the end of every CTA's slice) marked to stay in L2 for sweep 2
  long long wait_cycles;   // limit of the scoring kernel's mbarrier waits (dkv_set_wait_limit)
  int withhold_sweep, withhold_tile;   // test hook of dkv_debug_withhold_tile (-1: off)
  // passes scored by score_sweep.cuh
  float2* d_stats;      // row sums of a head's segments (null where only passes with given log-denominators are)
  int planes, plane_rows;  // window rows of a head: planes of at most 128
  float2* d_tc_stats;   // [3][stats_rows][256]: partial softmax statistics, three jobs in rotation, each [heads][slots][256]
  // host state
  uint8_t scored[DKV_MAX_LAYERS], gathered[DKV_MAX_LAYERS];
  uint8_t selected[DKV_MAX_LAYERS];     // 1: by scores (dkv_select_topk), 2: by position (dkv_select_positions)
  int sel_n[DKV_MAX_LAYERS];            // positions selected per head: Blc, or what dkv_select_positions kept
  // decoding over the compressed cache
  float* d_dec_scratch;                 // parts of heads that lie in more than one block's slice (allocated on first use, grown on demand)
  size_t dec_scratch_floats;
  unsigned int* d_dec_tickets;          // [L][Bt*Hkv], zero between launches
  long long launches;
  int last_cuda;
  // optional per-step timing with CUDA events (dkv_profile)
  bool prof_on;
  std::vector<ProfRec>* prof_recs;
  size_t prof_used;
  double prof_ms[DKV_N_STEPS];
  long long prof_launches[DKV_N_STEPS];
  // staging for the host-buffer pass (allocated on first use)
  bool staged;
  void *st_q[2], *st_k[2], *st_v[2];
  void *st_kb[DKV_MAX_LAYERS], *st_vb[DKV_MAX_LAYERS];
  cudaStream_t st_copy, st_comp;
  cudaEvent_t ev_copied[2], ev_consumed[2];
};

namespace {

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// A failed call is reported once: the runtime keeps its code until it is read, and the next check after a launch would
// otherwise take it for its own, in this context or another.
int cuda_fail(dkv_ctx* c, cudaError_t e) {
  if (c) c->last_cuda = (int)e;
  cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? DKV_ERR_NOMEM : DKV_ERR_CUDA;
}
#define DKV_CUDA(ctx, call)                                   \
  do {                                                        \
    cudaError_t e__ = (call);                                 \
    if (e__ != cudaSuccess) return cuda_fail(ctx, e__);       \
  } while (0)
#define DKV_LAUNCH(ctx, call)                                 \
  do {                                                        \
    DKV_CUDA(ctx, call);                                      \
    (ctx)->launches++;                                        \
  } while (0)
#define DKV_LAUNCHED(ctx)                                     \
  do {                                                        \
    DKV_CUDA(ctx, cudaGetLastError());                        \
    (ctx)->launches++;                                        \
  } while (0)

// Event pair around one step's launches; read back by dkv_profile_read.
struct ProfScope {
  dkv_ctx* c; cudaStream_t st; ProfRec* r;
  ProfScope(dkv_ctx* c_, int step, int launches, cudaStream_t st_) : c(c_), st(st_), r(nullptr) {
    if (!c->prof_on) return;
    if (c->prof_used == c->prof_recs->size()) {
      ProfRec n; n.step = 0; n.launches = 0;
      if (cudaEventCreate(&n.a) != cudaSuccess || cudaEventCreate(&n.b) != cudaSuccess) return;
      c->prof_recs->push_back(n);
    }
    r = &(*c->prof_recs)[c->prof_used++];
    r->step = step; r->launches = launches;
    cudaEventRecord(r->a, st);
  }
  ~ProfScope() { if (r) cudaEventRecord(r->b, st); }
};

// Launch with programmatic stream serialisation (the kernel waits for its predecessor itself, so that its scheduling
// overlaps the predecessor's end) and, if cluster > 1, clusters of that many blocks along x.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, int cluster, cudaStream_t st, const Args&... args) {
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cfg.attrs = at; cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

size_t layer_scores(const Shape& s) { return (size_t)s.Bt * s.Hkv * s.P; }
size_t layer_idx(const Shape& s) { return (size_t)s.Bt * s.Hkv * s.Blc; }
size_t layer_kv_bytes(const Shape& s) { return (size_t)s.Bt * s.Hkv * s.S * s.D * 2; }
size_t layer_q_bytes(const Shape& s) { return (size_t)s.Bt * s.Hq * s.ws * s.D * 2; }
size_t layer_buf_bytes(const Shape& s) { return (size_t)s.Bt * s.Hkv * s.rows * s.D * 2; }

int validate(const dkv_config* c) {
  if (!c) return DKV_ERR_INVALID_ARG;
  if (c->n_layers < 1 || c->n_q_heads < 1 || c->n_kv_heads < 1 || c->batch < 1) return DKV_ERR_INVALID_ARG;
  if (c->n_q_heads % c->n_kv_heads != 0) return DKV_ERR_INVALID_ARG;
  if (c->window < 1 || c->seq_len <= c->window) return DKV_ERR_INVALID_ARG;
  if (c->pool_kernel < 1 || c->pool_kernel % 2 == 0) return DKV_ERR_INVALID_ARG;
  if (c->pool_kernel > 255) return DKV_ERR_UNSUPPORTED;
  if (c->avg_budget < 1 || c->layer_max < c->avg_budget || c->update_interval < 1) return DKV_ERR_INVALID_ARG;
  if (c->flags & ~DKV_F_ALL) return DKV_ERR_INVALID_ARG;
  if (c->pool_kind != 0 && c->pool_kind != 1) return DKV_ERR_UNSUPPORTED;
  if (c->n_layers > DKV_MAX_LAYERS || c->layer_max > DKV_MAX_LAYER_BUDGET) return DKV_ERR_UNSUPPORTED;
  if (c->head_dim != 64 && c->head_dim != 128) return DKV_ERR_UNSUPPORTED;
  if ((long long)c->window * (c->n_q_heads / c->n_kv_heads) > DKV_MAX_WINDOW_ROWS) return DKV_ERR_UNSUPPORTED;
  if ((long long)c->n_layers * c->batch * c->n_kv_heads * (long long)c->seq_len >= (1ll << 31)) return DKV_ERR_UNSUPPORTED;
  return DKV_OK;
}

// Measurement overrides from the environment, read once per context in dkv_create: an integer inside
// [lo, hi], anything else (unset, not a number, out of range) gives the default.
int env_int(const char* name, int dflt, int lo, int hi) {
  const char* e = getenv(name);
  if (!e || !*e) return dflt;
  char* end = nullptr;
  const long v = strtol(e, &end, 10);
  if (end == e || *end != '\0' || v < lo || v > hi) return dflt;
  return (int)v;
}

int check_layer(const dkv_ctx* c, int layer) {
  if (!c) return DKV_ERR_INVALID_ARG;
  if (layer < 0 || layer >= c->s.L) return DKV_ERR_INVALID_ARG;
  return DKV_OK;
}

// ---- step (1): scores of one layer -------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr) == cudaSuccess &&
        qr == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// bf16 tensor [heads][rows][D] seen as (D, rows, heads); boxes of 64 columns x `box_rows` rows, 128-byte swizzle,
// rows past the end of a head read as zero.
bool make_map(CUtensorMap* m, const void* base, int D, int rows, int heads, int box_rows = 128) {
  EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)rows, (cuuint64_t)heads};
  const cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)rows * D * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Copies of the queries in sweep 1's 128-row operand (score_tc.cuh): as many as fit, up to four.
int query_copies(int M) { return M <= 32 ? 4 : M <= 64 ? 2 : 1; }

uint32_t make_idesc(int M, int N) {
  // fp32 accumulator, bf16 A and B, both K-major
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Statistics slots a head of a job needs: thread blocks that can share it (its share of the grid, one cut at either end).
int stats_slots(int n_sms, int job_heads) { return n_sms / job_heads + 2; }

// Parameters of one sweep over the `nl` consecutive layers that start at `layer` (q, k: their nl device
// pointers); `buf` picks the statistics scratch (jobs in flight rotate).  In sweep 2 every CTA walks its slice of the
// key space from the end to the start: sweep 1 cut the same space into the same slices, so each CTA begins with
// the keys that were streamed last and may still be in L2.
// `grid`: thread blocks of the launch; `stats_grid`: of the launch that ran sweep 1 for these layers (sweep 2).
template <int NL>
bool make_job(dkv_ctx* c, int mode, int layer, int nl, const void* const* q, const void* const* k, float* scores_out,
              int buf, int grid, int stats_grid, bool hist, tc::Maps<NL>* maps, tc::Params* p, const float* const* lse = nullptr) {
  const Shape& s = c->s;
  const int heads = s.Bt * s.Hkv;
  for (int i = 0; i < nl; ++i)
    if (!make_map(&maps->q[i], q[i], s.D, s.M, heads, 128 / query_copies(s.M)) || !make_map(&maps->k[i], k[i], s.D, s.S, heads)) return false;
  for (int i = 0; i < nl; ++i) maps->lse[i] = lse ? lse[i] : nullptr;      // (entries past nl are never read)
  p->S = s.S; p->P = s.P; p->ws = s.ws; p->M = s.M; p->D = s.D; p->heads = nl * heads; p->half = s.pool / 2;
  p->nl = nl; p->hpl = heads;
  p->back = (mode == tc::kEmit && c->emit_backward) ? 1 : 0;
  p->retain_tiles = (int)((long long)c->retain_mb * (1 << 20) / ((long long)grid * tc::kTileKeys * s.D * 2));
  p->wait_cycles = c->wait_cycles;
  p->withhold_tile = c->withhold_sweep == mode ? c->withhold_tile : -1;
  p->tph = (s.S + tc::kTileKeys - 1) / tc::kTileKeys;
  p->nq16 = (s.M + 15) / 16 * 16;
  p->nmblk = (s.M + 127) / 128;
  p->slots = stats_slots(c->n_sms, nl * heads); p->m_stride = 256;
  p->scale2 = kLog2e / sqrtf((float)s.D);
  p->stats = c->d_tc_stats + (size_t)buf * c->stats_rows * 256;
  p->scores = c->d_scores + (size_t)layer * layer_scores(s);
  p->copy_out = scores_out;
  p->status = c->d_status;
  p->stats_grid = stats_grid;
  p->layer_hist = hist ? c->d_layer_hist + (size_t)layer * s.Bt * kBins : nullptr;
  p->hkv = s.Hkv;
  p->mode = mode;
  p->out_scale = (c->cfg.flags & DKV_F_WINDOW_MEAN) ? 1.0f / (float)s.M : 1.0f;
  p->pool_avg = c->cfg.pool_kind == 1;
  p->idesc = mode == tc::kStats ? make_idesc(128, 128) : make_idesc(128, p->nq16);
  return true;
}

// The scoring kernel for two jobs (either may be kNone) of the same shape: the specialised build for exactly 128 window rows
// of 128 dims, builds with two or four copies of the queries for up to 64 or 32 window rows, the general one otherwise.  Groups of
// layers have 128 rows of 128 dims or more than 128 rows (pass_by_sweeps).
template <int NL>
auto score_kernel(int M, int D) {
  if constexpr (NL > 1) return M == 128 && D == 128 ? tc::score_tc_kernel<NL, true, 1> : tc::score_tc_kernel<NL, false, 1>;
  else return M == 128 && D == 128 ? tc::score_tc_kernel<NL, true, 1> : query_copies(M) == 4 ? tc::score_tc_kernel<NL, false, 4>
       : query_copies(M) == 2 ? tc::score_tc_kernel<NL, false, 2> : tc::score_tc_kernel<NL, false, 1>;
}
// The build's shared memory, per function and device: set before its first launch, and only for the builds that a caller can
// reach, since each is loaded onto the device by it.
template <int NL>
cudaError_t set_score_attribute(int M, int D) {
  return cudaFuncSetAttribute(score_kernel<NL>(M, D), cudaFuncAttributeMaxDynamicSharedMemorySize, tc::kSmemBytes);
}
template <int NL>
cudaError_t launch_tc(int grid, cudaStream_t st, const tc::Maps<NL>& m0, const tc::Maps<NL>& m1, const tc::Params& j0, const tc::Params& j1) {
  const tc::Params& j = j0.mode == tc::kNone ? j1 : j0;
  return launch_pdl(score_kernel<NL>(j.M, j.D), dim3(grid), tc::kThreads, (size_t)tc::kSmemBytes, 1, st, m0, m1, j0, j1);
}

// Thread blocks of a scoring launch over `nl` layers: one an SM, fewer if there are fewer key tiles.
int score_grid(const dkv_ctx* c, int nl) {
  const long long tiles = (long long)nl * c->s.Bt * c->s.Hkv * ((c->s.S + tc::kTileKeys - 1) / tc::kTileKeys);
  return (int)(tiles < c->n_sms ? tiles : c->n_sms);
}

// A group of consecutive layers that is scored together: its first layer, how many, the statistics scratch its sweep 1
// writes and the grid it ran on.
struct ScoreGroup { int first, n, buf, grid; };

// One launch: sweep 2 of group `e` (if not null), then sweep 1 of group `s` (if not null), whose grid it sets.  `q`, `k`,
// `lse`: all layers' pointers, indexed by layer (lse: null, or the caller's normalisers instead of sweep 1).
template <int NL>
int launch_score(dkv_ctx* c, const ScoreGroup* e, ScoreGroup* s, const void* const* q, const void* const* k, const float* const* lse,
                 float* scores_out, bool hist, cudaStream_t st) {
  tc::Maps<NL> m0, m1;                       // only the layers of the jobs are filled in and read
  tc::Params j0, j1;
  memset(&j0, 0, sizeof j0); memset(&j1, 0, sizeof j1);
  j0.mode = j1.mode = tc::kNone;
  // No more blocks than sweep 1 has tiles, whatever sweep 2 has: a block without a tile would leave a gap among its head's statistics.
  const int grid = score_grid(c, (s ? s : e)->n);
  if (s) s->grid = grid;
  if (e && !make_job(c, tc::kEmit, e->first, e->n, q + e->first, k + e->first, scores_out, e->buf, grid, e->grid, hist, &m0, &j0, lse ? lse + e->first : nullptr)) return DKV_ERR_CUDA;
  if (s && !make_job(c, tc::kStats, s->first, s->n, q + s->first, k + s->first, nullptr, s->buf, grid, grid, hist, &m1, &j1)) return DKV_ERR_CUDA;
  j0.inputs_ready = e && !lse;               // sweep 1 of group `e` was in the launch before
  ProfScope ps(c, s ? DKV_STEP_SCORE_STATS : DKV_STEP_SCORE_EMIT, 1, st);
  DKV_LAUNCH(c, launch_tc(grid, st, e ? m0 : m1, s ? m1 : m0, j0, j1));
  return DKV_OK;
}

// ---- scoring of a pass (score_sweep.cuh) ---------------------------------------------------------
int tiles_per_head(const Shape& s) { return (s.S + tc::kTileKeys - 1) / tc::kTileKeys; }
bool long_heads(const dkv_ctx* c) { return tiles_per_head(c->s) > sweep::kRowTiles; }
int row_blocks(const dkv_ctx* c) { return (c->plane_rows + 15) / 16 * 2; }              // the kernel's NB
int most_layers(const dkv_ctx* c) { return c->s.L < tc::kMaxGroup ? c->s.L : tc::kMaxGroup; }
// Segments a (head, plane) can have in a launch over nl layers: its share of the pipes, one cut at either end.
int stats_places(const dkv_ctx* c, int nl) { return 2 * c->n_sms / (nl * c->s.Bt * c->s.Hkv * c->planes) + 2; }

// Calls f with the kernel of this context's shape for one sweep, and its shared memory.
template <int kSweep, typename F>
cudaError_t with_sweep_kernel(int nb, F f) {
  switch (nb) {
    case 2: return f(score_sweep_kernel<2, kSweep>, (int)sweep::Shape1<2>::kSmem);
    case 4: return f(score_sweep_kernel<4, kSweep>, (int)sweep::Shape1<4>::kSmem);
    case 6: return f(score_sweep_kernel<6, kSweep>, (int)sweep::Shape1<6>::kSmem);
    case 8: return f(score_sweep_kernel<8, kSweep>, (int)sweep::Shape1<8>::kSmem);
    case 10: return f(score_sweep_kernel<10, kSweep>, (int)sweep::Shape1<10>::kSmem);
    case 12: return f(score_sweep_kernel<12, kSweep>, (int)sweep::Shape1<12>::kSmem);
    case 14: return f(score_sweep_kernel<14, kSweep>, (int)sweep::Shape1<14>::kSmem);
    default: return f(score_sweep_kernel<16, kSweep>, (int)sweep::Shape1<16>::kSmem);
  }
}
// The builds' shared memory, per function and device: set before their first launch, and only for the builds that a caller can
// reach, since each is loaded onto the device by it.  all: passes without the caller's normalisers too (pass_by_sweeps).
cudaError_t set_sweep_attributes(int nb, bool all, bool long_rows) {
  auto set = [](auto kernel, int smem) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); };
  cudaError_t e = set(pool_kernel, 0);
  if (e == cudaSuccess && all) e = long_rows ? with_sweep_kernel<sweep::kLongRowSums>(nb, set) : with_sweep_kernel<sweep::kRowSums>(nb, set);
  if (e == cudaSuccess && all) e = with_sweep_kernel<sweep::kKeySums>(nb, set);
  return e != cudaSuccess ? e : with_sweep_kernel<sweep::kGivenSums>(nb, set);
}

// Which of the two scoring kernels takes a pass.  With the caller's normalisers it is always score_sweep.cuh (128 rows of 128 dims, whole
// passes against the library that scored them with score_tc.cuh: 4 layers of 700 keys 32.5 -> 30.1 us, 8 of 4K 42.5 -> 37.0, 32 of 1K /
// 4K / 16K 60 / 96 / 247 -> 51 / 85 / 221), and for one layer at a
// time always score_tc.cuh, which has a launch less and pools in it (a layer of 32K with normalisers 18.3 us a call, by sweeps 23.1;
// without, 8 layers of 4K call by call 253-298 us against 278-328).  score_tc.cuh remains for 128 window rows of 128 dims, for
// which it has a build, while an SM has few tiles (8 layers of 4K, 4 heads: 58 us against 65; 32 of 8K, 110 tiles an SM: 285 / 283;
// 32 of 32K, 443: 1046 / 1024; 4 x 16K, 886: 2013 / 1955), and for more than 128 rows (two planes, whose pooling takes a launch)
// while an SM has at most two tiles (4 layers of 1K, 4 heads, 224 rows, 128 tiles in all: 48.3 / 50.2; 8 of 2K, 512 tiles:
// 60.8 / 58.7; 28 of 16K: 388 / 364 in bursts and the same, 408-418, at the power cap; 16 of 16K, 4 heads of 64, 140 rows: 207 / 168).
// So do 208 rows and more over heads of two tiles whose scored positions, with their neighbours in the pooling, fill one: sweep 2 of
// score_tc.cuh reads that one only.  32 layers of B samples of 8 heads of 130 keys (score_tc.cuh / sweeps), B = 3, 4, 8: 224 rows of 128 dims
// 110 / 104, 133 / 137, 228 / 240; 256 rows of 128 dims 112 / 110, 135 / 143, 233 / 251 (150 keys); 256 of 64 dims B = 6, 8 179 / 177, 222 / 238.  With
// fewer rows or longer heads the sweeps are faster again: 192 rows 225 / 221, 224 rows of 160 keys, B = 6, 193 / 186.
bool pass_by_sweeps(const dkv_ctx* c) {
  const Shape& s = c->s;
  const long long tiles = (long long)s.L * s.Bt * s.Hkv * tiles_per_head(s);
  if (s.M >= 208 && tiles_per_head(s) == 2 && s.P + s.pool / 2 * 2 <= tc::kTileKeys && tiles >= (s.D == 128 ? 12ll : 24ll) * c->n_sms) return false;
  return tiles >= (s.M == 128 && s.D == 128 ? 200ll : c->planes > 1 ? 2ll : 0ll) * c->n_sms;
}

// Scores of a pass's `nl` consecutive layers from `layer`, and their digits: row sums, key sums and pooling, or with the caller's
// normalisers the last two.  q, k, lse (or null): the layers' pointers.
int launch_sweeps(dkv_ctx* c, int layer, int nl, const void* const* q, const void* const* k, const float* const* lse, cudaStream_t st) {
  const Shape& s = c->s;
  const int heads = s.Bt * s.Hkv, nb = row_blocks(c), tph = tiles_per_head(s);
  sweep::Layers maps;                        // only the first nl entries are filled in and read
  for (int i = 0; i < nl; ++i) {
    if (!make_map(&maps.q[i], q[i], s.D, s.M, heads, 8 * nb) || !make_map(&maps.k[i], k[i], s.D, s.S, heads)) return DKV_ERR_CUDA;
    maps.lse[i] = lse ? lse[i] : nullptr;
  }
  sweep::Args a;
  memset(&a, 0, sizeof a);
  a.S = s.S; a.P = s.P; a.ws = s.ws; a.M = s.M; a.D = s.D;
  a.planes = c->planes; a.plane_rows = c->plane_rows;
  a.tph = tph;
  a.hpl = heads; a.vheads = nl * heads * c->planes;
  a.scale2 = kLog2e / sqrtf((float)s.D);
  a.post = (c->cfg.flags & DKV_F_WINDOW_MEAN) ? 1.0f / (float)s.M : 1.0f;
  a.idesc = make_idesc(128, 8 * nb);         // columns past the window rows are zero logits
  a.raw = reinterpret_cast<float*>(c->d_cand);
  a.stats = c->d_stats; a.slots = stats_places(c, nl);
  a.hist = c->d_layer_hist + (size_t)layer * s.Bt * kBins;
  a.hist_n = (size_t)nl * s.Bt * kBins;
  a.status = c->d_status;
  a.wait_cycles = c->wait_cycles;
  a.segment_cycles = c->wait_cycles > INT64_MAX / (2 * tph) ? INT64_MAX : c->wait_cycles * (2 * tph);      // a segment swept twice
  const long long tiles = (long long)a.vheads * tph;
  const dim3 grid((unsigned int)((tiles + 1) / 2 < c->n_sms ? (tiles + 1) / 2 : c->n_sms));
  auto launch = [&](auto score_kernel, int smem) { return launch_pdl(score_kernel, grid, sweep::kOneThreads, (size_t)smem, 1, st, maps, a); };
  if (!lse) {
    a.withhold_tile = c->withhold_sweep == tc::kStats ? c->withhold_tile : -1;
    ProfScope ps(c, DKV_STEP_SCORE_STATS, 1, st);
    DKV_LAUNCH(c, long_heads(c) ? (with_sweep_kernel<sweep::kLongRowSums>(nb, launch)) : (with_sweep_kernel<sweep::kRowSums>(nb, launch)));
  }
  a.withhold_tile = c->withhold_sweep == tc::kEmit ? c->withhold_tile : -1;
  {
    ProfScope ps(c, DKV_STEP_SCORE_EMIT, 1, st);
    DKV_LAUNCH(c, lse ? (with_sweep_kernel<sweep::kGivenSums>(nb, launch)) : (with_sweep_kernel<sweep::kKeySums>(nb, launch)));
  }
  ProfScope ps(c, DKV_STEP_SCORE_EMIT, 1, st);
  int seg = sweep::kPoolSeg;
  while (seg > sweep::kPoolThreads && (long long)nl * heads * ((s.P + seg - 1) / seg) < 2 * c->n_sms) seg /= 2;
  const int segs = (s.P + seg - 1) / seg;
  DKV_LAUNCH(c, launch_pdl(pool_kernel, dim3(segs * nl * heads), sweep::kPoolThreads, 0, 1, st, (const float*)a.raw,
                           c->d_scores + (size_t)layer * layer_scores(s), a.hist, s.P, tph * tc::kTileKeys, c->planes, s.pool / 2,
                           (int)(c->cfg.pool_kind == 1), s.Hkv, seg, segs));
  return DKV_OK;
}

// One layer on its own; lse: as for dkv_score_lse, or null.
int do_score(dkv_ctx* c, int layer, const void* q, const void* k, const float* lse, float* scores_out, cudaStream_t st) {
  ScoreGroup g = {layer, 1, layer % 3, 0};
  const void *qs[DKV_MAX_LAYERS], *ks[DKV_MAX_LAYERS];      // indexed by layer
  const float* ls[DKV_MAX_LAYERS];
  qs[layer] = q; ks[layer] = k; ls[layer] = lse;
  int rc;
  if (!lse && (rc = launch_score<1>(c, nullptr, &g, qs, ks, nullptr, nullptr, false, st))) return rc;
  if ((rc = launch_score<1>(c, &g, nullptr, qs, ks, lse ? ls : nullptr, scores_out, false, st))) return rc;
  c->scored[layer] = 1;
  c->selected[layer] = c->gathered[layer] = 0;
  return DKV_OK;
}

// ---- step (2): per-head top-Bl' ----------------------------------------------------------------
// Positions of a layer's idx in ascending order and their places, see sort_positions_kernel.
int do_sort_positions(dkv_ctx* c, int layer, const int* held, int keep, int* sorted_out, int* rank_out, cudaStream_t st) {
  const Shape& s = c->s;
  size_t smem = 16;
  while (smem < (size_t)keep * 8) smem <<= 1;
  sort_positions_kernel<<<s.Bt * s.Hkv, kSelThreads, smem, st>>>(c->d_idx + (size_t)layer * layer_idx(s), held, keep, sorted_out, rank_out,
                                                                 s.Blc, s.Hkv, s.L, layer);
  DKV_LAUNCHED(c);
  return DKV_OK;
}

int do_select(dkv_ctx* c, int layer, int* sorted_out, int* rank_out, cudaStream_t st) {
  const Shape& s = c->s;
  {
    ProfScope ps(c, DKV_STEP_SELECT, 1, st);
    unsigned int* lh = c->d_layer_hist + (size_t)layer * s.Bt * kBins;
    DKV_CUDA(c, cudaMemsetAsync(lh, 0, sizeof(unsigned int) * s.Bt * kBins, st));
    // A cluster a head from the length where its exchanges (about 2 us) cost less than the passes over the scores that it
    // saves, while the heads leave half of the SMs idle: 4 blocks from 8192 positions, 8 from 24576 (a call, heads of
    // 6300/10000/16352/32736 scores, 1 block: 12.3/14.3/16.4/22.6 us; 4: 12.3/12.3/14.3/14.4; 8 with 8 heads: 32736: 14.3;
    // 8 with 18 heads: 17 to 18 at any length; 2 never pays).
    const int heads = s.Bt * s.Hkv;
    const int parts = s.P >= 24576 && heads * 16 <= c->n_sms ? 8 : s.P >= 8192 && heads * 8 <= c->n_sms ? 4 : 1;
    DKV_LAUNCH(c, launch_pdl(parts > 1 ? select_topk_kernel<true> : select_topk_kernel<false>, dim3(heads * parts), kSelThreads, select_smem(c->sel_cap),
                             parts, st, (const float*)(c->d_scores + (size_t)layer * layer_scores(s)), c->d_idx + (size_t)layer * layer_idx(s), lh, s.P,
                             s.Blc, c->sel_cap, c->d_count, s.Hkv, s.L, layer, parts));
  }
  c->selected[layer] = 1;
  c->sel_n[layer] = s.Blc;
  c->gathered[layer] = 0;
  return sorted_out || rank_out ? do_sort_positions(c, layer, nullptr, s.Blc, sorted_out, rank_out, st) : DKV_OK;
}

// ---- step (3): Update_Buffer_Length ------------------------------------------------------------
// The updates after l[0] < l[1] < ... layers.  fill > 0: the counts of all layers start at `fill` (else they are what
// the selections and earlier updates left).  The last update's integers are left in d_dbg.
int do_rebudget(dkv_ctx* c, const int* l, int n, int fill, int* counts_out, cudaStream_t st) {
  const Shape& s = c->s;
  ProfScope ps(c, DKV_STEP_REBUDGET, 3 * ((n + kRbUpdates - 1) / kRbUpdates), st);
  const size_t per_layer = (size_t)s.Hkv * s.P, cand_stride = (size_t)s.L * per_layer, bl = (size_t)s.Bt * s.L;
  int slices = (int)((per_layer + kRbChunk - 1) / kRbChunk);
  if (slices > 64) slices = 64;
  for (int u0 = 0; u0 < n; u0 += kRbUpdates) {
    RbBatch batch = {};
    batch.n = n - u0 < kRbUpdates ? n - u0 : kRbUpdates;
    for (int u = 0; u < batch.n; ++u) {
      batch.l[u] = l[u0 + u];
      batch.k[u] = (long long)s.N * s.Hkv * batch.l[u];
      const long long pop = (long long)batch.l[u] * s.Hkv * s.P;
      if (batch.k[u] > pop) batch.k[u] = pop;
    }
    DKV_LAUNCH(c, launch_pdl(rb_locate_kernel, dim3(batch.n, s.Bt), 1024, 0, 1, st, batch, (const unsigned int*)c->d_layer_hist, c->d_rb_state,
                             c->d_rb_above, c->d_cand_n, c->d_count, u0 == 0 ? fill : 0, s.Bt, s.Hkv, s.L, s.P));
    DKV_LAUNCH(c, launch_pdl(rb_collect_kernel, dim3(slices, batch.l[batch.n - 1], s.Bt), kRbThreads, 0, 1, st, batch, (const float*)c->d_scores,
                             (const RbState*)c->d_rb_state, c->d_cand, c->d_cand_n, s.Bt, per_layer, cand_stride));
    DKV_LAUNCH(c, launch_pdl(rb_finish_kernel, dim3(kRbCluster, batch.n, s.Bt), 1024, 0, kRbCluster, st, batch, (const RbState*)c->d_rb_state,
                             (const unsigned int*)c->d_rb_above, (const uint2*)c->d_cand, (const unsigned int*)c->d_cand_n, cand_stride, c->d_count,
                             c->d_dbg, c->d_dbg + bl, c->d_dbg + 2 * bl, u0 + batch.n == n ? batch.n - 1 : -1, counts_out, s.Bt, s.L, s.Bl, s.N,
                             (int)((c->cfg.flags & DKV_F_PRORATA) != 0), (int)((c->cfg.flags & DKV_F_NORM_MINMAX) != 0)));
  }
  return DKV_OK;
}

// ---- step (4): gather / shrink ------------------------------------------------------------------
int do_shrink(dkv_ctx* c, int layer0, int n, void* const* kb, void* const* vb, cudaStream_t st) {
  const Shape& s = c->s;
  LayerPtrs ptrs;
  for (int i = 0; i < n; ++i) { ptrs.kb[layer0 + i] = kb[i]; ptrs.vb[layer0 + i] = vb[i]; }
  ProfScope ps(c, DKV_STEP_SHRINK, 1, st);
  DKV_LAUNCH(c, launch_pdl(shrink_kernel, dim3(s.Bt * s.Hkv, n, 2), kShrinkThreads, 0, 1, st, ptrs, layer0, (const int*)c->d_count, c->d_held,
                           c->d_shrink_tickets, s.Hkv, s.L, s.ws, s.rows, s.D * 2 / 16));
  return DKV_OK;
}

int do_gather(dkv_ctx* c, int layer, const void* k_src, const void* v_src, void* kb, void* vb, cudaStream_t st) {
  const Shape& s = c->s;
  const int vec = s.D * 2 / 16, rpb = kGatherThreads / vec * kGatherRows;
  const dim3 grid((s.rows + rpb - 1) / rpb, s.Bt * s.Hkv);
  ProfScope ps(c, DKV_STEP_GATHER, 1, st);
  DKV_LAUNCH(c, launch_pdl(gather_rows_kernel, grid, kGatherThreads, 0, 1, st, static_cast<const uint4*>(k_src), static_cast<const uint4*>(v_src),
                           static_cast<uint4*>(kb), static_cast<uint4*>(vb), (const int*)(c->d_idx + (size_t)layer * layer_idx(s)),
                           (const int*)c->d_count, c->sel_n[layer], s.Blc, s.S, s.P, s.ws, s.rows, vec, c->d_held, s.Hkv, s.L, layer));
  c->gathered[layer] = 1;
  return DKV_OK;
}

// The end of a pass: select and gather every layer with its final count.
int do_select_gather(dkv_ctx* c, const void* const* k, const void* const* v, void* const* kb, void* const* vb, cudaStream_t st) {
  const Shape& s = c->s;
  PassPtrs ptrs;
  for (int l = 0; l < s.L; ++l) { ptrs.k[l] = k[l]; ptrs.v[l] = v[l]; ptrs.kb[l] = kb[l]; ptrs.vb[l] = vb[l]; }
  ProfScope ps(c, DKV_STEP_SELECT, 1, st);
  // A cluster a head, as in do_select, while all blocks fit on the SMs at once, two to each: the blocks share the copying
  // too, so that the line depends on the rows to copy as well (one costs about as much as 16 positions).  Per pass with
  // 1 / 4 / 8 blocks a head and B^l = 128 | 1024: 8 heads of 6144 47 / 49 / 49 | 57 / 51 / 50 us, of 16352 55 / 54 / 55 | 67 / 58 / 57,
  // of 32736 72 / 66 / 65 | 83 / 70 / 67; 32 heads of 16352 90 / 91 / 92 | 102 / 97 / 95; 64 heads of 6144 75 / 79 / 86 | 88 / 85 / 100, of
  // 32736 234 / 233 / 264 | 248 / 237 / 260; 112 heads need two waves: slower.
  const int heads = s.Bt * s.Hkv * s.L;
  const int parts = s.P >= 24576 && heads * 4 <= c->n_sms ? 8 : s.P + 16 * s.Blc >= 20480 && heads * 2 <= c->n_sms ? 4 : 1;
  DKV_LAUNCH(c, launch_pdl(parts > 1 ? select_gather_cluster_kernel : select_gather_kernel, dim3(s.Bt * s.Hkv * parts, s.L), kSelThreads,
                           select_smem(c->sel_cap), parts, st, ptrs, (const float*)c->d_scores,
                           c->d_idx, (const int*)c->d_count, c->d_held, s.P, s.ws, s.Blc, c->sel_cap, s.S, s.D * 2 / 16, s.Hkv, s.L));
  return DKV_OK;
}

// The address under which kernels can use page-locked host memory, if `host` is that (and 16-byte aligned).
bool host_view(const void* host, void** dev) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, host) == cudaSuccess && at.type == cudaMemoryTypeHost && at.devicePointer && aligned16(at.devicePointer)) {
    *dev = at.devicePointer;
    return true;
  }
  cudaGetLastError();                          // an unregistered pointer is not an error here
  return false;
}

// Layer counts after which Algorithm 1 updates the budgets: every m layers, and after the last.
int update_points(const Shape& s, int* l) {
  int n = 0;
  for (int u = s.m; u < s.L; u += s.m) l[n++] = u;
  l[n++] = s.L;
  return n;
}

// What the host knows of the layers.
void forget_layers(dkv_ctx* c) {
  memset(c->scored, 0, sizeof c->scored);
  memset(c->selected, 0, sizeof c->selected);
  memset(c->gathered, 0, sizeof c->gathered);
}

int do_reset(dkv_ctx* c, cudaStream_t st) {
  const Shape& s = c->s;
  forget_layers(c);
  DKV_CUDA(c, cudaMemsetAsync(c->d_count, 0, sizeof(int) * s.Bt * s.L, st));
  DKV_CUDA(c, cudaMemsetAsync(c->d_held, 0, sizeof(int) * s.Bt * s.L, st));
  DKV_CUDA(c, cudaMemsetAsync(c->d_dbg, 0, sizeof(int) * 3 * s.Bt * s.L, st));
  return DKV_OK;
}

// What the host knows after a pass.
void mark_pass_done(dkv_ctx* c) {
  for (int l = 0; l < c->s.L; ++l) { c->scored[l] = c->selected[l] = c->gathered[l] = 1; c->sel_n[l] = c->s.Blc; }
}

// ---- decoding ------------------------------------------------------------------------------------
// QB = 8: up to 8 queries a head group; 16: more than 8, 16 at a time.
template <int D, int QB>
cudaError_t launch_decode(const DecodePtrs& ptrs, const DecodeArgs& a, int cluster, int split_grid, cudaStream_t st) {
  constexpr int NW = QB == 8 ? 8 : 4;
  if (split_grid > 0)
    return launch_pdl(decode_split_kernel<D, QB, 4>, dim3(split_grid), 128, (size_t)(a.nl * a.Bt + 1) * 4, 1, st, ptrs, a);
  return launch_pdl(decode_cluster_kernel<D, QB, NW>, dim3(cluster, a.Bt * a.Hkv, a.nl), NW * 32, 0, cluster, st, ptrs, a);
}

int do_decode(dkv_ctx* c, int layer0, int nl, int nq, const void* const* q, const void* const* kb, const void* const* vb,
              float* const* out, cudaStream_t st) {
  const Shape& s = c->s;
  const int BH = s.Bt * s.Hkv, heads = BH * nl, GQ = s.G * nq;
  DecodeArgs a;
  a.layer0 = layer0; a.nl = nl; a.Bt = s.Bt; a.Hkv = s.Hkv; a.GQ = GQ; a.L = s.L; a.ws = s.ws; a.row_stride = s.rows;
  a.scale2 = kLog2e / sqrtf((float)s.D);
  a.held = c->d_held; a.scratch = nullptr; a.tickets = nullptr;
  // A cluster per head while the heads alone leave SMs idle (as many blocks a head as fit one wave, at most the
  // portable 8, and one row block a warp at least); equal slices of all rows from a head per four SMs on.
  int cluster = 1, split_grid = 0;
  const int warps = GQ <= 8 ? 8 : 4;
  while (cluster < 8 && heads * cluster * 2 <= c->n_sms && cluster * warps * kDecRowBlock < s.rows) cluster *= 2;
  if (heads * 4 > c->n_sms && nl * s.Bt <= kDecMaxPairs) {
    // as many blocks of four warps as are resident at once, but no more warps than there can be row blocks
    const long long most = ((long long)heads * ((s.rows + kDecRowBlock - 1) / kDecRowBlock) + 3) / 4;
    split_grid = c->n_sms * 2;
    if (split_grid > most) split_grid = (int)most;
    const int qb = GQ <= 8 ? 8 : 16;
    const size_t need = (size_t)split_grid * 4 * 2 * ((GQ + qb - 1) / qb) * (qb * s.D + qb * 2);
    if (need > c->dec_scratch_floats) {
      if (c->d_dec_scratch) { DKV_CUDA(c, cudaDeviceSynchronize()); cudaFree(c->d_dec_scratch); c->d_dec_scratch = nullptr; c->dec_scratch_floats = 0; }
      DKV_CUDA(c, cudaMalloc(&c->d_dec_scratch, need * sizeof(float)));
      c->dec_scratch_floats = need;
    }
    a.scratch = c->d_dec_scratch; a.tickets = c->d_dec_tickets + (size_t)layer0 * BH;
  }
  DecodePtrs ptrs;
  for (int i = 0; i < nl; ++i) { ptrs.q[i] = q[i]; ptrs.kb[i] = kb[i]; ptrs.vb[i] = vb[i]; ptrs.out[i] = out[i]; }
  ProfScope ps(c, DKV_STEP_DECODE, 1, st);
  cudaError_t e;
  if (s.D == 128) e = GQ <= 8 ? launch_decode<128, 8>(ptrs, a, cluster, split_grid, st) : launch_decode<128, 16>(ptrs, a, cluster, split_grid, st);
  else e = GQ <= 8 ? launch_decode<64, 8>(ptrs, a, cluster, split_grid, st) : launch_decode<64, 16>(ptrs, a, cluster, split_grid, st);
  DKV_LAUNCH(c, e);
  return DKV_OK;
}

// Algorithm 1's loop, one chain of launches on `st`.
//   scoring   by score_sweep.cuh, up to 32 layers at a time: row sums, key sums, pooling; with `lse` (the window rows'
//             log-denominators of every layer) the last two.  Or by score_tc.cuh (pass_by_sweeps): launch g runs sweep 2 of layer
//             group g-1 and then sweep 1 of group g (a group = up to `pass_group` layers, so that the fixed cost of a launch is
//             paid once per group).  Either counts the scores' digits.
//   updates   all of Eq. 4-6's updates together: their order does not matter, a layer's count is the minimum over them
//             and nothing reads an intermediate one.
//   select, gather   with the final counts.
// (Selecting and gathering B^l rows of each layer and truncating them at every update, on side streams beside the
// scoring, took 32 of the 148 SMs from the scoring kernel and still left a tail of 0.1 ms after the last layer.)
int do_pass(dkv_ctx* c, const void* const* q, const void* const* k, const void* const* v, const float* const* lse,
            void* const* kb, void* const* vb, cudaStream_t st) {
  const Shape& s = c->s;
  const int most = most_layers(c);
  int rc, l[DKV_MAX_LAYERS];
  if (lse || pass_by_sweeps(c)) {
    for (int i = 0; i < s.L; i += most) {
      const int nl = s.L - i < most ? s.L - i : most;
      if ((rc = launch_sweeps(c, i, nl, q + i, k + i, lse ? lse + i : nullptr, st))) return rc;
    }
  } else {
    ScoreGroup prev = {}, cur = {};
    for (int g = 0, done = 0; done < s.L || prev.n; ++g) {
      cur.first = done; cur.n = s.L - done < c->pass_group ? s.L - done : c->pass_group; cur.buf = g % 3;
      done += cur.n;
      if ((rc = launch_score<tc::kMaxGroup>(c, prev.n ? &prev : nullptr, cur.n ? &cur : nullptr, q, k, nullptr, nullptr, true, st))) return rc;
      prev = cur;
    }
  }
  if ((rc = do_rebudget(c, l, update_points(s, l), s.Blc, nullptr, st))) return rc;
  if ((rc = do_select_gather(c, k, v, kb, vb, st))) return rc;
  mark_pass_done(c);
  return DKV_OK;
}

// All of it, or as much as there is of it.
void free_staging(dkv_ctx* c) {
  for (int i = 0; i < 2; ++i) {
    for (void** p : {&c->st_q[i], &c->st_k[i], &c->st_v[i]}) { cudaFree(*p); *p = nullptr; }
    for (cudaEvent_t* e : {&c->ev_copied[i], &c->ev_consumed[i]}) if (*e) { cudaEventDestroy(*e); *e = nullptr; }
  }
  for (int l = 0; l < c->s.L; ++l) for (void** p : {&c->st_kb[l], &c->st_vb[l]}) { cudaFree(*p); *p = nullptr; }
  for (cudaStream_t* s : {&c->st_copy, &c->st_comp}) if (*s) { cudaStreamDestroy(*s); *s = nullptr; }
  c->staged = false;
}

void free_all(dkv_ctx* c) {
  cudaFree(c->d_scores); cudaFree(c->d_idx); cudaFree(c->d_count); cudaFree(c->d_held); cudaFree(c->d_dbg);
  cudaFree(c->d_rb_state); cudaFree(c->d_rb_above); cudaFree(c->d_layer_hist); cudaFree(c->d_shrink_tickets);
  cudaFree(c->d_cand); cudaFree(c->d_cand_n); cudaFree(c->d_status); cudaFree(c->d_tc_stats); cudaFree(c->d_stats);
  cudaFree(c->d_dec_scratch); cudaFree(c->d_dec_tickets);
  if (c->prof_recs) {
    for (ProfRec& r : *c->prof_recs) { cudaEventDestroy(r.a); cudaEventDestroy(r.b); }
    delete c->prof_recs;
  }
  free_staging(c);
}

int make_staging(dkv_ctx* c) {
  const Shape& s = c->s;
  for (int i = 0; i < 2; ++i) {
    DKV_CUDA(c, cudaMalloc(&c->st_q[i], layer_q_bytes(s)));
    DKV_CUDA(c, cudaMalloc(&c->st_k[i], layer_kv_bytes(s)));
    DKV_CUDA(c, cudaMalloc(&c->st_v[i], layer_kv_bytes(s)));
    DKV_CUDA(c, cudaEventCreateWithFlags(&c->ev_copied[i], cudaEventDisableTiming));
    DKV_CUDA(c, cudaEventCreateWithFlags(&c->ev_consumed[i], cudaEventDisableTiming));
  }
  for (int l = 0; l < s.L; ++l) {
    DKV_CUDA(c, cudaMalloc(&c->st_kb[l], layer_buf_bytes(s)));
    DKV_CUDA(c, cudaMalloc(&c->st_vb[l], layer_buf_bytes(s)));
  }
  DKV_CUDA(c, cudaStreamCreateWithFlags(&c->st_copy, cudaStreamNonBlocking));
  DKV_CUDA(c, cudaStreamCreateWithFlags(&c->st_comp, cudaStreamNonBlocking));
  return DKV_OK;
}

int ensure_staging(dkv_ctx* c) {
  if (c->staged) return DKV_OK;
  const int rc = make_staging(c);
  if (rc) free_staging(c);                     // a later call starts anew
  c->staged = rc == DKV_OK;
  return rc;
}

}  // namespace

extern "C" {

int dkv_version(void) { return 1000; }

const char* dkv_strerror(int code) {
  switch (code) {
    case DKV_OK: return "ok";
    case DKV_ERR_INVALID_ARG: return "invalid argument";
    case DKV_ERR_STATE: return "call out of order for this layer";
    case DKV_ERR_CUDA: return "CUDA runtime error";
    case DKV_ERR_TIMEOUT: return "device-side wait timed out";
    case DKV_ERR_UNSUPPORTED: return "shape not supported";
    case DKV_ERR_NOMEM: return "out of memory";
    case DKV_ERR_TOO_LARGE: return "problem needs more scratch than the static array holds";
    default: return "unknown error";
  }
}

int dkv_create(const dkv_config* cfg, dkv_ctx** out) {
  if (!out) return DKV_ERR_INVALID_ARG;
  *out = nullptr;
  int rc = validate(cfg);
  if (rc) return rc;
  dkv_ctx* c = new (std::nothrow) dkv_ctx;
  if (!c) return DKV_ERR_NOMEM;
  memset(c, 0, sizeof *c);
  c->cfg = *cfg;
  c->prof_recs = new (std::nothrow) std::vector<ProfRec>();
  if (!c->prof_recs) { delete c; return DKV_ERR_NOMEM; }
  Shape& s = c->s;
  s.L = cfg->n_layers; s.Hq = cfg->n_q_heads; s.Hkv = cfg->n_kv_heads; s.D = cfg->head_dim; s.Bt = cfg->batch;
  s.S = cfg->seq_len; s.ws = cfg->window; s.pool = cfg->pool_kernel; s.N = cfg->avg_budget; s.Bl = cfg->layer_max;
  s.m = cfg->update_interval;
  s.G = s.Hq / s.Hkv; s.P = s.S - s.ws; s.M = s.ws * s.G; s.Blc = s.Bl < s.P ? s.Bl : s.P; s.rows = s.Blc + s.ws;
  const int heads = s.Bt * s.Hkv;
  c->planes = (s.M + 127) / 128;
  c->plane_rows = c->planes == 1 ? s.M : (s.M + 31) / 32 * 16;
  c->sel_cap = 1024;                                       // a quarter more than B^l for the rest of the threshold's digit
  while (c->sel_cap < s.Blc + s.Blc / 4 && c->sel_cap < DKV_MAX_LAYER_BUDGET) c->sel_cap <<= 1;

  cudaError_t e = cudaGetDevice(&c->device);
  {
    int sms = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
    c->n_sms = sms > 0 ? sms : 1;
    // Layers per scoring launch of a pass that score_tc.cuh scores: enough that a thread block has about 110 tiles a sweep.  A launch costs some 8 us
    // (fill, drain, statistics) whatever it does: 32 layers of 8K in launches of 8 / 16 / 32 layers take 299 / 290 / 286 us;
    // at 32K eight layers are as good as more.
    const long long tiles = (long long)heads * ((s.S + tc::kTileKeys - 1) / tc::kTileKeys), want = (110ll * c->n_sms + tiles - 1) / tiles;
    int g = want < s.L ? (int)want : s.L;
    if (g > tc::kMaxGroup) g = tc::kMaxGroup;
    const int launches = (s.L + g - 1) / g;
    c->pass_group = env_int("DKV_PASS_GROUP", (s.L + launches - 1) / launches, 1, tc::kMaxGroup);
    // (stats_slots of a job's heads; score_tc.cuh's jobs are single layers where passes are scored by score_sweep.cuh)
    c->stats_rows = (size_t)c->n_sms + 2 * (size_t)(pass_by_sweeps(c) ? 1 : c->pass_group) * heads;
    c->emit_backward = env_int("DKV_EMIT_FORWARD", 0, 0, 1) == 0;
    // Sweep 2 starts on the keys sweep 1 streamed last: that much of a job (4/7 of L2, 72 of 126 MB) is loaded with
    // an evict-last policy, every other key tile and the gather's rows evict-first, so that the rest of the
    // stream does not push it out before it is read again.
    int l2_bytes = 0;
    if (cudaDeviceGetAttribute(&l2_bytes, cudaDevAttrL2CacheSize, c->device) != cudaSuccess) l2_bytes = 0;
    c->retain_mb = c->emit_backward ? env_int("DKV_L2_RETAIN_MB", (int)(((long long)l2_bytes * 4 / 7) >> 20), 0, 1024) : 0;
    c->host_v_staged = env_int("DKV_HOST_V_STAGED", 0, 0, 1) != 0;
    c->host_h2d = c->host_d2h = 0;
    c->wait_cycles = tc::kDefaultWaitCycles;
    c->withhold_sweep = c->withhold_tile = -1;
  }
  const size_t bl = (size_t)s.Bt * s.L;
#define TRY(call) if (e == cudaSuccess) e = (call)
  TRY(cudaMalloc(&c->d_scores, sizeof(float) * s.L * layer_scores(s)));
  TRY(cudaMalloc(&c->d_idx, sizeof(int) * s.L * layer_idx(s)));
  TRY(cudaMalloc(&c->d_count, sizeof(int) * bl));
  TRY(cudaMalloc(&c->d_held, sizeof(int) * bl));
  TRY(cudaMalloc(&c->d_dbg, sizeof(int) * 3 * bl));
  TRY(cudaMalloc(&c->d_rb_state, sizeof(RbState) * kRbUpdates * s.Bt));
  TRY(cudaMalloc(&c->d_rb_above, sizeof(unsigned int) * kRbUpdates * bl));
  TRY(cudaMalloc(&c->d_shrink_tickets, sizeof(unsigned int) * bl));
  TRY(cudaMemset(c->d_shrink_tickets, 0, sizeof(unsigned int) * bl));
  TRY(cudaMalloc(&c->d_layer_hist, sizeof(unsigned int) * s.L * s.Bt * kBins));
  {
    const int most = most_layers(c);
    TRY(cudaMalloc(&c->d_cand, std::max(sizeof(uint2) * s.L * layer_scores(s), sizeof(float) * most * heads * c->planes * tiles_per_head(s) * tc::kTileKeys)));
    // Row sums; a launch over fewer layers than `most` (the last of a pass) has more segments a head, but no more in all.
    if (pass_by_sweeps(c)) TRY(cudaMalloc(&c->d_stats, sizeof(float2) * c->plane_rows * (2 * c->n_sms + 2 * most * heads * c->planes)));
    TRY(set_sweep_attributes(row_blocks(c), pass_by_sweeps(c), long_heads(c)));
  }
  TRY(cudaMalloc(&c->d_cand_n, sizeof(unsigned int) * s.Bt));
  TRY(cudaMalloc(&c->d_tc_stats, sizeof(float2) * 3 * c->stats_rows * 256));
  TRY(set_score_attribute<1>(s.M, s.D));
  if (!pass_by_sweeps(c)) TRY(set_score_attribute<tc::kMaxGroup>(s.M, s.D));
  TRY(cudaMalloc(&c->d_status, sizeof(int) * 8));
  TRY(cudaMemset(c->d_status, 0, sizeof(int) * 8));
  TRY(cudaMemset(c->d_count, 0, sizeof(int) * bl));
  TRY(cudaMemset(c->d_held, 0, sizeof(int) * bl));
  TRY(cudaMemset(c->d_dbg, 0, sizeof(int) * 3 * bl));
  TRY(cudaMalloc(&c->d_dec_tickets, sizeof(unsigned int) * s.L * heads));
  TRY(cudaMemset(c->d_dec_tickets, 0, sizeof(unsigned int) * s.L * heads));
  // The words above are cleared on the legacy default stream, for which the first kernel of a caller's non-blocking stream
  // does not wait.
  TRY(cudaStreamSynchronize(cudaStreamLegacy));
  // The attributes belong to the functions, not to this context: always the most any valid configuration needs, so that
  // contexts do not undo each other.
  {
    const int most = (int)(select_smem(kMaxCountingList) > select_smem(DKV_MAX_LAYER_BUDGET) ? select_smem(kMaxCountingList) : select_smem(DKV_MAX_LAYER_BUDGET));
    TRY(cudaFuncSetAttribute(select_topk_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    TRY(cudaFuncSetAttribute(select_topk_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    TRY(cudaFuncSetAttribute(select_gather_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    TRY(cudaFuncSetAttribute(select_gather_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    TRY(cudaFuncSetAttribute(sort_positions_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DKV_MAX_LAYER_BUDGET * 8));
  }
#undef TRY
  if (e != cudaSuccess) {
    rc = e == cudaErrorMemoryAllocation ? DKV_ERR_NOMEM : DKV_ERR_CUDA;
    cudaGetLastError();
    free_all(c);
    delete c;
    return rc;
  }
  *out = c;
  return DKV_OK;
}

int dkv_destroy(dkv_ctx* c) {
  if (!c) return DKV_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  free_all(c);
  delete c;
  return DKV_OK;
}

int dkv_reset(dkv_ctx* c, void* stream) {
  if (!c) return DKV_ERR_INVALID_ARG;
  return do_reset(c, as_stream(stream));
}

int dkv_score(dkv_ctx* c, int32_t layer, const void* q_win, const void* k, float* scores_out, void* stream) {
  int rc = check_layer(c, layer);
  if (rc) return rc;
  if (!q_win || !k || !aligned16(q_win) || !aligned16(k) || !aligned16(scores_out)) return DKV_ERR_INVALID_ARG;
  return do_score(c, layer, q_win, k, nullptr, scores_out, as_stream(stream));
}

int dkv_score_lse(dkv_ctx* c, int32_t layer, const void* q_win, const void* k, const float* lse, float* scores_out,
                  void* stream) {
  int rc = check_layer(c, layer);
  if (rc) return rc;
  if (!q_win || !k || !lse || !aligned16(q_win) || !aligned16(k) || !aligned16(scores_out) || ((uintptr_t)lse & 3))
    return DKV_ERR_INVALID_ARG;
  return do_score(c, layer, q_win, k, lse, scores_out, as_stream(stream));
}

int dkv_set_scores(dkv_ctx* c, int32_t layer, const float* scores, void* stream) {
  int rc = check_layer(c, layer);
  if (rc) return rc;
  if (!scores) return DKV_ERR_INVALID_ARG;
  const size_t n = layer_scores(c->s);
  DKV_CUDA(c, cudaMemcpyAsync(c->d_scores + (size_t)layer * n, scores, n * sizeof(float), cudaMemcpyDeviceToDevice,
                              as_stream(stream)));
  c->scored[layer] = 1;
  c->selected[layer] = c->gathered[layer] = 0;
  return DKV_OK;
}

int dkv_select_topk(dkv_ctx* c, int32_t layer, int32_t* idx_out, int32_t* rank_out, void* stream) {
  int rc = check_layer(c, layer);
  if (rc) return rc;
  if (!c->scored[layer]) return DKV_ERR_STATE;
  return do_select(c, layer, idx_out, rank_out, as_stream(stream));
}

int dkv_rebudget(dkv_ctx* c, int32_t upto_layer, int32_t* counts_out, void* stream) {
  if (!c || upto_layer < 1 || upto_layer > c->s.L) return DKV_ERR_INVALID_ARG;
  for (int i = 0; i < upto_layer; ++i) if (!c->scored[i] || c->selected[i] != 1) return DKV_ERR_STATE;
  return do_rebudget(c, &upto_layer, 1, 0, counts_out, as_stream(stream));
}

int dkv_compact(dkv_ctx* c, int32_t layer, const void* k_src, const void* v_src, void* kb, void* vb, int32_t* len_out,
                void* stream) {
  int rc = check_layer(c, layer);
  if (rc) return rc;
  if (!kb || !vb || !aligned16(kb) || !aligned16(vb)) return DKV_ERR_INVALID_ARG;
  if ((k_src == nullptr) != (v_src == nullptr)) return DKV_ERR_INVALID_ARG;
  if (!aligned16(k_src) || !aligned16(v_src)) return DKV_ERR_INVALID_ARG;
  cudaStream_t st = as_stream(stream);
  if (k_src) {
    if (!c->selected[layer]) return DKV_ERR_STATE;
    rc = do_gather(c, layer, k_src, v_src, kb, vb, st);
  } else {
    if (!c->gathered[layer]) return DKV_ERR_STATE;
    rc = do_shrink(c, layer, 1, &kb, &vb, st);
  }
  if (rc) return rc;
  if (len_out) {
    const Shape& s = c->s;
    write_len_kernel<<<(s.Bt * s.Hkv + 127) / 128, 128, 0, st>>>(len_out, c->d_held, s.Bt, s.Hkv, s.L, layer, s.ws);
    DKV_LAUNCHED(c);
  }
  return DKV_OK;
}

int dkv_compact_all(dkv_ctx* c, int32_t upto_layer, void* const* kb, void* const* vb, void* stream) {
  if (!c || !kb || !vb || upto_layer < 1 || upto_layer > c->s.L) return DKV_ERR_INVALID_ARG;
  for (int i = 0; i < upto_layer; ++i) {
    if (!kb[i] || !vb[i] || !aligned16(kb[i]) || !aligned16(vb[i])) return DKV_ERR_INVALID_ARG;
    if (!c->gathered[i]) return DKV_ERR_STATE;
  }
  return do_shrink(c, 0, upto_layer, kb, vb, as_stream(stream));
}

static int run_pass(dkv_ctx* c, const void* const* q_win, const void* const* k, const void* const* v,
                    const float* const* lse, void* const* kb, void* const* vb, void* stream) {
  if (!c || !q_win || !k || !v || !kb || !vb) return DKV_ERR_INVALID_ARG;
  for (int l = 0; l < c->s.L; ++l) {
    if (!q_win[l] || !k[l] || !v[l] || !kb[l] || !vb[l]) return DKV_ERR_INVALID_ARG;
    if (!aligned16(q_win[l]) || !aligned16(k[l]) || !aligned16(v[l]) || !aligned16(kb[l]) || !aligned16(vb[l]))
      return DKV_ERR_INVALID_ARG;
    if (lse && (!lse[l] || ((uintptr_t)lse[l] & 3))) return DKV_ERR_INVALID_ARG;
  }
  // A pass overwrites every word of the counts, the held rows and the update's integers itself, so that the reset it begins
  // with is needed on the device only if a launch is refused midway.
  cudaStream_t st = as_stream(stream);
  forget_layers(c);
  const int rc = do_pass(c, q_win, k, v, lse, kb, vb, st);
  if (rc) {
    const int why = c->last_cuda;
    do_reset(c, st);
    c->last_cuda = why;
  }
  return rc;
}

int dkv_run_prefill_pass(dkv_ctx* c, const void* const* q_win, const void* const* k, const void* const* v,
                         void* const* kb, void* const* vb, void* stream) {
  return run_pass(c, q_win, k, v, nullptr, kb, vb, stream);
}

int dkv_run_prefill_pass_lse(dkv_ctx* c, const void* const* q_win, const void* const* k, const void* const* v,
                             const float* const* lse, void* const* kb, void* const* vb, void* stream) {
  if (!lse) return DKV_ERR_INVALID_ARG;
  return run_pass(c, q_win, k, v, lse, kb, vb, stream);
}

// The host-buffer pass up to its results, on the context's own streams.
static int host_pass(dkv_ctx* c, const void* const* q_win, const void* const* k, const void* const* v, void* const* kb,
                     void* const* vb, int32_t* counts_out) {
  const Shape& s = c->s;
  int rc;
  cudaStream_t cp = c->st_copy, st = c->st_comp;
  if ((rc = do_reset(c, st))) return rc;
  // Only the kept rows of V are ever needed on the device (count + ws of S per head).  Where the caller's V is
  // page-locked host memory that kernels can address, the gather reads exactly those rows over the bus instead of
  // V being copied in full first; pageable memory (or DKV_HOST_V_STAGED=1) takes the full copy.
  const void* v_dev[DKV_MAX_LAYERS];
  for (int l = 0; l < s.L; ++l) {
    void* p = nullptr;
    v_dev[l] = !c->host_v_staged && host_view(v[l], &p) ? p : nullptr;
  }
  // Page-locked output buffers are written by one kernel at the end.
  PassPtrs out;
  bool out_mapped = true;
  for (int l = 0; l < s.L && out_mapped; ++l) {
    out.k[l] = c->st_kb[l]; out.v[l] = c->st_vb[l];
    out_mapped = host_view(kb[l], &out.kb[l]) && host_view(vb[l], &out.vb[l]);
  }
  const long long row_bytes = (long long)s.D * 2;
  long long h2d = 0;
  for (int l = 0; l < s.L; ++l) {
    const int slot = l & 1;
    if (l >= 2) DKV_CUDA(c, cudaStreamWaitEvent(cp, c->ev_consumed[slot], 0));
    DKV_CUDA(c, cudaMemcpyAsync(c->st_q[slot], q_win[l], layer_q_bytes(s), cudaMemcpyHostToDevice, cp));
    DKV_CUDA(c, cudaMemcpyAsync(c->st_k[slot], k[l], layer_kv_bytes(s), cudaMemcpyHostToDevice, cp));
    h2d += (long long)layer_q_bytes(s) + (long long)layer_kv_bytes(s);
    if (!v_dev[l]) {
      DKV_CUDA(c, cudaMemcpyAsync(c->st_v[slot], v[l], layer_kv_bytes(s), cudaMemcpyHostToDevice, cp));
      h2d += (long long)layer_kv_bytes(s);
    }
    DKV_CUDA(c, cudaEventRecord(c->ev_copied[slot], cp));
    DKV_CUDA(c, cudaStreamWaitEvent(st, c->ev_copied[slot], 0));
    if ((rc = do_score(c, l, c->st_q[slot], c->st_k[slot], nullptr, nullptr, st))) return rc;
    if ((rc = do_select(c, l, nullptr, nullptr, st))) return rc;
    if ((rc = do_gather(c, l, c->st_k[slot], v_dev[l] ? v_dev[l] : c->st_v[slot], c->st_kb[l], c->st_vb[l], st))) return rc;
    if (v_dev[l]) h2d += (long long)(c->sel_n[l] + s.ws) * s.Bt * s.Hkv * row_bytes;
    DKV_CUDA(c, cudaEventRecord(c->ev_consumed[slot], st));
  }
  // all updates together, as in do_pass
  int upd[DKV_MAX_LAYERS];
  if ((rc = do_rebudget(c, upd, update_points(s, upd), 0, nullptr, st))) return rc;
  if ((rc = do_shrink(c, 0, s.L, c->st_kb, c->st_vb, st))) return rc;
  if (out_mapped) {
    const int per_block = kGatherThreads / (s.D * 2 / 16) * kGatherRows;
    DKV_LAUNCH(c, launch_pdl(copy_valid_kernel, dim3((s.rows + per_block - 1) / per_block, s.Bt * s.Hkv, s.L), kGatherThreads, 0, 1, st, out,
                             (const int*)c->d_held, s.ws, s.rows, s.D * 2 / 16, s.Hkv, s.L));
  }
  std::vector<int> counts((size_t)s.Bt * s.L);
  DKV_CUDA(c, cudaMemcpyAsync(counts.data(), c->d_count, sizeof(int) * s.Bt * s.L, cudaMemcpyDeviceToHost, st));
  DKV_CUDA(c, cudaStreamSynchronize(st));
  if (!out_mapped) {                           // one strided copy of the valid rows per (layer, sample, tensor)
    const size_t row = (size_t)s.D * 2, head_pitch = (size_t)s.rows * row, sample = (size_t)s.Hkv * head_pitch;
    for (int l = 0; l < s.L; ++l)
      for (int b = 0; b < s.Bt; ++b) {
        const size_t valid = (size_t)(counts[(size_t)b * s.L + l] + s.ws) * row;
        DKV_CUDA(c, cudaMemcpy2DAsync(static_cast<char*>(kb[l]) + b * sample, head_pitch,
                                      static_cast<const char*>(c->st_kb[l]) + b * sample, head_pitch, valid, s.Hkv,
                                      cudaMemcpyDeviceToHost, st));
        DKV_CUDA(c, cudaMemcpy2DAsync(static_cast<char*>(vb[l]) + b * sample, head_pitch,
                                      static_cast<const char*>(c->st_vb[l]) + b * sample, head_pitch, valid, s.Hkv,
                                      cudaMemcpyDeviceToHost, st));
      }
    DKV_CUDA(c, cudaStreamSynchronize(st));
  }
  if (counts_out) memcpy(counts_out, counts.data(), sizeof(int) * s.Bt * s.L);
  long long d2h = (long long)sizeof(int) * s.Bt * s.L;
  for (size_t i = 0; i < counts.size(); ++i) d2h += 2ll * (counts[i] + s.ws) * s.Hkv * row_bytes;
  c->host_h2d = h2d; c->host_d2h = d2h;
  DKV_CUDA(c, cudaStreamSynchronize(cp));
  return DKV_OK;
}

int dkv_run_prefill_pass_host(dkv_ctx* c, const void* const* q_win, const void* const* k, const void* const* v,
                              void* const* kb, void* const* vb, int32_t* counts_out) {
  if (!c || !q_win || !k || !v || !kb || !vb) return DKV_ERR_INVALID_ARG;
  for (int l = 0; l < c->s.L; ++l)
    if (!q_win[l] || !k[l] || !v[l] || !kb[l] || !vb[l]) return DKV_ERR_INVALID_ARG;
  int rc = ensure_staging(c);
  if (!rc) rc = host_pass(c, q_win, k, v, kb, vb, counts_out);
  if (rc && c->staged) {
    // what was enqueued before the refused call still reads and writes the caller's buffers: it ends before the call does
    const int why = c->last_cuda;
    cudaStreamSynchronize(c->st_copy);
    cudaStreamSynchronize(c->st_comp);
    do_reset(c, c->st_comp);
    cudaStreamSynchronize(c->st_comp);
    cudaGetLastError();
    c->last_cuda = why;
  }
  return rc;
}

int dkv_host_pass_bytes(dkv_ctx* c, int64_t* h2d, int64_t* d2h) {
  if (!c || !h2d || !d2h) return DKV_ERR_INVALID_ARG;
  *h2d = c->host_h2d; *d2h = c->host_d2h;
  return DKV_OK;
}

int dkv_apply_policy(dkv_ctx* c, int32_t policy, int32_t* counts_out, void* stream) {
  if (!c || (policy != DKV_POLICY_UNIFORM && policy != DKV_POLICY_PYRAMID)) return DKV_ERR_INVALID_ARG;
  const Shape& s = c->s;
  for (int i = 0; i < s.L; ++i) if (!c->selected[i]) return DKV_ERR_STATE;
  policy_counts_kernel<<<(s.Bt * s.L + 127) / 128, 128, 0, as_stream(stream)>>>(c->d_count, counts_out, s.Bt, s.L, s.N, policy);
  DKV_LAUNCHED(c);
  return DKV_OK;
}

int dkv_select_positions(dkv_ctx* c, int32_t layer, int32_t n_sink, int32_t n_recent, void* stream) {
  int rc = check_layer(c, layer);
  if (rc) return rc;
  const Shape& s = c->s;
  if (n_sink < 0 || n_recent < 0) return DKV_ERR_INVALID_ARG;
  if (n_sink > s.P) n_sink = s.P;
  if (n_recent > s.P) n_recent = s.P;
  const int first_recent = s.P - n_recent > n_sink ? s.P - n_recent : n_sink;
  const int n = n_sink + (s.P - first_recent);
  if (n > s.Blc) return DKV_ERR_INVALID_ARG;
  {
    const dim3 grid((n + 255) / 256 > 0 ? (n + 255) / 256 : 1, s.Bt * s.Hkv);
    positions_kernel<<<grid, 256, 0, as_stream(stream)>>>(c->d_idx + (size_t)layer * layer_idx(s), c->d_count, s.P, s.Blc, n_sink,
                                                         first_recent, n, s.Hkv, s.L, layer);
    DKV_LAUNCHED(c);
  }
  c->selected[layer] = 2;
  c->sel_n[layer] = n;
  c->gathered[layer] = 0;
  return DKV_OK;
}

int dkv_decode_attend(dkv_ctx* c, int32_t layer0, int32_t n_layers, int32_t nq, const void* const* q_dec,
                      const void* const* kb, const void* const* vb, float* const* out, void* stream) {
  if (!c || !q_dec || !kb || !vb || !out) return DKV_ERR_INVALID_ARG;
  const Shape& s = c->s;
  if (layer0 < 0 || n_layers < 1 || layer0 + n_layers > s.L || nq < 1 || (long long)nq * s.G > 64) return DKV_ERR_INVALID_ARG;
  for (int i = 0; i < n_layers; ++i) {
    if (!q_dec[i] || !kb[i] || !vb[i] || !out[i]) return DKV_ERR_INVALID_ARG;
    if (!aligned16(q_dec[i]) || !aligned16(kb[i]) || !aligned16(vb[i]) || !aligned16(out[i])) return DKV_ERR_INVALID_ARG;
    if (!c->gathered[layer0 + i]) return DKV_ERR_STATE;
  }
  cudaStream_t st = as_stream(stream);
  for (int l0 = 0; l0 < n_layers; l0 += kDecMaxLayers) {
    const int nl = n_layers - l0 < kDecMaxLayers ? n_layers - l0 : kDecMaxLayers;
    const int rc = do_decode(c, layer0 + l0, nl, nq, q_dec + l0, kb + l0, vb + l0, out + l0, st);
    if (rc) return rc;
  }
  return DKV_OK;
}

int dkv_get_counts(dkv_ctx* c, int32_t* host_counts, void* stream) {
  if (!c || !host_counts) return DKV_ERR_INVALID_ARG;
  DKV_CUDA(c, cudaMemcpyAsync(host_counts, c->d_count, sizeof(int) * c->s.Bt * c->s.L, cudaMemcpyDeviceToHost,
                              as_stream(stream)));
  DKV_CUDA(c, cudaStreamSynchronize(as_stream(stream)));
  return DKV_OK;
}

int dkv_layer_views(dkv_ctx* c, int32_t layer, const float** scores, const int32_t** idx) {
  int rc = check_layer(c, layer);
  if (rc) return rc;
  if (scores) *scores = c->d_scores + (size_t)layer * layer_scores(c->s);
  if (idx) *idx = c->d_idx + (size_t)layer * layer_idx(c->s);
  return DKV_OK;
}

int dkv_kept_sorted(dkv_ctx* c, int32_t layer, int32_t* sorted_out, void* stream) {
  int rc = check_layer(c, layer);
  if (rc) return rc;
  if (!sorted_out) return DKV_ERR_INVALID_ARG;
  if (!c->gathered[layer]) return DKV_ERR_STATE;
  return do_sort_positions(c, layer, c->d_held, c->sel_n[layer], sorted_out, nullptr, as_stream(stream));
}

int dkv_budget_views(dkv_ctx* c, const int32_t** cnt, const int32_t** z, const int32_t** zp, const int32_t** held) {
  if (!c) return DKV_ERR_INVALID_ARG;
  const size_t bl = (size_t)c->s.Bt * c->s.L;
  if (cnt) *cnt = c->d_dbg;
  if (z) *z = c->d_dbg + bl;
  if (zp) *zp = c->d_dbg + 2 * bl;
  if (held) *held = c->d_held;
  return DKV_OK;
}

// ---- scoring for callers that cannot allocate ------------------------------------------------------
// Scratch of dkv_score_static: [0, 256) status words, then the partial softmax statistics of
// sweep 1.  The array lives in every GPU that loads the library, from load to exit.  In host code
// its name is only a handle: the device address comes from cudaGetSymbolAddress, once per device.
static __device__ __align__(256) unsigned char g_static_scratch[DKV_STATIC_SCRATCH_BYTES];

namespace {
struct StaticSetup { bool done; unsigned char* ptr; int sms; };
StaticSetup g_static_setup[64];
std::mutex g_static_mutex;
}  // namespace

int dkv_score_static(const dkv_config* cfg, const void* q_win, const void* k, float* scores_out, void* stream) {
  int rc = validate(cfg);
  if (rc) return rc;
  if (!q_win || !k || !scores_out || !aligned16(q_win) || !aligned16(k) || !aligned16(scores_out))
    return DKV_ERR_INVALID_ARG;
  int dev = -1;
  DKV_CUDA(nullptr, cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return DKV_ERR_CUDA;
  StaticSetup su;
  {
    std::lock_guard<std::mutex> lock(g_static_mutex);
    StaticSetup& g = g_static_setup[dev];
    if (!g.done) {                           // first call on this device
      void* ptr = nullptr;
      DKV_CUDA(nullptr, cudaGetSymbolAddress(&ptr, g_static_scratch));
      int sms = 0;
      DKV_CUDA(nullptr, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
      if (!ptr || sms < 1) return DKV_ERR_CUDA;
      for (const int* m : (const int[][2]){{128, 128}, {32, 128}, {64, 128}, {256, 128}})      // later calls may have any shape
        DKV_CUDA(nullptr, set_score_attribute<1>(m[0], m[1]));
      g.ptr = static_cast<unsigned char*>(ptr);
      g.sms = sms;
      g.done = true;
    }
    su = g;
  }
  const int G = cfg->n_q_heads / cfg->n_kv_heads, heads = cfg->batch * cfg->n_kv_heads;
  const int S = cfg->seq_len, P = S - cfg->window, M = cfg->window * G, D = cfg->head_dim;
  const int tph = (S + tc::kTileKeys - 1) / tc::kTileKeys;
  const long long total_tiles = (long long)heads * tph;
  const int grid = (int)(total_tiles < su.sms ? total_tiles : su.sms);
  int slots = 1;
  for (int bh = 0; bh < heads; ++bh) {
    const int lo = tc::tile_owner((long long)bh * tph, total_tiles, grid);
    const int hi = tc::tile_owner((long long)(bh + 1) * tph - 1, total_tiles, grid);
    if (hi - lo + 1 > slots) slots = hi - lo + 1;
  }
  const unsigned long long need = 256ull + (unsigned long long)heads * slots * 256ull * sizeof(float2);
  if (need > DKV_STATIC_SCRATCH_BYTES) return DKV_ERR_TOO_LARGE;
  cudaStream_t st = as_stream(stream);
  tc::Maps<1> maps;
  maps.lse[0] = nullptr;
  if (!make_map(&maps.q[0], q_win, D, M, heads, 128 / query_copies(M)) || !make_map(&maps.k[0], k, D, S, heads)) return DKV_ERR_CUDA;
  DKV_CUDA(nullptr, cudaMemsetAsync(su.ptr, 0, 256, st));   // status words start at zero
  tc::Params p, none;
  memset(&p, 0, sizeof p);
  memset(&none, 0, sizeof none);
  none.mode = tc::kNone;
  p.S = S; p.P = P; p.ws = cfg->window; p.M = M; p.D = D; p.heads = heads; p.half = cfg->pool_kernel / 2;
  p.nl = 1; p.hpl = heads;
  p.back = 0;
  p.wait_cycles = tc::kDefaultWaitCycles;
  p.withhold_tile = -1;
  p.tph = tph; p.nq16 = (M + 15) / 16 * 16; p.nmblk = (M + 127) / 128;
  p.slots = slots; p.m_stride = 256;
  p.scale2 = kLog2e / sqrtf((float)D);
  p.out_scale = (cfg->flags & DKV_F_WINDOW_MEAN) ? 1.0f / (float)M : 1.0f;
  p.pool_avg = cfg->pool_kind == 1;
  p.stats = reinterpret_cast<float2*>(su.ptr + 256);
  p.scores = scores_out; p.copy_out = nullptr;
  p.status = reinterpret_cast<int*>(su.ptr);
  p.stats_grid = grid;
  p.mode = tc::kStats;
  p.idesc = make_idesc(128, 128);
  DKV_CUDA(nullptr, launch_tc(grid, st, maps, maps, p, none));
  p.mode = tc::kEmit;
  p.idesc = make_idesc(128, p.nq16);
  DKV_CUDA(nullptr, launch_tc(grid, st, maps, maps, none, p));
  return DKV_OK;
}

int dkv_memcpy_to_host(dkv_ctx* c, void* host_dst, const void* dev_src, uint64_t bytes, void* stream) {
  if (!c || !host_dst || !dev_src) return DKV_ERR_INVALID_ARG;
  DKV_CUDA(c, cudaMemcpyAsync(host_dst, dev_src, bytes, cudaMemcpyDeviceToHost, as_stream(stream)));
  DKV_CUDA(c, cudaStreamSynchronize(as_stream(stream)));
  return DKV_OK;
}

int dkv_last_status(dkv_ctx* c, int32_t* host_status) {
  if (!c || !host_status) return DKV_ERR_INVALID_ARG;
  DKV_CUDA(c, cudaDeviceSynchronize());
  DKV_CUDA(c, cudaMemcpy(host_status, c->d_status, sizeof(int) * 8, cudaMemcpyDeviceToHost));
  if (host_status[0] != 0) {                   // reported once
    DKV_CUDA(c, cudaMemset(c->d_status, 0, sizeof(int) * 8));
    DKV_CUDA(c, cudaStreamSynchronize(cudaStreamLegacy));     // (as in dkv_create)
  }
  host_status[1] = (int32_t)(c->launches & 0x7FFFFFFF);
  return host_status[0] == 0 ? DKV_OK : DKV_ERR_TIMEOUT;
}

int dkv_static_last_status(int32_t* host_status) {
  if (!host_status) return DKV_ERR_INVALID_ARG;
  DKV_CUDA(nullptr, cudaDeviceSynchronize());
  DKV_CUDA(nullptr, cudaMemcpyFromSymbol(host_status, g_static_scratch, sizeof(int) * 8));
  host_status[1] = 0;
  return host_status[0] == 0 ? DKV_OK : DKV_ERR_TIMEOUT;
}

int dkv_set_wait_limit(dkv_ctx* c, int64_t clock_ticks) {
  if (!c || clock_ticks < 1000) return DKV_ERR_INVALID_ARG;
  c->wait_cycles = clock_ticks;
  return DKV_OK;
}

int dkv_debug_withhold_tile(dkv_ctx* c, int32_t sweep, int32_t tile) {
  if (!c || (tile >= 0 && sweep != 1 && sweep != 2)) return DKV_ERR_INVALID_ARG;
  c->withhold_sweep = tile >= 0 ? sweep : -1;
  c->withhold_tile = tile >= 0 ? tile : -1;
  return DKV_OK;
}

int dkv_profile(dkv_ctx* c, int enable) {
  if (!c) return DKV_ERR_INVALID_ARG;
  c->prof_on = enable != 0;
  return DKV_OK;
}

int dkv_profile_read(dkv_ctx* c, double* ms, int64_t* launches) {
  if (!c || !ms || !launches) return DKV_ERR_INVALID_ARG;
  DKV_CUDA(c, cudaDeviceSynchronize());
  for (size_t i = 0; i < c->prof_used; ++i) {
    const ProfRec& r = (*c->prof_recs)[i];
    float t = 0.f;
    if (cudaEventElapsedTime(&t, r.a, r.b) == cudaSuccess) {
      c->prof_ms[r.step] += t;
      c->prof_launches[r.step] += r.launches;
    }
  }
  c->prof_used = 0;
  for (int i = 0; i < DKV_N_STEPS; ++i) {
    ms[i] = c->prof_ms[i]; launches[i] = c->prof_launches[i];
    c->prof_ms[i] = 0; c->prof_launches[i] = 0;
  }
  return DKV_OK;
}

int64_t dkv_launch_count(dkv_ctx* c) { return c ? (int64_t)c->launches : -1; }

int dkv_last_cuda_error(dkv_ctx* c) { return c ? c->last_cuda : 0; }

}  // extern "C"
