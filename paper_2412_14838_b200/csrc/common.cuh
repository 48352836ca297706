// Shared definitions of the libdkv kernels: problem shape, small device helpers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace dkv {

// Derived problem shape (names follow the paper: L layers, Hkv = H heads scored, G query heads per
// KV head, ws window, P = S - ws prefix tokens, N = wt - ws, Bl = B^l, m update interval).
struct Shape {
  int L, Hq, Hkv, D, Bt, S, ws, pool, N, Bl, m;
  int G;      // Hq / Hkv
  int P;      // S - ws
  int M;      // ws * G window-query rows per KV head
  int Blc;    // min(Bl, P)
  int rows;   // Blc + ws : row stride of the budget buffers
};

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Programmatic dependent launch: the kernel may have been scheduled while its predecessor on the stream still ran.  What that
// predecessor may have written is not touched before pdl_wait.  What kernels before the predecessor wrote may be, where the
// predecessor calls pdl_launch only after its own pdl_wait: all of its blocks have then waited, so what came before it is complete.
// Early readers, what they read, and the predecessor they count on for that:
//   score_sweep_kernel, key sums   queries and keys        score_sweep_kernel, row sums
//   rb_collect_kernel              scores                  rb_locate_kernel
//   select_gather_kernel,          scores                  rb_finish_kernel
//   select_gather_cluster_kernel
// (decode_cluster_kernel only asks for lines to be brought to L2.)  Such memory is not read-only for the lifetime of the grid: a
// kernel with pdl_wait takes its pointers without __restrict__ and reads with plain loads (no __ldg), which the compiler may
// neither turn into non-coherent loads nor move above the wait.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Per-layer device pointers passed by value to kernels that work on several layers at once.
struct LayerPtrs {
  void* kb[128];
  void* vb[128];
};

}  // namespace dkv
