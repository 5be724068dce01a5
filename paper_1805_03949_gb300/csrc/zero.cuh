// zero.cuh -- clearing a system before an assembly, and the launch of the tile
// kernels that add into it.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

namespace fea {

// Systems up to this size are cleared by one kernel in the launches per
// element type, which fea_assemble_launches counts, and the tile kernel that
// follows may start while it runs and wait for it only before its first
// addition: on small meshes the launches and the tiles' gathers take longer
// than the work (22,950 tet4, Poisson: 16.4 us per step with two memsets, 14.0
// with the kernel, 12.7 with the early start).
// Larger ones keep cudaMemsetAsync, which writes at 7.5 TB/s where the kernel
// reaches 5.8.
constexpr int64_t kSmallSystemBytes = 32ll << 20;

inline bool small_system(int64_t nnz) { return nnz * (int64_t)sizeof(double) <= kSmallSystemBytes; }

// Whether a tile kernel of `grid` CTAs starts early.  CTAs that start while
// another kernel still holds SMs are packed on the free ones, which costs more
// than the early start gains when they would fill each SM once to a few times
// and are bound by the FP64 unit (hex8, FP64 elasticity, us per step, early
// against not: 57 CTAs 31 / 33, 108 CTAs 47 / 34, 635 CTAs 119 / 105, 1,014
// CTAs 139 / 143).  So it does with few CTAs or with several per SM, or, right
// after the clearing, if its tiles are light (few FP64 instructions: tet4
// diffusion 12.7 / 14.0 up to 813 CTAs).  The types of a small mixed mesh
// overlap in turn: 1,630 elements, diffusion 20 / 39 us.
inline bool starts_early(unsigned grid, bool after_clearing, bool light) {
  return grid <= 64 || (after_clearing && (light || grid >= 1024));
}

// Clear A [nnz] and b [nb].
int zero_system(double* A, int64_t nnz, double* b, int64_t nb, cudaStream_t s);

// Device side of the early start: let the next kernel of the stream start; wait
// until the kernels before have finished and their writes are visible (nothing
// to wait for in a kernel launched without it).
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch, with `early` before the stream's previous kernel has finished: the
// kernel must call wait_for_previous() before it touches what that one writes.
template <class Kernel, class... Args>
cudaError_t launch_tiles(Kernel kern, unsigned grid, unsigned threads, size_t smem, cudaStream_t s, bool early,
                         const Args&... args) {
  if (!early) {
    kern<<<grid, threads, smem, s>>>(args...);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace fea
