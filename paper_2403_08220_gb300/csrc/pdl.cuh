// Programmatic dependent launch: a kernel's CTAs may be placed while the kernel
// before it on the stream still runs, which takes the launch and the ramp of
// its grid off the step's chain of short kernels.
//
// Rules, for every kernel that launch_pdl starts:
//  - pdl_wait (all earlier kernels of the stream complete, their writes visible)
//    comes before its first access to memory that an earlier kernel writes, or
//    before its first write to memory that an earlier kernel reads, in every
//    thread that makes one, and in every CTA before it exits.  So a kernel that
//    has ended has all earlier ones behind it, whether they were started this
//    way or not.
//  - pdl_launch comes after pdl_wait.  So only one kernel that has not waited is
//    resident beside the running one.
// Both are without effect in a kernel started the ordinary way.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace dino {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void pdl_launch() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void pdl_begin() {
  pdl_wait();
  pdl_launch();
}

// After pdl_wait: hands back a pointer: the compiler may move a load through a
// const __restrict__ parameter over an assembly statement, but not over the one
// that its address comes from.
template <class T>
__device__ __forceinline__ const T *pdl_after(const T *p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}

// Starts the kernel this way when it is short: its `ctas` (the tiles of a
// persistent kernel) are at most kPdlMaxCtas, four an SM.  A longer one gains
// nothing from an early start, and CTAs that sit on an SM waiting take it from
// the running kernel (all launches this way: 16384 chains, r = 200, 10.74 ->
// 11.07 ms a step, 1024 chains with the eigen map 2.35 -> 2.94; bounded: 64
// chains, r = 200, 319 -> 282 us a step; 64 chains in FP64, r = 16, 185 -> 128;
// 4096 chains of six layers of 400 1.45 -> 1.43 ms).  Kernels whose loads lose
// by pdl_after (k_rowprod: 490 -> 650 us) are started the ordinary way.
constexpr long kPdlMaxCtas = 4 * 152;

// Kernels of a CTA per chain that runs for tens of microseconds: only while each
// CTA has an SM of its own.  Placed early, several land on each of the SMs that
// are free by then, and the others stay idle (256 chains, r = 200, eight steps:
// 4.17 ms, with the bound 4.07).
inline long chain_ctas(int C) { return 4L * C; }

template <class... P, class... A>
cudaError_t launch_pdl_n(long ctas, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                         cudaStream_t st, A &&...args) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = ctas <= kPdlMaxCtas;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       A &&...args) {
  return launch_pdl_n((long)grid.x * grid.y * grid.z, kernel, grid, block, smem, st,
                      std::forward<A>(args)...);
}

}  // namespace dino
