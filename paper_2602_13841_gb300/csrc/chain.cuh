// Chained launches (programmatic dependent launch).  A V-cycle and an FGMRES iteration are hundreds of
// kernels of a few microseconds, each reading what the one before wrote, so the time between two of
// them counts.  A chained kernel may be scheduled while its predecessor's last blocks run: its first
// statement, chain_begin(), waits until that grid has ended and its writes are visible, then lets the
// next one be scheduled (the operator's kernels of one time node do so at their end).  Nothing is read or written before it, so every order of a plain launch holds: a
// grid ends only after its own wait, hence after all grids before it.  A predecessor without
// a wait, a copy, a memset or an event wait is ordered as by a plain launch; a chained launch
// captures into a graph like a plain one.  No pointer of a chained kernel is declared __restrict__, const
// or not: the compiler may take it that the wait does not change what such a pointer points to, and move
// loads above it.
// Plain -> chained: 2D 8^2 Q2/P1 DG(1) FP64 apply 30.7 -> 27.1 us, 2D 256^2 Q3/P2 DG(2) FP32 apply 57.3 ->
// 52.8, 2D 32^2 Q2/P1 DG(1) slab solve 7.52 -> 6.71 ms.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace stmg {

// chain_wait() opens a chained kernel; chain_release() lets the next one be scheduled once every block has
// called it (or ended).  Right after the wait (chain_begin) the next kernel's blocks come early, late in the
// kernel they do not take room from blocks of this grid that have yet to start.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_begin() {
  chain_wait();
  chain_release();
}

// Launch a kernel that opens with chain_wait() or chain_begin(), chained or plainly.  An error is left for cudaGetLastError.
template <typename... P, typename... A>
static void launch_if_chained(bool chained, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              A&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = chained ? 1 : 0;
  cudaLaunchKernelEx(&c, kern, std::forward<A>(args)...);
}

template <typename... P, typename... A>
static void launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  launch_if_chained(true, kern, grid, block, smem, s, std::forward<A>(args)...);
}

}  // namespace stmg
