// Programmatic dependent launch.  The kernels of a call run one after another
// on one stream, and between two of them a plain launch leaves 2.5 to 3.5 us
// in which nothing runs (measured between the projection and the product at
// every size).  A kernel launched by launch_pdl may start while its predecessor
// drains: it sets up its barriers and tensor memory, then waits for the
// predecessor to complete (with its writes visible) before it touches global
// memory.
//
// Only kernels whose grid fills the chip once (persistent blocks, as many per SM
// as fit) are launched this way.  The blocks of any other grid go to whichever
// SMs the predecessor leaves first and crowd there: the FP64 product of 256
// blocks took 276 us a call instead of 103 and the correlation's projection of
// 570 blocks 15 us instead of 11.5.  Those go through launch_plain.
//
// Every kernel of either kind calls pdl_begin() in every thread before its first
// access to global memory.  Each waits for its predecessor in full, so it also
// runs after everything before that; a predecessor that is no kernel of this
// library is waited for like any other.
#pragma once

#include <cuda_runtime.h>

namespace pj {

// Lets the next kernel of the stream be scheduled as this one's blocks leave,
// and waits for the previous one.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// A launch that the runtime refuses also leaves its error behind for whoever asks for the
// last one next (the caller's framework after a launch of its own): it is taken back here,
// and returned.
inline cudaError_t launched(cudaError_t e) {
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e;
}

template <typename... P, typename... A>
inline cudaError_t launch_plain(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                                const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  return launched(cudaLaunchKernelEx(&cfg, kernel, args...));
}

template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, int cluster,
                              const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = static_cast<unsigned>(cluster);
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return launched(cudaLaunchKernelEx(&cfg, kernel, args...));
}

}  // namespace pj
