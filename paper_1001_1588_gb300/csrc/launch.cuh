// Kernel launches of the analysis passes: dynamic shared memory allowed once per (device, kernel), and
// launches whose latency overlaps the kernel before them (programmatic dependent launch).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fftenkf {

// Allows `kern` `smem` bytes of dynamic shared memory on the current device.  The attribute call costs
// more host time than a launch, so it is made once per (device, kernel) and larger request.
cudaError_t allow_smem(const void* kern, size_t smem);

// In a kernel launched with launch_overlapped: returns once every earlier kernel of the stream has
// finished and its writes are visible; nothing of an earlier kernel is read or overwritten before it.
// Data of earlier kernels is read by plain loads: the compiler may move __ldg and loads through const
// __restrict__ pointers, which it takes for loads of constants, ahead of this wait.
__device__ __forceinline__ void stream_order_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next kernel of the stream be brought onto SMs that have room, where it waits in stream_order_wait(),
// once every CTA of this one has called it or left (without it: once every CTA has left).  For kernels that leave
// the SM's on-chip memory alone, as the network's.  The split and sine passes do without: the next pass's waiting
// CTAs hold shared memory, which is then missing as first-level cache for spills and instructions of the pass that
// runs (called at the start of each: 48 x 128, N = 25, 2 of 4 blocks observed 66 us, 34 without; 1024 x 48, N = 25,
// 4 blocks 346 and 259; 64^2 14 us both; called before a CTA's last stores: 35, 270, 14).
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch (of clusters of `cluster` CTAs) with the stream's order kept by stream_order_wait() at the kernel's start: the launch latency
// of a kernel overlaps the one before it (2-3 us between dependent kernels otherwise).
template <typename P>
inline cudaError_t launch_overlapped(void (*kern)(const P), dim3 grid, int threads, size_t smem, cudaStream_t st,
                                     const P& p, unsigned cluster = 1) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, p);
}

}  // namespace fftenkf
