// Host-side launch helper shared by the actor kernels.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace marl {

constexpr int SMEM_OPTIN_DEVICES = 64;

// A kernel's opt-in dynamic shared-memory size is a per-device setting.  `table` (one per kernel variant, zero
// initialised) remembers the largest size set on each device, so that the attribute call is made once per device
// and size instead of once per launch; devices beyond the table are set on every launch.
inline cudaError_t ensure_dynamic_smem(const void* kernel, uint32_t bytes, uint32_t (&table)[SMEM_OPTIN_DEVICES]) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool tracked = dev >= 0 && dev < SMEM_OPTIN_DEVICES;
  if (tracked && table[dev] >= bytes) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && tracked) table[dev] = bytes;
  return e;
}

// Launches a kernel that may start while the kernel before it in the stream is still running (programmatic dependent
// launch).  Such a kernel does what does not depend on earlier work - barriers, tensor memory, its weights - and then
// executes grid_wait() in every thread that touches anything earlier work reads or writes.  early = false: an ordinary
// launch (the step that first uses a newly uploaded weight image).
// Whatever share of the blocks has a tile more than the others: pipelined kernel, some thirty launches with 50 to 100 % such blocks, the
// early start costs or saves less than 1 % (683 tiles of 128 steps on 148 blocks, 91 with a fifth: 2490 us, ordinary 2494);
// split-operand kernel, 20 launches of fp32, hidden 128 and per-type networks, likewise (547 tiles of 64 steps in fp32 2101 us,
// ordinary 2104; 556 tiles of hidden 128 1956 against 1954).  One-step launches gain 2.5 to 3.5 us of 11 to 41.
template <typename... P>
inline cudaError_t launch_overlapped(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t stream, bool early, const P&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)grid);
  c.blockDim = dim3((unsigned)block);
  c.dynamicSmemBytes = smem;
  c.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, args...);
}

#ifdef __CUDACC__
// Waits until all earlier work of the stream is done and visible.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The next kernel's blocks may be scheduled once some thread of every block has come here (or the block has ended): to be
// called when a block's last step begins or a little before.  Waiting blocks hold an SM each; released at the start of a
// long launch they took the SMs that it leaves free from the kernels of other streams.
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

}  // namespace marl
