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

// Whether a pipelined-kernel launch of T steps over blocks that take `tiles` in turn should start early.  Early blocks take
// the SMs that the kernel before leaves idle first, so where more than half of the blocks, but not nearly all, have a tile
// more than the others, those end up side by side instead of spread over the chip: 683 tiles of 128 steps on 148 blocks (91
// with a fifth tile) 2885 us, against 2743 started after the kernel before.  Other shares gain: 293 tiles (145 with a second)
// 1580 -> 1557 us, 342 tiles (46 with a third) 753 -> 740, 64 tiles 414 -> 409; and so do short launches, where start-up
// weighs more.
inline bool early_pays(int tiles, int grid, int T) {
  const int rest = tiles % grid;  // blocks with a tile more than the others
  return T < 8 || rest <= grid / 2 || rest > grid - grid / 8;
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
