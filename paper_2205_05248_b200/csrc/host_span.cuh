// Which host arrays a kernel may read or write in place of a copy (marl_actor_step_host).
#pragma once
#include <cstddef>
#include <cstdint>

namespace marl {

// What the driver says about an address: whether it is pinned host memory, where kernels find it, and the one allocation
// or registration around it (size 0: not known).
struct HostRange {
  bool pinned;
  const void* device;
  uintptr_t start;
  size_t size;
};

// The device's address of the array [host, host + bytes), or null where a kernel could not touch all of it: an array that is
// pinned in part only (a copy turns that into an error, a kernel would fault on the rest), or one whose address has not
// the alignment that the kernels rely on (copies go to aligned memory).
inline const void* kernel_span(const HostRange& r, const void* host, size_t bytes, size_t align) {
  const uintptr_t h = reinterpret_cast<uintptr_t>(host);
  if (!r.pinned || !r.device || h % align || reinterpret_cast<uintptr_t>(r.device) % align) return nullptr;
  if (h < r.start || h - r.start > r.size || bytes > r.size - (h - r.start)) return nullptr;
  return r.device;
}

}  // namespace marl
